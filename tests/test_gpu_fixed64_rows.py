"""FP64 form on grids beyond the line (2 x SMs x 7 x 10 coverage words) up to
which one kernel takes every cell: the staged kernel's row widths beside the
covered-cell kernel, and grids on either side of the line, against the FP64
oracle.  Tolerance as in tests/test_gpu_parity.py: 1e-12 relative on PDFs, 1e-12
of the largest component on forces and torques."""
import numpy as np
import pytest

from oracle import Oracle
from paper_2303_11811_gb300 import inputs

pytestmark = pytest.mark.gpu

REST = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12).reshape(19, 1, 1, 1)
SMS = 152
LINE = 2 * SMS * 7 * 10


@pytest.fixture(scope="module")
def capi():
    import torch
    assert torch.cuda.is_available()
    from paper_2303_11811_gb300 import build, capi as c
    build.build()
    return c


def _run(capi, nx, ny, nz, walls, streaming, steps):
    """Moving spheres across the periodic x face, at a segment's edge and near
    the far wall; noise on the field."""
    kw = dict(tau=0.6, relax="trt", walls=walls, fbody=(1e-6, -2e-6, 3e-6), weighting="nt",
              eps_mode="supersample", eps_n=4, bc_velocity=(0.0, 0.0, 1e-3))
    rng = np.random.default_rng(nx)
    f = REST * (1.0 + 1e-3 * (2.0 * rng.random((19, nz, ny, nx)) - 1.0))
    x = np.array([[0.3 if not walls[0] else 2.4, 5.2, 4.4],
                  [min(128.4, nx / 2 + 0.1), ny / 2 + 0.4, nz / 2 + 0.2],
                  [nx - 6.6, ny - 5.3, nz - 4.5]])
    u = inputs.random_velocities(3, 1e-3, 7)
    e = capi.Engine(nx, ny, nz, streaming=streaming, **kw)
    o = Oracle(nx, ny, nz, **kw)
    for s in (e, o):
        s.set_pdfs(f)
        s.set_particles(x, np.array([2.1, 3.3, 1.9]), u=u, omega=0.1 * u, density=np.full(3, 2.0),
                        fixed=np.ones(3, np.uint8))
        s.step(steps)
    fg, fo = e.pdfs(), o.pdfs()
    assert np.max(np.abs(fg - fo) / np.abs(fo)) < 1e-12
    for a, b in zip(e.force_torque(), o.force_torque()):
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))


PERIODIC, OPEN, CHANNEL = (0,) * 6, (1, 1, 1, 1, 2, 3), (1, 1, 0, 0, 0, 0)


@pytest.mark.parametrize("nx,ny,nz", [(31, 147, 145), (33, 104, 103), (64, 103, 104), (70, 85, 84),
                                      (127, 74, 73), (255, 52, 52), (257, 49, 49), (320, 47, 46),
                                      (513, 36, 35), (545, 35, 34)])
@pytest.mark.parametrize("walls,streaming,steps", [(PERIODIC, "aa", 3), (OPEN, "pull", 2)])
def test_staged_rows(capi, nx, ny, nz, walls, streaming, steps):
    assert (nx + 31) // 32 * ny * nz > LINE
    _run(capi, nx, ny, nz, walls, streaming, steps)


@pytest.mark.parametrize("nx,ny,nz", [(32, 133, 160), (32, 133, 161), (61, 76, 140), (61, 76, 141)])
@pytest.mark.parametrize("walls,streaming,steps", [(PERIODIC, "pull", 2), (CHANNEL, "aa", 3)])
def test_either_side(capi, nx, ny, nz, walls, streaming, steps):
    _run(capi, nx, ny, nz, walls, streaming, steps)
    count = {}
    for precision in ("fp64", "fp32"):
        e = capi.Engine(nx, ny, nz, 0.6, precision=precision)
        e.set_particles(np.array([[9.0, 9.0, 9.0]]), np.array([3.0]), fixed=np.ones(1, np.uint8))
        e.step(1)
        e.step(1)  # fixed spheres: no mapping, the collision and the force
        count[precision] = e.last_launch_count()
    # the FP32 form's collision is one launch
    assert count["fp64"] - count["fp32"] == (0 if (nx + 31) // 32 * ny * nz <= LINE else 1)


@pytest.mark.parametrize("nx,ny,nz", [(40, 40, 40), (70, 85, 84)])
@pytest.mark.parametrize("streaming,steps", [("pull", 2), ("aa", 2), ("aa", 3)])
def test_all_paths(capi, nx, ny, nz, streaming, steps):
    """Quiescent cells, ordinary ones and ones outside the fixed-point range in
    one warp, covered and not, in one kernel and in two; bounds as in
    tests/test_gpu_fixed64.py::test_value_ranges, per step."""
    kw = dict(tau=0.8, relax="srt", weighting="eps", eps_mode="supersample", eps_n=4)
    rng = np.random.default_rng(4)
    d = np.zeros((19, nz, ny, nx))
    d[..., 8:22] = 1e-3 * (2.0 * rng.random((19, nz, ny, 14)) - 1.0)
    d[..., 14:18] = 0.45 * (2.0 * rng.random((19, nz, ny, 4)) - 1.0)
    f = REST * (1.0 + d)
    x = np.array([[16.0, 20.0, 20.0], [22.3, 20.4, 21.1], [33.0, 10.0, 10.0], [9.0, 31.0, 30.0]])
    u = np.array([[0.01, 0.02, -0.01], [-0.03, 0.0, 0.01], [0.0, 0.0, 0.0], [0.4, 0.0, 0.1]])
    e = capi.Engine(nx, ny, nz, streaming=streaming, **kw)
    o = Oracle(nx, ny, nz, **kw)
    for s in (e, o):
        s.set_pdfs(f)
        s.set_particles(x, np.array([3.6, 4.2, 3.0, 4.0]), u=u, density=np.ones(4),
                        fixed=np.ones(4, np.uint8))
        s.step(steps)
    assert np.max(np.abs(e.pdfs() - o.pdfs())) < steps * 1e-12 / 36.0
    for a, b in zip(e.force_torque(), o.force_torque()):
        assert np.max(np.abs(a - b)) <= steps * (1e-12 * np.max(np.abs(b)) + 1e-15 * 4000.0)
