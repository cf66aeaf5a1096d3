"""FP64 form: the staged kernel of the uncovered cells and the kernel of the
covered cells, at the sizes and values where their paths change, against the
FP64 oracle.  Tolerance as in tests/test_gpu_parity.py: 1e-12 relative on PDFs,
1e-12 of the largest component on forces and torques."""
import numpy as np
import pytest

from oracle import Oracle
from paper_2303_11811_gb300 import inputs

pytestmark = pytest.mark.gpu

REST = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12).reshape(19, 1, 1, 1)


@pytest.fixture(scope="module")
def capi():
    import torch
    assert torch.cuda.is_available()
    from paper_2303_11811_gb300 import build, capi as c
    build.build()
    return c


def _check(e, o, steps):
    e.step(steps)
    o.step(steps)
    fg, fo = e.pdfs(), o.pdfs()
    assert np.max(np.abs(fg - fo) / np.abs(fo)) < 1e-12
    if e.np:
        for a, b in zip(e.force_torque(), o.force_torque()):
            assert np.max(np.abs(a - b)) <= 1e-12 * max(np.max(np.abs(b)), 1e-300)


# row widths around the tiles: one word, a padded word, whole tiles of several
# rows, rows of one tile, two and three segments, a last segment of one word
@pytest.mark.parametrize("nx", [31, 32, 33, 64, 127, 255, 256, 257, 320, 513, 545])
@pytest.mark.parametrize("walls,streaming", [((0,) * 6, "pull"), ((0,) * 6, "aa"),
                                             ((1, 1, 0, 0, 0, 0), "aa"),
                                             ((1, 1, 1, 1, 2, 3), "pull")])
def test_row_widths(capi, nx, walls, streaming):
    """Moving spheres across the periodic x face, at a segment's edge and near
    the far wall; noise on the field; an odd and an even number of steps."""
    ny, nz = 11, 9
    kw = dict(tau=0.6, relax="trt", walls=walls, fbody=(1e-6, -2e-6, 3e-6), weighting="nt",
              eps_mode="supersample", eps_n=4, bc_velocity=(0.0, 0.0, 1e-3))
    rng = np.random.default_rng(nx)
    f = REST * (1.0 + 1e-3 * (2.0 * rng.random((19, nz, ny, nx)) - 1.0))
    x0 = 0.3 if not walls[0] else 2.4
    x = np.array([[x0, 5.2, 4.4], [min(128.4, nx / 2 + 0.1), 5.9, 4.6], [nx - 6.6, 4.7, 4.5]])
    r = np.array([2.1, 2.3, 1.9])
    u = inputs.random_velocities(3, 1e-3, 7)
    for steps in (2, 3):
        e = capi.Engine(nx, ny, nz, streaming=streaming, **kw)
        o = Oracle(nx, ny, nz, **kw)
        for s in (e, o):
            s.set_pdfs(f)
            s.set_particles(x, r, u=u, omega=0.1 * u, density=np.full(3, 2.0),
                            fixed=np.ones(3, np.uint8))
        _check(e, o, steps)


@pytest.mark.parametrize("scale", [1e-14, 1e-6, 0.05, 0.2, 0.45])
@pytest.mark.parametrize("force", [0.0, 1e-9, 1e-4])
def test_value_ranges(capi, scale, force):
    """Deviations from far below the force to beyond the fixed-point range (the
    FP64 form), beside quiescent cells; a sphere moving as fast as the fluid,
    one in contact reach of it (cells of two particles)."""
    n = 40
    kw = dict(tau=0.8, relax="srt", fbody=(force, 0.0, -force), weighting="eps",
              eps_mode="supersample", eps_n=4)
    rng = np.random.default_rng(3)
    d = np.zeros((19, n, n, n))
    d[:, :, :, 12:30] = scale * (2.0 * rng.random((19, n, n, 18)) - 1.0)
    f = REST * (1.0 + d)
    x = np.array([[14.0, 20.0, 20.0], [22.3, 20.4, 20.1], [34.0, 10.0, 10.0]])
    r = np.array([3.6, 4.2, 3.0])
    u = np.array([[0.1, 0.2, -0.1], [-0.3, 0.0, 0.1], [0.0, 0.0, 0.0]]) * scale
    e = capi.Engine(n, n, n, **kw)
    o = Oracle(n, n, n, **kw)
    for s in (e, o):
        s.set_pdfs(f)
        s.set_particles(x, r, u=u, density=np.ones(3), fixed=np.ones(3, np.uint8))
    e.step(1)
    o.step(1)
    fg, fo = e.pdfs(), o.pdfs()
    # relative to the field's smallest weight: deviations of any sign make
    # single PDFs small
    assert np.max(np.abs(fg - fo)) < 1e-12 / 36.0
    for a, b in zip(e.force_torque(), o.force_torque()):
        # a force is a sum of thousands of cells' momenta of the size of scale
        # (and of f), each rounded like the oracle's PDFs: 2^-53 of w_q
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b)) + 1e-15 * 4000.0


@pytest.mark.parametrize("nx", [40, 300])
def test_rest_stays_exact(capi, nx):
    """Fluid at rest without forces around resting spheres: the lattice weights
    and zero forces, to the last bit."""
    e = capi.Engine(nx, 24, 20, 0.7, relax="trt", weighting="nt")
    e.set_particles(np.array([[10.0, 12.0, 10.0], [nx - 11.3, 12.2, 9.7]]), np.array([4.0, 5.1]),
                    fixed=np.ones(2, np.uint8))
    e.step(5)
    assert np.array_equal(e.pdfs(), np.broadcast_to(REST, (19, 20, 24, nx)))
    F, T = e.force_torque()
    assert not F.any() and not T.any()


def test_nonfinite_is_reported(capi):
    """A NaN and an infinity next to a sphere reach the force."""
    for bad in (np.nan, np.inf):
        e = capi.Engine(32, 32, 32, 0.6)
        e.set_particles(np.array([[16.0, 16.0, 16.0]]), np.array([4.0]),
                        fixed=np.ones(1, np.uint8))
        f = np.broadcast_to(REST, (19, 32, 32, 32)).copy()
        f[3, 16, 16, 11] = bad
        e.set_pdfs(f)
        assert e.step_status(3) == capi.PSM_ERR_NONFINITE
