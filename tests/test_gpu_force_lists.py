"""The force reduction's walk over the particles' cell lists: lists shorter than
a round of the block, at its edges and of many rounds, with cells shared between
two particles (their slots ordered either way), against FP64 sums of the slot
forces (bounds of test_gpu_force_reduction.py); and a grid longer than 2^23
cells, whose offsets are converted to FP64 another way, against the same sphere
in a short one, bit for bit.
"""
import numpy as np
import pytest

from tests.test_gpu_force_reduction import _check, capi  # noqa: F401

pytestmark = pytest.mark.gpu


class _Box:
    nx, ny, nz = 64, 40, 36
    walls = (0, 0, 0, 0, 1, 1)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "df64"])
@pytest.mark.parametrize("radii", [(1.0, 1.3), (2.4, 2.6), (2.9, 3.6), (7.5, 5.2)])
def test_lists_with_shared_cells(capi, precision, radii):  # noqa: F811
    w = _Box()
    e = capi.Engine(w.nx, w.ny, w.nz, 0.6, walls=w.walls, fbody=(1e-4, 2e-5, -3e-5),
                    precision=precision)
    a, b = radii
    # two touching pairs, one across the periodic faces; the larger sphere
    # comes first in one and second in the other
    x = np.array([[20.3, 18.6, 14.2], [20.3 + a + b - 0.7, 18.6, 14.2],
                  [0.4, 0.2, 22.5], [0.4 - (a + b - 0.6), 0.2, 22.5]])
    x[3, 0] += w.nx
    e.set_particles(x, np.array([b, a, a, b]), density=np.full(4, 2.0), fixed=np.ones(4, bool),
                    omega=1e-3 * np.arange(12.0).reshape(4, 3))
    e.step(4)
    assert (e.slots()[2] >= 0).any()
    _check(e, w, precision, x)
    e.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "df64"])
@pytest.mark.parametrize("n", [1023, 1024])
def test_many_particles(capi, precision, n):  # noqa: F811
    """The last number of particles with blocks of 128 threads, the first with
    blocks of 64: lists below and above a round of either."""
    w = _Box()
    w.nx, w.ny, w.nz, w.walls = 88, 64, 64, (0,) * 6
    rng = np.random.default_rng(n)
    x = np.stack(np.meshgrid(np.arange(16), np.arange(8), np.arange(8), indexing="ij"), -1)
    x = (x.reshape(-1, 3)[:n] * [5.5, 8.0, 8.0]) + [2.5, 4.0, 4.0] + 0.4 * rng.random((n, 3))
    e = capi.Engine(w.nx, w.ny, w.nz, 0.6, fbody=(1e-4, 2e-5, -3e-5), precision=precision)
    e.set_particles(x, 0.9 + 2.0 * rng.random(n), density=np.full(n, 2.0), fixed=np.ones(n, bool))
    e.step(2)
    _check(e, w, precision, x)
    e.close()


def test_long_grid(capi):  # noqa: F811
    got = []
    for nx in (64, (1 << 23) + 64):
        e = capi.Engine(nx, 6, 6, 0.6, fbody=(1e-4, 2e-5, -3e-5), streaming="aa")
        e.set_particles(np.array([[33.3, 1.8, 2.1]]), np.array([1.0]), density=np.array([2.0]),
                        fixed=np.ones(1, bool))
        e.step(2)
        got.append(e.force_torque())
        e.close()
    assert np.any(got[0][1] != 0.0)
    for s, t in zip(*got):
        assert np.array_equal(s, t)
