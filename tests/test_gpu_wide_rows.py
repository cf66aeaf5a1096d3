"""FP64 form on rows of more than 65,536 cells: a cell's place in its tile is
listed in 16 bits, relative to the tile.  Against the FP64 oracle, with spheres
at the ends of the row and on either side of cell 65,536; tolerance of
tests/test_gpu_fixed64.py."""
import numpy as np
import pytest

from oracle import Oracle
from paper_2303_11811_gb300 import inputs
from tests.test_gpu_fixed64 import REST, _check, capi  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls,streaming", [((0,) * 6, "pull"), ((1, 1, 0, 0, 0, 0), "aa")])
def test_wide_rows(capi, walls, streaming):  # noqa: F811
    nx, ny, nz = 65536 + 300, 7, 8
    kw = dict(tau=0.6, relax="trt", walls=walls, fbody=(1e-6, -2e-6, 3e-6), eps_mode="supersample",
              eps_n=4)
    rng = np.random.default_rng(1)
    f = REST * (1.0 + 1e-3 * (2.0 * rng.random((19, nz, ny, nx)) - 1.0))
    x = np.array([[2.4, 3.2, 4.4], [65534.1, 2.9, 4.6], [65539.2, 3.4, 3.6], [nx - 2.6, 3.7, 4.5]])
    u = inputs.random_velocities(4, 1e-3, 7)
    e = capi.Engine(nx, ny, nz, streaming=streaming, **kw)
    o = Oracle(nx, ny, nz, **kw)
    for s in (e, o):
        s.set_pdfs(f)
        s.set_particles(x, np.array([1.3, 1.4, 1.2, 1.3]), u=u, omega=0.1 * u,
                        density=np.full(4, 2.0), fixed=np.ones(4, np.uint8))
    _check(e, o, 3)
