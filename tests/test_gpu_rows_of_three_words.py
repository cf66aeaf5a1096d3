"""FP64 form on rows of 65 to 96 cells (three coverage words): the cases and
tolerances of tests/test_gpu_fixed64.py's row widths.  tests/test_gpu_force_lists.py
has such rows among spheres that leave most words without cells of the staged
kernel, so that its warps run through many tiles at once."""
import pytest

from tests.test_gpu_fixed64 import capi, test_row_widths as _row_widths  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [65, 88, 96])
@pytest.mark.parametrize("walls,streaming", [((0,) * 6, "pull"), ((0,) * 6, "aa"),
                                             ((1, 1, 1, 1, 2, 3), "pull")])
def test_three_words(capi, nx, walls, streaming):  # noqa: F811
    _row_widths(capi, nx, walls, streaming)
