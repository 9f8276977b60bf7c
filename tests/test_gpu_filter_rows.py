"""The field marches where the filter's FP64 split ends: rows of 16 - 2H of a
CTA (14, 12, 10, 8), warps without a row in the grid, long strips of two warps
a CTA; against the FP64 oracle with the single-phase tolerances."""
import pytest

from test_gpu_edges import FP32, FP64, O, test_field_marches as marches  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("size", [(30, 8, 70), (25, 9, 33), (33, 17, 12), (9, 25, 40), (57, 40, 18), (65, 700), (30, 1201)])
def test_rows(O, size, bc, prec):  # noqa: F811
    marches(O, size, bc, prec)
