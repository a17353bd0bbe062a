"""The autotuner times every launch shape once: what a precision's kernels do not
read stays at its default, and values that select the same shapes are not both
tried."""

import pytest

from paper_1908_03121_gb300 import autotune as A
from paper_1908_03121_gb300 import fmm as B

SMS = 152


def _shape(c, precision, order, n):
    """What the launches read of a tuning (the multipole items as they resolve)."""
    items = c["mp_items"]
    if precision == B.FMM_MIXED:
        if order == 3 and c["mp_pair_targets"]:
            items = "pairs"
        elif items == 0 and n > SMS:
            cap = c["ctas_per_sm"] if 0 < c["ctas_per_sm"] < 3 else 3
            items = 2 if n < 2 * cap * SMS else 1
        return c["mono_subgrids"] or 2, c["ctas_per_sm"], c["dataflow"], items
    if 4 * n < SMS:
        items = 16
    elif items == 0:
        items = 2 if n < 8 * SMS else 1
    return c["ctas_per_sm"], c["dataflow"], items


@pytest.mark.parametrize("precision", [B.FMM_MIXED, B.FMM_DFLOAT, B.FMM_FP64])
@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("n", [0, 8, 37, 38, 76, 152, 153, 700, 1216, 5000])
def test_every_shape_once(precision, order, n):
    c = A.candidates(precision, order, n, SMS)
    shapes = [_shape(x, precision, order, n) for x in c]
    assert len(set(shapes)) == len(shapes)
    assert {x["ctas_per_sm"] for x in c} == set(A.CTAS_PER_SM) and {x["dataflow"] for x in c} == set(A.DATAFLOW)
    if precision == B.FMM_MIXED:
        assert {x["mono_subgrids"] for x in c} == set(A.MONO_SUBGRIDS)
        assert ("pairs" in {s[3] for s in shapes}) == (order == 3)
    assert set(c[0]) == {"mono_subgrids", "ctas_per_sm", "dataflow", "mp_pair_targets", "mp_items"}
