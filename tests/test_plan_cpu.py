"""What the planner decides, on the CPU."""
import pytest

from paper_2310_04559_gb300 import binding as B

GIB = 1 << 30


def _plan(o, v, n, budget, **kw):
    kw = dict(dict(mode="ozaki_bf16", symmetric=True, order="integral_first"), **kw)
    ws = B.workspace_size(o, v, n, budget=int(budget), **kw)
    assert ws <= budget
    return dict(B.plan(o, v, n, ws_bytes=ws, **kw), ws=ws)


# L is read over the host link once per block.  Seven digit slices take no fewer blocks than the default's six.
@pytest.mark.parametrize("o,v,n,gib", [(10, 100, 500, 0.1), (10, 100, 500, 0.2), (20, 160, 800, 0.4), (20, 160, 800, 2.0),
                                       (40, 400, 2000, 8.0), (40, 400, 2000, 48.0), (6, 200, 1200, 1.0)])
def test_streamed_L_is_not_read_far_more_often_than_digit_slices_would(o, v, n, gib):
    default = _plan(o, v, n, gib * GIB, host_L=True)
    digits = _plan(o, v, n, gib * GIB, host_L=True, slices=7)
    assert default["n_blocks"] <= 3 * digits["n_blocks"]
