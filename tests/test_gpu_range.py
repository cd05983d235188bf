"""Results at the ends of the range of doubles.

The emulated mode scales every row by a power of two, so inputs times powers of two give the same bits times a power of
two, as long as the result is a normal number; below that only the last rounding is coarser (one of R+ and one of R-,
2^-1074 each at most)."""
import numpy as np
import pytest
import torch

from paper_2310_04559_gb300 import binding as B
from paper_2310_04559_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda", 0)


def _calls(L, t2, W, order, sym):
    yield "R", B.ladder_forward(L, t2, symmetric=sym, order=order)
    if order == "integral_first":
        dL, dt2 = B.ladder_backward(L, t2, W, symmetric=sym)
        yield "dL", dL
        yield "dt2", dt2
        o, v = t2.shape[0], t2.shape[2]
        Lov = L[:, :o].contiguous()
        yield "ijkl", B.tijkl(Lov, t2)
        yield "ijbk", B.tijbk(Lov, L, t2)


@pytest.mark.parametrize("order", ["integral_first", "cholesky_first"])
@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("top", [970, 973, 1000, 1022, -900, -1022, -1040])
def test_emulated_results_scale_with_the_inputs(dev, order, sym, top):
    o, v, n = 3, 21, 40
    L, t2 = synth.ladder_inputs_torch(o, v, n, seed=6, device="cuda")
    W = torch.randn(t2.shape, dtype=torch.float64, device=dev, generator=torch.Generator(device=dev).manual_seed(2))
    want = dict(_calls(L, t2, W, order, sym))
    # L by 2^l and t2, W by 2^t: R, dt2 and the terms by 2^(2 l + t), dL by 2^(l + 2 t); the largest entry near 2^top
    at = max(int(torch.frexp(w.abs().max())[1]) for w in want.values())
    l = t = (top - at) // 3
    Ls, ts, Ws = (x * 2.0 ** k for x, k in ((L, l), (t2, t), (W, t)))
    assert torch.isfinite(Ls).all() and torch.isfinite(ts).all()
    for name, got in _calls(Ls, ts, Ws, order, sym):
        ref = np.ldexp(want[name].cpu().numpy(), 3 * l)
        g = got.cpu().numpy()
        assert np.isfinite(ref).all()
        tiny = 2.0 ** -1073 if top < 0 else 0.0
        assert np.all(np.abs(g - ref) <= tiny), (name, np.abs(g - ref).max())
