"""Results at the ends of the range of doubles.

The emulated mode scales every row by a power of two, so inputs times powers of two give the same bits times a power of
two, as long as the result is a normal number; below that only the last rounding is coarser (one of R+ and one of R-,
2^-1074 each at most)."""
import numpy as np
import pytest
import torch

from paper_2310_04559_gb300 import _lib
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


@pytest.mark.parametrize("mode,u", [("bf16", 2.0 ** -8), ("tf32", 2.0 ** -11)])
def test_mixed_integrals_above_half_of_the_largest_float(dev, mode, u):
    """Integrals of 1.9e38 to 3.2e38, whose sums pass FP32's range and whose half sums V+ do not.  Bound as in
    test_gpu_mixed: L rounded twice per product, V+- and T+- once each."""
    o, v, n = 2, 35, 1
    rng = np.random.default_rng(8)
    L = rng.uniform(1.0, 1.29, (n, v, v))
    L = 0.5 * (L + L.transpose(0, 2, 1)) * np.sqrt(1.9e38)
    t2 = np.zeros((o, o, v, v))
    for i in range(o):
        for j in range(i, o):
            for c, d in ((0, 34), (7, 7), (3, 20)):
                t2[i, j, c, d] = t2[j, i, d, c] = 1e-3 * rng.uniform(0.5, 2.0)
    V = np.einsum("nac,nbd->abcd", L, L)
    assert 3.4e38 < 2 * V.min() and V.max() < 3.25e38
    ref = np.einsum("abcd,ijcd->ijab", V, t2)
    bound = 4.1 * u * np.einsum("abcd,ijcd->ijab", V + V.transpose(0, 1, 3, 2), np.abs(t2))
    R = B.ladder_forward(torch.from_numpy(L).to(dev), torch.from_numpy(t2).to(dev), mode=mode, symmetric=True,
                         order="integral_first").cpu().numpy()
    assert np.all(np.abs(R - ref) <= bound)


@pytest.mark.parametrize("mode", ["bf16", "tf32"])
@pytest.mark.parametrize("e", [0, -50, -62, -66, -70])
def test_mixed_denormal_integrals_round_once(dev, mode, e):
    """Streamed L keeps its integral block in FP64, where V+- are exact before their one rounding: the FP32 block of
    resident L gives the same bits, also where the integrals (about 2^(2 e)) are denormal in FP32."""
    o, v, n = 2, 97, 4
    L, t2 = synth.ladder_inputs_torch(o, v, n, seed=12, device="cpu")
    L, t2 = L * 2.0 ** e, t2 * 2.0 ** 20
    R = B.ladder_forward(L.to(dev), t2.to(dev), mode=mode, symmetric=True, order="integral_first")
    S = B.ladder_forward(L.pin_memory(), t2.to(dev), mode=mode, symmetric=True, host_L=True, chol_chunk=n)
    assert torch.equal(R, S), float((R - S).abs().max() / S.abs().max())


@pytest.mark.parametrize("a_block", [0, 5])
@pytest.mark.parametrize("exchange", [False, True])
def test_fp64_general_amplitudes_propagate_as_the_plain_product(dev, a_block, exchange):
    """Infinite and NaN amplitudes, and finite ones whose sum t_cd + t_dc overflows, give the entries of the plain
    product sum_cd (ac|bd) t_ijcd: infinities of its sign, NaN where it is NaN, else finite within FP64's rounding."""
    o, v, n = 3, 37, 6
    rng = np.random.default_rng(5)
    L = rng.uniform(0.1, 1.0, (n, v, v)) * rng.choice([-1.0, 1.0], (n, v, v))
    t2 = rng.standard_normal((o, o, v, v))
    t2[0, 1, 4, 30] = np.inf
    t2[1, 0, 7, 7] = -np.inf
    t2[1, 2, 3, 5], t2[1, 2, 5, 3] = np.inf, -np.inf
    t2[2, 1, 9, 8] = np.nan
    t2[2, 2, 10, 36] = t2[2, 2, 36, 10] = 1.5e308
    L *= 0.02  # |(ac|bd)| <= 2.4e-3: those results stay finite
    V = np.einsum("nac,nbd->abcd", L, L)
    t = t2.transpose(0, 1, 3, 2) if exchange else t2
    with np.errstate(invalid="ignore", over="ignore"):
        ref = (V.reshape(v * v, 1, v * v) * t.reshape(1, o * o, v * v)).sum(-1).T.reshape(o, o, v, v)
        mag = (np.abs(V).reshape(v * v, 1, v * v) * np.abs(t).reshape(1, o * o, v * v)).sum(-1).T.reshape(o, o, v, v)
    assert np.isinf(ref[0, 1]).all() and np.isnan(ref[2, 1]).all() and np.isfinite(ref[2, 2]).all()
    assert 0 < np.isnan(ref[1, 2]).sum() < v * v
    R0 = rng.standard_normal(ref.shape)
    for acc in (False, True):
        R = torch.from_numpy(R0.copy()).to(dev)
        B.ladder_forward(torch.from_numpy(L).to(dev), torch.from_numpy(t2).to(dev), R=R, mode="fp64", symmetric=False,
                         order="integral_first", a_block=a_block, exchange=exchange, accumulate=acc)
        R = R.cpu().numpy() - (R0 if acc else 0.0)
        fin = np.isfinite(ref)
        assert np.array_equal(np.isnan(R), np.isnan(ref))
        assert np.array_equal(R[np.isinf(ref)], ref[np.isinf(ref)])
        assert np.all(np.abs(R[fin] - ref[fin]) <= 1e-13 * mag[fin] + (1e-13 if acc else 0.0))


@pytest.mark.parametrize("v", [9, 37, 160])
def test_emulated_general_amplitudes_up_to_the_largest_double(dev, v):
    """Finite amplitudes whose sums t_cd + t_dc pass 2^1024 are no infinities: the same bits as their 2^-200th, times
    2^200 (v = 160: rows walked by a cluster); infinite ones are still refused."""
    o, n = 2, 5
    L, _ = synth.ladder_inputs_torch(o, v, n, seed=3, device="cuda")
    L *= 2.0 ** -80
    g = torch.Generator(device=dev).manual_seed(v)
    t2 = (0.5 + 0.49 * torch.rand((o, o, v, v), dtype=torch.float64, device=dev, generator=g)) * 2.0 ** 824
    t2[1, 1] *= 2.0 ** -30  # a row without such sums
    want = B.ladder_forward(L, t2, symmetric=False, order="integral_first")
    huge = t2 * 2.0 ** 200
    assert torch.isfinite(huge).all() and torch.isinf(huge[0, 0] + huge[0, 0].T).any()
    got = B.ladder_forward(L, huge, symmetric=False, order="integral_first")
    assert torch.isfinite(got).all() and torch.equal(got, want * 2.0 ** 200)
    huge[1, 0, 3, 5] = float("inf")
    with pytest.raises(_lib.LadderError) as e:
        B.ladder_forward(L, huge, symmetric=False, order="integral_first")
    assert e.value.status == -11
