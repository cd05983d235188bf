"""The residue form of the emulated-FP64 mode (CRT over bf16 GEMMs): its kernels at the sizes where they can go wrong.

Bounds.  Every FP64 operand row is rounded once to 2^-42 of twice its largest magnitude at most, everything after that is
exact up to the FP64 conversion, so an entry of a GEMM is off by at most K (maxA maxB) (2 * 2^-41 + 2^-82) plus its own
FP64 rounding: `bound` below, with 2^-40 for the product of both.  A second contraction adds the rounding of the
intermediate rows (at least 42 bits of the row's largest entry) in the same way."""
import ctypes

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


def cu(x, dev):
    return torch.from_numpy(np.ascontiguousarray(x)).to(dev)


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


# tile edges (256 rows, columns in units of 32), K-steps of 64, passes of 1024, moduli 12 -> 13 at K = 3574
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (255, 33, 63), (256, 256, 64), (257, 31, 65), (300, 290, 1023),
                                   (64, 513, 1024), (129, 97, 1025), (40, 300, 3574), (300, 40, 3575), (70, 65, 70001)])
def test_gemm_edges(dev, M, N, K):
    rng = np.random.default_rng(M * 7 + N * 3 + K)
    A = rng.standard_normal((M, K)) * np.exp(rng.uniform(-20, 20, (M, 1)))
    Bm = rng.standard_normal((N, K)) * np.exp(rng.uniform(-20, 20, (N, 1)))
    ref = A @ Bm.T
    C = B.gemm(cu(A, dev), cu(Bm, dev)).cpu().numpy()
    bound = K * np.abs(A).max(1)[:, None] * np.abs(Bm).max(1)[None, :] * 2.0 ** -40 + 1e-13 * (np.abs(A) @ np.abs(Bm).T)
    assert np.all(np.abs(C - ref) <= bound)
    # one sign: every residue sum grows linearly, and integers come out exactly
    Ai, Bi = rng.integers(1, 400, (M, K)).astype(np.float64), rng.integers(1, 400, (N, K)).astype(np.float64)
    Ci = B.gemm(cu(Ai, dev), cu(Bi, dev)).cpu().numpy()
    assert np.array_equal(Ci, Ai @ Bi.T)


def test_gemm_smaller_workspace_runs_digit_slices(dev):
    """A workspace of the digit slices' size is still taken (with the digit slices), one byte less is refused."""
    lib = _lib.load()
    M, N, K = 200, 130, 900
    rng = np.random.default_rng(1)
    A, Bm = cu(rng.standard_normal((M, K)), dev), cu(rng.standard_normal((N, K)), dev)
    al = lambda x: (x + 255) & ~255  # noqa: E731
    digits = 256 + al(2 * 6 * M * 904) + al(4 * M) + al(2 * 6 * N * 904) + al(4 * N)
    full = ctypes.c_size_t()
    assert lib.cc_ladder_gemm_workspace_size(1, M, N, K, 0, ctypes.byref(full)) == 0 and full.value > digits
    out = []
    for nbytes in (full.value, digits, digits - 1):
        C = torch.zeros((M, N), dtype=torch.float64, device=dev)
        ws = B.alloc_workspace(nbytes, dev)
        st = lib.cc_ladder_gemm(1, M, N, K, B._ptr(A), K, B._ptr(Bm), K, B._ptr(C), N, 0, 0, B._ptr(ws), nbytes, B._stream(dev))
        out.append((st, C.cpu().numpy()))
    ref = (A @ Bm.T).cpu().numpy()
    assert [s for s, _ in out] == [0, 0, -4]
    assert rel(out[0][1], ref) < 1e-11 and rel(out[1][1], ref) < 1e-10


# v odd, even, a multiple of 4, of 16, beyond one 32-tile and beyond a cluster's share; o = 1 has no antisymmetric part
@pytest.mark.parametrize("o,v,n", [(1, 1, 3), (1, 33, 20), (3, 2, 5), (2, 31, 65), (3, 36, 70), (4, 48, 30), (2, 101, 40)])
@pytest.mark.parametrize("sym", [True, False])
def test_ladder_sizes_against_oracle(dev, oracle, o, v, n, sym):
    rng = np.random.default_rng(o * 100 + v)
    L = synth.cholesky_vectors(n, v, symmetric=False, rng=rng)
    t2 = synth.amplitudes(o, v, symmetric=sym, rng=rng)
    ref = oracle.ladder(L, t2)
    for order in ("integral_first", "cholesky_first"):
        R = B.ladder_forward(cu(L, dev), cu(t2, dev), symmetric=sym, order=order).cpu().numpy()
        assert rel(R, ref) < 2e-11, (order, rel(R, ref))


@pytest.mark.parametrize("sym", [True, False])
def test_rows_of_very_different_size(dev, oracle, sym):
    """Orbitals scaled over 60 orders of magnitude: integral rows far below the range of the integers take the second,
    exact walk for their exponent, and every a, b keeps its own relative accuracy."""
    o, v, n = 2, 40, 50
    rng = np.random.default_rng(9)
    s = np.exp2(rng.integers(-100, 100, v).astype(np.float64))
    L = synth.cholesky_vectors(n, v, symmetric=False, rng=rng) * s[None, :, None]
    L[:, 3, :] *= np.exp2(-60.0) * (np.arange(v) == 7)  # one non-zero column, tiny
    L[:, 5, :] = 0.0
    t2 = synth.amplitudes(o, v, symmetric=sym, rng=rng)
    ref = oracle.ladder(L, t2)
    R = B.ladder_forward(cu(L, dev), cu(t2, dev), symmetric=sym, order="integral_first").cpu().numpy()
    for a in range(v):
        for b in range(v):
            nr = np.linalg.norm(ref[:, :, a, b])
            assert np.linalg.norm(R[:, :, a, b] - ref[:, :, a, b]) <= 1e-10 * nr, (a, b)


def test_streamed_L_equals_resident_L(dev):
    """Chunks of Cholesky vectors add their residues, so the streamed result is the resident one, bit for bit."""
    o, v, n = 3, 40, 150
    L, t2 = synth.ladder_inputs(o, v, n, seed=3)
    want = B.ladder_forward(cu(L, dev), cu(t2, dev), symmetric=True, order="integral_first").cpu().numpy()
    for chunk in (33, 64, 150):
        R = B.ladder_forward(torch.from_numpy(L).pin_memory(), cu(t2, dev), symmetric=True, host_L=True, chol_chunk=chunk)
        assert np.array_equal(R.cpu().numpy(), want), chunk


def test_wait_expiry_in_the_ladder(dev):
    lib = _lib.load()
    L, t2 = synth.ladder_inputs(4, 40, 80, seed=5)
    Lg, tg = cu(L, dev), cu(t2, dev)
    want = B.ladder_forward(Lg, tg, symmetric=True).cpu().numpy()
    try:
        lib.cc_ladder_set_wait_limit_ns(1)
        with pytest.raises(_lib.LadderError) as e:
            B.ladder_forward(Lg, tg, symmetric=True)
        assert e.value.status == -8
    finally:
        lib.cc_ladder_set_wait_limit_ns(0)
    assert np.array_equal(B.ladder_forward(Lg, tg, symmetric=True).cpu().numpy(), want)


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 127, 128, 129, 255, 256, 257])
def test_short_rows(dev, K):
    """Rows up to 256 elements are split by a warp each, longer ones by a CTA; integers come out exactly."""
    rng = np.random.default_rng(K)
    A, Bm = rng.integers(-999, 1000, (13, K)).astype(np.float64), rng.integers(-999, 1000, (7, K)).astype(np.float64)
    A[3] = 0.0
    A[5] *= 2.0 ** -300
    C = B.gemm(cu(A, dev), cu(Bm, dev)).cpu().numpy()
    assert np.array_equal(C, A @ Bm.T)
    A[12, K - 1] = np.nan
    with pytest.raises(_lib.LadderError):
        B.gemm(cu(A, dev), cu(Bm, dev))


@pytest.mark.parametrize("o,v,n", [(1, 3, 2), (2, 5, 3), (3, 9, 7), (2, 33, 7), (2, 67, 4)])
def test_short_rows_of_several_segments(dev, o, v, n):
    """Cholesky-first order: L rows of v and of n segments of v entries, one side and the other of 256 elements."""
    L, t2 = (x.numpy() for x in synth.ladder_inputs_torch(o, v, n, device="cpu"))
    R = B.ladder_forward(cu(L, dev), cu(t2, dev), symmetric=True, order="cholesky_first").cpu().numpy()
    ref = np.einsum("Pac,Pbd,ijcd->ijab", L, L, t2, optimize=True)
    # two roundings of rows of v, and of n v, elements to 42 bits of their largest entry
    scale = np.abs(L).max() ** 2 * np.abs(t2).max() * n * v * v
    assert np.abs(R - ref).max() <= scale * 2.0 ** -38


@pytest.mark.parametrize("M,N,K", [(300, 257, 20480), (260, 300, 20481), (300, 513, 41000), (257, 300, 61441)])
def test_long_k_is_split(dev, M, N, K):
    """More than 256 columns and more than 20480 elements: partial residues of uneven splits, summed by the conversion."""
    rng = np.random.default_rng(K)
    A, Bm = rng.integers(-400, 400, (M, K)).astype(np.float64), rng.integers(-400, 400, (N, K)).astype(np.float64)
    assert np.array_equal(B.gemm(cu(A, dev), cu(Bm, dev)).cpu().numpy(), A @ Bm.T)
