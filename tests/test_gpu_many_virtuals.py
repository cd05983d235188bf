"""Many virtual orbitals in the emulated-FP64 mode: the integral rows' split keeps the exponents of a row's c and d in
dynamic shared memory beside its tiles, so from v = 953 on the two together pass the 48 KB that a launch gets unasked.

Bound: operand rows carry 42 bits, intermediate rows 43 bits of their largest entry and an error of 2^-38 of
max|L|^2 at most, so an entry of R is off by at most n v^2 max|L|^2 max|t2| 2^-38 * 4 (n >= 3: all roundings and the FP64
conversion)."""
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


# the last size whose shared memory stays within 48 KB, the first beyond, one no multiple of four, a larger one
@pytest.mark.parametrize("v", [952, 956, 957, 1000])
@pytest.mark.parametrize("sym", [True, False])
def test_range_of_a(dev, v, sym):
    o, n, a = 2, 3, (v - 2, v - 1)
    L, t2 = synth.ladder_inputs_torch(o, v, n, seed=v, device="cuda")
    if not sym:
        t2 = torch.randn(t2.shape, dtype=torch.float64, device=dev, generator=torch.Generator(device=dev).manual_seed(v))
    R = torch.zeros_like(t2)
    B.ladder_forward(L, t2, R=R, symmetric=sym, order="integral_first", a_range=a, budget=48 << 30)
    # R[i,j,a,b] = sum_P (L_P[a,:] t_ij) . L_P[b,:]
    X = torch.einsum("Pc,ijcd->Pijd", L[:, a[0]], t2)
    ref = torch.einsum("Pijd,Pbd->ijb", X, L)
    got = R[:, :, a[0]]
    if sym:  # written for b >= a only
        got, ref = got[:, :, a[0]:], ref[:, :, a[0]:]
    bound = n * v * v * float(L.abs().max()) ** 2 * float(t2.abs().max()) * 2.0 ** -36
    assert float((got - ref).abs().max()) <= bound
    assert float(ref.abs().max()) > 0 and np.isfinite(bound)
    # and close in the norm, far below that worst case
    assert float((got - ref).norm() / ref.norm()) < 1e-10


@pytest.mark.parametrize("n", [12275, 12276, 12280, 12283, 12284])
def test_digit_rows_of_many_segments(dev, n):
    """Cholesky-first in digit slices: the exponents of n + v segments beside 32 bytes of static shared memory."""
    o, v = 1, 5
    L, t2 = synth.ladder_inputs_torch(o, v, n, seed=1, device="cuda")
    R = B.ladder_forward(L, t2, symmetric=True, order="cholesky_first", slices=7)
    ref = torch.einsum("Pad,Pbd->ab", torch.einsum("Pac,cd->Pad", L, t2[0, 0]), L)
    assert float((R[0, 0] - ref).norm() / ref.norm()) < 1e-10
