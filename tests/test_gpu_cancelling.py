"""Integral rows whose terms cancel.  Up to 3574 Cholesky vectors the integrals are put together from 64-bit fractions of
P = 256 255 253 ... 217 (12 moduli), each off by at most 12 * 128 units of P 2^-64 in units of the product of two 42-bit rows.
That error is absolute: it is set by the largest entries of the two rows of L, not by what is left of their products.

With rows of L that are integers of at most 2^21 nothing else is rounded before the integral rows are, so, 2^e > max |row|,
  |V - exact| <= 2^(eA + eB - 82) 1536 P 2^-64  (+ 2^-41 of the row's largest |V|, its rounding to 43 bits)
for the halves V+- together, times sum |t_ij|, and as much again for their sum and the conversion to FP64."""
import math

import numpy as np
import pytest
import torch

from paper_2310_04559_gb300 import binding as B

pytestmark = pytest.mark.gpu

P12 = math.prod((256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217))


@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("v,n,left", [(24, 60, 1), (33, 200, 3), (40, 3574, 1)])
def test_cancelling_integrals(v, n, left, sym):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    o = 2
    rng = np.random.default_rng(v)
    # pairs of Cholesky vectors, equal but for a sign in the columns a < v / 2 and for `left` in the others:
    # (ac|bd) of a < v / 2 <= b is a sum of products that cancel down to `left` / 2^20 of them
    half = v // 2
    base = rng.integers(-2 ** 20, 2 ** 20, (n // 2, v, v))
    L = np.empty((n // 2, 2, v, v))
    L[:, 0] = base
    L[:, 1, :half] = -base[:, :half]
    L[:, 1, half:] = base[:, half:] + rng.integers(-left, left + 1, (n // 2, v - half, v))
    L = L.reshape(n // 2 * 2, v, v)
    t2 = rng.integers(-3, 4, (o, o, v, v)).astype(np.float64)
    if sym:
        t2 = t2 + t2.transpose(1, 0, 3, 2)
    dev = torch.device("cuda", 0)
    R = B.ladder_forward(torch.from_numpy(L).to(dev), torch.from_numpy(t2).to(dev), symmetric=sym,
                         order="integral_first").cpu().numpy()
    Ld, td = torch.from_numpy(L).to(dev), torch.from_numpy(t2).to(dev)
    # all integers: |V| < n 2^42 < 2^54, R < v^2 6 2^54: FP64 sums are off by far less than the bound
    V = torch.einsum("Pac,Pbd->abcd", Ld, Ld)
    ref = torch.einsum("abcd,ijcd->ijab", V, td).cpu().numpy()
    top = V.abs().amax(dim=(2, 3))
    top = torch.maximum(top, top.T).cpu().numpy()
    e = np.frexp(np.abs(L).max(axis=(0, 2)))[1]  # per orbital a: 2^e > the largest entry of its rows
    unit = 2.0 ** (e[:, None] + e[None, :] - 82.0) * 1536 * (P12 * 2.0 ** -64)
    bound = 2 * np.abs(t2).sum(axis=(2, 3))[:, :, None, None] * (unit + 2.0 ** -41 * top)[None, None]
    bound += 1e-13 * (v * v * 6 * top)[None, None]
    assert np.all(np.abs(R - ref) <= bound)
    # the cancelling rows are those the absolute part is there for
    mixed = (slice(0, half), slice(half, v))
    assert top[mixed].max() < 2.0 ** -12 * top[:half, :half].max()
