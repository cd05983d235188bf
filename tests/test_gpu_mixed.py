"""Packed rows of the mixed modes (FP32 integral block, V+- rounded once to bf16 or tf32) at tile edges and odd sizes.

With one nonzero amplitude per pair, R_ijab is one integral (two for i = j) times it, so every packed position is read back.
Bound: L is rounded twice per product, V+- and T+- once each, and |V+| + |V-| <= V_1 + V_2 for the two integrals of a
position, all of one sign: at most (2 + 1 + 1) u (V_1 + V_2) |t| to first order, u = 2^-8 (bf16) or 2^-11 (tf32), FP32 sums far below."""
import numpy as np
import pytest
import torch

from paper_2310_04559_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,u", [("bf16", 2.0 ** -8), ("tf32", 2.0 ** -11)])
@pytest.mark.parametrize("v,a_block", [(1, 0), (2, 1), (31, 0), (32, 5), (33, 0), (64, 0), (65, 7), (97, 0)])
def test_every_packed_position(mode, u, v, a_block):
    o, n = 4, 5
    rng = np.random.default_rng(v)
    L = rng.uniform(0.05, 1.0, (n, v, v))
    L = 0.5 * (L + L.transpose(0, 2, 1))
    edge = [min(x, v - 1) for x in (0, 31, 32, 33, 63, 64, v - 1)]
    t2 = np.zeros((o, o, v, v))
    for i in range(o):
        for j in range(i, o):
            c, d = (rng.choice(edge, 2) if rng.random() < 0.5 else rng.integers(0, v, 2))
            t2[i, j, c, d] = t2[j, i, d, c] = x = rng.uniform(0.5, 2.0) * rng.choice([-1, 1])
            if i == j:
                t2[i, i, d, c] = x
    V = np.einsum("nac,nbd->abcd", L, L)
    ref = np.einsum("abcd,ijcd->ijab", V, t2)
    bound = 4.1 * u * np.einsum("abcd,ijcd->ijab", V + V.transpose(0, 1, 3, 2), np.abs(t2))
    dev = torch.device("cuda", 0)
    R = B.ladder_forward(torch.from_numpy(L).to(dev), torch.from_numpy(t2).to(dev), mode=mode, symmetric=True,
                         order="integral_first", a_block=a_block, budget=1 << 28).cpu().numpy()
    assert np.all(np.abs(R - ref) <= bound)
