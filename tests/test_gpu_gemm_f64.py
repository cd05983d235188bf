"""The FP64 GEMM at the edges of its shapes: rows around 8, 16 and 32 (warps side by side or splitting K), columns
around 8 NT, K shorter than a tile and split over a cluster, against numpy's FP64 product.  An FP64 sum of K terms is off
by at most K 2^-53 sum |a b| in either order."""
import numpy as np
import pytest
import torch

from paper_2310_04559_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(1, 8, 1), (8, 9, 15), (9, 65, 17), (16, 300, 300), (17, 7, 2000), (32, 64, 16), (33, 1, 33),
                                   (63, 257, 5000), (8, 3000, 40), (200, 190, 31)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_gemm_f64_shapes(M, N, K, accumulate):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(M + 3 * N + 5 * K)
    A, Bm, C0 = rng.standard_normal((M, K)), rng.standard_normal((N, K)), rng.standard_normal((M, N))
    g = lambda x: torch.from_numpy(x).to("cuda")  # noqa: E731
    C = B.gemm(g(A), g(Bm), mode="fp64", C=g(C0), accumulate=accumulate).cpu().numpy()
    ref = A @ Bm.T + (C0 if accumulate else 0.0)
    bound = 2 * (K + 1) * 2.0 ** -53 * (np.abs(A) @ np.abs(Bm).T + np.abs(C0))
    assert np.all(np.abs(C - ref) <= bound)
    again = B.gemm(g(A), g(Bm), mode="fp64", C=g(C0), accumulate=accumulate).cpu().numpy()
    assert np.array_equal(C, again)
