"""Streamed L in the residue form at odd sizes: every chunk after the first adds to the residue planes, whose rows are
padded to 16 bytes, so the sums of ragged tiles have to come out as those of resident L, bit for bit."""
import pytest
import torch

from paper_2310_04559_gb300 import binding as B
from paper_2310_04559_gb300 import synth

pytestmark = pytest.mark.gpu


# one column, one tile, columns beside a half tile (128) and a tile (256), rows that end off 16 bytes
@pytest.mark.parametrize("o,v,n,chunk", [(1, 1, 5, 2), (2, 7, 20, 3), (2, 11, 70, 64), (3, 16, 40, 7), (2, 33, 30, 8), (2, 50, 1500, 1100)])
def test_chunks_add_up(o, v, n, chunk):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    L, t2 = synth.ladder_inputs_torch(o, v, n, seed=v, device="cpu")
    R = B.ladder_forward(L.cuda(), t2.cuda(), symmetric=True, order="integral_first")
    S = B.ladder_forward(L.pin_memory(), t2.cuda(), symmetric=True, host_L=True, chol_chunk=chunk)
    assert torch.equal(R, S)
