"""What the planner decides, on the CPU."""
import ctypes

import pytest

from paper_2310_04559_gb300 import _lib
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


# Amplitudes without pair symmetry: packed, a call issues little more than half of 2 (o^2 + n) v^4 per product, else all of it.
@pytest.mark.parametrize("mode,o,v,n", [("ozaki_bf16", 128, 16, 336), ("ozaki_bf16", 300, 8, 20), ("ozaki_bf16", 128, 48, 200),
                                        ("fp64", 300, 8, 20), ("fp64", 64, 4, 40)])
def test_far_more_occupied_than_virtual_orbitals_run_unpacked(mode, o, v, n):
    p = _plan(o, v, n, 64 * GIB, mode=mode, symmetric=False)
    products = 1 if mode == "fp64" else 12  # at least 12 residues
    assert p["flops_issued"] >= products * p["flops_algorithmic"]


# A range of `a` without pair symmetry builds the integrals (a, all b): the work of the plain product, wherever it lies.
@pytest.mark.parametrize("mode,a_range", [("ozaki_bf16", (0, 7)), ("ozaki_bf16", (90, 100)), ("fp64", (90, 100)), ("bf16", (90, 100))])
def test_flops_of_a_range_without_pair_symmetry(mode, a_range):
    p = _plan(6, 100, 300, 8 * GIB, mode=mode, symmetric=False, a_range=a_range)
    products = 12 if mode == "ozaki_bf16" else 1  # at least 12 residues
    assert p["flops_issued"] >= products * p["flops_algorithmic"]


# The GEMM building block's workspace is what its caller allocates, beside 8 (M K + N K + M N) bytes of its own.
@pytest.mark.parametrize("M,N,K", [(60000, 60000, 60000), (125000, 125000, 1000), (50000, 50000, 50000), (8192, 8192, 8192)])
def test_gemm_workspace_leaves_room_for_the_operands(M, N, K):
    out = ctypes.c_size_t()
    assert _lib.load().cc_ladder_gemm_workspace_size(1, M, N, K, 0, ctypes.byref(out)) == 0
    digits = 2 * 6 * (M + N) * (K + 8) + 4 * (M + N) + 5 * 256
    assert out.value <= max(150 * GIB, digits)
    assert out.value + 8 * (M * K + N * K + M * N) < 275e9
