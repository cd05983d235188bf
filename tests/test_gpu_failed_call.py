"""A call that the CUDA runtime refuses returns CC_ERR_CUDA and leaves nothing behind: the next call is judged by itself.
The refusal here is the runtime's own answer on the host, a synchronising call while its stream is being captured."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2310_04559_gb300 import _lib
from paper_2310_04559_gb300 import binding as B
from paper_2310_04559_gb300 import synth

pytestmark = pytest.mark.gpu


def cudart():
    for name in ("libcudart.so.13", "libcudart.so", "/usr/local/cuda/lib64/libcudart.so"):
        try:
            return ctypes.CDLL(name)
        except OSError:
            continue
    pytest.skip("no CUDA runtime library to capture a stream with")


@pytest.mark.parametrize("mode", ["fp64", "ozaki_bf16", "bf16"])
def test_next_call_after_a_refused_one(mode):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rt = cudart()
    o, v, n = 2, 24, 30
    L, t2 = synth.ladder_inputs_torch(o, v, n, seed=4, device="cuda")
    R = torch.empty_like(t2)
    ws = B.alloc_workspace(B.workspace_size(o, v, n, mode=mode, symmetric=True), L.device)
    call = lambda: B.ladder_forward(L, t2, R=R, workspace=ws, mode=mode, symmetric=True)  # noqa: E731
    want = call().clone()
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        call()
        assert rt.cudaStreamBeginCapture(ctypes.c_void_p(s.cuda_stream), ctypes.c_int(2)) == 0  # relaxed
        try:
            with pytest.raises(_lib.LadderError) as e:
                call()
        finally:
            graph = ctypes.c_void_p()
            assert rt.cudaStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(graph)) != 0
            rt.cudaGetLastError()  # (that runtime's own record of the invalidated capture)
    assert e.value.status == -7
    torch.cuda.synchronize()
    R.zero_()
    assert np.array_equal(call().cpu().numpy(), want.cpu().numpy())
