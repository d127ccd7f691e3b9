"""A refused launch of a matrix product is reported by the call it belongs to
and leaves no error behind for the next one.  The launch is refused on the host:
its stream is in a capture that an unsupported call has invalidated."""
import ctypes

import numpy as np
import pytest

import paper_2409_10399_gb300 as lbm

pytestmark = pytest.mark.gpu


def _cudart():
    import torch
    torch.cuda.current_stream()
    for line in open("/proc/self/maps"):
        if "libcudart" in line:
            return ctypes.CDLL(line.split()[-1])
    pytest.skip("no shared CUDA runtime in the process")


@pytest.mark.parametrize("dtype", ["float32", "bfloat16"])
def test_refused_product_leaves_no_error_pending(dtype):
    import torch
    rt = _cudart()
    a = torch.randn(64, 64, device="cuda").bfloat16()
    c = torch.zeros(64, 64, device="cuda", dtype=getattr(torch, dtype))
    lbm.fno_gemm(a, a, c)  # a good call first
    want = c.clone()
    pops = torch.full((6, 9, 32), 0.1, dtype=torch.float64, device="cuda")
    out = np.zeros(8)
    lbm.diag_populations_noalloc("D2Q9", 2, pops.data_ptr(), 32, out.ctypes.data, 0)
    torch.cuda.synchronize()
    raw = ctypes.c_void_p()
    assert rt.cudaStreamCreateWithFlags(ctypes.byref(raw), 1) == 0
    st = type("Stream", (), {"cuda_stream": raw.value})()
    graph = ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(raw, 1) == 0
    try:
        assert rt.cudaStreamSynchronize(raw) != 0  # not allowed in a capture, which it invalidates
        rt.cudaGetLastError()
        with pytest.raises(lbm.LBMError) as e:
            lbm.fno_gemm(a, a, c, stream=st)
        assert e.value.code == -3
    finally:
        assert rt.cudaStreamEndCapture(raw, ctypes.byref(graph)) != 0
        rt.cudaGetLastError()
        assert rt.cudaStreamDestroy(raw) == 0
    again = np.zeros(8)
    lbm.diag_populations_noalloc("D2Q9", 2, pops.data_ptr(), 32, again.ctypes.data, 0)
    assert np.array_equal(out, again)
    c.zero_()
    lbm.fno_gemm(a, a, c)
    assert torch.equal(c, want)
