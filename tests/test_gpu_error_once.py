"""A call that fails in the CUDA runtime reports its error once: the next call
starts clean.  The failure is made on the host, by calling entry points that
synchronise while their stream is being captured (which the runtime refuses).
(-m gpu)"""
import ctypes

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entry", ["decode_all", "decode_noalloc"])
def test_a_refused_call_leaves_no_error_behind(entry):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_10188_gb300 as acx
    acx.build.build()
    rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    data = synth.dna(200_000, 3)
    arc = acx.encode(data)
    assert np.array_equal(oracle.decode(arc), data)
    h = np.frombuffer(arc, np.uint8).copy()
    d = torch.from_numpy(h).cuda()
    out = torch.zeros(data.size, dtype=torch.uint8, device="cuda")
    ctx = acx.Context(0)
    A = acx.Archive(ctx, d.data_ptr(), h, h.size)

    def call(st):
        if entry == "decode_noalloc":
            return acx.lib.decode_noalloc(d.data_ptr(), h.size, out.data_ptr(), out.numel(), st)
        return acx.decode_all(ctx, A, out.data_ptr(), out.numel(), st)

    try:
        s = torch.cuda.Stream()
        assert call(s.cuda_stream) == 0  # (allocates the scratch)
        torch.cuda.synchronize()
        st, graph = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p()
        assert rt.cudaStreamBeginCapture(st, 2) == 0  # relaxed mode
        assert call(s.cuda_stream) == acx.lib.E_CUDA
        assert rt.cudaStreamEndCapture(st, ctypes.byref(graph)) != 0 and not graph.value
        rt.cudaGetLastError()
        out.zero_()
        assert call(torch.cuda.current_stream().cuda_stream) == 0, ctx.last_error()
        assert np.array_equal(out.cpu().numpy(), data)
    finally:
        A.close()
        ctx.close()
