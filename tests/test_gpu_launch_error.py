"""A launch that the runtime refuses."""
import ctypes as C

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["append", "few rows", "tcgen05", "empty cache"])
def test_a_refused_launch_leaves_no_error_for_the_next_call(call):
    """A capture that a synchronisation has invalidated refuses every launch, on the host.  The call reports it, and the next one, on another
    stream, is not told of it again."""
    from paper_2605_26266_b200 import binding as B
    cudart = C.CDLL("libcudart.so.12")
    heads, m = 4, {"few rows": 16, "empty cache": 700}.get(call, 400)
    cache = B.Cache(1, heads, 128, 2, 64, 1024)
    x = torch.randn(1, heads, 512, 128, device="cuda").bfloat16()
    q, out = x[:, :, :m].contiguous() if m <= 512 else torch.randn(1, heads, m, 128, device="cuda").bfloat16(), None
    out = torch.empty_like(q)
    n = 0 if call == "empty cache" else 512
    B.kvq_quantize_append(cache, x, x)
    attend = lambda: B.kvq_attn_corrected(cache, q, q, q, 0.1, cache_len=n, out=out)
    attend()
    want, codes = out.clone(), B.kvq_unpack_codes(cache, 0, 0, 512)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    handle, graph = C.c_void_p(stream.cuda_stream), C.c_void_p()
    with torch.cuda.stream(stream):
        assert cudart.cudaStreamBeginCapture(handle, 2) == 0             # relaxed
        try:
            assert cudart.cudaStreamSynchronize(handle) != 0
            with pytest.raises(B.KvqError) as e:
                B.kvq_quantize_append(cache, x, x, cache_len=0) if call == "append" else attend()
            assert e.value.status == B.KVQ_ERR_CUDA
        finally:
            cudart.cudaStreamEndCapture(handle, C.byref(graph))
            cudart.cudaGetLastError()
    assert torch.equal(B.kvq_unpack_codes(cache, 0, 0, 512), codes)     # an ordinary launch, which looks at the last error
    attend()
    assert torch.equal(out.view(torch.int16), want.view(torch.int16))
