"""The calls only enqueue work on the caller's stream (no allocation, no synchronisation), so a step
(attention over the cache, then quantize-append of the chunk) can be captured in a CUDA graph and replayed.
The replayed step must give the bytes of the eager one."""
import math

import numpy as np
import pytest
import torch

from paper_2605_26266_b200 import inputs
from tests import kvq_testlib as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["KVQ_KERNEL_TCGEN05", "KVQ_KERNEL_TCGEN05_PAIR"])
@pytest.mark.parametrize("heads,tokens", [(4, 600), (40, 1560)])   # units split over the SMs + merge / persistent rounds of whole units
def test_step_replayed_from_a_graph_equals_the_eager_step(heads, tokens, kernel):
    from paper_2605_26266_b200 import binding as B
    w = inputs.WORKLOADS["sweep_int2"]
    sigma = 1.0 / math.sqrt(w.head_dim)
    reps = -(-heads // w.heads)                  # more heads than the workload has: its heads again
    chunks = [[T.to_dev(np.ascontiguousarray(np.tile(a, (1, reps, 1, 1))[:, :heads]))
               for a in inputs.make_chunk(w, c, tokens=tokens)] for c in range(3)]

    def fresh():
        cache = B.Cache(1, heads, w.head_dim, w.bits, w.group, 5120)
        for q, k, v in chunks[:2]:
            B.kvq_quantize_append(cache, k, v)
        return cache

    q, k, v = chunks[2]
    flags = B.KVQ_CORRECTION_ON | getattr(B, kernel)

    eager = fresh()
    n = eager.length
    out_e = B.kvq_attn_corrected(eager, q, k, v, sigma, flags)
    B.kvq_quantize_append(eager, k, v)
    torch.cuda.synchronize()

    cache = fresh()
    out_g = torch.zeros_like(out_e)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    # the workspace is sized before the capture: nothing may allocate inside it
    need = B.kvq_attn_workspace_bytes(cache, n, tokens, tokens, flags)
    cache.workspace = torch.empty(max(need, 16), dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            B.kvq_attn_corrected(cache, q, k, v, sigma, flags, cache_len=n, out=out_g, status_word=status)
            B.kvq_quantize_append(cache, k, v, cache_len=n)
    torch.cuda.synchronize()
    for _ in range(2):                       # a replay writes the same slots again
        out_g.zero_()
        graph.replay()
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert torch.equal(out_g.view(torch.int16), out_e.view(torch.int16))
    for a, b in zip(cache.buffers, eager.buffers):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


@pytest.mark.parametrize("d,heads,tokens", [(64, 4, 300), (64, 8, 16), (128, 8, 16)])
def test_auto_kernels_replayed_from_a_graph(d, heads, tokens):
    """The kernels KVQ_KERNEL_AUTO takes for 64 channels and for a few rows; their kernels of one call overlap in the graph too."""
    from paper_2605_26266_b200 import binding as B
    w = inputs.Workload("graph", 870 + d + tokens, 1, heads, d, 32, 0, 2, 64, 1)
    cache = B.Cache(1, heads, d, 2, 64, 4096)
    _, k, v = inputs.make_chunk(w, 0, tokens=3000)
    B.kvq_quantize_append(cache, T.to_dev(k), T.to_dev(v))
    q, k, v = (T.to_dev(x) for x in inputs.make_chunk(w, 1, tokens=tokens))
    flags, sigma = B.KVQ_CORRECTION_ON, 1.0 / math.sqrt(d)
    assert B.kvq_attn_kernel_launches(cache, 3000, tokens, tokens, flags) >= 2
    cache.workspace = torch.empty(B.kvq_attn_workspace_bytes(cache, 3000, tokens, tokens, flags), dtype=torch.uint8, device="cuda")
    want = B.kvq_attn_corrected(cache, q, k, v, sigma, flags)
    out = torch.zeros_like(want)
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            B.kvq_attn_corrected(cache, q, k, v, sigma, flags, out=out)
            B.kvq_attn_corrected(cache, out, k, v, sigma, flags, out=out)      # the next call of the step, in place
    torch.cuda.synchronize()
    again = B.kvq_attn_corrected(cache, want, k, v, sigma, flags)
    for _ in range(3):
        out.zero_()
        cache.workspace.fill_(0xFF)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out.view(torch.int16), again.view(torch.int16))


@pytest.mark.parametrize("d,heads,m,n", [(64, 2, 256, 1024), (128, 32, 16, 8192), (128, 16, 300, 3072), (128, 24, 1024, 2048), (128, 40, 700, 0), (64, 40, 300, 1024)])
def test_calls_behind_joins(d, heads, m, n):
    """Calls whose first kernel follows two nodes (a join of two streams) or a copy: the bytes of the synchronised chain, eager and
    replayed."""
    from paper_2605_26266_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(31)
    draw = lambda t: torch.randn(1, heads, t, d, device="cuda", generator=g).bfloat16()
    cache = B.Cache(1, heads, d, 2, 64, (max(n, 128) + 127) // 128 * 128 + 1024)
    past = draw(max(n, 16)), draw(max(n, 16))
    q0, k0, v0 = draw(m), draw(m), draw(m)
    q, k, v, q2 = (torch.empty_like(q0) for _ in range(4))
    outs = [torch.empty_like(q0) for _ in range(4)]
    big = torch.zeros(1 << 24, device="cuda")
    side = torch.cuda.Stream()

    def chain(sync):
        main = torch.cuda.current_stream()
        for a, b in ((q, q0), (k, k0), (v, v0)):
            a.copy_(b)
        if n:
            B.kvq_quantize_append(cache, *past, cache_len=0)
        for i in range(4):
            side.wait_stream(main)
            big.add_(1.0)
            q.mul_(1.03125)                                       # main: the queries
            with torch.cuda.stream(side):                         # side: the chunk, quantized into the window
                k.neg_()
                sync()
                if n:
                    B.kvq_quantize_append(cache, k, v, cache_len=0)
                if i == 2:
                    k.zero_()
            sync()
            main.wait_stream(side)
            B.kvq_attn_corrected(cache, q, k, v, d ** -0.5, cache_len=n, out=outs[i])     # behind both
            sync()
            q2.copy_(outs[i])
            v.copy_(q2)                                           # a copy node right before the next call on this stream
            sync()
            k.copy_(k0)
            B.kvq_attn_corrected(cache, q2, k, v, d ** -0.5, cache_len=n, out=outs[i])
            sync()
    chain(torch.cuda.synchronize)
    torch.cuda.synchronize()
    want = [o.clone() for o in outs] + [b.clone() for b in cache.buffers]
    chain(lambda: None)
    torch.cuda.synchronize()
    assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(outs + cache.buffers, want))
    graph = torch.cuda.CUDAGraph()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=stream):
        chain(lambda: None)
    for _ in range(4):
        for o in outs:
            o.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(outs + cache.buffers, want))
