"""Repeated launches on the same inputs give the same bytes: nothing on the path depends on the order in which
CTAs, warps or copies happen to run (split units are merged in a fixed order, no atomics touch the data).  A missing
fence or a reused buffer released too early would show up here as a rare difference."""
import math

import numpy as np
import pytest
import torch

from paper_2605_26266_b200 import inputs
from tests import kvq_testlib as T

pytestmark = pytest.mark.gpu

CASES = [
    # workload, heads, tokens per chunk, cached chunks, launches
    ("sweep_int2", 16, 1560, 4, 60),     # every unit split over the SMs, ragged last query block
    ("dit", 24, 1560, 3, 40),            # a round of 148 whole units, then 20 units split; two groups per key
    ("pipeline", 6, 300, 5, 60),         # four groups per key, heavy-tailed keys, 12 units split
    ("sweep_int4", 3, 129, 2, 60),       # INT4, three whole units, one row past a tile in both directions
]


@pytest.mark.parametrize("kernel", ["KVQ_KERNEL_TCGEN05", "KVQ_KERNEL_TCGEN05_PAIR"])
@pytest.mark.parametrize("name,heads,tokens,chunks,launches", CASES, ids=[c[0] for c in CASES])
def test_repeated_launches_give_identical_bytes(name, heads, tokens, chunks, launches, kernel):
    from paper_2605_26266_b200 import binding as B
    w = inputs.WORKLOADS[name]
    sigma = 1.0 / math.sqrt(w.head_dim)
    cut = lambda a: T.to_dev(np.ascontiguousarray(a[:1, :heads]))
    cache = B.Cache(1, heads, w.head_dim, w.bits, w.group, 128 * (-(-tokens * (chunks + 1) // 128)))
    first_bytes = None
    for c in range(chunks):
        _, k, v = (cut(a) for a in inputs.make_chunk(w, c, tokens=tokens))
        B.kvq_quantize_append(cache, k, v)
    q, k, v = (cut(a) for a in inputs.make_chunk(w, chunks, tokens=tokens))
    n = cache.length
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ref_out = ref_lse = None
    for i in range(launches):
        out = torch.empty_like(q)
        lse = torch.empty(q.shape[:3], dtype=torch.float32, device="cuda")
        B.kvq_attn_corrected(cache, q, k, v, sigma, B.KVQ_CORRECTION_ON | getattr(B, kernel), cache_len=n,
                             out=out, lse=lse, status_word=status)
        B.kvq_quantize_append(cache, k, v, cache_len=n)          # the append of the step, every time at the same place
        if ref_out is None:
            ref_out, ref_lse = out, lse
            first_bytes = [b.clone() for b in cache.buffers]
        else:
            assert torch.equal(out.view(torch.int16), ref_out.view(torch.int16)), f"launch {i}"
            assert torch.equal(lse.view(torch.int32), ref_lse.view(torch.int32)), f"launch {i}"
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for a, b in zip(cache.buffers, first_bytes):
        assert torch.equal(a, b)


@pytest.mark.parametrize("bits,group", [(2, 32), (2, 128), (4, 32)])
def test_pair_ranges_that_start_in_the_cache_give_identical_bytes(bits, group):
    """More units than SM pairs, so that the last round is cut into ranges: most of them start in the cache, where the
    TMA thread waits for the dequantizing warps to give back a stage of packed tiles and refills it at once."""
    from paper_2605_26266_b200 import binding as B
    b, h, m, n, d = 2, 32, 2048, 8192, 128
    g = torch.Generator(device="cuda").manual_seed(7)
    draw = lambda t: torch.randn(b, h, t, d, device="cuda", generator=g)
    cache = B.Cache(b, h, d, bits, group, n)
    heavy = draw(n) / (sum(draw(n).square() for _ in range(3)) / 3).sqrt()           # Student-t(3) keys
    heavy[..., :8] *= 10.0                                                           # a few keys carry a row: one wrong value row shows
    B.kvq_quantize_append(cache, heavy.to(torch.bfloat16), draw(n).to(torch.bfloat16))
    del heavy
    q, k, v = (draw(m).to(torch.bfloat16) for _ in range(3))
    first = None
    for i in range(60):
        out = B.kvq_attn_corrected(cache, q, k, v, d ** -0.5, B.KVQ_CORRECTION_ON | B.KVQ_KERNEL_TCGEN05_PAIR)
        first = out if first is None else first
        assert torch.equal(out.view(torch.int16), first.view(torch.int16)), f"launch {i}"


@pytest.mark.parametrize("d,heads,rows,n,bits,kernel", [
    (64, 2, 256, 1024, 2, "KVQ_KERNEL_AUTO"), (64, 16, 300, 3000, 4, "KVQ_KERNEL_AUTO"),      # tcgen05, every unit split
    (64, 80, 300, 700, 2, "KVQ_KERNEL_AUTO"),                                                 # whole units
    (64, 8, 16, 3000, 2, "KVQ_KERNEL_AUTO"), (128, 8, 16, 3000, 4, "KVQ_KERNEL_AUTO"), (128, 3, 30, 2000, 2, "KVQ_KERNEL_AUTO"),   # a few rows, split
    (128, 8, 48, 3000, 2, "KVQ_KERNEL_TCGEN05"), (128, 8, 128, 3000, 4, "KVQ_KERNEL_TCGEN05"),   # one query tile
])
def test_overlapping_kernels_on_a_poisoned_workspace(d, heads, rows, n, bits, kernel):
    """The kernels of a call overlap: one that read what the one before it has not written yet would find NaN (the workspace is
    filled with it before each call) or the other problem's data (two problems in turn, back to back on one workspace)."""
    from paper_2605_26266_b200 import binding as B
    w = inputs.Workload("overlap", 880 + d + rows, 1, heads, d, 32, 0, bits, 32, 1, k_outliers=2, k_outlier_scale=4.0)
    cache = B.Cache(1, heads, d, bits, 32, 4096)
    _, k, v = inputs.make_chunk(w, 0, tokens=n)
    B.kvq_quantize_append(cache, T.to_dev(k), T.to_dev(v))
    flags, sigma = B.KVQ_CORRECTION_ON | getattr(B, kernel), 1.0 / math.sqrt(d)
    chunks = [[T.to_dev(x) for x in inputs.make_chunk(w, 1 + i, tokens=rows)] for i in range(2)]
    cache.workspace = torch.empty(B.kvq_attn_workspace_bytes(cache, n, rows, rows, flags), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")

    def call(i):
        lse = torch.empty(1, heads, rows, dtype=torch.float32, device="cuda")
        return B.kvq_attn_corrected(cache, *chunks[i], sigma, flags, lse=lse, status_word=status), lse

    first, got = [call(0), call(1)], []
    for _ in range(40):
        cache.workspace.fill_(0xFF)
        got.append((0, call(0)))
        got.append((1, call(1)))                             # straight behind, on the other's leftovers
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and torch.isfinite(first[0][0].float()).all()
    for i, (out, lse) in got:
        assert torch.equal(out.view(torch.int16), first[i][0].view(torch.int16)) and torch.equal(lse, first[i][1])
