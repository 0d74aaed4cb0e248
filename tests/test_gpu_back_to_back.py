"""Calls one right behind another: the first kernel of a call is placed while the kernel before it in the stream still runs, and waits
there.  Chains of appends, attention calls and other kernels that write their inputs and read their outputs in place, without any
synchronisation, give the bytes that the same chain gives with the device idle between all of its steps."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads,m,past,rotate_v", [
    (64, 2, 256, 1024, False), (128, 4, 16, 2000, False), (64, 40, 300, 700, False), (128, 6, 256, 3000, False), (128, 3, 1000, 1500, False),
    (128, 20, 700, 0, False), (128, 4, 300, 500, True), (64, 3, 100, 600, True)])
def test_chains_without_synchronisation(d, heads, m, past, rotate_v):
    from paper_2605_26266_b200 import binding as B

    def chain(sync):
        g = torch.Generator(device="cuda").manual_seed(11)
        draw = lambda t: torch.randn(1, heads, t, d, device="cuda", generator=g).bfloat16()
        cache = B.Cache(1, heads, d, 2, 64, (past + 8 * m + 127) // 128 * 128 + 128, rotate_v=rotate_v)
        if past:
            B.kvq_quantize_append(cache, draw(past), draw(past))
        q, k, v, out = draw(m), draw(m), draw(m), torch.empty(1, heads, m, d, device="cuda", dtype=torch.bfloat16)
        big, seen = torch.zeros(1 << 24, device="cuda"), []
        for i in range(6):
            steps = [lambda: big.add_(1.0),                            # a kernel that is still running when the next is placed
                     lambda: q.mul_(1.0625),
                     lambda: B.kvq_attn_corrected(cache, q, k, v, d ** -0.5, cache_len=past if past == 0 else None, out=out),
                     lambda: k.copy_(out).add_(q),                     # the chunk's keys: read by the call before, appended next
                     lambda: B.kvq_quantize_append(cache, k, v, cache_len=past if past == 0 else None),
                     lambda: B.kvq_attn_corrected(cache, q, k, v, d ** -0.5, cache_begin=0, cache_len=past if past == 0 else None, out=out),
                     lambda: seen.append(out.clone()),
                     lambda: v.neg_()]
            for step in steps:
                step()
                if sync:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        return seen + cache.buffers
    for a, b in zip(chain(False), chain(True)):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


# Chains of the library's calls alone: a kernel of another kind in between is never released early, and would hide a missing wait.
# d, heads, rows, cached tokens: few-row kernel in clusters and with its merge kernel, one CTA split and whole, pairs, no cached
# keys (no pre-pass), 64 channels
SHAPES = [(64, 2, 256, 1024), (128, 32, 16, 8192), (128, 16, 300, 3072), (128, 24, 1024, 2048), (128, 40, 700, 0), (64, 40, 300, 1024)]


def setup(d, heads, m, n, ring=False, seed=23):
    from paper_2605_26266_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(seed)
    draw = lambda t: torch.randn(1, heads, t, d, device="cuda", generator=g).bfloat16()
    cache = B.Cache(1, heads, d, 2, 64, (max(n, 128) + 127) // 128 * 128 + (0 if ring else 1024), ring=ring)
    if n:
        B.kvq_quantize_append(cache, draw(n), draw(n))
    return B, draw, cache


def same_bytes(chain, *args):
    """chain(step) runs its calls through step(); with the device idle between all of them it has to give the same bytes."""
    def run(sync):
        torch.cuda.synchronize()

        def step(call):
            call()
            if sync:
                torch.cuda.synchronize()
        out = chain(step, *args)
        torch.cuda.synchronize()
        return [t.view(torch.uint8) for t in out]
    want = run(True)
    for _ in range(3):
        assert all(torch.equal(a, b) for a, b in zip(run(False), want))


@pytest.mark.parametrize("d,heads,m,n", SHAPES)
def test_calls_that_share_a_workspace_and_read_each_others_outputs(d, heads, m, n):
    """The next call's pre-pass or attention kernel writes the workspace that the merge before it reads; outputs come back as the next
    call's queries, and as its current keys."""
    def chain(step):
        B, draw, cache = setup(d, heads, m, n)
        qs, k, v = [draw(m) for _ in range(3)], draw(m), draw(m)
        outs = [torch.empty_like(k) for _ in range(9)]
        attend = lambda q, kc, out: step(lambda: B.kvq_attn_corrected(cache, q, kc, v, d ** -0.5, cache_len=n, out=out))
        step(lambda: None)
        for i in range(3):
            attend(qs[i], k, outs[i])
        for i in range(3, 6):
            attend(outs[i - 1], k, outs[i])
        for i in range(6, 9):
            attend(qs[i - 6], outs[i - 1], outs[i])
        return outs
    same_bytes(chain)


@pytest.mark.parametrize("d,heads,m,n", [s for s in SHAPES if s[3]])
def test_appends_that_overwrite_what_the_call_before_reads(d, heads, m, n):
    """A full ring: every append overwrites tokens of the window that the attention call before it reads, and the call after it reads them."""
    def chain(step):
        B, draw, cache = setup(d, heads, m, n, ring=True)
        size = cache.desc.capacity
        rows = (min(m, size) + 15) // 16 * 16                                # windows start on multiples of 16
        q, chunks = draw(m), [(draw(rows), draw(rows)) for _ in range(4)]
        outs = [torch.empty_like(q) for _ in range(8)]
        step(lambda: None)
        for i in range(8):
            k, v = chunks[i % 4]
            begin = cache.length - min(cache.length, size) // 16 * 16
            step(lambda: B.kvq_attn_corrected(cache, q, k, v, d ** -0.5, cache_begin=begin, cache_len=cache.length - begin, out=outs[i]))
            step(lambda: B.kvq_quantize_append(cache, k, v))
        return outs + cache.buffers
    same_bytes(chain)


@pytest.mark.parametrize("d,heads,tokens", [(128, 24, 4680), (64, 2, 256), (128, 3, 33)])
def test_appends_to_the_same_slots(d, heads, tokens):
    """The last of several appends to one place is the one that stays, whatever each warp's share of the time."""
    def chain(step):
        B, draw, cache = setup(d, heads, 0, 0)
        cache = B.Cache(1, heads, d, 2, 64, 4736)
        chunks = [(draw(tokens), draw(tokens)) for _ in range(4)]
        step(lambda: None)
        for i in range(12):
            k, v = chunks[i % 4]
            step(lambda: B.kvq_quantize_append(cache, k, v, cache_len=0))
        return cache.buffers
    same_bytes(chain)


@pytest.mark.parametrize("d,heads,m,n", SHAPES)
def test_streams_ordered_by_events(d, heads, m, n):
    """Append on one stream, attention on another, an event from each to the next."""
    def chain(step):
        B, draw, cache = setup(d, heads, m, n)
        q, k, v = draw(m), draw(m), draw(m)
        outs = [torch.empty_like(q) for _ in range(6)]
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        torch.cuda.synchronize()
        for i in range(6):
            with torch.cuda.stream(streams[0]):
                streams[0].wait_stream(streams[1])
                step(lambda: B.kvq_quantize_append(cache, k if i % 2 else v, v, cache_len=0))
            with torch.cuda.stream(streams[1]):
                streams[1].wait_stream(streams[0])
                step(lambda: B.kvq_attn_corrected(cache, q, k, v, d ** -0.5, cache_begin=0, cache_len=max(n, m // 16 * 16) if n else 0, out=outs[i]))
        return outs
    same_bytes(chain)
