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
