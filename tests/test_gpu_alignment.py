"""Rows that start on 16-byte boundaries only (what the interface asks for) give the bytes of rows on 32-byte boundaries, which the
attention kernel's stores and the append kernel's loads take 32 bytes at a time."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def layouts(x, how):
    """x in memory of its own: "dense", every token 16 bytes longer, or the whole tensor 16 bytes further on."""
    b, h, t, d = x.shape
    if how == "dense":
        return x.clone()
    if how == "rows":
        y = torch.full((b, h, t, d + 8), 7.0, dtype=x.dtype, device=x.device)[..., :d]
    else:
        y = torch.full((x.numel() + 8,), 7.0, dtype=x.dtype, device=x.device)[8:].view(b, h, t, d)
    assert (y.data_ptr() | y.stride(2) * 2) % 16 == 0 and (y.data_ptr() % 32 or y.stride(2) * 2 % 32)
    return y.copy_(x)


@pytest.mark.parametrize("how", ["rows", "start"])
@pytest.mark.parametrize("d,heads,m,n", [(128, 40, 1024, 0), (128, 160, 200, 130), (64, 160, 300, 129)])
def test_16_byte_boundaries(d, heads, m, n, how):
    from paper_2605_26266_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(d + m)
    draw = lambda t: torch.randn(1, heads, t, d, device="cuda", generator=g).bfloat16()
    pk, pv, q, k, v = draw(max(n, 37)), draw(max(n, 37)), draw(m), draw(m), draw(m)
    results = []
    for l in ("dense", how):
        cache = B.Cache(1, heads, d, 2, 32, 256)
        B.kvq_quantize_append(cache, layouts(pk, l), layouts(pv, l))
        out = layouts(torch.zeros_like(q), l)
        B.kvq_attn_corrected(cache, q, k, v, d ** -0.5, cache_len=n, out=out)
        results.append([out.contiguous().view(torch.int16), *cache.buffers])
        if l == "rows":
            assert bool((out.as_strided((heads * m, 8), (d + 8, 1), out.storage_offset() + d) == 7.0).all())     # nothing behind a row
    assert all(torch.equal(a, b) for a, b in zip(*results))
