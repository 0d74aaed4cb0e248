"""A last round with fewer tile steps than CTAs: some of the ranges it is cut into are empty, and the slots of their CTAs must not
reach the merge.  The workspace is filled with NaN, or with the finite partial rows of another problem, before the call.  Nor do the
places beyond the last range."""
import numpy as np
import pytest
import torch

from oracle import kvq_oracle as O
from paper_2605_26266_b200 import inputs
from tests import kvq_testlib as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads,m,n,bits,kernel", [
    (64, 80, 300, 700, 2, "KVQ_KERNEL_AUTO"),                  # 160 units of 9 tiles on 148 SMs: 108 steps
    (64, 152, 130, 400, 4, "KVQ_KERNEL_AUTO"),                 # 152 of 6: 24 steps
    (128, 160, 200, 1280, 2, "KVQ_KERNEL_TCGEN05"),            # 160 of 12: 144 steps
    (128, 76, 512, 1300, 4, "KVQ_KERNEL_TCGEN05_PAIR"),        # 76 of 15 on 74 pairs: 30 steps
    (128, 155, 90, 1500, 4, "KVQ_KERNEL_TCGEN05"),             # 155 of 13, one query tile: 91 steps
])
def test_empty_ranges_of_the_last_round(d, heads, m, n, bits, kernel):
    from paper_2605_26266_b200 import binding as B
    picked = sorted({0, heads - 1, heads - 2, heads - 4, heads // 2} | set(range(max(0, heads - 13), heads, 3)))
    w = inputs.Workload("sparse", 890 + heads, 1, heads, d, 32, 0, bits, 64, 1)
    g, o = B.Cache(1, heads, d, bits, 64, 1536), O.Cache(1, len(picked), d, bits, 64, 1536)
    _, k, v = inputs.make_chunk(w, 0, tokens=n)
    B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v))
    O.quantize_append(o, 0, k[:, picked], v[:, picked])
    q, kc, vc = inputs.make_chunk(w, 1, tokens=m)
    flags, sigma = B.KVQ_CORRECTION_ON | getattr(B, kernel), T.sigma_of(d)
    rows = np.unique(np.r_[0, 1, 127 % m, 128 % m, 255 % m, m - 1])
    want = O.attn_corrected(o, 0, n, q[:, picked], kc[:, picked], vc[:, picked], sigma, rows=rows)
    args = (g, T.to_dev(q), T.to_dev(kc), T.to_dev(vc), sigma, flags)
    g.workspace = torch.empty(B.kvq_attn_workspace_bytes(g, n, m, m, flags), dtype=torch.uint8, device="cuda")
    first = None
    # NaN bytes; FP32 1.9 everywhere (maxima above, sums and rows of the size of real ones); zeros
    for fill in (0xFF, 0x3F, 0x00):
        g.workspace.fill_(fill)
        lse = torch.empty(1, heads, m, dtype=torch.float32, device="cuda")
        out = B.kvq_attn_corrected(*args, lse=lse)
        got = T.from_dev_bf16(out)[0][picked][:, rows]
        T.assert_attn_close(got, want["out"], f"fill {fill:#x}")
        assert np.abs(lse.cpu().numpy()[0][picked][:, rows] - want["lse"]).max() < 2e-2
        first = out if first is None else first
        assert torch.equal(out.view(torch.int16), first.view(torch.int16))


@pytest.mark.parametrize("d,heads,m,n,n_cur", [(64, 8, 300, 0, 4000), (64, 8, 300, 256, 2000), (128, 8, 300, 0, 4000), (128, 8, 300, 0, 2000), (128, 3, 600, 0, 5000)])
def test_infinite_values_in_the_last_range_of_a_unit(d, heads, m, n, n_cur):
    """Ranges are merged four at a time, and the places of the last four that are empty repeat the last range with weight zero."""
    from paper_2605_26266_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(4)
    draw = lambda t: torch.randn(1, heads, t, d, device="cuda", generator=g).bfloat16()
    cache = B.Cache(1, heads, d, 2, 64, 256)
    if n:
        B.kvq_quantize_append(cache, draw(n), draw(n))
    q, k, v = draw(m), draw(n_cur), draw(n_cur)
    v[..., n_cur - 1, 3], v[..., n_cur - 1, d - 2], v[..., 0, 5] = float("inf"), float("-inf"), float("inf")
    want = B.kvq_attn_corrected(cache, q, k, v, d ** -0.5, B.KVQ_CORRECTION_OFF | B.KVQ_KERNEL_MMA_SYNC)
    assert torch.isposinf(want[..., 3]).all() and torch.isneginf(want[..., d - 2]).all() and torch.isposinf(want[..., 5]).all()
    kernels = [0] if d == 64 else [0, B.KVQ_KERNEL_TCGEN05, B.KVQ_KERNEL_TCGEN05_PAIR]
    for kernel in kernels:
        got = B.kvq_attn_corrected(cache, q, k, v, d ** -0.5, B.KVQ_CORRECTION_OFF | kernel)
        for same in (torch.isposinf, torch.isneginf, torch.isnan):
            assert torch.equal(same(got), same(want))
