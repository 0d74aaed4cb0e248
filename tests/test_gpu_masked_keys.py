"""Keys that a caller masks through one channel: the query holds 1 there, masked current keys the lowest BF16 number or -inf,
so that their scores are about -4e37 or -inf and their weight is zero.  Whole tiles, steps and ranges of masked keys come
before others.  Expected: attention over the keys that are left."""
import numpy as np
import pytest
import torch

from oracle import kvq_oracle as O
from paper_2605_26266_b200 import inputs
from tests import kvq_testlib as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mask", [0xFF7F, 0xFF80], ids=["lowest", "-inf"])
@pytest.mark.parametrize("d,heads,m,n", [(64, 2, 129, 1000), (64, 40, 300, 130), (64, 2, 16, 1000), (64, 3, 30, 40), (128, 2, 16, 1000), (128, 200, 7, 40)])
def test_masked_keys_have_no_weight(d, heads, m, n, mask):
    from paper_2605_26266_b200 import binding as B
    n_cur = 420
    w = inputs.Workload("masked", 950 + d + m, 1, heads, d, 32, 0, 2, 64, m)
    g, o = (X.Cache(1, heads, d, 2, 64, 1024) for X in (B, O))
    _, k, v = inputs.make_chunk(w, 0, tokens=n)
    B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v))
    O.quantize_append(o, 0, k, v)
    q, _, _ = inputs.make_chunk(w, 1, tokens=m)
    _, kc, vc = inputs.make_chunk(w, 2, tokens=n_cur)
    q[..., -1] = 0x3F80
    masked = (np.arange(n_cur) < 300) | (np.arange(n_cur) % 3 == 0)
    kc[..., -1] = 0
    kept_k, kept_v = kc[:, :, ~masked], vc[:, :, ~masked]
    kc[:, :, masked, -1] = mask
    sigma = T.sigma_of(d)
    lse = torch.empty(1, heads, m, dtype=torch.float32, device="cuda")
    mass = torch.empty_like(lse)
    out = B.kvq_attn_corrected(g, T.to_dev(q), T.to_dev(kc), T.to_dev(vc), sigma, B.KVQ_CORRECTION_ON, cache_len=n, lse=lse, cached_mass=mass)
    want = O.attn_corrected(o, 0, n, q, kept_k, kept_v, sigma, correction=True)
    T.assert_attn_close(T.from_dev_bf16(out).reshape(want["out"].shape), want["out"])
    assert np.abs(lse.cpu().numpy().reshape(want["lse"].shape) - want["lse"]).max() < 2e-2
    assert np.abs(mass.cpu().numpy().reshape(want["cached_mass"].shape) - want["cached_mass"]).max() < 1e-2


@pytest.mark.parametrize("mask", [0xFF7F, 0xFF80], ids=["lowest", "-inf"])
@pytest.mark.parametrize("kernel,heads,m,n_cur,n,bits,first,last", [
    ("KVQ_KERNEL_TCGEN05", 16, 700, 700, 700, 2, 512, 700),         # 48 units of 12 tiles in ranges of four: the second starts with two masked tiles
    ("KVQ_KERNEL_TCGEN05", 16, 256, 896, 384, 4, 256, 896),         # 16 of 10: ranges of four, tiles 2 to 6 masked: one range has no other key
    ("KVQ_KERNEL_TCGEN05", 2, 300, 1100, 1000, 2, 400, 1100),       # 4 of 17, BF16 rows
    ("KVQ_KERNEL_TCGEN05_PAIR", 32, 300, 512, 1279, 2, 128, 512),   # 32 pair units of 14 tiles over 74 pairs
    ("KVQ_KERNEL_TCGEN05_PAIR", 3, 600, 2000, 500, 4, 100, 2000),   # 6 of 20, BF16 rows, ranges without another key
])
def test_ranges_that_start_with_masked_keys(kernel, heads, m, n_cur, n, bits, first, last, mask):
    """128 channels: where a unit's tiles are split, a range may start with masked keys, or hold no others; computed whole, the
    keys before them have given the row its maximum."""
    from paper_2605_26266_b200 import binding as B
    picked = sorted({0, 1, heads // 2, heads - 1})
    w = inputs.Workload("maskedrange", 2050 + heads + m, 1, heads, 128, 32, 0, bits, 64, m)
    g, o = B.Cache(1, heads, 128, bits, 64, 1280), O.Cache(1, len(picked), 128, bits, 64, 1280)
    _, k, v = inputs.make_chunk(w, 0, tokens=n)
    B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v))
    O.quantize_append(o, 0, k[:, picked], v[:, picked])
    q, _, _ = inputs.make_chunk(w, 1, tokens=m)
    _, kc, vc = inputs.make_chunk(w, 2, tokens=n_cur)
    q[..., -1], kc[..., -1] = 0x3F80, 0
    masked = (np.arange(n_cur) >= first) & (np.arange(n_cur) < last)
    kc[:, :, masked, -1] = mask
    sigma = T.sigma_of(128)
    lse = torch.empty(1, heads, m, dtype=torch.float32, device="cuda")
    mass = torch.empty_like(lse)
    out = B.kvq_attn_corrected(g, T.to_dev(q), T.to_dev(kc), T.to_dev(vc), sigma, B.KVQ_CORRECTION_ON | getattr(B, kernel), lse=lse, cached_mass=mass)
    rows = np.unique(np.r_[0, 31, 127, 128, 255, m - 1])
    want = O.attn_corrected(o, 0, n, q[:, picked], kc[:, picked][:, :, ~masked], vc[:, picked][:, :, ~masked], sigma, correction=True, rows=rows)
    T.assert_attn_close(T.from_dev_bf16(out)[0][picked][:, rows], want["out"])
    assert torch.isfinite(out.float()).all()
    assert np.abs(lse.cpu().numpy()[0][picked][:, rows] - want["lse"].reshape(len(picked), -1)).max() < 2e-2
    assert np.abs(mass.cpu().numpy()[0][picked][:, rows] - want["cached_mass"].reshape(len(picked), -1)).max() < 1e-2
