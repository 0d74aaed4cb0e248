"""Heads of 64 channels on the tcgen05 kernel: weights far below the largest of their row, and values that are not finite or
the largest a BF16 holds."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1024, 65536])
@pytest.mark.parametrize("bits_below", [0.0, 9.7, 16.3, 24.3, 25.2, 30.0, 60.4])
def test_one_strong_key_over_many_weak_ones(n, bits_below):
    """One current key whose value is zero, and n cached keys that many bits below it: the output is all theirs.  Each weight has
    eight bits or more whatever its size, and their sum is counted in FP32, so the bound is that of a BF16 output, and twice over
    for the FP32 score (an error of 2^-24 of 60 bits)."""
    from paper_2605_26266_b200 import binding as B
    heads, m = max(1, 16384 // n) * 5, 200                        # beyond the few-row kernel: more than 8 192 steps
    assert heads * -(-m // 16) * (n // 32 + 1) > 8192
    cache = B.Cache(1, heads, 64, 2, 64, n, rotate_k=False)
    k = torch.zeros(1, heads, n, 64, device="cuda", dtype=torch.bfloat16)              # scores 0
    v = (torch.arange(64, device="cuda") % 4).to(torch.bfloat16).expand(1, heads, n, 64).contiguous()      # step 1, zero-point 0: exact
    B.kvq_quantize_append(cache, k, v)
    q, kc, vc = (torch.zeros(1, heads, t, 64, device="cuda", dtype=torch.bfloat16) for t in (m, 1, 1))
    q[..., 0], kc[..., 0] = 8.0, float(bits_below) * np.log(2.0)
    lse = torch.zeros(1, heads, m, dtype=torch.float32, device="cuda")
    mass = torch.zeros_like(lse)
    out = B.kvq_attn_corrected(cache, q, kc, vc, 0.125, B.KVQ_CORRECTION_OFF, lse=lse, cached_mass=mass)
    score = kc[0, 0, 0, 0].double().cpu()                                              # q . k / 8
    weak = n * torch.exp(-score)
    want = (weak / (1 + weak) * (torch.arange(64) % 4)).expand(1, heads, m, 64)
    assert torch.equal(out.cpu()[..., ::4], torch.zeros(1, heads, m, 16, dtype=torch.bfloat16))
    assert ((out.cpu().double() - want).abs() <= 2.0 ** -8 * want).all()
    assert ((mass.cpu().double() - weak / (1 + weak)).abs() <= 1e-4 * weak).all()
    assert ((lse.cpu().double() - (score + torch.log1p(weak))).abs() <= 1e-4).all()


@pytest.mark.parametrize("kind", ["equal", "random", "one"])
def test_infinite_values_stay_infinite(kind):
    """A weight that is exactly 1, or has no more than eight bits, leaves nothing for its second part, and 0 * inf is NaN."""
    from paper_2605_26266_b200 import binding as B
    heads, m, n, n_cur = 75, 200, 200, 1 if kind == "one" else 130
    g = torch.Generator(device="cuda").manual_seed(3)
    draw = lambda t: torch.randn(1, heads, t, 64, device="cuda", generator=g).bfloat16()
    cache = B.Cache(1, heads, 64, 2, 64, 256)
    B.kvq_quantize_append(cache, draw(n), draw(n))
    q, k, v = draw(m), draw(n_cur), draw(n_cur)
    if kind == "equal":
        q.zero_()                                                                      # every weight is 1
    at = n_cur // 2
    v[..., at, 3], v[..., at, 7], v[..., at, 40] = float("inf"), float("-inf"), float("nan")
    v[..., 0, 50], v[..., n_cur - 1, 51] = float("inf"), float("-inf")
    want = B.kvq_attn_corrected(cache, q, k, v, 0.125, B.KVQ_CORRECTION_ON | B.KVQ_KERNEL_MMA_SYNC)
    got = B.kvq_attn_corrected(cache, q, k, v, 0.125, B.KVQ_CORRECTION_ON)
    assert torch.isposinf(want[..., 3]).all() and torch.isneginf(want[..., 7]).all() and torch.isnan(want[..., 40]).all()
    for same in (torch.isposinf, torch.isneginf, torch.isnan):
        assert torch.equal(same(got), same(want))
    finite = torch.isfinite(want)
    assert (got[finite].float() - want[finite].float()).norm() < 1e-2 * want[finite].float().norm()


@pytest.mark.parametrize("heads,m,n_cur", [(75, 200, 130), (8, 300, 2000)])           # whole units, split ones
@pytest.mark.parametrize("rise", [1.0, 3.5, 7.5, 20.0])
def test_the_largest_values_stay_finite(rise, heads, m, n_cur):
    """A key some bits above those before it has a weight of at most 1, so that its value may be the largest BF16 number."""
    from paper_2605_26266_b200 import binding as B
    n = 64
    cache = B.Cache(1, heads, 64, 2, 64, 128)
    zeros = lambda t: torch.zeros(1, heads, t, 64, device="cuda", dtype=torch.bfloat16)
    B.kvq_quantize_append(cache, zeros(n), zeros(n))
    q, k, v = zeros(m), zeros(n_cur), zeros(n_cur)
    q[..., 0], k[..., 100, 0] = 8.0, rise * np.log(2.0)                               # the other scores are 0
    largest = torch.finfo(torch.bfloat16).max
    v[..., 100, 3], v[..., 100, 7] = largest, -largest
    want = B.kvq_attn_corrected(cache, q, k, v, 0.125, B.KVQ_CORRECTION_OFF | B.KVQ_KERNEL_MMA_SYNC)
    got = B.kvq_attn_corrected(cache, q, k, v, 0.125, B.KVQ_CORRECTION_OFF)
    assert torch.isfinite(want).all() and torch.isfinite(got).all()
    assert ((got - want).double().abs() <= 2.0 ** -7 * want.double().abs()).all()
