"""The few-row kernel's products of the keys' codes (at most two groups a head): every format with windows that end inside a step,
start at another slot and wrap, against the oracle; and query rows of any size, which it brings to one scale by a power of two."""
import numpy as np
import pytest
import torch

from oracle import kvq_oracle as O
from paper_2605_26266_b200 import inputs
from tests import kvq_testlib as T

pytestmark = pytest.mark.gpu

FORMATS = [(128, 2, 64), (128, 2, 128), (128, 4, 64), (128, 4, 128), (64, 2, 32), (64, 2, 64), (64, 4, 32), (64, 4, 64)]


@pytest.mark.parametrize("m,n,begin", [(16, 383, 112), (5, 33, 368), (1, 16, 0), (23, 384, 48)])      # a ring of 384 slots
@pytest.mark.parametrize("d,bits,group", FORMATS)
def test_every_format(d, bits, group, m, n, begin):
    from paper_2605_26266_b200 import binding as B
    w = inputs.Workload("codes", 1700 + m + d + group, 1, 3, d, 32, 0, bits, group, bits, k_outliers=2, k_outlier_scale=4.0)
    g, o = (X.Cache(1, 3, d, bits, group, 384, ring=True) for X in (B, O))
    _, k, v = inputs.make_chunk(w, 0, tokens=n)
    B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v), cache_len=begin)
    O.quantize_append(o, begin, k, v)
    q, _, _ = inputs.make_chunk(w, 1, tokens=m)
    _, kc, vc = inputs.make_chunk(w, 2, tokens=m)
    lse = torch.empty(1, 3, m, dtype=torch.float32, device="cuda")
    mass = torch.empty_like(lse)
    out = B.kvq_attn_corrected(g, T.to_dev(q), T.to_dev(kc), T.to_dev(vc), T.sigma_of(d), B.KVQ_CORRECTION_ON, cache_begin=begin, cache_len=n,
                               lse=lse, cached_mass=mass)
    want = O.attn_corrected(o, begin, n, q, kc, vc, T.sigma_of(d), correction=True)
    T.assert_attn_close(T.from_dev_bf16(out).reshape(want["out"].shape), want["out"])
    # products of codes leave the rotated query's FP16: 2^-12 / sqrt(3) of sigma |q| |k|, below 3 here, for the mean of a row's keys; five times that
    assert np.abs(lse.cpu().numpy().reshape(want["lse"].shape) - want["lse"]).max() < 2e-3
    assert np.abs(mass.cpu().numpy().reshape(want["cached_mass"].shape) - want["cached_mass"]).max() < 1e-2


@pytest.mark.parametrize("d,bits,group", FORMATS)
def test_queries_of_any_size(d, bits, group):
    """2^e times the query under 2^-e times the scale are the same scores, and every factor is a power of two: the same bits while the
    row's largest channel is at 2^-10 or more.  2^-30 is below that and the unit stops at 2^24: q 2^24 keeps, under the lowest code's place
    at 2^8, four bits and more of its FP16, and the scores are off by less than 2^-5 of their size."""
    from paper_2605_26266_b200 import binding as B
    heads, m, n = 3, 16, 500
    w = inputs.Workload("sizes", 1800 + d + group, 1, heads, d, 32, 0, bits, group, bits)
    g = B.Cache(1, heads, d, bits, group, 512)
    _, k, v = (T.to_dev(x) for x in inputs.make_chunk(w, 0, tokens=n))
    B.kvq_quantize_append(g, k, v)
    q, kc, vc = (T.to_dev(x) for x in inputs.make_chunk(w, 1, tokens=m))

    def run(e):
        lse = torch.empty(1, heads, m, dtype=torch.float32, device="cuda")
        out = B.kvq_attn_corrected(g, q * 2.0 ** e, kc, vc, T.sigma_of(d) * 2.0 ** -e, B.KVQ_CORRECTION_ON, lse=lse)
        return out, lse

    want = run(0)
    for e in (-8, 9, 40):
        got = run(e)
        assert torch.equal(got[0].view(torch.int16), want[0].view(torch.int16)) and torch.equal(got[1], want[1]), e
    got = run(-30)
    assert torch.isfinite(got[0].float()).all() and (got[1] - want[1]).abs().max() <= 2.0 ** -5 * want[1].abs().max()


@pytest.mark.parametrize("bits,group", [(2, 64), (2, 128), (4, 64), (4, 128)])
def test_zero_points_that_are_no_numbers(bits, group):
    """A key appended with an infinite channel has an infinite zero-point; with 128 channels its scores stay finite (as where FP16 keys
    saturate) and it takes all of a row's weight or none, exactly as a zero-point of 2^96."""
    from paper_2605_26266_b200 import binding as B
    heads, m, n = 3, 16, 200
    w = inputs.Workload("zeros", 1900 + bits + group, 1, heads, 128, 32, 0, bits, group, bits)
    _, k, v = inputs.make_chunk(w, 0, tokens=n)
    q, kc, vc = (T.to_dev(x) for x in inputs.make_chunk(w, 1, tokens=m))
    outs = []
    for bad in ((float("inf"), -float("inf"), float("nan")), (2.0 ** 96, -2.0 ** 96, 2.0 ** 96)):
        g = B.Cache(1, heads, 128, bits, group, 256)
        B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v))
        bits16 = torch.tensor(bad, device="cuda").bfloat16().view(torch.int16)
        for h in range(heads):
            g.views()["k_zero"][0, h, 40 + 60 * h, 0] = bits16[h]
        outs.append(B.kvq_attn_corrected(g, q, kc, vc, T.sigma_of(128), B.KVQ_CORRECTION_ON))
    assert torch.isfinite(outs[0].float()).all() and torch.equal(outs[0].view(torch.int16), outs[1].view(torch.int16))


@pytest.mark.parametrize("d,bits,group", FORMATS)
def test_large_queries_under_the_largest_scales(d, bits, group):
    """Where a scale near 1e30 leaves no room above them, channels beyond FP16's largest number count as that number, as with FP16 keys: scores
    stay below 2^127 and the row is the same bits as that of the clamped query."""
    from paper_2605_26266_b200 import binding as B
    heads, m, n = 3, 16, 500
    w = inputs.Workload("extreme", 1850 + d + group, 1, heads, d, 32, 0, bits, group, bits)
    g = B.Cache(1, heads, d, bits, group, 512, rotate_k=False)
    _, k, v = (T.to_dev(x) for x in inputs.make_chunk(w, 0, tokens=n))
    B.kvq_quantize_append(g, k, v)
    q = T.to_dev(inputs.make_chunk(w, 1, tokens=m)[0]) * 2.0 ** 19
    kc, vc = torch.zeros(2, 1, heads, 1, d, dtype=torch.bfloat16, device="cuda")
    got = []
    for rows in (q, q.clamp(-65536, 65536)):
        lse = torch.empty(1, heads, m, dtype=torch.float32, device="cuda")
        got.append((B.kvq_attn_corrected(g, rows, kc, vc, 9e29, B.KVQ_CORRECTION_OFF, lse=lse), lse))
    assert torch.isfinite(got[0][0].float()).all() and torch.isfinite(got[0][1]).all()
    assert torch.equal(got[0][0].view(torch.int16), got[1][0].view(torch.int16)) and torch.equal(got[0][1], got[1][1])


@pytest.mark.parametrize("mean", [0.0, 12.0, -30.0, 80.0, 3000.0, 65300.0])
@pytest.mark.parametrize("bits,group", [(2, 64), (2, 128), (4, 64), (4, 128)])
def test_keys_far_from_zero(bits, group, mean):
    """128 channels, a chunk of their own for all heads.  step (sum_c q_c code_c) and step zero (sum_c q_c) are then far larger than their
    difference.  One cached key carries the whole weight, so that the log-sum-exp is its score; queries are exact in FP16, and
    what is left are the roundings of the FP32 sums: 2^-23 for each of eight products of 16 channels, 2^-24 for each of seven additions of the query's
    channels, for step and zero, twice for their products, for the two groups and for scale and base, of step (code + zero) |q|.
    FP16 keys would be off by some 2^-13 of it."""
    from paper_2605_26266_b200 import binding as B
    heads, m, d = 24, 16, 128
    r = np.random.default_rng(int(abs(mean)) + bits + group)
    sign = -1.0 if mean < 0 else 1.0
    # every other group at the mean, another one from head to head
    shift = np.where((np.arange(d) // 64 + np.arange(heads)[:, None]) % 2, np.float32(mean), np.float32(0))[None, :, None, :]
    k = inputs.f32_to_bf16_bits(r.standard_normal((1, heads, 1, d), dtype=np.float32) + shift)
    v = inputs.f32_to_bf16_bits(r.standard_normal((1, heads, 1, d), dtype=np.float32))
    q = inputs.f32_to_bf16_bits((sign * (0.1 + np.abs(r.standard_normal((1, heads, m, d))))).astype(np.float32))
    g, o = (X.Cache(1, heads, d, bits, group, 128, rotate_k=False) for X in (B, O))
    B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v))
    O.quantize_append(o, 0, k, v)
    kc = torch.full((1, heads, 1, d), -1000.0 * sign, dtype=torch.bfloat16, device="cuda")
    lse = torch.empty(1, heads, m, dtype=torch.float32, device="cuda")
    sigma = T.sigma_of(d)
    B.kvq_attn_corrected(g, T.to_dev(q), kc, torch.ones_like(kc), sigma, B.KVQ_CORRECTION_OFF, cache_len=1, lse=lse)
    code = O.unpack_codes(o.k_codes[:, :, 0], bits).reshape(1, heads, d // group, group).astype(np.float64)
    step, zero = (np.repeat(x[:, :, 0], group, -1) for x in (O.e4m3_decode(o.k_scale), O.bf16_bits_to_f64(o.k_zero)))
    code, qf = code.reshape(1, heads, d), O.bf16_bits_to_f64(q)
    want = sigma * np.einsum("bhmd,bhd->bhm", qf, (code - zero) * step)
    size = sigma * np.einsum("bhmd,bhd->bhm", np.abs(qf), (code + np.abs(zero)) * step)
    err = np.abs(lse.cpu().numpy() - want) / size
    assert err.max() <= (8 * 2 + 7 + 2 + 2 + 1 + 3) * 2.0 ** -24, err.max()


@pytest.mark.parametrize("bits,group", [(2, 64), (2, 128), (4, 64), (4, 128)])
def test_keys_far_from_zero_among_others(bits, group):
    """Tokens from 40 on lie far from zero, in several steps and warps; the bound of the test above for keys of size 40."""
    from paper_2605_26266_b200 import binding as B
    heads, n, m, d = 6, 700, 16, 128
    r = np.random.default_rng(d + bits + group)
    far = (40.0 * (np.arange(n) >= 40)[:, None] * np.where(np.arange(heads) % 2, 1.0, -1.0)[:, None, None])[None].astype(np.float32)
    draw = lambda t, x=0: inputs.f32_to_bf16_bits((r.standard_normal((1, heads, t, d)) + x).astype(np.float32))
    g, o = (X.Cache(1, heads, d, bits, group, 768, rotate_k=False) for X in (B, O))
    k, v = draw(n, far), draw(n)
    B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v))
    O.quantize_append(o, 0, k, v)
    q, kc, vc = draw(m), draw(33), draw(33)
    lse = torch.empty(1, heads, m, dtype=torch.float32, device="cuda")
    sigma = 0.25 * T.sigma_of(d)
    out = B.kvq_attn_corrected(g, T.to_dev(q), T.to_dev(kc), T.to_dev(vc), sigma, B.KVQ_CORRECTION_ON, cache_len=n, lse=lse)
    want = O.attn_corrected(o, 0, n, q, kc, vc, sigma, correction=True)
    T.assert_attn_close(T.from_dev_bf16(out).reshape(want["out"].shape), want["out"])
    # 31 * 2^-24 of sigma (40 + 15 steps of 0.4 or 3 of 2) |q|, |q| at most 130 in sum
    assert np.abs(lse.cpu().numpy().reshape(want["lse"].shape) - want["lse"]).max() < 31 * 2.0 ** -24 * sigma * 46 * 130
