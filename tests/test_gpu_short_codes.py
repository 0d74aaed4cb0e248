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
    assert np.abs(lse.cpu().numpy().reshape(want["lse"].shape) - want["lse"]).max() < 2e-2
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
