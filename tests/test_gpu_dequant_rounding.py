"""Dequantized keys and values are (code - zero) * step rounded once (FP16 keys, saturated there; BF16 values), also for
groups far from zero, whose zero-points lie far outside the code range.  One cached token carries the whole weight of every
row: the output is then its dequantized value, and the log-sum-exp of a row whose query is a unit vector one channel of its
dequantized key.  The kernels for heads of 64 channels, and the one for few rows where it takes a chunk shared by all heads."""
import numpy as np
import pytest
import torch

from oracle import kvq_oracle as O
from paper_2605_26266_b200 import inputs
from tests import kvq_testlib as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mean", [0.0, 12.0, -30.0, 80.0, 3000.0, 65300.0])
@pytest.mark.parametrize("d,bits,group,m", [(64, 2, 32, 129), (64, 4, 32, 300), (64, 4, 64, 129), (64, 2, 64, 16), (64, 4, 32, 16),
                                            (128, 2, 32, 16), (128, 4, 64, 16), (128, 2, 128, 16)])
def test_one_rounding(d, bits, group, m, mean):
    from paper_2605_26266_b200 import binding as B
    batch, heads = 2, 24
    r = np.random.default_rng(int(abs(mean)) + d + bits + group)
    shape = (batch, heads, 1, d)
    # every other group of a token sits at the mean, so that exact and inexact ones meet in a warp
    shift = np.where((np.arange(d) // 32 + np.arange(heads)[:, None]) % 2, np.float32(mean), np.float32(0))[None, :, None, :]
    k, v = (inputs.f32_to_bf16_bits(r.standard_normal(shape, dtype=np.float32) + shift) for _ in range(2))
    g, o = B.Cache(batch, heads, d, bits, group, 128, rotate_k=False), O.Cache(batch, heads, d, bits, group, 128, rotate_k=False)
    B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v))
    O.quantize_append(o, 0, k, v)

    def hat(which):
        code, byte, zero = (getattr(o, which + s)[:, :, 0] for s in ("_codes", "_scale", "_zero"))
        x = O.unpack_codes(code, bits).reshape(batch, heads, d // group, group).astype(np.float64)
        return ((x - O.bf16_bits_to_f64(zero)[..., None]) * O.e4m3_decode(byte)[..., None]).reshape(batch, heads, d)

    want_k = np.clip(hat("k"), -65504.0, 65504.0).astype(np.float16).astype(np.float64)
    want_v = inputs.f32_to_bf16_bits(hat("v").astype(np.float32))        # up to 24 significant bits: exact in float32
    kc = torch.full((batch, heads, 1, d), -1000.0, dtype=torch.bfloat16, device="cuda")      # weight 2^-1300
    vc = torch.ones_like(kc)
    if d == 128:
        kc, vc = (t[:, :1].expand(-1, heads, -1, -1) for t in (kc, vc))                       # no tensor map can address it
    for first in range(0, d, m):
        channels = (first + np.arange(m)) % d
        q = np.zeros((batch, heads, m, d), dtype=np.float32)
        q[:, :, np.arange(m), channels] = 1.0
        lse = torch.empty(batch, heads, m, dtype=torch.float32, device="cuda")
        out = B.kvq_attn_corrected(g, T.to_dev(inputs.f32_to_bf16_bits(q)), kc, vc, 1.0, B.KVQ_CORRECTION_OFF, cache_len=1, lse=lse)
        got_v = out.view(torch.int16).cpu().numpy().view(np.uint16)
        bad = (got_v != want_v[:, :, None]) & ((got_v | want_v[:, :, None]) != 0x8000)       # either sign of zero
        assert not bad.any(), f"{bad.sum()} of {bad.size} values"
        s, got_s = want_k[:, :, channels], lse.cpu().numpy().astype(np.float64)
        # scale_log2, its product with the score and the one with ln 2: three roundings of 2^-24
        assert (np.abs(got_s - s) <= 4 * 2.0 ** -24 * np.abs(s) + 1e-30).all(), np.abs(got_s / np.where(s == 0, 1, s) - 1).max()


@pytest.mark.parametrize("d,bits,group,m", [(64, 2, 32, 16), (64, 4, 32, 30), (64, 4, 64, 200), (64, 2, 64, 300), (128, 4, 32, 16), (128, 2, 64, 16)])
def test_groups_far_from_zero_among_others(d, bits, group, m):
    """Only tokens from 40 on lie far from zero: a warp of the few-row kernel meets them after steps it has already summed."""
    from paper_2605_26266_b200 import binding as B
    heads, n, n_cur = 6, 700, 33
    r = np.random.default_rng(d + bits + group)
    far = (40.0 * (np.arange(n) >= 40)[:, None] * np.where(np.arange(heads) % 2, 1.0, -1.0)[:, None, None])[None].astype(np.float32)
    draw = lambda t, x=0: inputs.f32_to_bf16_bits((r.standard_normal((1, heads, t, d)) + x).astype(np.float32))
    g, o = (X.Cache(1, heads, d, bits, group, 768, rotate_k=False) for X in (B, O))
    k, v = draw(n, far), draw(n, far)
    B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v))
    O.quantize_append(o, 0, k, v)
    q, kc, vc = draw(m), draw(n_cur), draw(n_cur)
    dq, dk, dv = (T.to_dev(x) for x in (q, kc, vc))
    if d == 128:
        kc, vc = (np.repeat(x[:, :1], heads, 1) for x in (kc, vc))
        dk, dv = (x[:, :1].expand(-1, heads, -1, -1) for x in (dk, dv))
    lse = torch.empty(1, heads, m, dtype=torch.float32, device="cuda")
    mass = torch.empty_like(lse)
    sigma = 0.25 * T.sigma_of(d)
    out = B.kvq_attn_corrected(g, dq, dk, dv, sigma, B.KVQ_CORRECTION_ON, cache_len=n, lse=lse, cached_mass=mass)
    want = O.attn_corrected(o, 0, n, q, kc, vc, sigma, correction=True)
    rel, _ = T.attn_errors(T.from_dev_bf16(out).reshape(want["out"].shape), want["out"])
    assert rel <= T.REL_L2_TOL, rel
    # FP16 keys of magnitude 40: sigma |q| 40 2^-12 / sqrt(3) = 1.4e-3 a score
    assert np.abs(lse.cpu().numpy().reshape(want["lse"].shape) - want["lse"]).max() < 2e-2
    assert np.abs(mass.cpu().numpy().reshape(want["cached_mass"].shape) - want["cached_mass"]).max() < 1e-2


@pytest.mark.parametrize("d,bits,group,m", [(64, 2, 32, 300), (64, 4, 64, 129), (64, 2, 64, 16), (64, 4, 32, 16), (128, 4, 32, 16), (128, 2, 128, 16)])
def test_bias_keeps_32_bits(d, bits, group, m):
    """One cached key that is zero wherever the query is not, with a large step: a row's score is its bias alone."""
    from paper_2605_26266_b200 import binding as B
    heads = 24
    r = np.random.default_rng(d + bits + group + m)
    k = np.zeros((1, heads, 1, d), dtype=np.float32)
    top = 20.0 * (1 + np.arange(heads))[None, :, None, None]
    k[..., 0::group], k[..., 1::group] = top, -top
    q = r.uniform(1.0, 2.0, (1, heads, m, d)).astype(np.float32)
    q[..., 0::group] = q[..., 1::group] = 0.0
    k, q = inputs.f32_to_bf16_bits(k), inputs.f32_to_bf16_bits(q)
    g, o = (X.Cache(1, heads, d, bits, group, 128, rotate_k=False) for X in (B, O))
    B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(k))
    O.quantize_append(o, 0, k, k)
    kc = np.full((1, 1 if d == 128 else heads, 1, d), 0xC900, dtype=np.uint16)                # -2^19: no weight on the current key
    dk = T.to_dev(kc).expand(-1, heads, -1, -1)
    lse = torch.empty(1, heads, m, dtype=torch.float32, device="cuda")
    sigma = T.sigma_of(d)
    B.kvq_attn_corrected(g, T.to_dev(q), dk, dk, sigma, B.KVQ_CORRECTION_ON, cache_len=1, lse=lse)
    nu = (O.bf16_bits_to_f64(q) ** 2).reshape(1, heads, m, d // group, group).sum(-1)
    step = O.e4m3_decode(o.k_scale[:, :, 0])
    want = -(np.float64(np.float32(sigma)) ** 2 / 24.0) * (nu * step[:, :, None] ** 2).sum(-1)
    # about ten roundings of 2^-24 (the sum of squares, the coefficient, the products, the change of base); a bias of 16
    # significant bits is off by up to 2^-17
    err = np.abs(lse.cpu().numpy() / want - 1).max()
    assert err <= 2.0 ** -20, err
