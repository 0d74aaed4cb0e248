"""The tcgen05 kernel for heads of 64 channels, which KVQ_KERNEL_AUTO takes for problems of more than a few thousand steps: enough
heads that every shape below runs on it, rows and keys at the edges of its tiles, whole and split units, against the oracle on three
of the heads.  Weights travel as two BF16 parts, so what is left of the error is the rounding of the output, which the test takes from the
oracle's own result, and the FP16 rounding of the rotated query (a few per cent of it); with weights in one BF16 part it is 1.2
times that rounding.  Values far from zero are rounded to BF16 themselves: as much again, at most, where a row has one key."""
import numpy as np
import pytest
import torch

from oracle import kvq_oracle as O
from paper_2605_26266_b200 import inputs
from tests import kvq_testlib as T

pytestmark = pytest.mark.gpu

# heads, rows, current keys, cached keys, bits, group, runs of 16 cached tokens, of six, whose values lie far from zero
CASES = [(150, 65, 1, 129, 2, 64, 0), (150, 128, 64, 127, 4, 32, 0), (90, 129, 65, 300, 2, 32, 0), (90, 256, 128, 64, 4, 64, 0), (60, 257, 63, 0, 2, 64, 0),
         (40, 300, 300, 1500, 2, 64, 0), (150, 65, 1, 129, 2, 64, 1), (90, 129, 65, 300, 4, 32, 1), (40, 300, 300, 1500, 2, 32, 3)]


@pytest.mark.parametrize("correction", [True, False])
@pytest.mark.parametrize("heads,m,n_cur,n,bits,group,far", CASES)
def test_units_of_64_channels(heads, m, n_cur, n, bits, group, far, correction):
    from paper_2605_26266_b200 import binding as B
    picked = [0, heads // 2, heads - 1]
    w = inputs.Workload("units64", 1200 + m, 1, heads, 64, 32, 0, bits, group, m, head_scale=True)
    g, o = B.Cache(1, heads, 64, bits, group, 2048), O.Cache(1, len(picked), 64, bits, group, 2048)
    if n:
        _, k, v = inputs.make_chunk(w, 0, tokens=n)
        shift = np.where(np.arange(n) // 16 % 6 < far, np.float32(40.0), np.float32(0))[None, None, :, None]
        v = inputs.f32_to_bf16_bits(O.bf16_bits_to_f64(v).astype(np.float32) + shift)
        B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v))
        O.quantize_append(o, 0, k[:, picked], v[:, picked])
    q, _, _ = inputs.make_chunk(w, 1, tokens=m)
    _, kc, vc = inputs.make_chunk(w, 2, tokens=n_cur)
    sigma, flags = T.sigma_of(64), B.KVQ_CORRECTION_ON if correction else B.KVQ_CORRECTION_OFF
    steps = -(-n // 32) + -(-n_cur // 32)
    assert heads * -(-m // 16) * steps > 8192 or heads * -(-m // 16) > 444          # beyond the few-row kernel
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    lse = torch.zeros(1, heads, m, dtype=torch.float32, device="cuda")
    mass = torch.full_like(lse, -1.0)
    out = B.kvq_attn_corrected(g, T.to_dev(q), T.to_dev(kc), T.to_dev(vc), sigma, flags, cache_len=n, lse=lse, cached_mass=mass, status_word=status)
    want = O.attn_corrected(o, 0, n, q[:, picked], kc[:, picked], vc[:, picked], sigma, correction=correction)
    assert int(status.item()) == 0
    got = T.from_dev_bf16(out)[:, picked]
    if not far:                                       # half a unit in the last place of an output of 40 is 0.125
        T.assert_attn_close(got, want["out"].reshape(got.shape))
    exact = want["out"].reshape(got.shape)
    rounded = torch.from_numpy(exact).to(torch.bfloat16).double().numpy()
    assert T.attn_errors(got, exact)[0] < 1.12 * (2.0 ** 0.5 if far else 1.0) * T.attn_errors(rounded, exact)[0]
    assert np.abs(lse.cpu().numpy()[:, picked] - want["lse"].reshape(1, 3, m)).max() < 2e-2
    assert np.abs(mass.cpu().numpy()[:, picked] - want["cached_mass"].reshape(1, 3, m)).max() < 1e-2
