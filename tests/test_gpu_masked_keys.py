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
