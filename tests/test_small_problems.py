"""Small problems of any number of rows on the few-row kernel: where KVQ_KERNEL_AUTO draws the line (host-side size query, no
GPU needed; on a machine without one it plans for 148 SMs), and results on either side of it against the oracle."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import kvq_oracle as O
from paper_2605_26266_b200 import inputs
from tests import kvq_testlib as T


@pytest.fixture(scope="module")
def B():
    from paper_2605_26266_b200 import build
    build.build_library()
    from paper_2605_26266_b200 import binding
    return binding


def workspace(B, d, heads, m, n, flags=1):
    desc, size = B.kvq_cache_desc(1, heads, d, 2, 64, B.KVQ_ROTATE_K, 65536), C.c_size_t(0)
    assert B.lib.kvq_attn_workspace_bytes(C.byref(desc), n, m, m, flags, C.byref(size)) == B.KVQ_OK
    return size.value


def partial_rows(d, heads, m, n):
    """Bytes of the few-row kernel's partial rows: 16 rows and 64 statistics a CTA, as many splits as let all CTAs run at once."""
    units, steps = heads * -(-m // 16), -(-n // 32) + -(-m // 32)
    splits = max(1, min(296 // units, steps // 8, 128))
    return 0 if splits == 1 else -(-units * splits * (16 * d + 64) * 4 // 256) * 256


@pytest.mark.parametrize("d,heads,m,n,few", [
    (64, 2, 256, 1024, True), (64, 1, 1024, 2048, True), (64, 16, 512, 0, True), (64, 27, 256, 0, True),
    (64, 64, 96, 512, True), (64, 32, 128, 896, True), (64, 32, 128, 897, False),      # 8 192 steps, and one more for each unit
    (64, 74, 96, 0, True), (64, 75, 96, 64, False),                                    # 444 CTAs
    (128, 2, 128, 4096, True), (128, 32, 96, 672, True), (128, 32, 96, 673, False),    # 4 608 steps
    (128, 37, 128, 0, True), (128, 38, 128, 128, False),                               # 296 CTAs
    (128, 2, 129, 4096, False),                                                        # a second query tile of the other kernel
])
def test_where_the_line_lies(B, d, heads, m, n, few):
    assert (workspace(B, d, heads, m, n) == partial_rows(d, heads, m, n)) == few


@pytest.mark.gpu
@pytest.mark.parametrize("heads,m,n_cur", [(150, 100, 5), (172, 111, 64), (149, 33, 1)])
def test_units_of_a_single_tile_match_the_oracle(B, heads, m, n_cur):
    """64 channels, more heads than processors, at most 128 rows and 64 current keys, no cache: on the few-row kernel whatever its number of CTAs."""
    w = inputs.Workload("single", 1500 + m, 1, heads, 64, 32, 0, 2, 64, m, head_scale=True)
    g, o = B.Cache(1, heads, 64, 2, 64, 128), O.Cache(1, heads, 64, 2, 64, 128)
    q, _, _ = inputs.make_chunk(w, 1, tokens=m)
    _, kc, vc = inputs.make_chunk(w, 2, tokens=n_cur)
    lse = torch.zeros(1, heads, m, dtype=torch.float32, device="cuda")
    out = B.kvq_attn_corrected(g, T.to_dev(q), T.to_dev(kc), T.to_dev(vc), T.sigma_of(64), cache_len=0, lse=lse)
    want = O.attn_corrected(o, 0, 0, q, kc, vc, T.sigma_of(64), correction=True)
    T.assert_attn_close(T.from_dev_bf16(out).reshape(want["out"].shape), want["out"])
    assert np.abs(lse.cpu().numpy().reshape(want["lse"].shape) - want["lse"]).max() < 2e-2


@pytest.mark.parametrize("d,heads,m,n,launches", [
    (64, 2, 256, 1024, 1), (64, 2, 16, 2032, 1), (64, 1, 16, 2300, 2),                 # 5 and 8 splits; 9
    (128, 2, 16, 1520, 1), (128, 2, 16, 1800, 2), (128, 3, 16, 100, 1),                # 6 splits; 7; 1
    (128, 22, 16, 2032, 2), (64, 44, 16, 1000, 1), (64, 45, 16, 1000, 2),              # 176 CTAs of 4 splits, 180
])
def test_clusters_merge_without_a_second_launch(B, d, heads, m, n, launches):
    desc, count = B.kvq_cache_desc(1, heads, d, 2, 64, B.KVQ_ROTATE_K, 65536), C.c_int(0)
    assert B.lib.kvq_attn_kernel_launches(C.byref(desc), n, m, m, 1, C.byref(count)) == B.KVQ_OK
    assert count.value == launches and workspace(B, d, heads, m, n) == partial_rows(d, heads, m, n)


# d, bits, group, heads, rows, current keys, cached keys
CASES = [(128, 2, 32, 2, 65, 1, 129), (128, 4, 64, 3, 100, 33, 1000), (128, 2, 128, 2, 128, 128, 31), (128, 4, 128, 1, 127, 64, 4001),
         (64, 2, 64, 3, 1000, 40, 300), (64, 4, 32, 60, 97, 31, 65), (64, 2, 32, 1, 513, 700, 0)]


@pytest.mark.gpu
@pytest.mark.parametrize("d,bits,group,heads,m,n_cur,n", CASES)
def test_small_problems_match_the_oracle(B, d, bits, group, heads, m, n_cur, n):
    w = inputs.Workload("small", 1300 + m, 1, heads, d, 32, 0, bits, group, m, k_outliers=2, k_outlier_scale=4.0, head_scale=True)
    g, o = B.Cache(1, heads, d, bits, group, 4224), O.Cache(1, heads, d, bits, group, 4224)
    if n:
        _, k, v = inputs.make_chunk(w, 0, tokens=n)
        B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v))
        O.quantize_append(o, 0, k, v)
    q, _, _ = inputs.make_chunk(w, 1, tokens=m)
    _, kc, vc = inputs.make_chunk(w, 2, tokens=n_cur)
    sigma = T.sigma_of(d)
    lse = torch.zeros(1, heads, m, dtype=torch.float32, device="cuda")
    mass = torch.full_like(lse, -1.0)
    out = B.kvq_attn_corrected(g, T.to_dev(q), T.to_dev(kc), T.to_dev(vc), sigma, cache_len=n, lse=lse, cached_mass=mass)
    want = O.attn_corrected(o, 0, n, q, kc, vc, sigma, correction=True)
    T.assert_attn_close(T.from_dev_bf16(out).reshape(want["out"].shape), want["out"])
    assert np.abs(lse.cpu().numpy().reshape(want["lse"].shape) - want["lse"]).max() < 2e-2
    assert np.abs(mass.cpu().numpy().reshape(want["cached_mass"].shape) - want["cached_mass"]).max() < 1e-2
