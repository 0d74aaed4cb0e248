"""Heads of 64 channels through KVQ_KERNEL_AUTO (the tcgen05 kernel with 64-channel tiles): edges of the query and key
tiles, split and whole units, every format, ring windows, rotated values, both corrections, against the oracle; and the
warp-level kernel where a call brings no workspace."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import kvq_oracle as O
from paper_2605_26266_b200 import inputs
from tests import kvq_testlib as T

pytestmark = pytest.mark.gpu

CASES = [
    # bits, group, batch, heads, rows, current keys, cached keys, options
    (2, 32, 1, 2, 1, 1, 1, {}),
    (2, 64, 2, 1, 128, 128, 128, dict(signs=True)),
    (4, 32, 1, 3, 129, 63, 127, dict(rotate_v=True)),
    (4, 64, 1, 2, 256, 129, 0, {}),
    (2, 64, 1, 1, 257, 64, 1000, dict(ring=True)),
    (4, 32, 2, 2, 300, 300, 2049, dict(ring=True, rotate_v=True)),
    (2, 32, 1, 2, 17, 16, 5000, dict(signs=True)),
    (2, 64, 1, 2, 256, 256, 1024, dict(rotate=False)),
    (2, 64, 2, 80, 65, 20, 130, {}),                       # more units than SMs
]


def problem(B, case, seed):
    bits, group, batch, heads, m, n_cur, n, opt = case
    d, cap, begin = 64, (n // 128 + 1) * 128, 16
    w = inputs.Workload("head64", 700 + seed, batch, heads, d, 32, 0, bits, group, seed, k_outliers=2, k_outlier_scale=4.0, head_scale=True)
    signs = np.random.default_rng(seed).choice([-1, 1], size=d).astype(np.int8) if opt.get("signs") else None
    kw = dict(rotate_k=opt.get("rotate", True), signs=signs, ring=opt.get("ring", False), rotate_v=opt.get("rotate_v", False))
    if not kw["ring"]:
        cap += 128
    g, o = B.Cache(batch, heads, d, bits, group, cap, **kw), O.Cache(batch, heads, d, bits, group, cap, **kw)
    if kw["ring"]:
        begin = cap - 48                                       # the window wraps
    if n:
        _, k, v = inputs.make_chunk(w, 0, tokens=n)
        B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v), cache_len=begin)
        O.quantize_append(o, begin, k, v)
    q, _, _ = inputs.make_chunk(w, 1, tokens=m)
    _, kc, vc = inputs.make_chunk(w, 2, tokens=n_cur)
    return g, o, begin, n, q, kc, vc


@pytest.mark.parametrize("correction", [True, False])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(x) for x in c[:7]))
def test_head64_matches_the_oracle(case, correction):
    from paper_2605_26266_b200 import binding as B
    g, o, begin, n, q, kc, vc = problem(B, case, CASES.index(case))
    sigma = T.sigma_of(64) * 1.25
    want = O.attn_corrected(o, begin, n, q, kc, vc, sigma, correction=correction)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    lse = torch.zeros(q.shape[:3], dtype=torch.float32, device="cuda")
    mass = torch.full_like(lse, -1.0)
    out = B.kvq_attn_corrected(g, T.to_dev(q), T.to_dev(kc), T.to_dev(vc), sigma, B.KVQ_CORRECTION_ON if correction else B.KVQ_CORRECTION_OFF,
                               cache_begin=begin, cache_len=n, lse=lse, cached_mass=mass, status_word=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    T.assert_attn_close(T.from_dev_bf16(out).reshape(want["out"].shape), want["out"])
    assert np.abs(lse.cpu().numpy().reshape(want["lse"].shape) - want["lse"]).max() < 2e-2
    assert np.abs(mass.cpu().numpy().reshape(want["cached_mass"].shape) - want["cached_mass"]).max() < 1e-2


def test_head64_without_workspace_runs_the_warp_level_kernel():
    from paper_2605_26266_b200 import binding as B
    g, _, begin, n, q, kc, vc = problem(B, CASES[7], 7)
    q, kc, vc = T.to_dev(q), T.to_dev(kc), T.to_dev(vc)
    sigma, m, n_cur = T.sigma_of(64), q.shape[2], kc.shape[2]
    assert B.kvq_attn_workspace_bytes(g, n, m, n_cur, B.KVQ_CORRECTION_ON) > 0
    want = B.kvq_attn_corrected(g, q, kc, vc, sigma, B.KVQ_CORRECTION_ON | B.KVQ_KERNEL_MMA_SYNC, cache_begin=begin, cache_len=n)
    out = torch.empty_like(q)
    st = B._strides
    r = B.lib.kvq_attn_corrected(C.byref(g.desc), begin, n, q.data_ptr(), st(q), kc.data_ptr(), vc.data_ptr(), st(kc), m, n_cur,
                                 out.data_ptr(), st(out), sigma, B.KVQ_CORRECTION_ON, None, None, None, 0, None, B._stream())
    torch.cuda.synchronize()
    assert r == B.KVQ_OK and torch.equal(out.view(torch.int16), want.view(torch.int16))
    for forced in (B.KVQ_KERNEL_TCGEN05, B.KVQ_KERNEL_TCGEN05_PAIR):
        with pytest.raises(B.KvqError) as e:
            B.kvq_attn_corrected(g, q, kc, vc, sigma, forced, cache_begin=begin, cache_len=n)
        assert e.value.status == B.KVQ_ERR_UNSUPPORTED


@pytest.mark.parametrize("m", [16, 256])
def test_head64_calls_on_several_streams_share_nothing(m):
    """Attention calls that only read one cache, on two streams at once: each stream has its workspace, results are those of
    calls one after the other.  More streams than buffers are kept; a captured call keeps none."""
    from paper_2605_26266_b200 import binding as B
    w = inputs.Workload("streams", 760 + m, 1, 8, 64, 32, 0, 2, 64, 1)
    g = B.Cache(1, 8, 64, 2, 64, 4096)
    _, k, v = inputs.make_chunk(w, 0, tokens=4000)
    B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v))
    chunks = [[T.to_dev(x) for x in inputs.make_chunk(w, 1 + i, tokens=m)] for i in range(2)]
    want = [B.kvq_attn_corrected(g, *c, T.sigma_of(64)) for c in chunks]
    assert g.workspace is None
    torch.cuda.synchronize()
    streams, got = [torch.cuda.Stream() for _ in chunks], [[], []]
    for _ in range(50):
        for i, c in enumerate(chunks):
            with torch.cuda.stream(streams[i]):
                got[i].append(B.kvq_attn_corrected(g, *c, T.sigma_of(64)))
    torch.cuda.synchronize()
    for i in range(2):
        assert all(torch.equal(o.view(torch.int16), want[i].view(torch.int16)) for o in got[i])
    kept = g._stream_workspaces
    assert len({w.data_ptr() for w in kept.values()}) == len(kept) == 3
    more = [torch.cuda.Stream() for _ in range(12)]
    for st in more:
        with torch.cuda.stream(st):
            got[0].append(B.kvq_attn_corrected(g, *chunks[0], T.sigma_of(64)))
    before = list(kept)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=more[-1]):
        got[1].append(B.kvq_attn_corrected(g, *chunks[1], T.sigma_of(64)))
    graph.replay()
    torch.cuda.synchronize()
    assert len(kept) == 8 and list(kept) == before
    for i in range(2):
        assert torch.equal(got[i][-1].view(torch.int16), want[i].view(torch.int16))


@pytest.mark.parametrize("m", [16, 200])
def test_head64_token_interleaved(m):
    """[batch, tokens, heads, head_dim] storage of inputs and output."""
    from paper_2605_26266_b200 import binding as B
    w = inputs.Workload("inter", 770 + m, 2, 3, 64, 32, 0, 2, 32, 1)
    g, o = (X.Cache(2, 3, 64, 2, 32, 1024) for X in (B, O))
    _, k, v = inputs.make_chunk(w, 0, tokens=900)
    B.kvq_quantize_append(g, *(T.to_dev(x).permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for x in (k, v)))
    O.quantize_append(o, 0, k, v)
    T.assert_cache_equal(T.gpu_cache_arrays(g, 900), o, 900)
    q, k, v = inputs.make_chunk(w, 1, tokens=m)
    qd, kd, vd = (T.to_dev(x).permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for x in (q, k, v))
    out = torch.empty_like(qd)
    assert not out.is_contiguous()
    B.kvq_attn_corrected(g, qd, kd, vd, T.sigma_of(64), out=out)
    want = O.attn_corrected(o, 0, 900, q, k, v, T.sigma_of(64), correction=True)["out"]
    T.assert_attn_close(T.from_dev_bf16(out).reshape(want.shape), want)
