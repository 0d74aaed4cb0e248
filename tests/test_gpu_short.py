"""Chunks of a few query rows (the kernel KVQ_KERNEL_AUTO takes for them): edges of its row blocks and key steps, splits that
leave a single step or end in the current chunk, every format, ring windows that wrap inside a step, rotated values, shared
(stride 0) and token-interleaved chunks, against the oracle; and the kernels that served such calls before where the
workspace is sized for them, or missing."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import kvq_oracle as O
from paper_2605_26266_b200 import inputs
from tests import kvq_testlib as T

pytestmark = pytest.mark.gpu

CASES = [
    # head_dim, bits, group, batch, heads, rows, current keys, cached keys, options
    (128, 2, 32, 1, 2, 1, 1, 1, {}),
    (128, 2, 64, 2, 1, 16, 16, 0, {}),
    (128, 4, 128, 1, 3, 16, 33, 31, dict(signs=True)),
    (128, 4, 32, 1, 2, 17, 17, 1000, dict(ring=True)),
    (128, 4, 64, 2, 2, 31, 300, 513, dict(rotate_v=True)),
    (128, 2, 128, 1, 1, 33, 1, 4097, dict(ring=True, rotate=False)),
    (128, 2, 128, 1, 2, 64, 64, 2000, {}),
    (64, 2, 32, 1, 2, 2, 15, 65, dict(signs=True, ring=True)),
    (64, 2, 64, 2, 3, 16, 1, 1999, {}),
    (64, 4, 32, 1, 1, 15, 700, 0, {}),
    (64, 4, 64, 1, 2, 48, 48, 1025, dict(rotate_v=True, ring=True)),
    (128, 2, 64, 1, 160, 5, 5, 300, {}),                   # more units than CTAs: nothing is split
]


def problem(B, case, seed):
    d, bits, group, batch, heads, m, n_cur, n, opt = case
    cap, begin = (n // 128 + 1) * 128, 16
    w = inputs.Workload("short", 800 + seed, batch, heads, d, 32, 0, bits, group, seed, k_outliers=2, k_outlier_scale=4.0, head_scale=True)
    signs = np.random.default_rng(seed).choice([-1, 1], size=d).astype(np.int8) if opt.get("signs") else None
    kw = dict(rotate_k=opt.get("rotate", True), signs=signs, ring=opt.get("ring", False), rotate_v=opt.get("rotate_v", False))
    if kw["ring"]:
        begin = cap - 48                                       # the window wraps after 48 tokens, inside a step of 32
    else:
        cap += 128
    g, o = B.Cache(batch, heads, d, bits, group, cap, **kw), O.Cache(batch, heads, d, bits, group, cap, **kw)
    for t in g.buffers:
        t.fill_(0x7F)                                          # tokens past the window hold NaN steps
    if n:
        _, k, v = inputs.make_chunk(w, 0, tokens=n)
        B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v), cache_len=begin)
        O.quantize_append(o, begin, k, v)
    q, _, _ = inputs.make_chunk(w, 1, tokens=m)
    _, kc, vc = inputs.make_chunk(w, 2, tokens=n_cur)
    return g, o, begin, n, q, kc, vc


@pytest.mark.parametrize("correction", [True, False])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(x) for x in c[:8]))
def test_short_chunks_match_the_oracle(case, correction):
    from paper_2605_26266_b200 import binding as B
    d = case[0]
    g, o, begin, n, q, kc, vc = problem(B, case, CASES.index(case))
    sigma = T.sigma_of(d) * 1.25
    want = O.attn_corrected(o, begin, n, q, kc, vc, sigma, correction=correction)
    flags = B.KVQ_CORRECTION_ON if correction else B.KVQ_CORRECTION_OFF
    rotv = 2 if g.desc.flags & B.KVQ_ROTATE_V and n else 0
    assert B.kvq_attn_kernel_launches(g, n, q.shape[2], kc.shape[2], flags) - rotv in (1, 2)   # no query pre-pass
    lse = torch.zeros(q.shape[:3], dtype=torch.float32, device="cuda")
    mass = torch.full_like(lse, -1.0)
    out = B.kvq_attn_corrected(g, T.to_dev(q), T.to_dev(kc), T.to_dev(vc), sigma, flags, cache_begin=begin, cache_len=n, lse=lse, cached_mass=mass)
    torch.cuda.synchronize()
    T.assert_attn_close(T.from_dev_bf16(out).reshape(want["out"].shape), want["out"])
    assert np.abs(lse.cpu().numpy().reshape(want["lse"].shape) - want["lse"]).max() < 2e-2
    assert np.abs(mass.cpu().numpy().reshape(want["cached_mass"].shape) - want["cached_mass"]).max() < 1e-2


def test_short_chunk_with_a_smaller_workspace_or_shared_heads():
    from paper_2605_26266_b200 import binding as B
    case = (128, 2, 64, 1, 2, 16, 16, 2000, {})
    g, o, begin, n, q, kc, vc = problem(B, case, 20)
    sigma, m, n_cur = T.sigma_of(128), 16, 16
    want = O.attn_corrected(o, begin, n, q, kc, vc, sigma)["out"]
    dq, dk, dv = T.to_dev(q), T.to_dev(kc), T.to_dev(vc)
    st, out = B._strides, torch.empty_like(dq)

    def call(flags, ws):
        return B.lib.kvq_attn_corrected(C.byref(g.desc), begin, n, dq.data_ptr(), st(dq), dk.data_ptr(), dv.data_ptr(), st(dk), m, n_cur,
                                        out.data_ptr(), st(out), sigma, flags, None, None, ws.data_ptr() if ws is not None else None,
                                        ws.numel() if ws is not None else 0, None, B._stream())

    need = B.kvq_attn_workspace_bytes(g, n, m, n_cur, B.KVQ_CORRECTION_ON)
    assert need > 0 and call(B.KVQ_CORRECTION_ON, None) == B.KVQ_ERR_WORKSPACE
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    assert call(B.KVQ_CORRECTION_ON, ws) == B.KVQ_OK
    T.assert_attn_close(T.from_dev_bf16(out).reshape(want.shape), want)
    # one chunk of keys and values for all heads (stride 0)
    shared_k, shared_v = (t[:, :1].expand(-1, 2, -1, -1) for t in (dk, dv))
    want = O.attn_corrected(o, begin, n, q, np.repeat(kc[:, :1], 2, 1), np.repeat(vc[:, :1], 2, 1), sigma)["out"]
    got = B.kvq_attn_corrected(g, dq, shared_k, shared_v, sigma, cache_begin=begin, cache_len=n)
    T.assert_attn_close(T.from_dev_bf16(got).reshape(want.shape), want)


@pytest.mark.parametrize("heads,n,opt", [(2, 1000, {}), (140, 2000, {}), (2, 1000, dict(rotate_v=True))])
def test_workspace_that_suits_only_the_former_kernel(heads, n, opt):
    """Few keys or many heads: the tcgen05 kernel needs less room than the splits of the few-row kernel.  A call that brings just
    that gets that kernel's bytes, and nothing behind the workspace is touched."""
    from paper_2605_26266_b200 import binding as B
    g, o, begin, n, q, kc, vc = problem(B, (128, 2, 64, 1, heads, 16, 16, n, opt), 21)
    sigma, flags = T.sigma_of(128), B.KVQ_CORRECTION_ON
    need, former = (B.kvq_attn_workspace_bytes(g, n, 16, 16, f) for f in (flags, flags | B.KVQ_KERNEL_TCGEN05))
    assert 0 < former < need
    dq, dk, dv = T.to_dev(q), T.to_dev(kc), T.to_dev(vc)
    want = B.kvq_attn_corrected(g, dq, dk, dv, sigma, flags | B.KVQ_KERNEL_TCGEN05, cache_begin=begin, cache_len=n)
    ws, out, st = torch.full((need,), 0xA5, dtype=torch.uint8, device="cuda"), torch.empty_like(dq), B._strides
    r = B.lib.kvq_attn_corrected(C.byref(g.desc), begin, n, dq.data_ptr(), st(dq), dk.data_ptr(), dv.data_ptr(), st(dk), 16, 16,
                                 out.data_ptr(), st(out), sigma, flags, None, None, ws.data_ptr(), former, None, B._stream())
    torch.cuda.synchronize()
    assert r == B.KVQ_OK and torch.equal(out.view(torch.int16), want.view(torch.int16)) and bool((ws[former:] == 0xA5).all())
    few = B.kvq_attn_corrected(g, dq, dk, dv, sigma, flags, cache_begin=begin, cache_len=n)
    assert not torch.equal(few.view(torch.int16), want.view(torch.int16))                  # another kernel, with the room it asks for
    if heads == 2:
        T.assert_attn_close(T.from_dev_bf16(few).reshape(1, 2, 16, 128), O.attn_corrected(o, begin, n, q, kc, vc, sigma)["out"].reshape(1, 2, 16, 128))


def test_64_channels_without_workspace_keep_the_warp_level_kernel():
    from paper_2605_26266_b200 import binding as B
    g, _, begin, n, q, kc, vc = problem(B, (64, 2, 64, 1, 2, 16, 16, 2000, {}), 22)
    dq, dk, dv = T.to_dev(q), T.to_dev(kc), T.to_dev(vc)
    sigma, st, out = T.sigma_of(64), B._strides, torch.empty_like(dq)
    want = B.kvq_attn_corrected(g, dq, dk, dv, sigma, B.KVQ_CORRECTION_ON | B.KVQ_KERNEL_MMA_SYNC, cache_begin=begin, cache_len=n)
    ws = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    for ptr, size in ((None, 0), (ws.data_ptr(), 256), (ws.data_ptr() + 16, 1 << 19)):       # none, too small, not aligned
        out.zero_()
        r = B.lib.kvq_attn_corrected(C.byref(g.desc), begin, n, dq.data_ptr(), st(dq), dk.data_ptr(), dv.data_ptr(), st(dk), 16, 16,
                                     out.data_ptr(), st(out), sigma, B.KVQ_CORRECTION_ON, None, None, ptr, size, None, B._stream())
        torch.cuda.synchronize()
        assert r == B.KVQ_OK and torch.equal(out.view(torch.int16), want.view(torch.int16))


def test_short_chunk_token_interleaved():
    from paper_2605_26266_b200 import binding as B
    g, o, begin, n, q, kc, vc = problem(B, (128, 4, 32, 2, 3, 20, 20, 700, dict(signs=True)), 23)
    qd, kd, vd = (T.to_dev(x).permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for x in (q, kc, vc))
    out = torch.empty_like(qd)
    assert not out.is_contiguous()
    B.kvq_attn_corrected(g, qd, kd, vd, T.sigma_of(128), cache_begin=begin, cache_len=n, out=out)
    want = O.attn_corrected(o, begin, n, q, kc, vc, T.sigma_of(128))["out"]
    T.assert_attn_close(T.from_dev_bf16(out).reshape(want.shape), want)
