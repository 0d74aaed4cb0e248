"""128 channels, few units of few tiles: split with FP32 partial rows, by both tcgen05 kernels, all units and a last round of them; against the
oracle and no further from it than the same call without room for them, whose units are not split, from workspaces full of NaN and of
another call's rows."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import kvq_oracle as O
from paper_2605_26266_b200 import inputs
from tests import kvq_testlib as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel,heads,m,n_cur,n,ctas", [
    ("KVQ_KERNEL_TCGEN05", 16, 700, 700, 700, 144),        # 48 units of 12 tiles, four tiles a CTA
    ("KVQ_KERNEL_TCGEN05", 30, 256, 129, 1000, 75),        # 30 of 10
    ("KVQ_KERNEL_TCGEN05", 180, 100, 100, 1020, 148),      # 32 of 9 behind a round of 148, one query tile
    ("KVQ_KERNEL_TCGEN05", 40, 64, 64, 1400, 120),         # 40 of 12: a chunk of few rows like any other
    ("KVQ_KERNEL_TCGEN05_PAIR", 32, 300, 512, 1279, 148),  # 32 of 14 on 74 pairs
    ("KVQ_KERNEL_TCGEN05_PAIR", 100, 513, 300, 600, 148),  # 52 of 8 behind two rounds: not split, the pair's line is higher
    ("KVQ_KERNEL_TCGEN05_PAIR", 100, 200, 300, 900, 148),  # 26 of 11 behind a round of 74
])
def test_fp32_parts(kernel, heads, m, n_cur, n, ctas):
    from paper_2605_26266_b200 import binding as B
    picked = [heads - 16, heads - 13, heads - 7, heads - 1]      # of units that are split
    w = inputs.Workload("wide", 1950 + heads + m, 1, heads, 128, 32, 0, 2, 64, 1, head_scale=True)
    g, o = B.Cache(1, heads, 128, 2, 64, 1408), O.Cache(1, len(picked), 128, 2, 64, 1408)
    _, k, v = inputs.make_chunk(w, 0, tokens=n)
    B.kvq_quantize_append(g, T.to_dev(k), T.to_dev(v))
    O.quantize_append(o, 0, k[:, picked], v[:, picked])
    q, _, _ = inputs.make_chunk(w, 1, tokens=m)
    _, kc, vc = inputs.make_chunk(w, 2, tokens=n_cur)
    flags, sigma = B.KVQ_CORRECTION_ON | getattr(B, kernel), T.sigma_of(128)
    need = B.kvq_attn_workspace_bytes(g, n, m, n_cur, flags)
    rotated = -(-heads * m * 272 // 256) * 256
    if torch.cuda.get_device_properties(0).multi_processor_count == 148 and m != 513:
        assert need - rotated == ctas * 2 * (256 * 128 * 4 + 3 * 256 * 4)
    want = O.attn_corrected(o, 0, n, q[:, picked], kc[:, picked], vc[:, picked], sigma, correction=True)
    args = (g, T.to_dev(q), T.to_dev(kc), T.to_dev(vc), sigma, flags)
    g.workspace = torch.empty(max(need, 16), dtype=torch.uint8, device="cuda")
    dq, dk, dv, st = *args[1:4], B._strides
    whole = torch.empty_like(dq)
    assert B.lib.kvq_attn_corrected(C.byref(g.desc), 0, n, dq.data_ptr(), st(dq), dk.data_ptr(), dv.data_ptr(), st(dk), m, n_cur, whole.data_ptr(), st(whole),
                                    sigma, flags, None, None, g.workspace.data_ptr(), rotated, None, B._stream()) == B.KVQ_OK
    error = lambda x: np.linalg.norm(T.from_dev_bf16(x)[0][picked] - want["out"]) / np.linalg.norm(want["out"])
    first = None
    for fill in (0xFF, 0x3F):
        g.workspace.fill_(fill)
        lse = torch.empty(1, heads, m, dtype=torch.float32, device="cuda")
        mass = torch.empty_like(lse)
        out = B.kvq_attn_corrected(*args, lse=lse, cached_mass=mass)
        got = T.from_dev_bf16(out)[0][picked]
        T.assert_attn_close(got, want["out"], f"fill {fill:#x}")
        # A split by itself lowers the error by 1 to 4 % (each part's largest weight is exact).  Rows rounded to BF16, 2^-9 / sqrt(3) of a value at most,
        # would add some 1e-3 in quadrature to 2.3e-3
        assert error(out) <= 1.01 * error(whole)
        assert np.abs(lse.cpu().numpy()[0][picked] - want["lse"].reshape(len(picked), -1)).max() < 2e-2
        assert np.abs(mass.cpu().numpy()[0][picked] - want["cached_mass"].reshape(len(picked), -1)).max() < 1e-2
        first = out if first is None else first
        assert torch.equal(out.view(torch.int16), first.view(torch.int16))


def test_a_workspace_without_room_for_them():
    """A call may bring what was asked for before there were FP32 partial rows, the rotated queries' room: the units are not split then, and
    nothing behind the workspace is touched."""
    from paper_2605_26266_b200 import binding as B
    heads, m, n = 16, 700, 700
    w = inputs.Workload("room", 1990, 1, heads, 128, 32, 0, 2, 64, 1)
    g = B.Cache(1, heads, 128, 2, 64, 768)
    _, k, v = (T.to_dev(x) for x in inputs.make_chunk(w, 0, tokens=n))
    B.kvq_quantize_append(g, k, v)
    q, kc, vc = (T.to_dev(x) for x in inputs.make_chunk(w, 1, tokens=m))
    flags, rotated, st = B.KVQ_CORRECTION_ON | B.KVQ_KERNEL_TCGEN05, heads * m * 272 // 256 * 256, B._strides
    assert rotated == heads * m * 272
    want = B.kvq_attn_corrected(g, q, kc, vc, T.sigma_of(128), flags)
    room, out = torch.full((rotated + 4096,), 0xAB, dtype=torch.uint8, device="cuda"), torch.empty_like(q)
    call = lambda size: B.lib.kvq_attn_corrected(C.byref(g.desc), 0, n, q.data_ptr(), st(q), kc.data_ptr(), vc.data_ptr(), st(kc), m, m, out.data_ptr(), st(out),
                                                 T.sigma_of(128), flags, None, None, room.data_ptr(), size, None, B._stream())
    assert call(rotated - 1) == B.KVQ_ERR_WORKSPACE
    assert call(rotated) == B.KVQ_OK
    torch.cuda.synchronize()
    assert (room[rotated:] == 0xAB).all()
    T.assert_attn_close(T.from_dev_bf16(out), T.from_dev_bf16(want))


@pytest.mark.parametrize("kernel,heads,m,n_cur,n", [
    ("KVQ_KERNEL_TCGEN05", 180, 100, 100, 1020),           # ranges of one and two tiles: a unit's last cached tile, then the next one's only current one
    ("KVQ_KERNEL_TCGEN05", 181, 200, 60, 1100),
    ("KVQ_KERNEL_TCGEN05_PAIR", 100, 300, 100, 1200),
])
def test_short_ranges_again_and_again(kernel, heads, m, n_cur, n):
    """A range may end one unit and begin another with a tile each: the bias rows of the one are all there before its scores are computed,
    whichever of the expanding warps is ahead."""
    from paper_2605_26266_b200 import binding as B
    w = inputs.Workload("again", 1960 + heads + m, 1, heads, 128, 32, 0, 2, 64, 1, head_scale=True)
    g = B.Cache(1, heads, 128, 2, 64, 1280)
    _, k, v = (T.to_dev(x) for x in inputs.make_chunk(w, 0, tokens=n))
    B.kvq_quantize_append(g, k, v)
    q = T.to_dev(inputs.make_chunk(w, 1, tokens=m)[0])
    kc, vc = (T.to_dev(x) for x in inputs.make_chunk(w, 2, tokens=n_cur)[1:])
    flags = B.KVQ_CORRECTION_ON | getattr(B, kernel)
    want, out = B.kvq_attn_corrected(g, q, kc, vc, T.sigma_of(128), flags), torch.empty_like(q)
    differ = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(1000):
        B.kvq_attn_corrected(g, q, kc, vc, T.sigma_of(128), flags, out=out)
        differ += (out.view(torch.int16) != want.view(torch.int16)).any()
    assert differ.item() == 0
