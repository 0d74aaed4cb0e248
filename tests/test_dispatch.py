"""Which kernel KVQ_KERNEL_AUTO plans for chunks of a few rows, read from the host-side size and launch-count queries (no GPU
needed; on a machine without one they plan for 148 SMs)."""
import ctypes as C

import pytest


@pytest.fixture(scope="module")
def B():
    from paper_2605_26266_b200 import build
    build.build_library()
    from paper_2605_26266_b200 import binding
    return binding


def plan(B, d, batch, heads, m, n_cur, n, flags):
    desc = B.kvq_cache_desc(batch, heads, d, 2, 64, B.KVQ_ROTATE_K, 65536)
    size, count = C.c_size_t(0), C.c_int(0)
    assert B.lib.kvq_attn_workspace_bytes(C.byref(desc), n, m, n_cur, flags, C.byref(size)) == B.KVQ_OK
    assert B.lib.kvq_attn_kernel_launches(C.byref(desc), n, m, n_cur, flags, C.byref(count)) == B.KVQ_OK
    return size.value, count.value


@pytest.mark.parametrize("batch,heads,m,n,few", [
    (1, 32, 1, 16384, True), (1, 160, 16, 8192, True), (8, 128, 16, 2048, True),         # one block of rows: always
    (1, 32, 32, 8000, True), (1, 64, 17, 2048, True), (1, 64, 48, 2048, True), (1, 8, 64, 2048, True), (1, 64, 64, 512, True),
    # several blocks of many heads: more CTAs than run at once
    (1, 160, 17, 0, False), (1, 160, 32, 8192, False), (4, 128, 32, 128, False), (4, 80, 48, 0, False), (8, 128, 64, 128, False),
    # several blocks over long caches
    (1, 32, 32, 32768, False), (1, 32, 48, 8192, False), (1, 32, 64, 2048, False), (1, 8, 65, 0, False),
])
def test_few_rows_take_their_kernel_where_it_is_faster(B, batch, heads, m, n, few):
    auto = plan(B, 128, batch, heads, m, m, n, B.KVQ_CORRECTION_ON)
    # the tcgen05 kernel that serves them otherwise: with a cache it has a pre-pass and room for the rotated queries
    tcgen05 = plan(B, 128, batch, heads, m, m, n, B.KVQ_CORRECTION_ON | B.KVQ_KERNEL_TCGEN05)
    assert (auto != tcgen05) if few else (auto == tcgen05)


@pytest.mark.parametrize("d,flags,offset,size,status", [
    (128, 0, 16, 0, "KVQ_ERR_ALIGNMENT"), (128, 0, 128, 4096, "KVQ_ERR_ALIGNMENT"), (128, 0, 0, -1, "KVQ_ERR_WORKSPACE"),
    (128, 0, 16, -1, "KVQ_ERR_WORKSPACE"), (128, 4, 16, 0, "KVQ_ERR_ALIGNMENT"), (64, 4, 16, 0, "KVQ_ERR_ALIGNMENT"),
])
def test_workspace_errors_of_a_few_rows(B, d, flags, offset, size, status):
    """A workspace of the size asked for that is not 256-byte aligned is an alignment error, a smaller one a size error (`size`:
    bytes beyond what kvq_attn_workspace_bytes asks for).  Refused on the host: the pointers are never used."""
    m = n_cur = 16
    desc = B.kvq_cache_desc(1, 2, d, 2, 64, B.KVQ_ROTATE_K | flags, 4096, *([1 << 20] * 6))
    need = C.c_size_t(0)
    assert B.lib.kvq_attn_workspace_bytes(C.byref(desc), 2000, m, n_cur, B.KVQ_CORRECTION_ON, C.byref(need)) == B.KVQ_OK
    st = B.kvq_strides(2 * m * d, m * d, d)
    r = B.lib.kvq_attn_corrected(C.byref(desc), 0, 2000, 1 << 20, st, 1 << 20, 1 << 20, st, m, n_cur, 1 << 20, st, 0.1,
                                 B.KVQ_CORRECTION_ON, None, None, (1 << 20) + offset, need.value + size, None, None)
    assert r == getattr(B, status)


def test_64_channels_beyond_the_counts_of_the_tcgen05_kernel(B):
    """More than 2^31 tile steps: the warp-level kernel, without a workspace, as before 64 channels had another kernel."""
    assert plan(B, 64, 1, 64, 1 << 20, 1 << 20, 65536, B.KVQ_CORRECTION_ON) == (0, 1)
    assert plan(B, 64, 1, 64, 1 << 18, 1 << 18, 65536, B.KVQ_CORRECTION_ON)[0] > 0
    desc, size = B.kvq_cache_desc(1, 64, 64, 2, 64, B.KVQ_ROTATE_K, 65536), C.c_size_t(0)
    for m in (1 << 18, 1 << 20):
        assert B.lib.kvq_attn_workspace_bytes(C.byref(desc), 65536, m, m, B.KVQ_KERNEL_TCGEN05, C.byref(size)) == B.KVQ_ERR_UNSUPPORTED


@pytest.mark.parametrize("kernel,heads,m,tiles,split", [
    # 148 CTAs, 74 pairs; tiles: the chunk's and the cache's.  Few units: from six idle tile steps a CTA on, seven a pair, and two ranges of four
    ("TCGEN05", 32, 256, 7, False), ("TCGEN05", 32, 256, 8, True), ("TCGEN05", 14, 256, 7, False), ("TCGEN05", 74, 256, 12, False), ("TCGEN05", 74, 256, 13, True),
    ("TCGEN05_PAIR", 37, 512, 14, False), ("TCGEN05_PAIR", 37, 512, 15, True),
    # left over by a whole round: only with a tile step for every CTA, and a step later with many units
    ("TCGEN05", 150, 256, 8, False), ("TCGEN05", 150, 120, 10, False), ("TCGEN05", 158, 256, 10, False), ("TCGEN05", 164, 256, 9, False),
    ("TCGEN05", 162, 256, 10, False), ("TCGEN05", 162, 256, 11, True), ("TCGEN05", 166, 256, 9, True), ("TCGEN05", 180, 100, 9, True),
    ("TCGEN05", 205, 256, 10, False), ("TCGEN05", 190, 256, 9, True), ("TCGEN05", 222, 256, 13, False), ("TCGEN05", 222, 256, 15, True),
    ("TCGEN05_PAIR", 76, 512, 10, False), ("TCGEN05_PAIR", 82, 512, 9, False), ("TCGEN05_PAIR", 82, 512, 10, True),
    ("TCGEN05_PAIR", 106, 512, 13, False), ("TCGEN05_PAIR", 106, 512, 15, True),
    ("TCGEN05", 300, 256, 9, False),                                                                                     # by several
])
def test_few_units_of_few_tiles_are_split_where_that_is_faster(B, kernel, heads, m, tiles, split):
    flags = B.KVQ_CORRECTION_ON | getattr(B, "KVQ_KERNEL_" + kernel)
    cached = 128 * (tiles - -(-m // 128)) - 5
    size, launches = plan(B, 128, 1, heads, m, m, cached, flags)
    rotated = -(-heads * m * 272 // 256) * 256
    assert (launches == 3) == split == (size > rotated)                      # pre-pass, attention, and a merge where units are split
    if split:
        assert (size - rotated) % (2 * 134144) == 0                          # FP32 rows
