"""Kernels overlap (programmatic dependent launch): blocks start while the grid before still runs, and wait there.  What that grid, or
one before it, may write - the workspace, and for a call's first kernel every tensor and the cache - must not be read through the
read-only path (`__ldg`, ld.global.nc), which is defined only for memory that nothing writes during the kernel.  Checked in
the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_26266_b200", "csrc")


def ldg_arguments(text):
    """The argument of every __ldg( ... ), parentheses matched."""
    for m in re.finditer(r"__ldg\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield text[m.end():i - 1]


# workspace memory written and read inside one call: bias rows and rotated queries of the pre-pass, partial rows for the merge
@pytest.mark.parametrize("name,pointers", [("attn_sm100.cu", ("ax_rows", "partial", "slot_of", "sl")), ("attn_short.cu", ("partial", "slots", "sl"))])
def test_workspace_is_not_read_through_the_read_only_path(name, pointers):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    assert "wait_for_previous_grid()" in text and all(p in text for p in pointers[:1])
    bad = [a for a in ldg_arguments(text) if any(re.search(rf"\b{p}\b", a) for p in pointers)]
    assert not bad, bad


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name", sorted(n for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh"))))
def test_kernels_that_wait_read_with_ordinary_loads(name):
    text = source(name)
    assert ".nc." not in text
    if "wait_for_previous_grid();" not in text:               # ordinary launches only
        return
    assert "launch_after(true" in text or name == "kvq_common.cuh"
    if name != "attn_sm100.cu":
        assert "__ldg(" not in text
        return
    # the cached tiles of the tcgen05 kernel: it starts behind the pre-pass, whose blocks have all waited before they let it start
    body = text[text.index("void load_raw("):text.index("void load_raw_staged(")]
    assert text.count("__ldg(") == body.count("__ldg(")
    pre_pass = text[text.index(" rotate_query_kernel(const RotParams p)"):]
    assert pre_pass.index("wait_for_previous_grid();") < pre_pass.index("allow_next_grid();") < pre_pass.index("load_coherent(")


def kernels(text):
    """(name, body) of every __global__ function."""
    for m in re.finditer(r"__global__ void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\(", text):
        i = text.index("{", text.index(") {", m.end()))
        depth, j = 1, i + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        yield m.group(1), text[i:j]


def without_wait(text):
    """Kernels that are not launched the ordinary way and touch memory, or let the next grid start, without having waited."""
    out = []
    for name, body in kernels(text):
        if re.search(rf"\b{name}(<[^;{{}}<>]*>)?<<<", text):
            continue
        wait = body.find("wait_for_previous_grid();")
        if wait < 0 or 0 <= body.find("allow_next_grid();") < wait:
            out.append(name)
    return out


def test_every_kernel_that_may_start_early_waits():
    found = set()
    for name in sorted(n for n in os.listdir(CSRC) if n.endswith(".cu")):
        text = source(name)
        assert without_wait(text) == []
        early = {k for k, body in kernels(text) if "wait_for_previous_grid();" in body}
        for m in [m.start() for m in re.finditer(r"wait_for_previous_grid\(\);", text)]:      # the check sees a missing one
            cut = text[:m] + text[m + len("wait_for_previous_grid();"):]
            kernel = next(k for k, body in kernels(text) if text.index(body) <= m < text.index(body) + len(body))
            assert without_wait(cut) == [kernel] or kernel == "attn_tcgen05_kernel"            # which waits in several roles
        found |= early
    assert found == {"attn_short_kernel", "attn_short_merge_kernel", "rotate_query_kernel", "attn_tcgen05_kernel", "attn_merge_kernel",
                     "quantize_append_kernel"}


def test_both_ctas_of_a_pair_wait_for_the_last_commits():
    """Commits of a pair (tc_commit_pair) arrive on the barriers of both CTAs at times of their own.  The leader drains its copy of
    the last ones; the peer has to drain its own before the cluster barrier that lets it leave."""
    with open(os.path.join(CSRC, "attn_sm100.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    end = text[text.rindex("++nseg;"):text.index("tmem_dealloc_pair(tmem")]
    # two warps of the peer's dequantizing role (warps 12 to 15), then the barrier
    assert re.search(r"rank != 0 && warp < 14\) cx\.drain\(kDrain \+ warp - 12, 0\);.*cluster_sync_all\(\);", end, re.S)
    assert re.search(r"commit\(kDrain \+ qt\);\s*cx\.drain\(kDrain \+ qt, 0\);", text)


def test_a_pair_is_there_while_its_tensor_memory_is_allocated_and_freed():
    """tcgen05.alloc and .dealloc with cta_group::2 concern the TMEM of both CTAs of a cluster.  CTAs of a cluster are placed together
    but do not start or end together, so a barrier of the cluster stands in front of the first and behind the second."""
    body = dict(kernels(source("attn_sm100.cu")))["attn_tcgen05_kernel"]
    before, rest = body.split("tmem_alloc_pair(")
    assert "cluster_sync_all();" in before
    inside, after = rest.split("tmem_dealloc_pair(")
    assert inside.count("cluster_sync_all();") == 2 and "wait_for_previous_grid" not in inside[inside.rindex("cluster_sync_all();"):]
    assert "cluster_sync_all();" in after


def test_every_barrier_that_is_committed_on_is_waited_for_before_the_exit():
    """Commits arrive on their barriers in no promised order, and where nobody waits for one it may arrive in the shared memory of the CTA
    that comes next.  Of the barriers the issuers commit on, the softmax groups wait for every phase of kSFull and for the last one of a
    segment on kODone + 2; the issuers drain kDrain; the last phases of all others are drained by the dequantizing warps.  Their parities, from the
    number of tiles and segments, against a count of the commits."""
    body = dict(kernels(source("attn_sm100.cu")))["attn_tcgen05_kernel"]
    committed = {re.match(r"k\w+", a).group(0) for a in re.findall(r"\bcommit\(([^()]+)\);", body)}
    assert committed == {"kSFull", "kODone", "kKEmpty", "kVEmpty", "kQEmpty", "kQCurDone", "kDrain"}
    tail = body[body.rindex("++nseg;"):body.rindex("wait_for_previous_grid();")]
    drained = dict(re.findall(r"cx\.drain\((k\w+) \+ i, ([^;]+)\);", tail))
    assert set(drained) == {"kKEmpty", "kVEmpty", "kODone"}
    assert "cx.drain(i == 0 ? kQEmpty : kQCurDone, (nseg - 1) & 1);" in tail
    assert "cx.wait(kSFull + 2 * hf + qt, it & 1, 301)" in body and "cx.wait(kODone + 2 + qt, (it - 1) & 1, 303)" in body
    parity = {k: eval("lambda it, i: " + v.replace("kODone", "")) for k, v in drained.items()}
    for tiles in range(1, 9):
        phases = {(k, i): 0 for k in drained for i in range(2)}
        for t in range(tiles):                            # tile t uses stage t % 2; a tile's first half of O is committed once
            phases["kKEmpty", t & 1] += 1
            phases["kVEmpty", t & 1] += 1
            phases["kODone", 0] += 1
            phases["kODone", 1] += 1
        for (k, i), n in phases.items():
            assert (n == 0) == (k != "kODone" and tiles <= i)
            if n:
                assert parity[k](tiles, i) == (n - 1) & 1, (k, i, tiles)


def test_a_warp_is_whole_where_it_allocates_and_frees_tensor_memory():
    """tcgen05.alloc, .relinquish_alloc_permit and .dealloc are .sync.aligned: all lanes of the warp execute them together.  Lane 0 has run code
    of its own before both, and nothing promises that the lanes have met again without a __syncwarp()."""
    body = dict(kernels(source("attn_sm100.cu")))["attn_tcgen05_kernel"]
    one_lane = body.index("if (tid == 0) {")
    before = body[one_lane:body.index("tmem_alloc(")]
    assert re.search(r"\n  __syncwarp\(\);\s*if constexpr \(PAIR\) cluster_sync_all\(\);\s*if \(warp == 0\) \{\s*if constexpr \(PAIR\) \{ tmem_alloc_pair", before)
    role = body.index("if (lane == 0) {", body.index("tmem_alloc("))
    assert re.search(r"if \(warp == 0\) \{\s*__syncwarp\(\);[^{}]*tmem_dealloc_pair\(tmem, 512\); else tmem_dealloc\(tmem, 512\);", body[role:])


def test_a_site_code_names_one_wait():
    """The code that an expired wait leaves in the status word tells which one it was; kvq.h lists them."""
    text = source("attn_sm100.cu")
    at = {}
    for m in re.finditer(r"cx\.wait\([^;]*?, (\d{3})\)", text):
        at.setdefault(int(m.group(1)), []).append(m.start())
    assert {c for c, places in at.items() if len(places) > 1} == {402}
    a, b = at[402]                                            # the two forms of one wait, a pair's and a CTA's
    assert text[a:b].count(";") == 1 and "else ok = " in text[a:b]
    with open(os.path.join(CSRC, "..", "..", "include", "kvq.h")) as f:
        header = f.read()
    listed = header[header.index("Site codes:"):header.index("kvq_status_word_result maps")]
    assert set(at) == {int(c) for c in re.findall(r"\b(\d{3}) \(", listed)}
