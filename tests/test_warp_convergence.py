"""The warp-wide instructions of tensor memory (tcgen05 .sync.aligned) and of
the named and cluster barriers (bar.sync, bar.red, barrier.cluster) need a converged warp.  Read off the
sources: each place where lanes of a warp part ways ahead of one -- the bounded
wait on a copy, the branch in which one thread issues copies, the allocation
behind a thread's own work -- ends in __syncwarp().  (Text only: a kernel that
broke this rule is not run to see what happens.)"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_14907_gb300", "csrc")


def _text(name):
    s = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", s)


def _block(s, at):
    """The braces that open at or after s[at]: (start, end)."""
    i = s.index("{", at)
    n = 0
    for j in range(i, len(s)):
        n += {"{": 1, "}": -1}.get(s[j], 0)
        if n == 0:
            return i, j + 1
    raise AssertionError("unbalanced")


def test_bounded_wait_ends_converged():
    s = _text("bulk.cuh")
    at = re.search(r"MPBP_DI bool bulk_wait_\w+\(", s).start()
    i, j = _block(s, at)
    body = s[i:j]
    assert "while" in body
    loop_end = _block(body, body.index("while"))[1]
    assert body.index("__syncwarp();") > loop_end
    assert "return" not in body[:body.index("__syncwarp();")]


ISSUE = re.compile(r"if \(([^{};]*(?:tid|threadIdx\.x) == 0[^{};]*)\)\s*(\{|bulk_)")


@pytest.mark.parametrize("name", ["frames.cuh", "frames_t4.cuh", "frames_x3.cuh"])
def test_issuing_thread_rejoins_its_warp(name):
    s = _text(name)
    found = 0
    for m in ISSUE.finditer(s):
        end = _block(s, m.start())[1] if m.group(2) == "{" else s.index(";", m.end()) + 1
        if not re.search(r"tile_load_|bulk_load|bulk_prefetch|mbar_arrive_tx", s[m.start():end]):
            continue
        found += 1
        assert s[end:].lstrip().startswith("__syncwarp();"), s[m.start():end + 80]
    assert found >= 1


@pytest.mark.parametrize("name", ["tmem.cuh", "frames_tc.cu"])
def test_allocation_starts_converged(name):
    s = _text(name)
    at = [m.start() for m in re.finditer(r"asm volatile\(\"tcgen05\.alloc", s)]
    assert at
    for a in at:
        assert s[:a].rstrip().endswith("__syncwarp();")


@pytest.mark.parametrize("name,fn", [("frames_tc.cu", "group_bar(int"), ("frames_tc.cu", "group_bar_and("),
                                     ("frames.cuh", "void sync()"), ("mpbp_unwrap.cu", "void cluster_sync(")])
def test_named_and_cluster_barriers_start_converged(name, fn):
    s = _text(name)
    i, j = _block(s, s.index(fn))
    body = s[i:j]
    assert "__syncwarp();" in body[:body.index("asm volatile")]


def test_no_guarded_store_ahead_of_tensor_memory():
    """The M = 64 kernel's resident-probe scatter and window write-back: the
    lanes' own conditions are predicates, or end before the next access."""
    s = _text("frames.cuh")
    i, j = _block(s, s.index("MPBP_DI void t2_win_flush"))
    body = s[i:j]
    guard = body.index("if (row >= w.wlo")
    assert guard < body.index("__syncwarp();") < body.index("tmem_st2(")
    for m in re.finditer(r"else if constexpr \(TPR\)", s):
        a, b = _block(s, m.start())
        assert "red_add_v2(" not in s[a:b]


def test_every_source_with_warp_wide_instructions_is_known():
    wide = re.compile(r"sync\.aligned|barrier\.cluster|bar\.sync|bar\.red")
    names = {os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*")) if wide.search(_text(os.path.basename(f)))}
    assert names == {"tmem.cuh", "frames_tc.cu", "frames.cuh", "mpbp_unwrap.cu"}
