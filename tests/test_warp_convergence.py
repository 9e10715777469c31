"""Instructions marked `.aligned` (tensor memory, cluster barriers) are undefined in a warp whose lanes have parted: lost lanes or a
hang.  Whether a compiler lets lanes meet again by itself cannot be provoked on demand, so the sources are read: the pieces of the
epilogue whose branches depend on the lane end with __syncwarp() and leave no other way, and the wrappers of the barriers begin with it."""
import os
import re

import pytest

from conftest import ROOT


def body(name, function):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(ROOT, "paper_2001_07710_b200", "csrc", name)).read())
    m = re.search(r"\b%s\(([^;{]*?)\)\s*\{" % function, text, re.S)
    depth, i = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[m.end():i - 1].strip()


@pytest.mark.parametrize("function", ["store_piece", "send_part"])
def test_lane_dependent_pieces_end_with_the_whole_warp(function):
    b = body("mma_tile.cuh", function)
    assert b.endswith("__syncwarp();") and not re.search(r"\breturn\b|\bgoto\b", b)


@pytest.mark.parametrize("name,function,first", [("mma_tile.cuh", "cluster_arrive", "__syncwarp"), ("mma_tile.cuh", "cluster_wait", "__syncwarp"),
                                                 ("mma_tile.cuh", "alloc_columns", "__syncwarp"), ("mma_tile.cuh", "free_columns", "__syncwarp"),
                                                 ("conv_tile.cuh", "tmem_alloc", "__syncwarp"), ("conv_tile.cuh", "tmem_dealloc", "__syncwarp"),
                                                 ("project.cu", "sel_barrier", "if constexpr")])
def test_aligned_barriers_begin_with_the_whole_warp(name, function, first):
    b = body(name, function)
    assert b.startswith(first) and 0 <= b.index("__syncwarp();") < b.index(".aligned")


def test_pooled_results_meet_with_the_whole_warp():
    b = body("mma_tile.cuh", "pool_results")
    assert re.search(r"__syncwarp\(\);\s*asm volatile\(\"bar\.sync 1[^;]*;[^;]*;$", b)


def test_consumer_warps_leave_a_wait_together():
    """Their waits end in warp-wide instructions: one lane that gives up by itself would leave the others there."""
    text = open(os.path.join(ROOT, "paper_2001_07710_b200", "csrc", "conv_f32_img.cu")).read()
    consumers = text[text.index("consumer warps\n"):]
    consumers = consumers[:consumers.index("tmem_dealloc(")]
    assert "__all_sync(0xFFFFFFFFu, mbar_wait" in body("conv_f32_img.cu", "warp_wait")
    assert consumers.count("warp_wait(") >= 6 and "mbar_wait<" not in consumers
