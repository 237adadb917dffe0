"""The kernels' bounded waits: a warp leaves a loop on the CTA's fail flag as a whole, or not at all.  Another warp sets the
flag at any time, so lanes that each read it may see different values; some would leave the loop while the others go on to
its next warp-wide barrier and wait there for good.  Read from the sources: no run could show it without a hang."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_24174_b200", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def code_lines(path):
    return [line.split("//", 1)[0] for line in open(path)]


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_lane_leaves_a_loop_on_its_own_reading_of_the_fail_flag(path):
    bad = [i + 1 for i, line in enumerate(code_lines(path))
           if re.search(r"\*failed|\bs_fail\b", line) and re.search(r"\bif\s*\(.*(\*failed|\bs_fail\b).*\)\s*\{?\s*break", line)]
    assert not bad, f"{os.path.basename(path)}: lines {bad} leave a loop on one lane's reading"


def test_the_flag_is_read_by_vote_where_the_whole_warp_loads_tiles():
    text = "".join(code_lines(os.path.join(CSRC, "attention_tc.cu")))
    assert len(re.findall(r"if \(warp_failed\(failed\)\) break;", text)) == 2
    vote = "".join(code_lines(os.path.join(CSRC, "common.cuh")))
    assert re.search(r"bool warp_failed\([^)]*\)\s*\{\s*return __any_sync\(0xFFFFFFFFu, \*failed != 0\);", vote)


@pytest.mark.parametrize("name", ["gemm_fused.cu", "gemm_tcgen05.cu"])
def test_the_accumulator_is_read_by_the_whole_warp(name):
    """A lane whose own wait for it ran out would stay away from the warp-wide loads that the others go on to: they depend on no lane's wait."""
    text = "".join(code_lines(os.path.join(CSRC, name)))
    assert len(re.findall(r"\bhave\b[^;]*mbar_wait\(bar_acc, 0\)|mbar_wait\(bar_acc, 0\)[^;]*;[^;]*\bhave\b", text)) == 1
    assert "tmem_ld16(" in text and not re.search(r"if \(have\) \{[^{}]*tmem_ld", text)
