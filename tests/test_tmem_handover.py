"""The tcgen05 attention keeps S, then P, in the same TMEM columns.  What orders the accesses to them is read from the sources: an MMA that overwrites
them waits for the one that read them, and a warp that does has the fence behind the barrier at which the other one's reads ended."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_24174_b200", "csrc")
TEXT = "\n".join(line.split("//", 1)[0] for line in open(os.path.join(CSRC, "attention_tc.cu")))


def between(a, b):
    assert TEXT.count(a) == 1
    i = TEXT.index(a)
    return TEXT[i:TEXT.index(b, i)]


def test_scores_are_written_when_the_tile_before_in_their_place_has_been_used():
    assert re.search(r"if \(u >= 2\) wait\(bar_o_full \+ 8u \* \(u & 1\), \(uint32_t\)\(\(u >> 1\) - 1\) & 1u\);", between("const int u = t + 1;", "umma_bf16_warp(d,"))


def test_probabilities_are_written_behind_barrier_and_fence():
    text = between("s_max[t & 1][half][rho] = mx;", "tmem_st8(")
    assert re.search(r'asm volatile\("bar\.sync %0, 64;"[^;]*;\s*tc_fence_after\(\);', text)
    assert "tc_fence_before();" in between("s[c + e] = __uint_as_float(r[e]);", "s_max[t & 1][half][rho] = mx;")


def test_lanes_that_waited_one_by_one_meet_before_tmem_is_read():
    waits = list(re.finditer(r"wait\(bar_[so]_full \+ 8u \* \(t & 1\)[^;]*;", TEXT))
    assert len(waits) == 2
    for m in waits:
        assert "__syncwarp();" in TEXT[m.end():TEXT.index("tmem_ld32(", m.end())]
