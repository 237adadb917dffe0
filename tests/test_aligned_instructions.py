"""Cluster barriers and TMEM allocation are .aligned instructions: the lanes of a warp have to reach them together, and their callers come from
loops and branches that lanes leave one by one.  Read from the sources: no run could show a lane that is missing without a hang."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_24174_b200", "csrc")
ALIGNED = r'"(barrier\.cluster\.[\w.]*aligned|tcgen05\.(?:alloc|dealloc|relinquish_alloc_permit)\.[\w.:]*aligned)'


def code(path):
    return "\n".join(line.split("//", 1)[0] for line in open(path))


def test_the_lanes_meet_right_before():
    """... but in the two that say so in their names."""
    text = code(os.path.join(CSRC, "common.cuh"))
    found = list(re.finditer(r"(\w+)\([^()]*\) \{\s*(__syncwarp\(\);\s*)?asm volatile\(\s*" + ALIGNED, text))
    assert len(found) == len(re.findall(ALIGNED, text)) == 9                     # cluster: arrive, wait, both, two converged; TMEM: two each for one CTA and for a pair
    assert {m.group(1) for m in found if not m.group(2)} == {"cluster_arrive_converged", "cluster_sync_converged"}


def test_who_is_converged():
    """The few-row GEMM, whose warps come from warp-wide barriers (its last barrier, behind the epilogue, is not among them)."""
    users = {os.path.basename(p): re.findall(r"\bcluster_\w+", code(p)) for p in glob.glob(os.path.join(CSRC, "*.cu"))}
    assert {p for p, names in users.items() if any(n.endswith("_converged") for n in names)} == {"gemm_fused.cu"}
    barriers = [n for n in users["gemm_fused.cu"] if n.startswith(("cluster_arrive", "cluster_sync", "cluster_wait"))]
    assert barriers == ["cluster_sync_converged", "cluster_arrive_converged", "cluster_wait"]


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_no_kernel_has_its_own(path):
    assert not re.search(ALIGNED, code(path))
