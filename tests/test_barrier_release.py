"""A warp that gives shared or tensor memory back through one lane's mbarrier arrival orders the other lanes'
accesses before it with __syncwarp() (a vote or a shuffle orders no memory).  Read from the sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_34045_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_lane_arrivals_follow_a_warp_barrier(path):
    code = [re.sub(r"//.*", "", line).strip() for line in open(path)]
    code = [(n, line) for n, line in enumerate(code, 1) if line]
    bare = [n for (_, before), (n, line) in zip(code, code[1:])
            if re.match(r"if \(lane == 0\) mbar_arrive\(", line) and before != "__syncwarp();"]
    assert not bare, f"{os.path.basename(path)}: lane 0 arrives without __syncwarp() before it, lines {bare}"
