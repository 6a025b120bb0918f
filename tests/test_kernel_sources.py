"""Rules of the CUDA sources that no run can show (CPU only)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1007_1609_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_aligned_cluster_barriers_follow_a_warp_barrier(path):
    """barrier.cluster.{arrive,wait}.aligned executed by a warp whose lanes
    have not met again is undefined: whatever the callers do, the statement
    before each of them is __syncwarp()."""
    text = re.sub(r"//[^\n]*", "", open(path).read())
    for m in re.finditer(r'asm volatile\(\s*"barrier\.cluster\.[a-z.]*\.aligned', text):
        assert text[:m.start()].rstrip().endswith("__syncwarp();"), text[m.start():m.end()]
