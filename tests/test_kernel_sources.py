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


def test_waits_of_the_on_chip_kernels_take_the_callers_limit():
    """CBDG_OPT_WAIT_LIMIT_MS reaches every wait of the on-chip recursions: no
    limit of their own, and every launch of a lattice passes the option on."""
    for name in ("cluster.cuh", "cluster_cplx.cuh", "adjoint_cluster.cuh"):
        text = open(os.path.join(CSRC, name)).read()
        assert "kWaitNs" not in text, name
        waits = re.findall(r"for \(unsigned it = 0; !mbar_try\(.*?;", text, re.S)
        assert waits
        assert len(re.findall(r"expired\w*\(t0, a\.wait_ns, a\.flags\)", text)) == len(waits), name
    api = open(os.path.join(CSRC, "api.cu")).read()
    structs = re.findall(r"\b(ClusterArgs|CplxClusterArgs|AdjointClusterArgs) c\{\};", api)
    assert len(structs) >= 4
    # the general lattice's launches share one place that fills the rest of the arguments
    assert api.count("c.wait_ns = static_cast<unsigned long long>(L->wait_ms) * 1000000ull;") == len(set(structs)) == 3


def test_destroy_frees_every_buffer_of_a_lattice():
    api = open(os.path.join(CSRC, "api.cu")).read()
    struct = api[api.index("struct cbdg_lattice {"):]
    struct = re.sub(r"//[^\n]*", "", struct[:struct.index("\n};")])
    members = [m for line in re.findall(r"\bDBuf ([^;()]*);", struct) for m in re.findall(r"\w+", line)]
    destroy = api[api.index("cbdg_status cbdg_destroy("):]
    freed = re.findall(r"&L->(\w+)", destroy[:destroy.index("b->release()")])
    assert len(members) > 40 and sorted(members) == sorted(freed)
