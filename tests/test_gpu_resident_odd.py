"""The shared-memory-resident recursion with an odd number of moments and enough
columns for slabs of two and four: its vectors lie behind a table of M entries of
8 bytes and are read 16 bytes at a time.  FP32 lattices reach this kernel with
hoppings that differ.  Tolerances are the repository's."""
import numpy as np
import pytest

from oracle import oracle as orc
from tests._common import as_oracle, gpu_available, max_abs
from tests.test_gpu_cluster import lattice
from tests.test_gpu_parity import K, TOL, gpu_lattice

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("columns,W", [(400, 2), (700, 4)])
def test_odd_number_of_moments(precision, columns, W):
    p = lattice(14, 12, 0, 0, 17, seed=21)
    p.hop = p.hop.copy()
    p.hop[5, 0] = p.hop[6, 1] = 0.7
    sites = np.random.default_rng(2).choice(p.N, columns).astype(np.int32)
    lat = gpu_lattice(p, precision)
    ee, eh = lat.moments(sites, p.M)
    assert lat.last_tile()[:2] == (W, 0)
    oee, oeh = orc.moments(as_oracle(p), lat.rescale, sites, p.M)
    assert max_abs(ee, oee) < TOL[precision][0] and max_abs(eh, oeh) < TOL[precision][0]
    d, n = lat.order_parameter(p.T, p.M)
    od, on = orc.order_parameter(as_oracle(p), lat.rescale, p.T, p.M, K)
    assert max_abs(d, od) < TOL[precision][1] and max_abs(n, on) < TOL[precision][1]
