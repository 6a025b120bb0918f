"""The FP64 recursion of lattices with one hopping in shared memory (walks along
(-1, +1) on the lattice with its zeros): moments and order parameter against the
oracle for every kind of edge, one and several cycles of walks, sides that are
coprime and equal, threads without sites, the largest lattice taken and the
first that is not, few columns; and the lattices that stay with the general kernel.
Tolerances are the repository's for FP64 (1e-11 on moments, 1e-10 on Delta)."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1007_1609_gb300 import cbdg
from tests._common import as_oracle, gpu_available, max_abs
from tests.test_gpu_cluster import lattice
from tests.test_gpu_parity import K, TOL, gpu_lattice

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("px,py", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("shape", [(52, 49, 17), (30, 44, 34), (61, 45, 20), (62, 65, 9), (1000, 3, 12), (3, 1000, 13)])
def test_moments_match_oracle(shape, px, py):
    Lx, Ly, M = shape
    p = lattice(Lx, Ly, px, py, M, seed=Lx + Ly)
    sites = np.random.default_rng(Ly).choice(p.N, 600).astype(np.int32)
    sites[:4] = [0, Lx - 1, p.N - Lx, p.N - 1]
    lat = gpu_lattice(p, "fp64")
    ee, eh = lat.moments(sites, M)
    assert lat.last_tile()[:2] == (1, 0)  # on chip, one column at a time
    few = lat.moments(sites[:20], M)
    oee, oeh = orc.moments(as_oracle(p), lat.rescale, sites[:20], M)
    for x, y in ((ee[:20], eh[:20]), few):
        assert max_abs(x, oee) < TOL["fp64"][0] and max_abs(y, oeh) < TOL["fp64"][0]


@pytest.mark.parametrize("shape", [(31, 30, 0, 0, 34), (30, 30, 1, 1, 67), (61, 45, 0, 1, 33)])
def test_order_parameter_matches_oracle(shape):
    Lx, Ly, px, py, M = shape
    p = lattice(Lx, Ly, px, py, M, seed=5)
    lat = gpu_lattice(p, "fp64")
    d, n = lat.order_parameter(p.T, M)
    assert lat.last_tile()[:2] == (1, 0)
    od, on = orc.order_parameter(as_oracle(p), lat.rescale, p.T, M, K)
    assert max_abs(d, od) < TOL["fp64"][1] and max_abs(n, on) < TOL["fp64"][1]


def test_other_lattices_keep_their_kernels():
    """64 x 64, or hoppings that differ."""
    p, q = lattice(64, 64, 1, 1, 9, seed=6), lattice(61, 45, 0, 0, 9, seed=6)
    q.hop = q.hop.copy()
    q.hop[5, 0] = q.hop[6, 1] = 0.7
    for prob in (p, q):
        lat = gpu_lattice(prob, "fp64")
        sites = np.arange(0, prob.N, 400, dtype=np.int32)
        ee, eh = lat.moments(sites, prob.M)
        assert lat.last_tile()[1] > 0
        oee, oeh = orc.moments(as_oracle(prob), lat.rescale, sites, prob.M)
        assert max_abs(ee, oee) < TOL["fp64"][0] and max_abs(eh, oeh) < TOL["fp64"][0]


def test_spectrum_violation_is_reported():
    p = lattice(40, 40, 0, 0, 64, seed=7)
    lat = gpu_lattice(p, "fp64", fixed_rescale_pico=int(0.5e12))  # a far inside the band
    for call in (lambda: lat.moments(np.arange(p.N, dtype=np.int32), 64), lambda: lat.order_parameter(p.T, 64)):
        with pytest.raises(cbdg.CbdgError) as ei:
            call()
        assert ei.value.status == cbdg.CBDG_ERR_SPECTRUM
