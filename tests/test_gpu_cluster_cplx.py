"""The register-resident recursion of general FP32 lattices (complex hoppings,
four or eight of them, on-site or bond pairing): matrix elements, moments and
currents against the FP64 oracle at the edges of its tiles (4 x 2 sites), of its
CTAs and of its clusters, for every kind of edge (periodic ones that the tiles
do not divide too), and against the streamed
kernels bit for bit; more targets than threads; and the calls it leaves to the
streamed kernels.  Tolerance: an update rounds at most
19 sums, each within 2^-24 of magnitudes that add up to at most 2, so 1.2e-6 a
step; the rounding errors of up to 41 steps add as a random walk (a factor of 6.4):
1e-5, the FP32 tolerance of the general recursion; twice that for a current,
which sums two spins."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1007_1609_gb300 import cbdg
from paper_1007_1609_gb300 import workloads as wl
from tests._common import as_oracle, gpu_available, max_abs
from tests.test_gpu_general import K, gpu_lattice

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]

TOL = 1e-5


def lattice(Lx, Ly, px, py, tp, bond, M, seed):
    """Hoppings with random phases, random complex pairing."""
    rng = np.random.Generator(np.random.PCG64(seed))
    N, site = Lx * Ly, np.arange(Lx * Ly)
    hop = wl.square_hops(Lx, Ly, px, py, t=1.0, tp=tp).astype(np.complex128)
    delta = np.zeros((N, 4), dtype=np.complex128)
    steps = [(1, 0), (0, 1), (1, 1), (1, -1)][: hop.shape[1] // 2]
    for k, (dx, dy) in enumerate(steps):  # directions 2 k and, seen from the neighbour, 2 k + 1
        x, y = site % Lx + dx, site // Lx + dy
        on = ((px == 1) | (x < Lx)) & ((py == 1) | ((y >= 0) & (y < Ly)))
        nb = (x % Lx + Lx * (y % Ly))[on]
        hop[on, 2 * k] *= np.exp(1j * rng.uniform(-1, 1, on.sum()))
        hop[nb, 2 * k + 1] = hop[on, 2 * k].conj()
        if k < 2:
            delta[on, 2 * k] = 0.2 * (rng.normal(size=on.sum()) + 1j * rng.normal(size=on.sum()))
            delta[nb, 2 * k + 1] = delta[on, 2 * k]
    return wl.Problem(name=f"g{Lx}x{Ly}", Lx=Lx, Ly=Ly, periodic_x=px, periodic_y=py,
                      eps=rng.uniform(-0.5, 0.5, N), mu=-0.4, hop=hop, pairing=wl.BOND if bond else wl.ONSITE,
                      coupling=1.2, delta0=delta if bond else delta[:, 0] + 0.3, T=0.02, M=M)


@pytest.mark.parametrize("tp,bond", [(0.0, 0), (0.0, 1), (-0.3, 0), (-0.3, 1)])
@pytest.mark.parametrize("shape", [(4, 4, 1, 1, 2), (5, 3, 0, 0, 3), (8, 6, 1, 0, 9), (7, 12, 0, 1, 41), (16, 10, 1, 1, 34),
                                   (33, 51, 0, 0, 33), (64, 64, 1, 1, 12), (60, 97, 1, 0, 10), (128, 128, 1, 1, 9),
                                   (3, 3, 1, 1, 6), (5, 7, 1, 1, 12), (6, 8, 1, 1, 8), (7, 12, 1, 0, 9), (9, 5, 0, 1, 9),
                                   (34, 47, 1, 1, 33), (64, 63, 1, 1, 12), (63, 98, 1, 0, 10), (125, 127, 1, 1, 9)])
def test_matrix_elements_match_oracle(shape, tp, bond):
    Lx, Ly, px, py, M = shape
    p = lattice(Lx, Ly, px, py, tp, bond, M, seed=Lx + 3 * Ly)
    rng = np.random.default_rng(Ly)
    sites = np.concatenate([[0, p.N - 1], rng.choice(p.N, 3)]).astype(np.int32)
    targets = np.concatenate([[p.N - 1, Lx - 1], rng.choice(p.N, 18)]).astype(np.int32)
    lat, ol = gpu_lattice(p, "fp32"), as_oracle(p)
    a11, a12 = lat.green_moments(sites, targets, M)
    assert lat.last_tile()[:2] == (2, 0)  # on chip, two columns a cluster
    o11, o12 = orc.green_moments(ol, lat.rescale, sites, targets, M)
    assert max_abs(a11, o11) < TOL and max_abs(a12, o12) < TOL
    streamed = gpu_lattice(p, "fp32", resident=0)
    for x, y in zip((a11, a12), streamed.green_moments(sites, targets, M)):  # the same sums in the same order
        assert np.array_equal(x, y)
    if bond:
        ee, eh = lat.moments(sites, M)
        assert lat.last_tile()[:2] == (2, 0)
        oee, oeh = orc.moments(ol, lat.rescale, sites, M)
        assert max_abs(ee, oee) < TOL and max_abs(eh, oeh) < TOL
        for x, y in zip((ee, eh), streamed.moments(sites, M)):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("tp", [0.0, -0.3])
def test_folds_match_oracle(tp):
    p = lattice(12, 14, 1, 0, tp, 1, 40, seed=3)
    lat, ol = gpu_lattice(p, "fp32"), as_oracle(p)
    d, n = lat.order_parameter(p.T, p.M)
    od, on = orc.order_parameter(ol, lat.rescale, p.T, p.M, K)
    assert max_abs(d, od) < TOL and max_abs(n, on) < TOL
    J = lat.bond_currents(p.T, p.M)
    assert lat.last_tile()[:2] == (2, 0)
    assert max_abs(J, 2.0 * orc.bond_currents(ol, lat.rescale, p.T, p.M, K)) < 2 * TOL


def test_more_targets_than_threads():
    """Every site of one start vector's lattice, some twice."""
    p = lattice(20, 20, 0, 0, -0.3, 1, 40, seed=4)
    sites = np.array([0, 210, 399], dtype=np.int32)
    targets = np.concatenate([np.arange(400), np.arange(399, -1, -1)]).astype(np.int32)
    lat = gpu_lattice(p, "fp32")
    a11, a12 = lat.green_moments(sites, targets, 40)
    assert lat.last_tile()[:2] == (2, 0)
    o11, o12 = orc.green_moments(as_oracle(p), lat.rescale, sites, targets, 40)
    assert max_abs(a11, o11) < TOL and max_abs(a12, o12) < TOL


@pytest.mark.parametrize("shape,n,n_t", [((180, 180, 1, 1), 4, 3), ((128, 128, 1, 1), 2000, 3), ((64, 64, 1, 1), 16, 4096)])
def test_other_calls_stay_streamed(shape, n, n_t):
    """A lattice that does not fit, and more columns of a large one, or more targets,
    than clusters take in good time."""
    p = lattice(*shape, -0.3, 1, 8, seed=5)
    rng = np.random.default_rng(6)
    sites, targets = rng.choice(p.N, n).astype(np.int32), rng.choice(p.N, n_t).astype(np.int32)
    lat = gpu_lattice(p, "fp32")
    a11, a12 = lat.green_moments(sites, targets, 8)
    assert lat.last_tile()[1] > 0
    o11, o12 = orc.green_moments(as_oracle(p), lat.rescale, sites[:4], targets, 8)
    assert max_abs(a11[:4], o11) < TOL and max_abs(a12[:4], o12) < TOL


def test_spectrum_violation_is_reported():
    p = lattice(24, 24, 1, 1, -0.3, 1, 64, seed=7)
    lat = gpu_lattice(p, "fp32", fixed_rescale_pico=int(0.5e12))  # a far inside the band
    sites = np.arange(8, dtype=np.int32)
    for call in (lambda: lat.moments(sites, 64), lambda: lat.green_moments(sites, sites, 64)):
        with pytest.raises(cbdg.CbdgError) as ei:
            call()
        assert ei.value.status == cbdg.CBDG_ERR_SPECTRUM
