"""The register-resident recursion of thread-block clusters (FP32 real on-site
lattices with one hopping): moments and order parameter against the FP64
oracle at the edges of its tiles (4 sites wide, 4, 6, 8 or 10 high), of its CTAs
and of its clusters, for every kind of edge, few and many start sites; the
lattices it does not take (hoppings that differ) against the streamed kernels.
Tolerances are those of the FP32 recursion: its column sums carry at most
38 * 2^-24 of the sum of magnitudes (<= 1), doubled in a moment: 4.5e-6."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1007_1609_gb300 import cbdg
from paper_1007_1609_gb300 import workloads as wl
from tests._common import as_oracle, gpu_available, max_abs
from tests.test_gpu_parity import K, TOL, gpu_lattice

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


def lattice(Lx, Ly, px, py, M, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    N = Lx * Ly
    return wl.Problem(name=f"c{Lx}x{Ly}", Lx=Lx, Ly=Ly, periodic_x=px, periodic_y=py,
                      eps=rng.uniform(-0.5, 0.5, size=N), mu=-0.5, hop=wl.square_hops(Lx, Ly, px, py),
                      pairing=wl.ONSITE, coupling=2.0, delta0=rng.uniform(0.2, 0.8, size=N).astype(np.complex128),
                      T=0.02, M=M)


@pytest.mark.parametrize("px,py", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("shape", [(3, 3, 2), (4, 8, 3), (5, 9, 37), (33, 49, 68), (65, 66, 35), (97, 95, 34),
                                   (130, 127, 36), (256, 250, 20), (500, 319, 21)])
def test_moments_match_oracle(shape, px, py):
    Lx, Ly, M = shape
    p = lattice(Lx, Ly, px, py, M, seed=Lx * 13 + Ly)
    sites = np.arange(p.N, dtype=np.int32)
    if p.N > 64:
        rng = np.random.default_rng(Ly)
        sites = np.concatenate([[0, Lx - 1, p.N - Lx, p.N - 1], rng.choice(p.N, 20)]).astype(np.int32)
    lat = gpu_lattice(p, "fp32")
    ee, eh = lat.moments(sites, M)
    assert lat.last_tile()[:2] == (1, 0)  # on chip, one column at a time
    oee, oeh = orc.moments(as_oracle(p), lat.rescale, sites, M)
    assert max_abs(ee, oee) < TOL["fp32"][0] and max_abs(eh, oeh) < TOL["fp32"][0]
    one = lat.moments(sites[-1:], M)  # a single start site, another plan
    assert max_abs(one[0], oee[-1:]) < TOL["fp32"][0] and max_abs(one[1], oeh[-1:]) < TOL["fp32"][0]


@pytest.mark.parametrize("shape", [(31, 30, 0, 0, 34), (22, 37, 1, 1, 67)])
def test_order_parameter_matches_oracle(shape):
    Lx, Ly, px, py, M = shape
    p = lattice(Lx, Ly, px, py, M, seed=5)
    lat = gpu_lattice(p, "fp32")
    d, n = lat.order_parameter(p.T, M)
    od, on = orc.order_parameter(as_oracle(p), lat.rescale, p.T, M, K)
    assert max_abs(d, od) < TOL["fp32"][1] and max_abs(n, on) < TOL["fp32"][1]


def test_hoppings_that_differ_take_the_general_path():
    """A lattice whose hoppings differ keeps the kernels that read each one;
    replacing the hoppings moves the lattice from one path to the other, also
    between replays of a captured iteration."""
    p = lattice(30, 70, 0, 0, 40, seed=6)
    q = lattice(30, 70, 0, 0, 40, seed=6)
    q.hop = p.hop.copy()
    q.hop[31, 0] = q.hop[32, 1] = 0.7  # the bond between sites 31 and 32
    lat = gpu_lattice(p, "fp32")
    for hop, prob in ((p.hop, p), (q.hop, q), (p.hop, p), (0.5 * p.hop, None)):
        cbdg.cbdg_set_hamiltonian(lat.handle, None, np.ascontiguousarray(hop))
        if prob is None:
            prob = lattice(30, 70, 0, 0, 40, seed=6)
            prob.hop = 0.5 * p.hop
        lat.delta = prob.delta0
        for _ in range(3):
            lat.scf_step(prob.T, prob.M, 0.5)
        ref, _, _, _ = orc.scf(as_oracle(prob), prob.T, prob.M, K, 0.5, 0.0, 3)
        assert max_abs(lat.delta, ref) < TOL["fp32"][1]


def test_spectrum_violation_is_reported():
    p = lattice(40, 40, 0, 0, 64, seed=7)
    lat = gpu_lattice(p, "fp32", fixed_rescale_pico=int(0.5e12))  # a far inside the band
    with pytest.raises(cbdg.CbdgError) as ei:
        lat.moments(np.arange(p.N, dtype=np.int32), p.M)
    assert ei.value.status == cbdg.CBDG_ERR_SPECTRUM


def test_ensemble_mixes_both_kernels():
    """Members with one hopping run in cluster registers, a member whose
    hoppings differ in the streaming kernel; all follow the oracle's loop."""
    ps = [lattice(24, 40, 0, 0, 48, seed=8), lattice(33, 21, 0, 0, 48, seed=9), lattice(40, 26, 0, 0, 48, seed=10)]
    ps[1].hop = ps[1].hop.copy()
    ps[1].hop[5, 0] = ps[1].hop[6, 1] = 1.3
    ens = cbdg.Ensemble(ps)
    ens.set_option(cbdg.CBDG_OPT_QUADRATURE_NODES, K)
    _, it, _ = ens.scf(0.02, 48, 0.5, 0.0, 2)
    assert it == 2
    for k, p in enumerate(ps):
        ref, _, _, _ = orc.scf(as_oracle(p), 0.02, 48, K, 0.5, 0.0, 2)
        assert max_abs(ens.delta(k), ref) < TOL["fp32"][1]
    ens.close()


@pytest.mark.parametrize("shape", [(3, 2, 0, 0, 2), (4, 4, 1, 1, 3), (9, 7, 0, 0, 10), (12, 8, 1, 0, 11),
                                   (33, 30, 0, 0, 20), (8, 36, 0, 1, 67), (66, 70, 0, 0, 66), (130, 67, 0, 0, 12)])
def test_backward_matches_oracle(shape):
    """The adjoint in cluster registers: every remainder of its kept pairs (8
    steps) and of its sums (64), one CTA and clusters, tiles that stick out,
    periodic sides.  Against the oracle's reverse mode within the FP32
    gradient tolerance (1e-3 of the largest component), and against the
    streamed adjoint within 2e-5 (both carry the rounding of M FP32 steps)."""
    Lx, Ly, px, py, M = shape
    p = lattice(Lx, Ly, px, py, M, seed=Lx + M)
    w = np.random.default_rng(M).normal(size=p.N)
    lat = gpu_lattice(p, "fp32")
    cbdg.cbdg_launch_count(lat.handle, reset=True)
    got = lat.backward(p.T, M, w.astype(np.complex128))
    assert cbdg.cbdg_launch_count(lat.handle) < 12  # one recursion launch, not one per step
    ref = gpu_lattice(p, "fp32", resident=0).backward(p.T, M, w.astype(np.complex128))
    for x, y in zip(got, ref):
        assert max_abs(x, y) <= 2e-5 * max(np.max(np.abs(y)), 1e-3)
    if p.N <= 1000:
        o = orc.scf_map_gradient(as_oracle(p), lat.rescale, orc.fold_coefficients(M, K, lat.rescale, p.T), w)
        for x, y in zip(got, o):
            assert max_abs(x.real.reshape(-1), np.asarray(y).reshape(-1)) <= 1e-3 * max(np.max(np.abs(y)), 1e-6)


def test_ldos_backward_matches_streamed():
    """The LDOS loss's source (the electron rows, a table per column) through
    the adjoint in cluster registers against the streamed one."""
    p = lattice(28, 20, 0, 0, 90, seed=12)
    lat, ref = gpu_lattice(p, "fp32"), gpu_lattice(p, "fp32", resident=0)
    sites = np.array([0, 27, 300, 559, 300], dtype=np.int32)
    E = np.linspace(-2.0, 2.0, 9)
    G = np.random.default_rng(4).normal(size=(5, 9))
    for x, y in zip(lat.ldos_backward(sites, 90, E, G), ref.ldos_backward(sites, 90, E, G)):
        assert max_abs(x, y) <= 2e-5 * np.max(np.abs(y))
