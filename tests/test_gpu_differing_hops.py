"""The kernels that lattices with differing hoppings, or with RESIDENT = 0, still
run: the streaming kernel of ensembles (one and two sites per thread, every
remainder of its three-step passes), the shared-memory recursion in both
precisions, and the FP32 adjoint's multi-step passes.  The tests of those
kernels in test_gpu_ensemble.py, test_gpu_resident.py and test_gpu_adjoint.py hold one hopping, which
the kernels in cluster registers now take.  Same shapes and tolerances."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1007_1609_gb300 import cbdg
from tests._common import as_oracle, gpu_available, max_abs
from tests.test_gpu_adjoint import rect_swave, rel
from tests.test_gpu_parity import K, TOL, gpu_lattice, rect

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


def one_weak_bond(p, t=0.9):
    """The same lattice with one hopping changed, near its middle."""
    x, y = (p.Lx - 1) // 2, (p.Ly - 1) // 2
    d = 0 if p.Lx > 1 else 2
    i = x + p.Lx * y
    j = i + (1 if d == 0 else p.Lx)
    p.hop = p.hop.copy()
    p.hop[i, d] = p.hop[j, d ^ 1] = t
    return p


@pytest.mark.parametrize("shapes", [[(96, 5), (5, 96), (70, 2), (13, 1), (33, 17), (1, 40)], [(64, 7), (5, 33), (40, 2), (9, 1)]])
@pytest.mark.parametrize("M", [64, 66, 68])
def test_ensemble_streaming_kernel(M, shapes):
    probs = [one_weak_bond(rect(lx, ly, M, seed=lx * 31 + ly + M, periodic=0)) for lx, ly in shapes]
    ens = cbdg.Ensemble(probs)
    ens.set_option(cbdg.CBDG_OPT_QUADRATURE_NODES, K)
    _, it, _ = ens.scf(0.02, M, 0.5, 0.0, 1)
    assert it == 1
    for s, p in enumerate(probs):
        ol = as_oracle(p)
        od, _ = orc.order_parameter(ol, orc.rescale(ol), p.T, M, K)
        assert max_abs(2 * ens.delta(s) - p.delta0, od) < 1e-5, p.name
    ens.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("Lx,Ly,M,periodic", [(16, 16, 256, 0), (7, 5, 33, 0), (6, 9, 64, 1), (1, 12, 20, 0), (13, 1, 21, 0),
                                              (40, 24, 48, 0), (48, 48, 64, 0)])
def test_shared_memory_recursion(Lx, Ly, M, periodic, precision):
    p = one_weak_bond(rect(Lx, Ly, M, seed=Lx + Ly, periodic=periodic))
    sites = np.arange(p.N, dtype=np.int32)
    lat = gpu_lattice(p, precision)
    ee, eh = lat.moments(sites, M)
    assert lat.last_tile()[1] == 0  # on chip
    oee, oeh = orc.moments(as_oracle(p), lat.rescale, sites, M)
    assert max_abs(ee, oee) < TOL[precision][0] and max_abs(eh, oeh) < TOL[precision][0]
    d, n = lat.order_parameter(p.T, M)  # the linear fold
    assert lat.last_tile()[1] == 0
    od, on = orc.order_parameter(as_oracle(p), lat.rescale, p.T, M, K)
    assert max_abs(d, od) < TOL[precision][1] and max_abs(n, on) < TOL[precision][1]


@pytest.mark.parametrize("route", ["resident0", "weak_bond"])
@pytest.mark.parametrize("Lx,Ly,M", [(20, 13, 40), (70, 9, 64), (33, 17, 101), (16, 40, 50), (128, 3, 23)])
def test_adjoint_multi_step_passes(Lx, Ly, M, route):
    p = rect_swave(Lx, Ly, M, seed=Lx + Ly + M)
    if route == "weak_bond":
        one_weak_bond(p)
    w = np.random.default_rng(M).normal(size=p.N)
    out, launches = {}, {}
    for steps in (0, 1):
        lat = gpu_lattice(p, "fp32", resident=0 if route == "resident0" else 1, temporal_steps=steps)
        cbdg.cbdg_launch_count(lat.handle, reset=True)
        out[steps] = lat.backward(p.T, M, w.astype(np.complex128))
        launches[steps] = cbdg.cbdg_launch_count(lat.handle)
        a = lat.rescale
        lat.close()
    assert M < launches[0] < launches[1]  # streamed, several steps per pass
    oe, oh, od = orc.scf_map_gradient(as_oracle(p), a, orc.fold_coefficients(M, K, a, p.T), w)
    ge, gh, gd = out[0]
    assert rel(ge, oe) < 1e-3 and rel(gh.real, oh) < 1e-3 and rel(gd.real, od) < 1e-3
    for x, y in zip(out[0], out[1]):
        assert rel(x, y) < 2e-5
