"""The contraction of gf1 on the tensor cores (M >= 64) against NumPy on the
moments that green_moments returns: every edge of its tiles (64 rows, 32
energies, K-blocks of 64 moments), rows of very different size, more rows and more
energies than one set of digit planes holds, and the FP64 kernel's side of
the rule.  Tolerance per output: both sides form w_n = .. exp(-i n arccos x) in
FP64, a phase rounded to n pi 2^-53 twice over, times a few roundings of the rest: 2^-52
sum_n (8 + 2 pi n) |a_n| |w_n| covers them, and NumPy's own sum (64 2^-53 of
the same sum)."""
import numpy as np
import pytest

from paper_1007_1609_gb300 import cbdg
from paper_1007_1609_gb300 import workloads as wl
from tests._common import gpu_available

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


def check(lat, sites, targets, M, E):
    G = lat.green_function(sites, targets, M, E)
    a = lat.green_moments(sites, targets, M)
    n = np.arange(M)
    x = (E / lat.rescale)[:, None]
    q = 1.0 / (M + 1.0)
    g = q * ((M - n + 1) * np.cos(np.pi * n * q) + np.sin(np.pi * n * q) / np.tan(np.pi * q))
    w = -2j * g * np.where(n == 0, 0.5, 1.0) * np.exp(-1j * n * np.arccos(x)) / (lat.rescale * np.sqrt(1.0 - x * x))
    c = 2.0**-52 * (64 + 8 + 2 * np.pi * n)
    for got, mom in zip(G, a):
        ref = np.einsum("smt,em->ste", mom, w, optimize=True)
        assert np.all(np.abs(got - ref) <= np.einsum("smt,em->ste", np.abs(mom), c * np.abs(w), optimize=True) + 1e-300)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n_s,n_t,M,n_E", [(1, 1, 64, 1), (3, 21, 65, 31), (5, 13, 128, 33), (2, 32, 129, 64), (64, 1, 127, 65),
                                           (1, 130, 192, 3), (7, 5, 63, 9)])
def test_contraction(precision, n_s, n_t, M, n_E):
    p = wl.random_dwave(12, M, seed=51, tp=-0.3)
    rng = np.random.default_rng(n_t)
    lat = cbdg.Lattice(p, precision=precision, complex_field=True)
    check(lat, rng.integers(0, p.N, n_s), rng.integers(0, p.N, n_t), M, rng.uniform(-0.99, 0.99, n_E) * lat.rescale)


def test_small_rows():
    """Distant targets of an open chain: rows whose entries stay zero for most of the
    recursion, beside the start site's row."""
    p = wl.random_swave(14, 64, seed=52, complex_delta=True)
    lat = cbdg.Lattice(p, precision="fp64", complex_field=True)
    targets = np.arange(0, p.N, 3)
    check(lat, np.array([0, p.N - 1]), targets, 64, np.linspace(-0.9, 0.9, 40) * lat.rescale)


@pytest.mark.parametrize("n_s,n_t,M,n_E", [(600, 230, 64, 2), (1, 3, 128, 66000), (1, 3, 64, 17000)])
def test_more_than_one_set_of_planes(n_s, n_t, M, n_E):
    """(the last one: the FP64 kernel)"""
    p = wl.random_dwave(16, M, seed=53)
    rng = np.random.default_rng(1)
    lat = cbdg.Lattice(p, precision="fp32", complex_field=True)
    check(lat, rng.integers(0, p.N, n_s), rng.integers(0, p.N, n_t), M, rng.uniform(-0.99, 0.99, n_E) * lat.rescale)
