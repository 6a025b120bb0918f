"""The on-chip adjoint is no further from the FP64 gradient than the streamed
adjoint, whose sums are compensated and whose vectors are the forward ones:
the root mean square distances, relative to each other, in the geometric mean
over shapes and inputs (one gradient alone varies by a fifth either way, with the
rounding of its matrix)."""
import numpy as np
import pytest

from paper_1007_1609_gb300 import cbdg
from tests._common import gpu_available
from tests.test_gpu_cluster import lattice
from tests.test_gpu_parity import gpu_lattice

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]

SHAPES = [(64, 64, 0, 0, 512), (47, 20, 0, 1, 152), (25, 38, 0, 0, 367), (30, 51, 0, 0, 369), (44, 28, 1, 1, 380),
          (52, 40, 1, 0, 260)]


def test_distance_from_fp64_is_not_larger_than_streamed():
    ratios = []
    for k, (Lx, Ly, px, py, M) in enumerate(SHAPES):
        for seed in (20 + k, 40 + k):
            p = lattice(Lx, Ly, px, py, M, seed=seed)
            w = (0.2 + 0.1 * np.random.default_rng(seed).normal(size=p.N)).astype(np.complex128)
            exact = gpu_lattice(p, "fp64").backward(p.T, M, w)
            lat = gpu_lattice(p, "fp32")
            cbdg.cbdg_launch_count(lat.handle, reset=True)
            here = lat.backward(p.T, M, w)
            assert cbdg.cbdg_launch_count(lat.handle) < 12  # on chip
            there = gpu_lattice(p, "fp32", resident=0).backward(p.T, M, w)
            ratios.append([np.linalg.norm(a - x) / np.linalg.norm(b - x) for x, a, b in zip(exact, here, there)])
    mean = np.exp(np.mean(np.log(ratios), axis=0))
    assert (mean <= 1.0).all(), mean
