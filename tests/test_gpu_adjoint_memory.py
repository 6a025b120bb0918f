"""The on-chip adjoint in little memory: with a workspace cap it runs as many
clusters as fit, or hands over to the streamed adjoint; with most of the device's memory
taken by someone else the call still answers.  Gradients agree within the
FP32 tolerance of the two adjoints (2e-5 of the largest component)."""
import numpy as np
import pytest

from paper_1007_1609_gb300 import cbdg
from tests._common import gpu_available, max_abs
from tests.test_gpu_cluster import lattice
from tests.test_gpu_parity import gpu_lattice

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


def gradient(lat, p, w):
    cbdg.cbdg_launch_count(lat.handle, reset=True)
    g = lat.backward(p.T, p.M, w)
    return g, cbdg.cbdg_launch_count(lat.handle)


def agree(a, b):
    return all(max_abs(x, y) <= 2e-5 * np.max(np.abs(y)) for x, y in zip(a, b))


@pytest.mark.parametrize("shape", [(64, 64, 0, 0, 100), (40, 72, 0, 1, 65)])
def test_workspace_caps_choose_the_clusters(shape):
    Lx, Ly, px, py, M = shape
    p = lattice(Lx, Ly, px, py, M, seed=3)
    w = np.random.default_rng(1).normal(size=p.N).astype(np.complex128)
    ref, on_chip = gradient(gpu_lattice(p, "fp32"), p, w)
    assert on_chip < 12  # one recursion launch
    routes = set()
    for mb in (1000, 600, 400, 300, 200, 150, 100, 70, 50, 30, 20):
        g, launches = gradient(gpu_lattice(p, "fp32", workspace_mb=mb), p, w)
        assert agree(g, ref), mb
        routes.add(launches < 12)
    assert routes == {True, False}


def test_gradient_with_little_free_memory():
    torch = pytest.importorskip("torch")
    p = lattice(64, 64, 0, 0, 512, seed=4)
    w = np.random.default_rng(2).normal(size=p.N).astype(np.complex128)
    ref, _ = gradient(gpu_lattice(p, "fp32"), p, w)
    lat = gpu_lattice(p, "fp32")
    lat.order_parameter(p.T, 2)  # its small buffers
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    taken = torch.empty(free - (400 << 20), dtype=torch.uint8, device="cuda")
    try:
        g, _ = gradient(lat, p, w)
    finally:
        del taken
        torch.cuda.empty_cache()
    assert agree(g, ref)
