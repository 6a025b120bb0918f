"""The Fermi coefficients by residues of the moment number (any K a multiple of
64) and node by node (other K), seen through the FP64 order parameter of a
3 x 4 lattice against the oracle: fewer nodes than one block takes, several
blocks, the last one partly filled; fewer moments than residues, every
residue, more turns than one pass of the block holds."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1007_1609_gb300 import cbdg
from tests._common import as_oracle, gpu_available, max_abs
from tests.test_gpu_parity import TOL, rect

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("nodes", [64, 512, 4096 + 192, 16384, 1040, 16399])
@pytest.mark.parametrize("M", [2, 3, 64, 129, 130, 4200])
def test_coefficients_match_oracle(M, nodes):
    p = rect(3, 4, M, seed=3, periodic=0)
    lat = cbdg.Lattice(p, precision="fp64")
    lat.set_option(cbdg.CBDG_OPT_QUADRATURE_NODES, nodes)
    for T in (0.0, 0.02):
        if T == 0.0 and nodes % 2:
            # the middle node is x = 0, where the library takes sign(x) = 0 and
            # the oracle the sign of a rounded cos(pi / 2): not the same sum
            continue
        for kernel, lam in (("jackson", 0.0), ("lorentz", 3.0)):
            d, n = lat.order_parameter(T, M, kernel=kernel, lam=lam)
            od, on = orc.order_parameter(as_oracle(p), lat.rescale, T, M, nodes, cbdg.KERNELS[kernel], lam)
            assert max_abs(d, od) < TOL["fp64"][1] and max_abs(n, on) < TOL["fp64"][1]
