"""The column sums of the register-resident recursion, apart from the rounding
of its vectors: on a torus without disorder the FP32 vectors of all start sites
are translations of one another bit for bit, so the moments of different
start sites differ by the rounding of the sums alone.

Expected of sums with compensation: chains of eight products (on these lattices,
whose tiles have four or six rows, sixteen in some) round with 0.7 (0.9) * 2^-24 of
the chain each (root mean square), independently, and nothing else rounds.  From the 32nd step on (moment 64) the weight lies on the whole lattice, 500 sites
and more, in 63 chains at least: with amplitudes that vary by a factor of a few,
2 * 0.7 * 2^-24 * 0.25 = 2.1e-8 at most for a moment.  Sums that round once or more at their own
size (over the lanes of a warp, say) give 2 * 0.4 * 2^-24 * sqrt(2) = 6.7e-8 for the two
warps of these lattices."""
import numpy as np
import pytest

from paper_1007_1609_gb300 import workloads as wl
from tests._common import gpu_available
from tests.test_gpu_parity import gpu_lattice

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("Lx,Ly", [(24, 24), (23, 22), (40, 36), (25, 70)])
def test_sums_of_translated_vectors_agree(Lx, Ly):
    N, M = Lx * Ly, 300
    p = wl.Problem(name=f"t{Lx}x{Ly}", Lx=Lx, Ly=Ly, periodic_x=1, periodic_y=1, eps=np.full(N, 0.21), mu=-0.5,
                   hop=wl.square_hops(Lx, Ly, 1, 1), pairing=wl.ONSITE, coupling=2.0,
                   delta0=np.full(N, 0.43, dtype=np.complex128), T=0.02, M=M)
    lat = gpu_lattice(p, "fp32")
    ee, eh = lat.moments(np.arange(N, dtype=np.int32), M)
    assert lat.last_tile()[:2] == (1, 0)  # on chip
    for mu in (ee[:, 64::2], ee[:, 65::2], eh[..., 0].real[:, 65::2]):
        off = mu - mu.mean(axis=0)
        assert np.sqrt(np.mean(off ** 2)) < 2.1e-8, np.sqrt(np.mean(off ** 2))
