"""Coded 2D lattices with one to three lattices per thread of the phase
kernel, groups that are not full and a last CTA that is partly empty, with slots whose thresholds are the extremes (beta = 0 and a beta
whose thresholds are 0), against int8 handles swept by the fused pass."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("L,n_lat", [(256, 1), (768, 2), (5888, 1), (4096, 2), (4096, 3), (3072, 4), (3072, 5), (2560, 7)])
def test_coded_phase_equals_the_int8_sweep(L, n_lat):
    betas = [[0.4407, 0.0, 30.0, 0.3, 0.5, 1.0, 0.4][k] for k in range(n_lat)]
    coded = sp.Lattice(B.SPIN_ISING, 2, L, B.SPIN_MSC1, n_temps=n_lat, seed=9)
    i8 = sp.Lattice(B.SPIN_ISING, 2, L, B.SPIN_I8, n_temps=n_lat, seed=9)
    i8.set_variant(1)
    for n in (1, 2):
        coded.sweep(betas, n)
        i8.sweep(betas, n)
    coded.sync()
    i8.sync()
    assert torch.equal(coded.unpack().view(-1), i8.spins)
    coded.close()
    i8.close()
