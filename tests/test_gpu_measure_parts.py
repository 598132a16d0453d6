"""E, M and Q of coded EA word-lattices at the sizes where the threads and parts
of a word-lattice change, against one spin per byte."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


# few and many word-lattices (n_real / 32 * T * 2) on both sides of 1024, 4096
# and 16384 sites; parts raised for few word-lattices, whole and partly filled
@pytest.mark.parametrize("dim,L,n_real,T", [
    (3, 10, 32, 2), (2, 32, 128, 100), (2, 34, 32, 3), (3, 12, 128, 94), (3, 12, 128, 96), (3, 16, 128, 96),
    (3, 16, 128, 160), (2, 66, 32, 400), (2, 128, 32, 3), (2, 130, 32, 1), (3, 18, 32, 2), (3, 22, 32, 2), (3, 22, 96, 16), (3, 26, 32, 2), (3, 28, 64, 32), (2, 130, 32, 400),
    (3, 32, 32, 1)])
def test_counts_equal_bytes(dim, L, n_real, T):
    coded = sp.Lattice(B.SPIN_EA, dim, L, B.SPIN_MSC1, n_real=n_real, n_temps=T, n_sets=2, seed=4)
    i8 = sp.Lattice(B.SPIN_EA, dim, L, B.SPIN_I8, n_real=n_real, n_temps=T, n_sets=2, seed=4)
    coded.sweep([0.8] * T, 1)
    i8.spins.copy_(coded.unpack().view(-1))
    for x, y in zip(coded.measure(), i8.measure()):
        assert torch.equal(x, y)
    # the energy alone, in more parts from 4097 sites on
    E = [torch.full((lat.n_lat,), 7, dtype=torch.int64, device="cuda") for lat in (coded, i8)]
    for lat, e in zip((coded, i8), E):
        B.spin_measure(lat.h, lat.couplings, E=e)
    assert torch.equal(*E)
    for lat in (coded, i8):
        lat.sync()
        lat.close()
