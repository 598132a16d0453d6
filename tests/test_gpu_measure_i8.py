"""Energy and magnetisation of int8 lattices from random configurations, at
the edges of the counting kernels' tiles (rows of 1 to many 8-byte chunks, a
last tile or segment that is partly empty, L that is no multiple of 8),
against the oracle's sums."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("dim,L,n_lat", [(2, 8, 3), (2, 24, 1), (2, 26, 2), (2, 136, 5), (2, 520, 2), (2, 1000, 3),
                                         (3, 8, 2), (3, 10, 2), (3, 24, 1), (3, 40, 3), (3, 72, 1), (3, 136, 1)])
def test_i8_energy_and_magnetisation(dim, L, n_lat):
    rng = np.random.default_rng(L)
    s = (1 - 2 * (rng.random((n_lat, L ** dim)) < 0.3)).astype(np.int8)
    s[0, -1] = s[0, 0] = -1  # bonds across the periodic boundary
    lat = sp.Lattice(B.SPIN_ISING, dim, L, B.SPIN_I8, n_temps=n_lat, seed=3)
    lat.pack(torch.from_numpy(s).cuda())
    E, M, _ = lat.measure()
    lat.sync()
    assert [int(v) for v in E.cpu()] == [oracle.ising_energy(dim, L, s[k]) for k in range(n_lat)]
    assert [int(v) for v in M.cpu()] == [int(s[k].sum()) for k in range(n_lat)]
    lat.close()
