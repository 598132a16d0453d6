"""Heisenberg sums whose partials are shared by clusters of 2, 4 and 8 CTAs, taken
again and again while another stream keeps the SMs busy (so that the CTAs of a
cluster start and finish at different times): the same bits every time, and
those of the allocation-free entry point."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("dim,L,n_lat", [(2, 726, 3), (3, 82, 3), (2, 1026, 2), (3, 102, 2), (2, 1450, 2), (3, 128, 2)])
def test_sums_do_not_depend_on_what_else_runs(dim, L, n_lat):
    lat = sp.Lattice(B.SPIN_HEISENBERG, dim, L, B.SPIN_F32X4, n_temps=n_lat, seed=L)
    other = torch.cuda.Stream()
    load = sp.Lattice(B.SPIN_HEISENBERG, 2, 260, B.SPIN_F32X4, seed=1, stream=other)
    E0, M0 = lat.measure()
    lat.sync()
    got = []
    for k in range(30):
        load.sweep([1.0], 1 + k % 3)
        got.append(lat.measure())
        E, M = torch.empty_like(E0), torch.empty_like(M0).view(-1)
        B.spin_heis_measure_noalloc(lat.spins, dim, L, n_lat, E, M, torch.cuda.current_stream().cuda_stream)
        got.append((E, M.view(n_lat, 3)))
    torch.cuda.synchronize()
    for E, M in got:
        assert torch.equal(E, E0) and torch.equal(M, M0)
    lat.close()
    load.close()
