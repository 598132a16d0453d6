"""Double checkerboard of the 2D int8 ferromagnet with the tiles as bits in
registers: lattices just large enough for each form (4 or 16 rows per thread,
1 to 32 lanes per tile), hits that are no multiple of the three drawn
together, both compound orders and extreme thresholds, against the oracle on
the lattice that the rest of the batch surrounds."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from graph_kernels import kernels  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


# n_lat L^2 / 512 >= 49152 takes the wide forms, >= 8192 (6144 at T = 8) the narrow ones
@pytest.mark.parametrize("T,L,n_lat,hits,order", [
    (8, 256, 48, 5, B.SPIN_ORDER_DCB), (8, 272, 80, 3, B.SPIN_ORDER_DCB_SYMMETRIC),
    (16, 256, 64, 4, B.SPIN_ORDER_DCB), (16, 512, 96, 1, B.SPIN_ORDER_DCB_SYMMETRIC), (16, 288, 310, 5, B.SPIN_ORDER_DCB),
    (32, 256, 64, 2, B.SPIN_ORDER_DCB), (32, 320, 250, 4, B.SPIN_ORDER_DCB_SYMMETRIC),
    (64, 256, 64, 7, B.SPIN_ORDER_DCB), (64, 384, 180, 3, B.SPIN_ORDER_DCB_SYMMETRIC)])
def test_bit_tiles_equal_the_oracle(T, L, n_lat, hits, order):
    betas = [0.4407] * n_lat
    betas[0], betas[1], betas[2] = 0.0, 30.0, 0.5
    lat = sp.Lattice(B.SPIN_ISING, 2, L, B.SPIN_I8, n_temps=n_lat, seed=17)
    lat.set_update_order(order, T, hits)
    lat.sweep(betas, 2 * hits)
    lat.sync()
    got = lat.spins.cpu().numpy().reshape(n_lat, -1)
    for t in (0, 1, 2, n_lat - 1):
        lid = oracle.lattice_id(0, 0, t)
        s = oracle.ising_init(2, L, 17, lid)
        oracle.dcb_sweeps(L, s, betas[t], 17, lid, 0, 2 * hits, T, hits, symmetric=order == B.SPIN_ORDER_DCB_SYMMETRIC)
        assert np.array_equal(got[t], s.ravel()), t
    lat.close()


# n_lat L^2 / 512 on both sides of 6144, 8192 and 13500
@pytest.mark.parametrize("T,L,n_lat,bits", [(8, 256, 47, False), (8, 256, 48, True), (16, 256, 63, False),
                                            (32, 256, 64, True), (64, 384, 46, False), (64, 384, 47, True)])
def test_form_and_equal_to_the_oracle_at_the_line(T, L, n_lat, bits, tmp_path):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        lat = sp.Lattice(B.SPIN_ISING, 2, L, B.SPIN_I8, n_temps=n_lat, seed=19)
        lat.set_update_order(B.SPIN_ORDER_DCB, T, 2)
        betas = [0.4407] * n_lat
        lat.sweep(betas, 2)
        lat.sync()
        got = lat.spins.cpu().numpy().reshape(n_lat, -1)[n_lat - 1]
        lid = oracle.lattice_id(0, 0, n_lat - 1)
        s = oracle.ising_init(2, L, 19, lid)
        oracle.dcb_sweeps(L, s, 0.4407, 19, lid, 0, 2, T, 2, symmetric=False)
        assert np.array_equal(got, s.ravel())
        names = kernels(torch, stream, lambda: lat.sweep(betas, 2), tmp_path / "graph.dot")
        assert any("dcb_bits" in name for name in names) == bits, names
        lat.close()
