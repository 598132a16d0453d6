"""Coded EA lattices with L % 8 != 0 (lanes take consecutive sites: last quads
that are not full, slot blocks that are not full, fewer sites than a warp)
against one spin per byte, and the batched launch against per-handle runs."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("dim,L,n_real,T", [(2, 4, 32, 2), (2, 6, 32, 3), (2, 10, 64, 5), (2, 14, 32, 1), (2, 18, 32, 9),
                                            (3, 4, 32, 2), (3, 6, 96, 5), (3, 10, 32, 7), (3, 12, 64, 6), (3, 14, 32, 4)])
def test_sites_equal_bytes(dim, L, n_real, T):
    betas = [0.0, 30.0, 0.7, 0.9, 0.5, 1.1, 1.3, 0.2, 0.4][:T]
    lats = [sp.Lattice(B.SPIN_EA, dim, L, layout, n_real=n_real, n_temps=T, n_sets=2, seed=7)
            for layout in (B.SPIN_MSC1, B.SPIN_I8)]
    for n in (1, 4):
        for lat in lats:
            lat.sweep(betas, n)
        assert torch.equal(lats[0].unpack().view(-1), lats[1].spins)
    for lat in lats:
        lat.sync()
        lat.close()


@pytest.mark.parametrize("L,n_real,T", [(4, 32, 8), (6, 64, 5), (10, 32, 33), (12, 96, 6), (14, 32, 3), (20, 32, 2)])
def test_batched_sites_equal_per_handle_runs(L, n_real, T):
    betas = [0.6 + 0.05 * t for t in range(T)]
    lats = [sp.Lattice(B.SPIN_EA, 3, L, B.SPIN_MSC1, n_real=n_real, n_temps=T, n_sets=2, seed=9) for _ in range(2)]
    for n, me, pt in ((3, 1, 1), (4, 2, 0), (2, 0, 0)):
        ref = lats[0].run(betas, n, measure_every=me, pt_every=pt)
        ser = lats[1].series_buffers(B._n_meas(lats[1].h, n, me)) if me else None
        sp.batch_run([lats[1].batch_item(betas, ser)], n, me, pt)
        for key in ref:
            assert torch.equal(ref[key], ser[key]), key
        assert torch.equal(lats[0].spins, lats[1].spins)
    for lat in lats:
        lat.sync()
        lat.close()
