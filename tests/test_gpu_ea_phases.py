"""Calls of two sweeps and of several on coded EA lattices, enqueued back to back
(each kernel starts while the one before it still runs), at grids below and
above one CTA per SM, against one spin per byte."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("dim,L,groups,T", [(3, 8, 2, 33), (2, 40, 4, 16), (3, 16, 2, 5), (3, 10, 3, 6), (3, 18, 4, 4),
                                            (2, 30, 8, 5), (2, 60, 6, 3), (2, 16, 40, 5), (2, 32, 6, 33),
                                            (2, 40, 18, 33), (3, 12, 5, 33), (3, 16, 9, 16), (3, 16, 10, 16)])
def test_calls_back_to_back_equal_bytes(dim, L, groups, T):
    betas = [0.3 + 0.05 * t for t in range(T)]
    lats = [sp.Lattice(B.SPIN_EA, dim, L, layout, n_real=32 * groups, n_temps=T, n_sets=2, seed=6)
            for layout in (B.SPIN_MSC1, B.SPIN_I8)]
    for n in (2, 6, 2):
        for lat in lats:
            for _ in range(8):
                lat.sweep(betas, n)
        assert torch.equal(lats[0].unpack().view(-1), lats[1].spins)
    for lat in lats:
        lat.sync()
        lat.close()
