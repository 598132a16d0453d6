"""Coded EA calls that keep the lattices in shared memory (several sweeps of
small lattices: full and partial slot blocks, row quads and single sites, one
and several rounds per thread, w = 64) against one spin per byte and against
calls of one sweep."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402

SHAPES = [(2, 4, 32, 1), (2, 6, 64, 5), (2, 8, 32, 3), (2, 16, 64, 9), (2, 30, 64, 4), (2, 64, 256, 30),
          (3, 4, 32, 2), (3, 6, 96, 5), (3, 8, 64, 6), (3, 10, 64, 4), (3, 12, 256, 7), (3, 14, 256, 30),
          (3, 16, 256, 30)]


@pytest.mark.parametrize("dim,L,n_real,T", SHAPES)
def test_long_calls_equal_bytes(dim, L, n_real, T):
    betas = [0.1 * t if t else 30.0 for t in range(T)]
    lats = [sp.Lattice(B.SPIN_EA, dim, L, layout, n_real=n_real, n_temps=T, n_sets=2, seed=5)
            for layout in (B.SPIN_MSC1, B.SPIN_I8)]
    for lat in lats:
        lat.sweep(betas, 16)
        lat.sweep(betas, 1)
        lat.sweep(betas, 5)
    assert torch.equal(lats[0].unpack().view(-1), lats[1].spins)
    for lat in lats:
        lat.sync()
        lat.close()


@pytest.mark.parametrize("dim,L", [(2, 14), (2, 32), (3, 6), (3, 8)])
@pytest.mark.parametrize("width", [32, 64])
def test_long_call_equals_single_sweeps(dim, L, width):
    """Past one launch's 1024 sweeps, with either number of spins per variable."""
    T, betas = 5, [0.3, 0.5, 0.7, 0.9, 1.1]
    lats = [sp.Lattice(B.SPIN_EA, dim, L, B.SPIN_MSC1, n_real=128, n_temps=T, n_sets=2, seed=6) for _ in range(2)]
    for lat in lats:
        if width == 64:
            lat.set_msc_width(64)
    lats[0].sweep(betas, 1030)
    for _ in range(515):
        lats[1].sweep(betas, 2)
    assert torch.equal(lats[0].spins, lats[1].spins)
    for lat in lats:
        lat.sync()
        lat.close()
