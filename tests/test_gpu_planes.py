"""Longer calls of int8 ferromagnets on bit planes (one or several rows per
block, pieces and row groups whose last is smaller, one to three lattices per
thread) against twin handles held to the in-place colour phases: lattices,
series, exchanges and labels, over calls of several lengths and schedules.  (2D
handles of few sites stay on bytes; test_gpu_planes_routes.py has the narrow
planes of those sizes, with more lattices.)"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


def twin(dim, L, n_temps, n_real, seed):
    lats = [sp.Lattice(B.SPIN_ISING, dim, L, B.SPIN_I8, n_temps=n_temps, n_real=n_real, seed=seed) for _ in range(2)]
    lats[1].set_variant(0)
    return lats


@pytest.mark.parametrize("dim,L,n_temps,n_real", [
    (2, 136, 3, 2), (2, 200, 1, 1), (2, 264, 2, 1), (2, 520, 5, 1), (2, 1000, 3, 1), (2, 512, 4, 1), (2, 2056, 40, 1),
    (3, 32, 4, 1), (3, 40, 3, 1), (3, 48, 1, 2), (3, 56, 1, 1), (3, 72, 2, 1), (3, 80, 3, 1), (3, 96, 1, 1),
    (3, 104, 1, 1), (3, 128, 1, 1), (3, 136, 2, 1), (3, 264, 1, 1), (3, 192, 5, 1),
    (2, 4096, 1, 1), (2, 4112, 1, 1), (2, 2832, 3, 1)])
def test_planes_equal_the_colour_phases(dim, L, n_temps, n_real):
    beta = 0.4407 if dim == 2 else 0.2216544
    betas = [beta * (1 + 0.02 * t) for t in range(n_temps)]
    lats = twin(dim, L, n_temps, n_real, 5)
    acc = [torch.zeros(n_temps, dtype=torch.int64, device="cuda") for _ in lats]
    lab = [lat.slot_labels() for lat in lats]
    for n, me, pt in ((1, 0, 0), (5, 0, 0), (6, 2, 3), (5, 1, 0), (4, 0, 2)):
        out = [lat.run(betas, n, measure_every=me, pt_every=pt, accepted=a, labels=l)
               for lat, a, l in zip(lats, acc, lab)]
        for key in out[0]:
            assert torch.equal(out[0][key], out[1][key]), key
        assert torch.equal(lats[0].spins, lats[1].spins)
    assert torch.equal(acc[0], acc[1]) and torch.equal(lab[0], lab[1])
    for lat in lats:
        lat.sync()
        lat.close()


@pytest.mark.parametrize("dim,L", [(2, 136), (3, 40)])
def test_planes_at_extreme_thresholds(dim, L):
    betas = [0.0, 30.0, 0.3]
    lats = twin(dim, L, 3, 1, 8)
    for lat in lats:
        lat.sweep(betas, 7)
    assert torch.equal(lats[0].spins, lats[1].spins)
    for lat in lats:
        lat.sync()
        lat.close()


def test_planes_stop_at_a_bad_exchange_table():
    """Adjacent betas too close for an exchange table: the sweeps up to the
    refused exchange stand, in the caller's bytes too."""
    betas = [0.4, 0.4 + 1e-9]
    lats = twin(2, 136, 2, 1, 3)
    for lat in lats:
        with pytest.raises(B.SpinError):
            lat.run(betas, 6, pt_every=3)
        lat.sync()
        assert lat.sweeps_done == 3
    assert torch.equal(lats[0].spins, lats[1].spins)
    for lat in lats:
        lat.close()
