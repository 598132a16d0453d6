"""Calls on either side of the lines between bytes, bit planes with a launch per
phase and masks drawn ahead (by sweeps, sites and lattices): the same chain as
twin handles held to the colour phases on bytes."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


def twins(dim, L, n_temps, n_real, seed=13):
    lats = [sp.Lattice(B.SPIN_ISING, dim, L, B.SPIN_I8, n_temps=n_temps, n_real=n_real, seed=seed) for _ in range(2)]
    lats[1].set_variant(0)
    return lats


@pytest.mark.parametrize("dim,L,n_temps,n_real,calls", [
    # 2D, L % 16 == 8: from 16, 6, 4, 3 and 2 sweeps by the sites of all lattices, never below
    (2, 136, 3, 9, (15, 40)), (2, 136, 3, 10, (15, 16)), (2, 200, 2, 9, (5, 6, 7)), (2, 264, 3, 5, (3, 4, 5)),
    (2, 520, 3, 3, (2, 3)), (2, 136, 5, 38, (1, 2, 3)), (2, 200, 8, 11, (1, 2, 5)), (2, 264, 6, 9, (2, 6)),
    (2, 1000, 2, 2, (2, 3)),
    # one CTA per lattice: few and many lattices, one and more per SM
    (2, 16, 2, 512, (31, 33)), (2, 16, 3, 400, (40,)), (2, 32, 2, 100, (22, 23, 48)), (2, 64, 2, 40, (8, 9, 12)),
    (2, 80, 3, 1000, (2, 3, 9)), (2, 128, 2, 60, (2, 3, 4, 5)), (2, 128, 3, 400, (2, 3, 9)), (3, 8, 2, 152, (26, 48)),
    (3, 8, 5, 61, (26, 48)), (3, 24, 2, 380, (2, 3, 5)), (3, 32, 2, 60, (2, 5, 6)), (3, 32, 2, 100, (2, 7))])
def test_both_sides_of_the_lines(dim, L, n_temps, n_real, calls):
    betas = [(0.4407 if dim == 2 else 0.2216544) * (1 + 0.02 * t) for t in range(n_temps)]
    lats = twins(dim, L, n_temps, n_real)
    acc = [torch.zeros(n_temps, dtype=torch.int64, device="cuda") for _ in lats]
    for n in calls:
        for me, pt in ((0, 0), (2, 3)):
            out = [lat.run(betas, n, measure_every=me, pt_every=pt, accepted=a) for lat, a in zip(lats, acc)]
            for key in out[0]:
                assert torch.equal(out[0][key], out[1][key]), (n, key)
            assert torch.equal(lats[0].spins, lats[1].spins), n
    assert torch.equal(acc[0], acc[1])
    for lat in lats:
        lat.sync()
        lat.close()


def test_extreme_thresholds_and_a_refused_exchange():
    betas = [0.0, 30.0, 0.3]
    lats = twins(2, 136, 3, 70)
    for lat in lats:
        lat.sweep(betas, 7)
    assert torch.equal(lats[0].spins, lats[1].spins)
    for lat in lats:  # adjacent betas too close for a table: the sweeps up to the exchange stand
        with pytest.raises(B.SpinError):
            lat.run([0.4, 0.4 + 1e-9, 0.5], 6, pt_every=3)
        lat.sync()
        assert lat.sweeps_done == 9
    assert torch.equal(lats[0].spins, lats[1].spins)
    for lat in lats:
        lat.close()
