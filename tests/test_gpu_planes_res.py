"""Small int8 ferromagnets with one CTA per lattice on bit planes and masks
drawn ahead (one, two and four words per thread, row groups whose last is
smaller, more rows than are kept before they are written, more sweeps than
the tape holds) against twin handles held to the in-place colour phases."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("dim,L,n_temps,n_real,long", [
    (2, 8, 3, 2, 70), (2, 16, 2, 1, 40), (2, 24, 5, 1, 40), (2, 32, 20, 1, 40), (2, 40, 3, 3, 33), (2, 64, 1, 1, 100),
    (2, 72, 4, 1, 40), (2, 120, 3, 1, 40), (2, 128, 40, 1, 250), (3, 8, 4, 2, 40), (3, 16, 3, 1, 70), (3, 24, 2, 2, 40),
    (3, 32, 3, 1, 40), (3, 40, 2, 1, 40), (3, 48, 1, 1, 40)])
def test_resident_planes_equal_the_colour_phases(dim, L, n_temps, n_real, long):
    beta = 0.4407 if dim == 2 else 0.2216544
    betas = [beta * (1 + 0.02 * t) for t in range(n_temps)]
    if n_temps > 3:
        betas[-1], betas[0] = 30.0, 0.0
    lats = [sp.Lattice(B.SPIN_ISING, dim, L, B.SPIN_I8, n_temps=n_temps, n_real=n_real, seed=6) for _ in range(2)]
    lats[1].set_variant(0)
    acc = [torch.zeros(n_temps, dtype=torch.int64, device="cuda") for _ in lats]
    lab = [lat.slot_labels() for lat in lats]
    for n, me, pt in ((5, 0, 0), (13, 2, 3), (long, 1, 0), (3, 1, 1), (20, 0, 4), (long, 7, 10)):
        out = [lat.run(betas, n, measure_every=me, pt_every=pt, accepted=a, labels=l)
               for lat, a, l in zip(lats, acc, lab)]
        for key in out[0]:
            assert torch.equal(out[0][key], out[1][key]), (n, key)
        assert torch.equal(lats[0].spins, lats[1].spins), n
        assert torch.equal(acc[0], acc[1]) and torch.equal(lab[0], lab[1]), n
    for lat in lats:
        lat.sync()
        lat.close()
