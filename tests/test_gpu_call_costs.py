"""A call takes about as long as its sweeps in shorter calls would at most: the
forms that prepare something for a whole call (masks drawn ahead, conversions)
are taken only where that pays, for few lattices and for many."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


def us(f):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    f()
    best = 1e30
    for _ in range(8):
        a.record()
        for _ in range(4):
            f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 250.0)
    return best


# a CTA per lattice with one or two lattices per SM, where its CTAs and those
# that draw its masks must not wait for one another
@pytest.mark.parametrize("L,n_lat,n,part", [(64, 152, 16, 8), (64, 152, 32, 8), (16, 304, 32, 8), (32, 304, 24, 8),
                                            (48, 200, 16, 4), (128, 100, 8, 2)])
def test_masks_ahead_pay_at_one_or_two_lattices_per_sm(L, n_lat, n, part):
    lat = sp.Lattice(B.SPIN_ISING, 2, L, B.SPIN_I8, n_real=n_lat, seed=1)
    whole = us(lambda: lat.sweep([0.4], n))
    parts = us(lambda: [lat.sweep([0.4], part) for _ in range(n // part)])
    assert whole < 1.2 * parts, (whole, parts)
    lat.sync()
    lat.close()
