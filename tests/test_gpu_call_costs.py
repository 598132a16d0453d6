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


def test_masks_ahead_stay_out_of_many_tiny_lattices():
    lat = sp.Lattice(B.SPIN_ISING, 3, 8, B.SPIN_I8, n_temps=4, n_real=2432, seed=1)
    betas = [0.2, 0.21, 0.22, 0.23]
    whole = us(lambda: lat.sweep(betas, 96))
    parts = us(lambda: [lat.sweep(betas, 8) for _ in range(12)])
    assert whole < 1.2 * parts, (whole, parts)
    lat.sync()
    lat.close()


# lattices that wait for launches in either form, one whose phases are longer
@pytest.mark.parametrize("L,n_lat,n", [(136, 1, 3), (520, 1, 3), (440, 3, 2), (1000, 1, 2), (1000, 3, 2), (1000, 3, 4),
                                       (264, 20, 2), (184, 20, 20)])
def test_conversions_pay(L, n_lat, n):
    lats = [sp.Lattice(B.SPIN_ISING, 2, L, B.SPIN_I8, n_real=n_lat, seed=1) for _ in range(2)]
    lats[1].set_variant(0)
    auto, phases = (us(lambda lat=lat: lat.sweep([0.4], n)) for lat in lats)
    assert auto < 1.12 * phases, (auto, phases)
    for lat in lats:
        lat.sync()
        lat.close()


@pytest.mark.parametrize("dim,L,n_lat", [(3, 32, 200), (3, 24, 600), (2, 128, 1216)])
def test_measuring_after_every_sweep_costs_little(dim, L, n_lat):
    """Large lattices, too many for the masks of many sweeps: a call that measures
    often still takes the form that measures in place."""
    lat = sp.Lattice(B.SPIN_ISING, dim, L, B.SPIN_I8, n_real=n_lat, seed=1)
    series = lat.series_buffers(30)

    def run(every):
        B.spin_run(lat.h, None, [0.3], 30, every, 0, *((series["E"], series["M"]) if every else (None, None)), None, None,
                   None, None, None)

    plain, measured = us(lambda: run(0)), us(lambda: run(1))
    assert measured < 1.6 * plain, (plain, measured)
    lat.sync()
    lat.close()
