"""The forms that prepare something for a whole call (masks drawn ahead,
conversions to bit planes) are taken only where that pays, for few lattices and
for many: the kernels that a call enqueues at sizes on either side, where the
other form was measured to be at least an eighth slower."""
import pytest

from tests.graph_kernels import kernels

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402

BYTES, PHASES, AHEAD = "bytes", "planes_phase_kernel", "planes_res_kernel"


def form(tmp_path, dim, L, n_temps, n_real, n, measure=0, swaps=0):
    s = torch.cuda.Stream()
    lat = sp.Lattice(B.SPIN_ISING, dim, L, B.SPIN_I8, n_temps=n_temps, n_real=n_real, seed=1, stream=s)
    betas = [0.3 + 0.01 * t for t in range(n_temps)]
    series = lat.series_buffers(n)
    out = (series["E"], series["M"]) if measure else (None, None)
    acc = torch.zeros(n_temps, dtype=torch.int64, device="cuda")

    def call():
        B.spin_run(lat.h, None, betas, n, measure, swaps, *out, None, None, None, acc if swaps else None, None)

    torch.cuda.synchronize()
    call()
    if swaps:  # (the tables are uploaded at a call's first exchange)
        call()
    lat.sync()
    names = kernels(torch, s, call, tmp_path / "graph.dot")
    lat.close()
    got = [k for k in (PHASES, AHEAD) if k in names]
    assert len(got) <= 1, names
    return got[0] if got else BYTES


@pytest.mark.parametrize("L,n_lat,n,want", [
    # both forms wait for launches; a launch per phase is enough work; in between
    (136, 1, 3, BYTES), (136, 1, 60, BYTES), (520, 1, 3, BYTES), (440, 3, 2, BYTES), (1000, 1, 2, BYTES), (1000, 3, 2, BYTES),
    (264, 20, 2, BYTES), (184, 20, 20, PHASES), (1000, 1, 6, PHASES), (1000, 3, 4, PHASES), (2008, 3, 2, PHASES),
    (1000, 20, 2, PHASES), (144, 1, 4, PHASES), (512, 20, 4, PHASES)])
def test_conversions(tmp_path, L, n_lat, n, want):
    assert form(tmp_path, 2, L, 1, n_lat, n) == want


@pytest.mark.parametrize("dim,L,n_temps,n_real,n,measure,swaps,want", [
    # few lattices: by the sweeps
    (2, 64, 1, 1, 4, 0, 0, BYTES), (2, 64, 1, 1, 32, 0, 0, AHEAD), (2, 128, 20, 1, 4, 0, 0, AHEAD), (3, 16, 1, 20, 32, 0, 0, AHEAD),
    # many tiny ones: bytes, but with exchanges or measurements in the call
    (3, 8, 4, 2432, 96, 0, 0, BYTES), (3, 8, 4, 2432, 33, 0, 8, AHEAD), (2, 16, 4, 2432, 100, 0, 0, BYTES),
    (2, 16, 4, 2432, 33, 0, 8, AHEAD), (2, 24, 4, 2432, 32, 0, 0, AHEAD), (2, 64, 1, 2432, 32, 0, 0, AHEAD),
    # many large ones: phases, but with frequent measurements
    (2, 128, 4, 512, 32, 0, 0, PHASES), (2, 128, 4, 512, 30, 1, 0, AHEAD), (2, 128, 1, 304, 32, 0, 0, AHEAD),
    (3, 32, 1, 452, 30, 0, 0, PHASES), (3, 32, 1, 452, 30, 1, 0, AHEAD), (3, 32, 1, 213, 65, 1, 0, AHEAD),
    (3, 32, 1, 20, 32, 0, 0, AHEAD), (3, 24, 1, 304, 32, 0, 0, AHEAD), (3, 24, 1, 2432, 32, 0, 0, PHASES),
    # too many for any masks
    (2, 64, 4, 2432, 32, 0, 0, BYTES), (2, 96, 4, 2432, 32, 0, 0, PHASES)])
def test_masks_ahead(tmp_path, dim, L, n_temps, n_real, n, measure, swaps, want):
    assert form(tmp_path, dim, L, n_temps, n_real, n, measure, swaps) == want


# one or two lattices per SM: the CTAs that update and those that draw their
# masks must not wait for one another's SMs (calls of 16 to 32 sweeps took 1.7
# to 4 times their parts)
@pytest.mark.parametrize("L,n_lat,n,part", [(64, 152, 16, 8), (16, 304, 32, 8), (32, 304, 24, 8)])
def test_masks_ahead_pay_at_one_or_two_lattices_per_sm(L, n_lat, n, part):
    lat = sp.Lattice(B.SPIN_ISING, 2, L, B.SPIN_I8, n_real=n_lat, seed=1)

    def us(f):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        f()
        best = 1e30
        for _ in range(12):
            a.record()
            for _ in range(10):
                f()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 100.0)
        return best

    whole = us(lambda: lat.sweep([0.4], n))
    parts = us(lambda: [lat.sweep([0.4], part) for _ in range(n // part)])
    assert whole < 1.4 * parts, (whole, parts)
    lat.sync()
    lat.close()
