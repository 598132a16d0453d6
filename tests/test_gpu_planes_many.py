"""Many small int8 ferromagnets in one handle, up to where the masks of two
sweeps are the most that is drawn ahead, and beyond: one chain with twin
handles held to the colour phases, odd numbers of sweeps included, and a
working buffer within what the header states."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


def handles(dim, L, n_temps, n_real, count=2):
    return [sp.Lattice(B.SPIN_ISING, dim, L, B.SPIN_I8, n_temps=n_temps, n_real=n_real, seed=11) for _ in range(count)]


# the last sweep that fits a half of the masks, one more lattice, many more
@pytest.mark.parametrize("dim,L,n_temps,n_real", [
    (2, 8, 16, 4095), (2, 16, 5, 3277), (2, 64, 2, 4096), (2, 64, 3, 2731), (2, 128, 2, 1024), (2, 128, 5, 410),
    (2, 40, 3, 4000), (3, 8, 4, 2730), (3, 8, 3, 3641), (3, 16, 2, 2730), (3, 16, 3, 1821), (3, 24, 1, 1213),
    (3, 24, 2, 607), (3, 32, 2, 341), (3, 32, 1, 683),
    # 15 to 17 sweeps in a half, with and without room for what is fetched ahead
    (2, 64, 1, 1084), (2, 64, 1, 1152), (2, 64, 1, 1153), (3, 16, 1, 723), (3, 16, 1, 768), (3, 16, 1, 769),
    (3, 24, 1, 170), (3, 24, 1, 171), (3, 32, 1, 96), (3, 32, 1, 97),
    # two and three sweeps
    (2, 64, 3, 3071), (3, 16, 2, 2047), (3, 16, 1, 4095)])
def test_many_lattices_equal_the_colour_phases(dim, L, n_temps, n_real):
    betas = [(0.4407 if dim == 2 else 0.2216544) * (1 + 0.02 * t) for t in range(n_temps)]
    lats = handles(dim, L, n_temps, n_real)
    lats[1].set_variant(0)
    acc = [torch.zeros(n_temps, dtype=torch.int64, device="cuda") for _ in lats]
    for n, me, pt in ((40, 0, 0), (9, 4, 0), (43, 7, 5)):
        out = [lat.run(betas, n, measure_every=me, pt_every=pt, accepted=a) for lat, a in zip(lats, acc)]
        for key in out[0]:
            assert torch.equal(out[0][key], out[1][key]), (n, key)
        assert torch.equal(lats[0].spins, lats[1].spins), n
    assert torch.equal(acc[0], acc[1])
    for lat in lats:
        lat.sync()
        lat.close()


@pytest.mark.parametrize("dim,L,n_temps,n_real", [(3, 8, 16, 4095), (3, 8, 3, 3500), (2, 64, 2, 4096), (3, 32, 2, 341),
                                                  (2, 128, 1, 1024), (2, 16, 1, 1)])
def test_working_buffer_is_bounded(dim, L, n_temps, n_real):
    lat, = handles(dim, L, n_temps, n_real, 1)
    betas = [0.3] * n_temps
    lat.sweep(betas, 1)
    lat.sync()
    free = torch.cuda.mem_get_info()[0]
    lat.sweep(betas, 5000 if n_temps * n_real < 100 else 50)
    lat.sync()
    took = free - torch.cuda.mem_get_info()[0]
    # 45 MB of masks, two copies of planes of at least 8 of 32 bits in use, 2 MB granules
    assert took <= (45 << 20) + 2 * 4 * lat.n_lat * lat.N // 8 + (4 << 20), took
    lat.close()
