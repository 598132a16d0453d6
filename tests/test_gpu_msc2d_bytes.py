"""Conversion of coded 2D lattices from and to one byte per spin: a buffer at
an odd address gives what an aligned one gives, and the bytes come back."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("L,n_lat", [(256, 1), (768, 3), (1024, 5)])
def test_bytes_at_any_address(L, n_lat):
    n = n_lat * L * L
    gen = torch.Generator(device="cuda")
    gen.manual_seed(L)
    s = 1 - 2 * torch.randint(0, 2, (n + 16,), dtype=torch.int8, device="cuda", generator=gen)
    lat = sp.Lattice(B.SPIN_ISING, 2, L, B.SPIN_MSC1, n_temps=n_lat, seed=2)
    words = []
    for off in (8, 3):
        B.spin_pack_i8(lat.h, s[off:off + n].clone() if off == 8 else s[off:off + n])
        words.append(lat.spins.clone())
        out = torch.zeros(n + 16, dtype=torch.int8, device="cuda")
        for o in (0, 8, 5):
            out.zero_()
            B.spin_unpack_i8(lat.h, out[o:o + n])
            lat.sync()
            assert torch.equal(out[o:o + n], s[off:off + n])
            assert not out[:o].any() and not out[o + n:].any()
    B.spin_pack_i8(lat.h, s[3:3 + n].clone())
    lat.sync()
    assert torch.equal(lat.spins, words[1])
    lat.close()
