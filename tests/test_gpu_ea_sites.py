"""Coded EA lattices with L % 8 != 0 (lanes take consecutive sites: last quads
that are not full, slot blocks that are not full, fewer sites than a warp)
against one spin per byte, and the batched launch against per-handle runs."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("dim,L,n_real,T", [(2, 4, 32, 2), (2, 6, 32, 3), (2, 10, 64, 5), (2, 14, 32, 1), (2, 18, 32, 9),
                                            (3, 4, 32, 2), (3, 6, 96, 5), (3, 10, 32, 7), (3, 12, 64, 6), (3, 14, 32, 4)])
def test_sites_equal_bytes(dim, L, n_real, T):
    betas = [0.0, 30.0, 0.7, 0.9, 0.5, 1.1, 1.3, 0.2, 0.4][:T]
    lats = [sp.Lattice(B.SPIN_EA, dim, L, layout, n_real=n_real, n_temps=T, n_sets=2, seed=7)
            for layout in (B.SPIN_MSC1, B.SPIN_I8)]
    for n in (1, 4):
        for lat in lats:
            lat.sweep(betas, n)
        assert torch.equal(lats[0].unpack().view(-1), lats[1].spins)
    for lat in lats:
        lat.sync()
        lat.close()


@pytest.mark.parametrize("L,n_real,T", [(4, 32, 8), (6, 64, 5), (10, 32, 33), (12, 96, 6), (14, 32, 3), (20, 32, 2)])
def test_batched_sites_equal_per_handle_runs(L, n_real, T):
    betas = [0.6 + 0.05 * t for t in range(T)]
    lats = [sp.Lattice(B.SPIN_EA, 3, L, B.SPIN_MSC1, n_real=n_real, n_temps=T, n_sets=2, seed=9) for _ in range(2)]
    for n, me, pt in ((3, 1, 1), (4, 2, 0), (2, 0, 0)):
        ref = lats[0].run(betas, n, measure_every=me, pt_every=pt)
        ser = lats[1].series_buffers(B._n_meas(lats[1].h, n, me)) if me else None
        sp.batch_run([lats[1].batch_item(betas, ser)], n, me, pt)
        for key in ref:
            assert torch.equal(ref[key], ser[key]), key
        assert torch.equal(lats[0].spins, lats[1].spins)
    for lat in lats:
        lat.sync()
        lat.close()


# last chunks of 128 sites that hold 100, 76, 84 and 60, couplings not staged
@pytest.mark.parametrize("L", [18, 22, 26, 30])
def test_batched_sites_with_couplings_in_l2_equal_per_handle_runs(L):
    lats = [sp.Lattice(B.SPIN_EA, 3, L, B.SPIN_MSC1, n_real=64, n_temps=3, n_sets=2, seed=5) for _ in range(2)]
    betas = [0.5, 0.8, 1.1]
    for n, me, pt in ((2, 0, 0), (3, 1, 1)):
        ref = lats[0].run(betas, n, measure_every=me, pt_every=pt)
        ser = lats[1].series_buffers(3) if me else None
        sp.batch_run([lats[1].batch_item(betas, ser)], n, me, pt)
        for key in ref:
            assert torch.equal(ref[key], ser[key]), key
        assert torch.equal(lats[0].spins, lats[1].spins)
    for lat in lats:
        lat.sync()
        lat.close()


@pytest.mark.parametrize("dim,L,n_real,T", [(2, 6, 32, 3), (2, 16, 64, 2), (2, 50, 32, 2), (2, 90, 32, 1), (3, 4, 32, 2),
                                            (3, 8, 32, 2), (3, 12, 64, 3), (3, 18, 32, 2), (3, 26, 32, 1)])
def test_counts_and_bytes_equal_bytes(dim, L, n_real, T):
    """E, M and Q (one and several parts per word-lattice), and the conversion
    from and to bytes at any address."""
    coded = sp.Lattice(B.SPIN_EA, dim, L, B.SPIN_MSC1, n_real=n_real, n_temps=T, n_sets=2, seed=4)
    i8 = sp.Lattice(B.SPIN_EA, dim, L, B.SPIN_I8, n_real=n_real, n_temps=T, n_sets=2, seed=4)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(L)
    n = i8.spins.numel()
    raw = 1 - 2 * (torch.rand(n + 4, device="cuda", generator=gen) < 0.3).to(torch.int8)
    words = []
    for off in (0, 1):
        s = raw[off:off + n]
        B.spin_pack_i8(coded.h, s)
        B.spin_pack_i8(i8.h, s.clone())
        for x, y in zip(coded.measure(), i8.measure()):
            assert torch.equal(x, y)
        words.append(coded.spins.clone())
        for o in (0, 2):
            out = torch.zeros(n + 4, dtype=torch.int8, device="cuda")
            B.spin_unpack_i8(coded.h, out[o:o + n])
            coded.sync()
            assert torch.equal(out[o:o + n], s) and not out[:o].any() and not out[o + n:].any()
    B.spin_pack_i8(coded.h, raw[1:1 + n].clone())
    coded.sync()
    assert torch.equal(coded.spins, words[1])
    for lat in (coded, i8):
        lat.close()
