"""Batched EA units with word-lattices kept in shared memory (units of three
and more CTAs on their own SMs: all, some or few of a CTA's word-lattices
resident, couplings staged or not, L % 8 != 0) against per-handle runs."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


# 152 SMs / groups CTAs per unit: between 3 and the number of slots
@pytest.mark.parametrize("L,groups,T,n_sets", [(4, 40, 6, 2), (8, 48, 33, 2), (8, 36, 9, 3), (10, 40, 8, 1),
                                               (12, 32, 30, 2), (16, 32, 32, 2), (16, 24, 7, 2), (20, 30, 6, 2)])
def test_resident_words_equal_per_handle_runs(L, groups, T, n_sets):
    betas = [1.2 - 0.8 * t / T for t in range(T)]
    lats = [sp.Lattice(B.SPIN_EA, 3, L, B.SPIN_MSC1, n_real=32 * groups, n_temps=T, n_sets=n_sets, seed=3)
            for _ in range(2)]
    acc = [torch.zeros(n_sets * T, dtype=torch.int64, device="cuda") for _ in lats]
    lab = [lat.slot_labels() for lat in lats]
    for n, me, pt in ((2, 0, 0), (3, 1, 1), (4, 2, 1), (3, 1, 0)):
        ref = lats[0].run(betas, n, measure_every=me, pt_every=pt, accepted=acc[0], labels=lab[0])
        ser = lats[1].series_buffers(B._n_meas(lats[1].h, n, me)) if me else None
        sp.batch_run([lats[1].batch_item(betas, ser, acc[1], lab[1])], n, me, pt)
        for key in ref:
            assert torch.equal(ref[key], ser[key]), key
        assert torch.equal(lats[0].spins, lats[1].spins)
        assert torch.equal(acc[0], acc[1]) and torch.equal(lab[0], lab[1])
    for lat in lats:
        lat.sync()
        lat.close()


def test_resident_words_go_home_after_a_timeout():
    """A wait that runs out ends the launch; the lattices hold a state that
    the chain can be restarted from, and the context goes on."""
    T, betas = 6, [0.5, 0.6, 0.7, 0.8, 0.9, 1.0]
    lats = [sp.Lattice(B.SPIN_EA, 3, 8, B.SPIN_MSC1, n_real=1280, n_temps=T, n_sets=2, seed=3) for _ in range(2)]
    B.spin_set_batch_options(lats[1].h, timeout_ns=50_000_000, missing_arrivals=1)
    sp.batch_run([lats[1].batch_item(betas)], 3, 0, 1)
    with pytest.raises(B.SpinError):
        lats[1].sync()
    # one sweep ran before the first barrier's wait gave up
    lats[0].sweep(betas, 1)
    lats[0].sync()
    assert torch.equal(lats[0].spins, lats[1].spins)
    for lat in lats:
        lat.close()
