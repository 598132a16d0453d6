"""Batches whose least teams (64 word-lattices per CTA at most) need more CTAs
than the GPU has SMs, but not more than two per SM: accepted, tuned, and equal
to per-handle runs, although their average share per unit would fit the form
with one CTA per SM."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


# least teams of 4 to 6 CTAs; groups x least team between 152 and 304
@pytest.mark.parametrize("L,groups,T,n_sets", [(8, 40, 100, 2), (4, 45, 100, 2), (6, 30, 170, 2), (4, 45, 70, 3),
                                               (4, 38, 100, 2)])
def test_least_teams_beyond_one_cta_per_sm(L, groups, T, n_sets):
    betas = [1.2 - 0.8 * t / T for t in range(T)]
    lats = [sp.Lattice(B.SPIN_EA, 3, L, B.SPIN_MSC1, n_real=32 * groups, n_temps=T, n_sets=n_sets, seed=9)
            for _ in range(2)]

    def compare():
        ref = lats[0].run(betas, 2, measure_every=1, pt_every=1)
        ser = lats[1].series_buffers(2)
        sp.batch_run([lats[1].batch_item(betas, ser)], 2, 1, 1)
        lats[1].sync()
        for key in ref:
            assert torch.equal(ref[key], ser[key]), key
        assert torch.equal(lats[0].spins, lats[1].spins)

    compare()
    assert B.spin_batch_tune([lats[1].batch_item(betas, lats[1].series_buffers(2))], 2, 1, 1,
                             torch.cuda.current_stream().cuda_stream) >= 1
    compare()
    for lat in lats:
        lat.close()
