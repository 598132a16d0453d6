"""Which of its two forms a batch of EA units takes (one CTA of 512 threads per
SM with word-lattices in shared memory, or two of 256) at shapes on both sides
of the line, and that both equal per-handle runs."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from graph_kernels import kernels  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


# of 152 SMs; the CTA with the most slots against an average one
@pytest.mark.parametrize("L,groups,T,n_sets,threads", [
    (4, 40, 6, 2, 256), (8, 20, 60, 2, 256), (8, 48, 60, 2, 512), (10, 40, 8, 1, 256), (10, 28, 60, 2, 512),
    (12, 28, 16, 2, 256), (12, 48, 33, 2, 512), (12, 32, 32, 3, 512), (14, 28, 60, 1, 512), (16, 24, 7, 2, 256),
    (16, 40, 8, 2, 512), (18, 40, 8, 2, 512), (20, 12, 32, 2, 512), (20, 40, 32, 2, 256), (22, 12, 32, 2, 256)])
def test_form_and_equal_per_handle_runs(L, groups, T, n_sets, threads, tmp_path):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("shapes chosen for 152 SMs")
    betas = [1.2 - 0.8 * t / T for t in range(T)]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        lats = [sp.Lattice(B.SPIN_EA, 3, L, B.SPIN_MSC1, n_real=32 * groups, n_temps=T, n_sets=n_sets, seed=3)
                for _ in range(2)]
        acc = [torch.zeros(n_sets * T, dtype=torch.int64, device="cuda") for _ in lats]
        lab = [lat.slot_labels() for lat in lats]
        for n, me, pt in ((2, 0, 0), (2, 1, 1), (3, 2, 1)):
            ref = lats[0].run(betas, n, measure_every=me, pt_every=pt, accepted=acc[0], labels=lab[0])
            ser = lats[1].series_buffers(B._n_meas(lats[1].h, n, me)) if me else None
            sp.batch_run([lats[1].batch_item(betas, ser, acc[1], lab[1])], n, me, pt)
            for key in ref:
                assert torch.equal(ref[key], ser[key]), key
            assert torch.equal(lats[0].spins, lats[1].spins)
            assert torch.equal(acc[0], acc[1]) and torch.equal(lab[0], lab[1])
        item = lats[1].batch_item(betas)
        dump = tmp_path / "graph.dot"
        assert "batch_kernel" in kernels(torch, stream, lambda: sp.batch_run([item], 2, 0, 1), dump)
        assert f"batch_kernelILi{threads}E" in dump.read_text()
        for lat in lats:
            lat.sync()
            lat.close()


def test_resident_words_of_an_uneven_share_go_home_after_a_timeout():
    """A wait that runs out ends the launch of the form with resident words;
    the lattices hold a state that the chain can be restarted from."""
    T, betas = 8, [0.5, 0.6, 0.7, 0.8, 0.9, 1.0, 1.1, 1.2]
    lats = [sp.Lattice(B.SPIN_EA, 3, 16, B.SPIN_MSC1, n_real=1280, n_temps=T, n_sets=2, seed=3) for _ in range(2)]
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
