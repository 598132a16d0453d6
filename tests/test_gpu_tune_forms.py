"""What the autotuner remembers serves later handles of the same shape without
changing what they are: a full-accuracy Heisenberg handle stays one after a
fast-math twin was tuned, and an int8 handle gets the fastest form, the default
one included, whatever variant the handle tuned first had been set to."""
import pytest

from tests.graph_kernels import kernels

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("tile", [0, 16])
def test_heisenberg_accuracy_is_kept(tile):
    for variant in (2, 0, 2):
        lat = sp.Lattice(B.SPIN_HEISENBERG, 2, 128, B.SPIN_F32X4, seed=2)
        lat.set_variant(variant)
        lat.set_update_order(B.SPIN_ORDER_DCB, tile, 3)
        assert lat.tune([1.1], 3)[0] == variant
        lat.close()


def test_default_form_is_tried_for_every_handle(tmp_path):
    """Three L = 1000: bit planes take half the time of the colour phases on bytes,
    all that set_variant(0) leaves."""
    L, n, betas = 1000, 40, [0.4, 0.42, 0.44]
    s = torch.cuda.Stream()
    first, second, plain = (sp.Lattice(B.SPIN_ISING, 2, L, B.SPIN_I8, n_temps=3, seed=7, stream=s) for _ in range(3))
    torch.cuda.synchronize()
    first.set_variant(0)
    first.tune(betas, n)
    second.tune(betas, n)
    for lat in (first, second, plain):
        lat.sweep(betas, n)
    torch.cuda.synchronize()
    assert torch.equal(first.spins, second.spins) and torch.equal(first.spins, plain.spins)
    for lat in (first, second, plain):
        assert "planes_phase_kernel" in kernels(torch, s, lambda: lat.sweep(betas, n), tmp_path / "graph.dot")
        lat.close()
