"""Captured calls of int8 ferromagnets hold the address of the handle's working
buffer: it stays theirs when later calls need a longer one (more sweeps of
masks, the fused pass), so that a replay neither reads nor writes memory that
something else owns by then."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


# sweeps before the capture, captured, after it (the call that needs more)
@pytest.mark.parametrize("dim,L,n_lat,first,captured,longer", [
    (2, 64, 1, 1000, 100, 2000), (2, 64, 1, 1000, 100, 5000), (3, 32, 2, 20, 7, 600), (2, 128, 3, 600, 40, 1500),
    (2, 256, 3, 8, 9, 2), (2, 512, 40, 5, 4, 3)])
def test_replay_after_a_longer_call(dim, L, n_lat, first, captured, longer):
    s = torch.cuda.Stream()
    betas = [0.1 + 0.3 * t / n_lat for t in range(n_lat)]
    a = sp.Lattice(B.SPIN_ISING, dim, L, B.SPIN_I8, n_temps=n_lat, seed=4, stream=s)
    b = sp.Lattice(B.SPIN_ISING, dim, L, B.SPIN_I8, n_temps=n_lat, seed=4, stream=s)
    for lat in (a, b):
        lat.sweep(betas, first)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        B.spin_sweep(a.h, None, betas, captured, a.seed)
    a.set_counters(first)  # the capture ran nothing
    a.sweep(betas, longer)
    # memory that may be handed out again if the old buffer was freed
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    others = [torch.full((1 << k,), 7, dtype=torch.uint8, device="cuda") for k in range(21, 27)]
    torch.cuda.synchronize()
    for _ in range(2):
        with torch.cuda.stream(s):
            g.replay()
    torch.cuda.synchronize()
    assert all(bool((t == 7).all()) for t in others)
    b.sweep(betas, longer)
    for _ in range(2):
        b.set_counters(first)
        b.sweep(betas, captured)
    b.sync()
    assert torch.equal(a.spins, b.spins)
    # and the handle goes on in its new buffer
    for lat in (a, b):
        lat.set_counters(first + longer)
        lat.sweep(betas, longer)
        lat.sync()
    assert torch.equal(a.spins, b.spins)
    a.close()
    b.close()
