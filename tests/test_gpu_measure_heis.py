"""Heisenberg energy and magnetisation on either side of the sizes (2^19, 2^20,
2^21 sites) from which clusters of 2, 4, 8 CTAs share each partial sum, against FP64
sums of the same FP32 spins, and bit for bit against the allocation-free
entry point."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("dim,L,n_lat", [(2, 4, 5), (2, 362, 2), (2, 724, 1), (2, 726, 2), (3, 52, 3), (3, 80, 1),
                                            (3, 82, 1), (3, 102, 2), (3, 126, 1), (3, 128, 1)])
def test_heisenberg_sums(dim, L, n_lat):
    N = L ** dim
    rng = np.random.default_rng(N)
    s = rng.standard_normal((n_lat, N, 3))
    s = (s / np.linalg.norm(s, axis=2, keepdims=True)).astype(np.float32)
    full = np.zeros((n_lat, N, 4), np.float32)
    full[:, :, :3] = s
    lat = sp.Lattice(B.SPIN_HEISENBERG, dim, L, B.SPIN_F32X4, n_temps=n_lat, seed=1)
    lat.spins.copy_(torch.from_numpy(full.reshape(-1)))
    Ef, Mf = lat.measure()
    Ef2, Mf2 = torch.empty_like(Ef), torch.empty_like(Mf).view(-1)
    B.spin_heis_measure_noalloc(lat.spins, dim, L, n_lat, Ef2, Mf2, torch.cuda.current_stream().cuda_stream)
    lat.sync()
    assert torch.equal(Ef, Ef2) and torch.equal(Mf.view(-1), Mf2)
    d = s.astype(np.float64).reshape((n_lat,) + (L,) * dim + (3,))
    E = -sum((d * np.roll(d, -1, ax)).sum(axis=tuple(range(1, dim + 2))) for ax in range(1, dim + 1))
    # at most ~100 additions from a term to the total (thread, warp, cluster,
    # partials), each within 2^-53 of sums of terms of size <= dim
    tol = 100 * 2.0 ** -53 * dim * N
    assert np.max(np.abs(Ef.cpu().numpy() - E)) <= tol
    assert np.max(np.abs(Mf.cpu().numpy() - d.reshape(n_lat, N, 3).sum(1))) <= tol
    lat.close()


def test_heisenberg_sums_are_correctly_rounded_per_thread():
    """One site per thread (N <= 64 x 256): the per-thread expansions are exact,
    so that only the FP64 tree's ~20 additions round -- against math.fsum of
    the exact products."""
    import math
    L, N = 24, 24 ** 3
    rng = np.random.default_rng(5)
    s = rng.standard_normal((N, 3))
    s = (s / np.linalg.norm(s, axis=1, keepdims=True)).astype(np.float32)
    full = np.zeros((N, 4), np.float32)
    full[:, :3] = s
    lat = sp.Lattice(B.SPIN_HEISENBERG, 3, L, B.SPIN_F32X4, seed=1)
    lat.spins.copy_(torch.from_numpy(full.reshape(-1)))
    Ef, Mf = lat.measure()
    lat.sync()
    d = s.astype(np.float64).reshape(L, L, L, 3)
    terms = np.concatenate([(d * np.roll(d, -1, ax)).ravel() for ax in range(3)])  # exact in FP64
    # partial sums of the tree stay below N / 64 until the last 64 additions
    tol = 2.0 ** -53 * (20 * N / 64 + 64 * abs(math.fsum(terms)) + N)
    assert abs(Ef.item() + math.fsum(terms)) <= tol
    for c in range(3):
        assert abs(Mf[0, c].item() - math.fsum(d[..., c].ravel())) <= tol
    lat.close()


def test_heisenberg_sums_of_spins_far_from_unit_length():
    """Lengths whose FP32 products overflow or vanish take the FP64 sums."""
    L = 8
    for scale in (1e25, 1e-25):
        full = np.zeros((L ** 3, 4), np.float32)
        full[:, 2] = scale
        lat = sp.Lattice(B.SPIN_HEISENBERG, 3, L, B.SPIN_F32X4, seed=1)
        lat.spins.copy_(torch.from_numpy(full.reshape(-1)))
        Ef, Mf = lat.measure()
        lat.sync()
        v = float(np.float32(scale))
        assert abs(Ef.item() / (-3 * L ** 3 * v * v) - 1) < 1e-12
        assert abs(Mf[0, 2].item() / (L ** 3 * v) - 1) < 1e-12
        lat.close()
