"""Heisenberg sums of lattices with at most a site per thread (CTAs, warps and
threads without one, the last of them partly full) against exact sums of the
same FP32 spins, and bit for bit between one lattice and many."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1101_1427_gb300 as sp  # noqa: E402
from paper_1101_1427_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("dim,L,n_lat", [(3, 4, 3), (3, 6, 5), (3, 8, 40), (2, 16, 3), (2, 18, 3), (3, 24, 2), (3, 26, 2),
                                         (2, 126, 2), (2, 128, 3), (2, 130, 2), (2, 180, 2)])
def test_sums_of_small_lattices(dim, L, n_lat):
    N = L ** dim
    rng = np.random.default_rng(L)
    s = rng.standard_normal((n_lat, N, 3))
    s = (s / np.linalg.norm(s, axis=2, keepdims=True)).astype(np.float32)
    full = np.zeros((n_lat, N, 4), np.float32)
    full[:, :, :3] = s
    lat = sp.Lattice(B.SPIN_HEISENBERG, dim, L, B.SPIN_F32X4, n_temps=n_lat, seed=1)
    lat.spins.copy_(torch.from_numpy(full.reshape(-1)))
    Ef, Mf = lat.measure()
    one = sp.Lattice(B.SPIN_HEISENBERG, dim, L, B.SPIN_F32X4, seed=1)
    one.spins.copy_(torch.from_numpy(full[-1].reshape(-1)))
    E1, M1 = one.measure()
    one.sync()
    assert E1[0] == Ef[-1] and torch.equal(M1[0], Mf[-1])
    # thread sums are exact to 2^-72; ~20 additions of the tree act on sums of at
    # most 256 threads' terms (2 sites each at most), 64 on those of the lattice
    for k in range(n_lat):
        d = s[k].astype(np.float64).reshape((L,) * dim + (3,))
        terms = np.concatenate([(d * np.roll(d, -1, ax)).ravel() for ax in range(dim)])  # exact in FP64
        E = math.fsum(terms)
        tol = 2.0 ** -53 * (20 * dim * min(2 * N, 64 * 512) + 64 * max(abs(E), math.sqrt(dim * N) * 4) + N)
        assert abs(Ef[k].item() + E) <= tol
        for c in range(3):
            M = math.fsum(d[..., c].ravel())
            assert abs(Mf[k, c].item() - M) <= tol
    lat.close()
    one.close()


def test_many_small_lattices_are_not_paid_by_the_thread():
    """The fixed cost of 64 CTAs per lattice: 1000 lattices of 8^3 spins take
    far less than 1000 times what a full CTA's reduction would."""
    lat = sp.Lattice(B.SPIN_HEISENBERG, 3, 8, B.SPIN_F32X4, n_real=1000, seed=1)
    full = sp.Lattice(B.SPIN_HEISENBERG, 3, 24, B.SPIN_F32X4, n_real=1000, seed=1)

    def us(h):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = 1e30
        for _ in range(6):
            a.record()
            h.measure()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    assert us(lat) < 0.5 * us(full)
    lat.close()
    full.close()
