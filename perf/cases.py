"""What is measured: the calls that a user of this library makes, through
``Lattice``, ``batch_run`` and the entry points below them, over the models,
layouts, sizes and schedules that it takes.

A case is one call of a running simulation (a few sweeps with its measurement
and exchange schedule) on lattices that the program already holds.  Ising and
Edwards-Anderson chains are whole-number functions of the seed and are compared
exactly; Heisenberg spins are FP32, and a decision that falls within rounding
of its threshold moves one spin by its own length.
"""
import math

import numpy as np
import torch

import paper_1101_1427_gb300 as sp
from paper_1101_1427_gb300 import _binding as B
from paper_1101_1427_gb300 import presets

I8, CODED = "i8", "coded"
CRITICAL_2D, CRITICAL_3D = 0.4407, 0.2216544


def _ising(name, dim, L, layout, slots, sweeps, measure=0, pt=0, beta=0.0, tile=0, hits=1, io=False):
    """slots > 1 with beta 0: the tempering benchmark's equally spaced betas.
    tile > 0: the double-checkerboard order.  io: the configuration comes from
    and goes back to one byte per spin around the sweeps."""
    c = {"kind": "ising", "dim": dim, "L": L, "layout": layout, "slots": slots, "sweeps": sweeps,
         "measure": measure, "pt": pt, "beta": beta, "tile": tile, "hits": hits, "io": io}
    return dict(c, name=name) if name else c


def _heis(name, dim, L, lattices, sweeps, done, beta, fast=False, tile=0, hits=1):
    """done: the handle's sweep count before the call (it renormalises the
    spins at every hundredth)."""
    c = {"kind": "heis", "dim": dim, "L": L, "lattices": lattices, "sweeps": sweeps, "done": done, "beta": beta,
         "fast": fast, "tile": tile, "hits": hits}
    return dict(c, name=name) if name else c


def _ea(name, dim, L, layout, real, slots, sweeps, measure, pt, batched=False, width=32, io=False):
    c = {"kind": "ea", "dim": dim, "L": L, "layout": layout, "real": real, "slots": slots, "sweeps": sweeps,
         "measure": measure, "pt": pt, "batched": batched, "width": width, "io": io}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest lattice of the presets, E and M after every sweep: one
        # block of work, all latency
        _ising("ising2d_L64_series", 2, 64, I8, 1, 1000, measure=1, beta=CRITICAL_2D),
        # the paper's tempering benchmark at its smallest quoted size: 20
        # replicas, one exchange per 10 sweeps
        _ising("ising2d_pt20_L64", 2, 64, I8, 20, 100, pt=10),
        # the same run in the middle of the range that the paper plots
        _ising("ising2d_pt20_L512", 2, 512, I8, 20, 20, pt=10),
        # the generator check of the paper (16 chains of L = 1024), its
        # configurations set from bytes before and read back as bytes after
        _ising("ising2d_coded_L1024_x16", 2, 1024, CODED, 16, 50, measure=10, beta=0.4, io=True),
        # a size that is no multiple of 256, so bytes are swept as bytes
        _ising("ising2d_L1000_x3", 2, 1000, I8, 3, 20, measure=10, beta=CRITICAL_2D),
        # the largest preset: 3 x 2^28 spins, measured every 10 sweeps
        _ising("ising2d_coded_L16384_x3", 2, 16384, CODED, 3, 10, measure=10, beta=CRITICAL_2D),
        # the paper's own update order: double checkerboard, 100 hits
        _ising("ising2d_dcb_L4096_x3", 2, 4096, I8, 3, 100, beta=CRITICAL_2D, tile=16, hits=100),
        # the paper's 3D workload
        _ising("ising3d_L512", 3, 512, I8, 1, 4, measure=4, beta=CRITICAL_3D),
        # the Heisenberg preset, full accuracy, up to a renormalisation
        _heis("heis3d_L128", 3, 128, 1, 20, 80, 0.693),
        # spin-glass tempering as the preset runs it: E, M, Q and an exchange
        # after every sweep, one persistent launch
        _ea("ea3d_L16_batched", 3, 16, CODED, 1024, 32, 8, 1, 1, batched=True),
        # an ordinary spin-glass call on one handle, and its configurations read out
        _ea("ea3d_L12_handle", 3, 12, CODED, 256, 30, 10, 5, 5, io=True),
        # ten handles of unequal sizes in one launch
        {"name": "uneven_batch", "kind": "mix", "scale": 1, "sweeps": 4},
    ]


# ------------------------------------------------------------------ drawn cases
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(n, lo=4):
    return max(lo, n + (n & 1))


def draw(rng):
    kind = rng.choice(["ising2d", "ising2d", "coded", "ising3d", "dcb", "heis", "heis", "ea", "ea", "batched", "mix"])
    if kind == "ising2d":  # odd multiples of 2, of 8 and of 256 alike
        L = _even(_log(rng, 8, 3000))
        step = rng.choice([2, 8, 8, 256])
        L = max(step, L // step * step, 4)
        slots = rng.choice([1, 3, 20, rng.randint(2, 40)])
        sweeps = max(2, min(400, int(4e9 / (slots * L * L * 15)), _log(rng, 4, 400)))
        every = rng.choice([0, 1, 5, 10])
        return _ising(None, 2, L, I8, slots, sweeps, measure=every, pt=rng.choice([0, 5, 10]) if slots > 1 else 0,
                      beta=0.0 if slots > 3 else rng.choice([0.4, CRITICAL_2D, 0.5]))
    if kind == "coded":
        L = 256 * _log(rng, 1, 32)
        slots = max(1, min(rng.choice([1, 2, 3, 16]), (3 << 28) // (L * L)))
        sweeps = max(2, min(100, int(6e9 / (slots * L * L)), _log(rng, 4, 100)))
        return _ising(None, 2, L, CODED, slots, sweeps, measure=rng.choice([0, 1, 10]), beta=CRITICAL_2D,
                      io=rng.random() < 0.3)
    if kind == "ising3d":
        L = _even(_log(rng, 6, 400))
        L = max(8, L // 8 * 8) if rng.random() < 0.6 else L
        slots = max(1, min(rng.choice([1, 3, 20]), int(1.2e8 / L ** 3)))
        sweeps = max(2, min(200, int(5e8 / (slots * L ** 3)), _log(rng, 4, 200)))
        return _ising(None, 3, L, I8, slots, sweeps, measure=rng.choice([0, 1, 10]), pt=rng.choice([0, 5]) if slots > 1 else 0,
                      beta=CRITICAL_3D)
    if kind == "dcb":
        dim = rng.choice([2, 2, 3])
        tile = rng.choice([8, 16, 32, 64]) if dim == 2 else rng.choice([8, 16])
        L = 2 * tile * _log(rng, 1, (4096 if dim == 2 else 256) // (2 * tile))
        hits = rng.choice([5, 10, 25, 100])
        return _ising(None, dim, L, I8, max(1, min(rng.choice([1, 3]), (1 << 25) // L ** dim)), hits,
                      beta=CRITICAL_2D if dim == 2 else CRITICAL_3D, tile=tile, hits=hits)
    if kind == "heis":
        dim, fast = rng.choice([2, 3, 3]), rng.random() < 0.5
        if dim == 2 and rng.random() < 0.5:
            tile, hits = rng.choice([8, 16, 32]), rng.choice([5, 10])
            return _heis(None, 2, 2 * tile * _log(rng, 1, 2048 // (2 * tile)), rng.choice([1, 2]), hits, 0, 1.1, fast, tile, hits)
        L = _even(_log(rng, 16, 1500)) if dim == 2 else rng.choice([_even(_log(rng, 8, 160)), 64, 128])
        lattices = max(1, min(rng.choice([1, 1, 4]), int(4e6 / L ** dim)))
        sweeps = max(1, min(rng.choice([2, 8, 20]), int(4e7 / (lattices * L ** dim))))
        return _heis(None, dim, L, lattices, sweeps, rng.choice([0, 95, 100 - sweeps]), 1.1 if dim == 2 else 0.693, fast)
    if kind == "ea":
        dim = rng.choice([2, 3, 3])
        if rng.random() < 0.2:  # one spin per byte
            return _ea(None, dim, _even(_log(rng, 4, 32 if dim == 2 else 16)), I8, rng.randint(1, 40), rng.choice([3, 8]),
                       _log(rng, 2, 20), rng.choice([0, 1, 5]), rng.choice([0, 1, 5]))
        L = _even(_log(rng, 6, 64 if dim == 2 else 32))
        real = 64 * max(1, min(16, int(3e5 / L ** dim)))
        return _ea(None, dim, L, CODED, _log(rng, 1, real // 64) * 64, rng.choice([2, 16, 32, 33]), _log(rng, 2, 20),
                   rng.choice([0, 1, 5]), rng.choice([0, 1, 5]), width=rng.choice([32, 32, 64]), io=rng.random() < 0.3)
    if kind == "batched":
        L = _even(_log(rng, 6, 32))
        groups = _log(rng, 1, max(1, min(32, int(1.4e5 / L ** 3))))
        return _ea(None, 3, L, CODED, 32 * groups, rng.choice([8, 24, 32]), _log(rng, 2, 10), rng.choice([0, 1, 1, 2]),
                   rng.choice([1, 1, 2]), batched=True)
    return {"kind": "mix", "scale": rng.choice([2, 4, 8]), "sweeps": rng.randint(2, 8)}


# ------------------------------------------------------------------ states
def _geometric(lo, hi, n):
    return list(1.0 / np.geomspace(lo, hi, n))


def _ising_betas(c):
    if c["beta"] == 0.0:
        return list(np.linspace(0.1, 0.15, c["slots"]))
    if c["pt"] and c["slots"] > 1:
        return list(np.linspace(0.98 * c["beta"], 1.02 * c["beta"], c["slots"]))
    return [c["beta"] * (1.0 + 0.05 * (t % 3 - 1)) if c["slots"] > 1 else c["beta"] for t in range(c["slots"])]


def _heis_start(c, seed):
    """Unit vectors about as aligned as neighbours are near the transition."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = torch.zeros(c["lattices"] * c["L"] ** c["dim"], 4, device="cuda")
    s[:, :3] = 0.75 * torch.randn(s.shape[0], 3, generator=gen, device="cuda")
    s[:, 2] += 1.0
    return s / s.norm(dim=1, keepdim=True)


def _mix_members(c):
    """The uneven batch of the presets (scale 1), or one with fewer realisations."""
    k = c["scale"]
    got = [("ea", L, max(32, R // k // 32 * 32), T) for L, R, T in presets.UNEVEN_EA]
    return got + [("ising", L, 1, 1) for L in presets.UNEVEN_ISING if L <= 4096 // k]


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = {"case": c}
    if kind == "mix":
        st["lats"], st["betas"] = [], []
        for k, (model, L, R, T) in enumerate(_mix_members(c)):
            if model == "ea":
                lat = sp.Lattice(B.SPIN_EA, 3, L, B.SPIN_MSC1, n_real=R, n_temps=T, n_sets=2, seed=seed + 50 + k)
            else:
                lat = sp.Lattice(B.SPIN_ISING, 2, L, B.SPIN_MSC1, seed=seed + 50 + k)
            st["lats"].append(lat)
            st["betas"].append(_geometric(0.8, 2.2, T) if model == "ea" else [CRITICAL_2D])
        return st
    if kind == "heis":
        lat = sp.Lattice(B.SPIN_HEISENBERG, c["dim"], c["L"], B.SPIN_F32X4, n_real=c["lattices"], seed=seed)
        lat.spins.copy_(_heis_start(c, seed).view(-1))
        lat.set_counters(c["done"])
        if c["fast"]:
            lat.set_variant(2)
        if c["tile"]:
            lat.set_update_order(B.SPIN_ORDER_DCB, c["tile"], c["hits"])
        st.update(lat=lat, betas=[c["beta"]])
        return st
    if kind == "ising":
        layout = B.SPIN_I8 if c["layout"] == I8 else B.SPIN_MSC1
        lat = sp.Lattice(B.SPIN_ISING, c["dim"], c["L"], layout, n_temps=c["slots"], seed=seed)
        st.update(lat=lat, betas=_ising_betas(c))
    else:
        layout = B.SPIN_I8 if c["layout"] == I8 else B.SPIN_MSC1
        lat = sp.Lattice(B.SPIN_EA, c["dim"], c["L"], layout, n_real=c["real"], n_temps=c["slots"], n_sets=2, seed=seed)
        if c["width"] == 64:
            lat.set_msc_width(64)
        st.update(lat=lat, betas=_geometric(0.9, 2.0, c["slots"]))
    if c.get("tile"):
        lat.set_update_order(B.SPIN_ORDER_DCB, c["tile"], c["hits"])
    if c["pt"]:
        st["accepted"] = torch.zeros(lat.n_sets * lat.n_temps, dtype=torch.int64, device="cuda")
    if c["io"] and kind == "ising":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        st["bytes"] = 1 - 2 * torch.randint(0, 2, (lat.n_lat * lat.N,), dtype=torch.int8, device="cuda", generator=gen)
    return st


def run(state):
    c = state["case"]
    if c["kind"] == "mix":
        items, out = [], []
        for lat, betas in zip(state["lats"], state["betas"]):
            series = lat.series_buffers(c["sweeps"])
            items.append(lat.batch_item(betas, series))
            out.append([lat.spins] + list(series.values()))
        sp.batch_run(items, c["sweeps"], 1, 1)
        return out
    lat = state["lat"]
    if c["kind"] == "heis":
        out = lat.run(state["betas"], c["sweeps"])
        out["spins"] = lat.spins
        out["Ef"], out["Mf"] = lat.measure()
        return out
    if "bytes" in state:
        lat.pack(state["bytes"])
    accepted = state.get("accepted")
    if c.get("batched"):
        out = lat.series_buffers(B._n_meas(lat.h, c["sweeps"], c["measure"]))
        sp.batch_run([lat.batch_item(state["betas"], out if c["measure"] else None, accepted)], c["sweeps"],
                     c["measure"], c["pt"])
    else:
        out = lat.run(state["betas"], c["sweeps"], measure_every=c["measure"], pt_every=c["pt"], accepted=accepted)
    out["spins"] = lat.spins
    if accepted is not None:
        out["accepted"] = accepted
    if c["io"]:
        out["bytes"] = lat.unpack()
    return {k: v for k, v in out.items() if v.numel()}


# ------------------------------------------------------------------ work
# 32-bit operations of one attempted update: Philox4x32-10 has 20 wide
# multiplies and 20 XORs per four words; the rest is the neighbour sum, the
# comparison and the flip.
_PHILOX_WORD, _ISING, _EA_WORD, _HEIS = 10, 15, 38, 40 + 70


def work(case):
    c = case
    if c["kind"] == "mix":
        b = f = 0
        for model, L, R, T in _mix_members(c):
            if model == "ea":
                words = 2 * T * (R // 32) * L ** 3
                b += 8 * words + 4 * 3 * (R // 32) * L ** 3 + c["sweeps"] * 8 * 5 * T * R
                f += c["sweeps"] * words * _EA_WORD
            else:
                b += L * L // 4 + c["sweeps"] * 16
                f += c["sweeps"] * L * L * _ISING
        return {"bytes": b, "flops": f}
    N = c["L"] ** c["dim"]
    if c["kind"] == "heis":
        return {"bytes": 32 * N * c["lattices"], "flops": N * c["lattices"] * c["sweeps"] * _HEIS}
    rows = c["sweeps"] // c["measure"] if c["measure"] else 0
    if c["kind"] == "ising":
        n = N * c["slots"]
        return {"bytes": (2 * n if c["layout"] == I8 else n // 4) + (2 * n if c["io"] else 0) + 16 * rows * c["slots"],
                "flops": n * c["sweeps"] * _ISING}
    n = 2 * c["slots"] * c["real"] * N
    series = 8 * 5 * rows * c["slots"] * c["real"]
    if c["layout"] == I8:
        return {"bytes": 2 * n + c["dim"] * c["real"] * N + series, "flops": n * c["sweeps"] * (_ISING + 6)}
    return {"bytes": n // 4 + c["dim"] * c["real"] * N // 8 + (n if c["io"] else 0) + series,
            "flops": n // 32 * c["sweeps"] * _EA_WORD}


def tolerance(case):
    # whole numbers are the same numbers; FP32 spins are compared with the
    # 64-bit chain below: 3.6e-8 off at L = 128 after 20 sweeps in full
    # accuracy, 1.7e-3 with the hardware approximations, where a few decisions
    # fall within rounding of their threshold (one spin of 128^3 decided
    # otherwise is 1e-3)
    if case["kind"] != "heis":
        return "exact"
    return {"rel": 7e-3 if case["fast"] else 4e-3, "max": 0.999}


# ------------------------------------------------------------------ the 64-bit chain
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words."""
    c = [torch.as_tensor(v, dtype=torch.int64, device="cuda") for v in (c0, c1, c2, c3)]
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & _M32) ^ c[1] ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c[3] ^ k1, p0 & _M32]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c


def _heis_exact(c, seed):
    dim, L, H = c["dim"], c["L"], c["L"] // 2
    s = _heis_start(c, seed)[:, :3].double().view([c["lattices"]] + [L] * dim + [3])
    axes = list(range(1, dim + 1))
    rows = torch.arange(L ** (dim - 1), device="cuda")
    par = rows if dim == 2 else rows // L + rows % L
    j = torch.arange(L ** dim // 2, dtype=torch.int64, device="cuda").view(-1, H)
    site = [(rows[:, None] * L + 2 * torch.arange(H, device="cuda") + ((par + col) & 1)[:, None]).view(-1) for col in (0, 1)]
    steps = [(None, h) for h in range(c["sweeps"])]
    if c["tile"]:
        T = c["tile"]
        coarse = [((site[col] // L) // T + (site[col] % L) // T) & 1 for col in (0, 1)]
        steps = [(a, m * c["hits"] + h) for m in range(c["sweeps"] // c["hits"]) for a in (0, 1) for h in range(c["hits"])]
    done = 0
    for n, (a, k) in enumerate(steps):
        for col in (0, 1):
            at, jj = site[col], j.view(-1)
            if a is not None:
                keep = coarse[col] == a
                at, jj = at[keep], jj[keep]
            field = torch.zeros_like(s)
            for ax in axes:
                field += s.roll(1, ax) + s.roll(-1, ax)
            for lat in range(c["lattices"]):
                w = _philox(jj, c["done"] + k, lat << 12, (4 << 28) | (col << 27), seed)
                u = [(x >> 8).double() / 2.0 ** 24 for x in w[:3]]
                z = 2.0 * u[0] - 1.0
                rho, phi = torch.sqrt((1.0 - z * z).clamp_min(0.0)), 2.0 * math.pi * u[1]
                new = torch.stack([rho * torch.cos(phi), rho * torch.sin(phi), z], 1)
                flat = s[lat].view(-1, 3)
                dE = ((flat[at] - new) * field[lat].view(-1, 3)[at]).sum(1)
                ok = (dE <= 0) | (u[2] < torch.exp(-c["beta"] * dE))
                flat[at[ok]] = new[ok]
        if not c["tile"]:
            done = k + 1
        elif (n + 1) % (2 * c["hits"]) == 0:
            done = k + 1
        else:
            continue
        if (c["done"] + done) // 100 != (c["done"] + done - c["hits"]) // 100:
            s /= s.norm(dim=-1, keepdim=True)
    bonds = torch.zeros_like(s[..., 0])
    for ax in axes:
        bonds += (s * s.roll(-1, ax)).sum(-1)
    flat = s.reshape(c["lattices"], -1, 3)
    spins = torch.cat([flat.reshape(-1, 3), torch.zeros(flat.shape[0] * flat.shape[1], 1, dtype=s.dtype, device="cuda")], 1)
    return {"spins": spins.reshape(-1), "Ef": -bonds.reshape(c["lattices"], -1).sum(1), "Mf": flat.sum(1)}


def exact(case, seed):
    if case["kind"] != "heis":
        return None  # whole numbers throughout
    return _heis_exact(case, seed)
