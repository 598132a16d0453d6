// +-J Edwards-Anderson glass in 3D (and on the square lattice of the
// paper's own Sec. 5 benchmark) with asynchronous multi-spin coding: bit b
// of a 32-bit word is the spin of realisation 32 g + b at one site, bit set
// <=> s = -1; word-lattices [n_sets][groups][n_temps], each stored
// colour-split (ea_cs.cuh).  Coupling words [groups][dim][colour][N/2], bit
// set <=> J = -1.  The 32 realisations of a word share one
// uniform per site and sweep (the paper's footnote to Sec. 5), so one Philox
// call serves four word-sites.
#include <algorithm>
#include <cmath>

#include "ea_cs.cuh"
#include "internal.h"

namespace spin {
namespace {

__global__ void init_msc_kernel(uint32_t *__restrict__ w, Geom g, RoundKeys rk) {
  const int G = g.n_real / 32;
  const int64_t quads = (g.N + 3) / 4;
  const int64_t n_wl = (int64_t)g.n_sets * G * g.n_temps;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n_wl * quads;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t wl = k / quads, q4 = k - wl * quads;
    const int t = (int)(wl % g.n_temps);
    const int grp = (int)((wl / g.n_temps) % G);
    const int a = (int)(wl / ((int64_t)g.n_temps * G));
    const uint4 r = philox(make_uint4((uint32_t)q4, 0u, lattice_id(a, grp, t), ctr_w(TAG_INIT, 0, 0)), rk);
    uint32_t *out = w + wl * g.N;
    const uint32_t half = (uint32_t)(g.N / 2);
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q) {
      const uint32_t i = (uint32_t)(4 * q4 + q);
      if (i < g.N) out[cs_word(i, colour_of(g, i), half)] = word_of(r, q);
    }
  }
}

__global__ void couplings_msc_kernel(uint32_t *__restrict__ J, Geom g, RoundKeys rk) {
  const int G = g.n_real / 32;
  const int64_t quads = (g.N + 3) / 4;
  const int64_t rows = (int64_t)G * g.dim;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < rows * quads;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t gd = k / quads, q4 = k - gd * quads;
    const int grp = (int)(gd / g.dim), d = (int)(gd % g.dim);
    const uint4 r = philox(make_uint4((uint32_t)q4, 0u, lattice_id(0, grp, 0),
                                      ctr_w(TAG_COUPLING, 0, (uint32_t)d)), rk);
    uint32_t *out = J + gd * g.N;
    const uint32_t half = (uint32_t)(g.N / 2);
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q) {
      const uint32_t i = (uint32_t)(4 * q4 + q);
      if (i < g.N) out[cs_word(i, colour_of(g, i), half)] = word_of(r, q);
    }
  }
}

struct NoAdd {
  __device__ void operator()(uint32_t, uint32_t, uint32_t) const {}
};

constexpr int kResThreads = 512;    // at most, msc_res_kernel
constexpr int64_t kResSweeps = 1024;  // sweeps per launch
constexpr size_t kResSmem = 227 * 1024 - 64;  // beside its thresholds
constexpr uint32_t kSlots = 4;  // slots of one (set, group) per thread of a colour phase

// Place of thread item k: (a, grp) and the first slot of its block, with the
// item's number among those of the slot block (fquads: quads per colour).
struct EaItem {
  uint32_t st, a, grp, t0, t1, j4;
};

__device__ __forceinline__ EaItem ea_item(const Geom &g, uint32_t k, const FastDiv &ftb) {
  const uint32_t quads = ((uint32_t)g.N / 2 + 3) / 4;
  const uint32_t G = (uint32_t)g.n_real / 32, T = (uint32_t)g.n_temps, TB = (T + kSlots - 1) / kSlots;
  EaItem x;
  const uint32_t sb = fdiv(k, g.fquads);
  x.j4 = k - sb * quads;
  x.st = fdiv(sb, ftb);  // sb = (a G + grp) TB + tb
  x.a = fdiv(x.st, g.fgrp);
  x.grp = x.st - x.a * G;
  x.t0 = (sb - x.st * TB) * kSlots;
  x.t1 = min(x.t0 + kSlots, T);
  return x;
}

// One colour phase over all word-lattices, L % 8 == 0.  Thread k takes one
// quad of colour sites (j4) in the word-lattices (a, grp, t) of kSlots
// consecutive slots t of one replica set a and group grp, one slot after the
// other.  Those updates share the quad's geometry and coupling words, read
// once (ea_cs.cuh); each word-lattice draws its own uniforms, so the mapping
// of updates to threads does not change the result.  kPair (w = 64, Sec. 5:
// 64 spins per variable): groups 2q and 2q + 1 of one (set, slot) share their
// uniforms, keyed by q.  ftb divides by the number of slot blocks.  Register
// bound: two CTAs per SM (the coupling words stay live across the slots).
// The geometry does not depend on the previous phase and comes before
// griddep_wait(); the next phase starts only then, since the CTAs of several
// phases that wait at once lie unevenly on the SMs.  10 sweeps in us, release
// first / here: 3D L = 8 32 groups x 33 slots x 2 (0.95 CTAs per SM) 95 / 68, 2D
// L = 40 14 x 33 (1.3) 89 / 65; 4 CTAs per SM and more are equal.
template <int kDim, bool kPair>
__global__ void __launch_bounds__(256, 2)
    msc_phase_kernel(uint32_t *__restrict__ w, const uint32_t *__restrict__ J, Geom g, uint32_t total,
                     FastDiv ftb, const uint32_t *__restrict__ thr, RoundKeys rk, uint32_t sweep, int colour) {
  const uint32_t N = (uint32_t)g.N, wctr = ctr_w(TAG_UPDATE, (uint32_t)colour, 0);
  const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= total) return;
  const EaItem x = ea_item(g, k, ftb);
  const uint32_t rkey = kPair ? x.grp >> 1 : x.grp;
  uint32_t *ws = w + (size_t)x.st * (uint32_t)g.n_temps * N;  // slot t of (a, grp) is word-lattice st T + t
  const EaQuadGeom q = ea_quad_geom<kDim>(x.j4, colour, (uint32_t)g.L, g.fL);
  griddep_wait();
  griddep_release();
  const EaQuadJ c = ea_quad_couplings<kDim>(J + (size_t)x.grp * kDim * N, q, colour, N);
#pragma unroll 1
  for (uint32_t t = x.t0; t < x.t1; ++t) {
    const uint4 r = philox(make_uint4(x.j4, sweep, lattice_id(x.a, rkey, t), wctr), rk);
    const uint32_t t4 = __ldg(thr + 4 * t + 1), t8 = __ldg(thr + 4 * t + 2);
    const uint32_t t12 = kDim == 3 ? __ldg(thr + 4 * t + 3) : 0u;
    ea_quad_update<kDim, false>(ws + (size_t)t * N, q, c, colour, N, r, t4, t8, t12, NoAdd());
  }
}

// The same for any even L.  Thread k takes one site (lanes consecutive colour
// indices, so that every load of a warp is contiguous) in up to kSlots slots,
// with its neighbour indices and coupling words found once; the four lanes of
// a quad draw the calls of four slots and exchange their words (quad_transpose).
// A thread per quad and slot read its words four apart from the next lane's and
// looked up each site's geometry and couplings again for every slot: 10 sweeps
// of 256 x 30 x 2 lattices of L = 12 with 2 measurements and exchanges took 151
// us, 135 here.  Draws before griddep_wait(), the next phase after it (10 sweeps
// in us, next phase first / here: 3D L = 18 20 x 4 x 2, 1.5 CTAs per SM, 73 / 49).
template <int kDim, bool kPair>
__global__ void __launch_bounds__(256)
    msc_site_phase_kernel(uint32_t *__restrict__ w, const uint32_t *__restrict__ J, Geom g, uint32_t total,
                          FastDiv ftb, const uint32_t *__restrict__ thr, RoundKeys rk, uint32_t sweep, int colour) {
  const uint32_t N = (uint32_t)g.N;
  const uint32_t id = blockIdx.x * blockDim.x + threadIdx.x, lane4 = id & 3u;
  const EaItem x = ea_item(g, min(id >> 2, total - 1), ftb);  // (lanes beyond the end draw the last quad again)
  const uint32_t rkey = kPair ? x.grp >> 1 : x.grp;
  uint32_t r[kSlots];
  {
    const uint4 v = philox(make_uint4(x.j4, sweep, lattice_id(x.a, rkey, min(x.t0 + lane4, x.t1 - 1)),
                                      ctr_w(TAG_UPDATE, (uint32_t)colour, 0)), rk);
    r[0] = v.x;
    r[1] = v.y;
    r[2] = v.z;
    r[3] = v.w;
  }
  quad_transpose(r);  // r[s]: the site's word in slot t0 + s
  const uint32_t j = 4 * x.j4 + lane4;
  if ((id >> 2) >= total || j >= N / 2) return;
  const EaSite e = ea_site<kDim>(j, colour, (uint32_t)g.L, g.fL);
  uint32_t *ws = w + (size_t)x.st * (uint32_t)g.n_temps * N;
  griddep_wait();
  griddep_release();
  const EaSiteJ c = ea_site_couplings<kDim>(J + (size_t)x.grp * kDim * N, e, colour, N);
  // all slots' words first, so that their latencies overlap
  EaSiteW v[kSlots];
#pragma unroll
  for (uint32_t s = 0; s < kSlots; ++s)
    v[s] = ea_site_words<kDim>(ws + (size_t)min(x.t0 + s, x.t1 - 1) * N, e, colour, N);
#pragma unroll
  for (uint32_t s = 0; s < kSlots; ++s) {
    const uint32_t t = x.t0 + s;
    if (t >= x.t1) break;
    const Flip f = ea_site_flip<kDim>(v[s], c, r[s], __ldg(thr + 4 * t + 1), __ldg(thr + 4 * t + 2),
                                      kDim == 3 ? __ldg(thr + 4 * t + 3) : 0u);
    ws[(size_t)t * N + (uint32_t)colour * (N / 2) + j] = v[s].S ^ f.F;
  }
}

// Several sweeps of lattices that fit in shared memory: a CTA holds the words
// of one slot block (kSlots slots of one set and group) and the group's
// couplings, and runs every sweep of the call with a barrier per colour phase
// instead of a launch.  Items, draws and updates are those of the phase kernels.
// Bound by the latency of a phase in one CTA (L = 12: 1.9 us for two sites per
// thread in four slots, 3.6 with a launch per phase): 10 sweeps of 256 x 30 x 2
// lattices of L = 12 with 2 measurements and exchanges 116 -> 100 us.  The next
// kernel starts after griddep_wait(): CTAs of several calls that wait at once
// pile up on some SMs (10 sweeps of 50 x 4 x 2 lattices of 2D L = 60 100 us, 70
// here).
template <int kDim, bool kPair, bool kRow>
__global__ void __launch_bounds__(kResThreads)
    msc_res_kernel(uint32_t *__restrict__ w, const uint32_t *__restrict__ J, Geom g, FastDiv ftb,
                   const uint32_t *__restrict__ thr, RoundKeys rk, uint32_t sweep0, uint32_t n_sweeps) {
  extern __shared__ uint4 msc_res_smem[];
  __shared__ uint32_t s_thr[kSlots][4];
  const uint32_t N = (uint32_t)g.N, half = N / 2, quads = (half + 3) / 4, lane4 = threadIdx.x & 3u;
  const uint32_t G = (uint32_t)g.n_real / 32, T = (uint32_t)g.n_temps, TB = (T + kSlots - 1) / kSlots;
  const uint32_t st = fdiv(blockIdx.x, ftb), a = fdiv(st, g.fgrp), grp = st - a * G;
  const uint32_t t0 = (blockIdx.x - st * TB) * kSlots, n_slots = min(kSlots, T - t0);
  const uint32_t rkey = kPair ? grp >> 1 : grp;
  uint32_t *sw = reinterpret_cast<uint32_t *>(msc_res_smem), *sJ = sw + kSlots * N;
  uint32_t *ws = w + ((size_t)st * T + t0) * N;
  const uint32_t *gJ = J + (size_t)grp * kDim * N;
  griddep_wait();
  griddep_release();
#pragma unroll 8
  for (uint32_t i = threadIdx.x; i < n_slots * N; i += blockDim.x) sw[i] = ws[i];
#pragma unroll 8
  for (uint32_t i = threadIdx.x; i < kDim * N; i += blockDim.x) sJ[i] = gJ[i];
  if (threadIdx.x < 4 * n_slots) s_thr[threadIdx.x >> 2][threadIdx.x & 3u] = thr[4 * t0 + threadIdx.x];
  __syncthreads();
  for (uint32_t k = 0; k < n_sweeps; ++k) {
    const uint32_t sweep = sweep0 + k;
#pragma unroll 1
    for (int colour = 0; colour < 2; ++colour) {
      const uint32_t wctr = ctr_w(TAG_UPDATE, (uint32_t)colour, 0);
      if (kRow) {
        for (uint32_t j4 = threadIdx.x; j4 < quads; j4 += blockDim.x) {
          const EaQuadGeom q = ea_quad_geom<kDim>(j4, colour, (uint32_t)g.L, g.fL);
          const EaQuadJ c = ea_quad_couplings<kDim>(sJ, q, colour, N);
#pragma unroll 1
          for (uint32_t s = 0; s < n_slots; ++s) {
            const uint4 r = philox(make_uint4(j4, sweep, lattice_id(a, rkey, t0 + s), wctr), rk);
            ea_quad_update<kDim, false>(sw + s * N, q, c, colour, N, r, s_thr[s][1], s_thr[s][2], s_thr[s][3],
                                        NoAdd());
          }
        }
      } else {
        // whole warps, for the exchange of words between lanes
        for (uint32_t id = threadIdx.x; (id & ~31u) < 4 * quads; id += blockDim.x) {
          const uint32_t j4 = min(id >> 2, quads - 1), j = id;
          const uint4 v = philox(make_uint4(j4, sweep, lattice_id(a, rkey, t0 + min(lane4, n_slots - 1)), wctr), rk);
          uint32_t r[kSlots] = {v.x, v.y, v.z, v.w};
          quad_transpose(r);  // r[s]: the site's word in slot t0 + s
          if (j >= half) continue;
          const EaSite e = ea_site<kDim>(j, colour, (uint32_t)g.L, g.fL);
          const EaSiteJ c = ea_site_couplings<kDim>(sJ, e, colour, N);
          EaSiteW x[kSlots];
#pragma unroll
          for (uint32_t s = 0; s < kSlots; ++s)
            x[s] = ea_site_words<kDim>(sw + min(s, n_slots - 1) * N, e, colour, N);
#pragma unroll
          for (uint32_t s = 0; s < kSlots; ++s) {
            if (s >= n_slots) break;
            const Flip f = ea_site_flip<kDim>(x[s], c, r[s], s_thr[s][1], s_thr[s][2], s_thr[s][3]);
            sw[s * N + (uint32_t)colour * half + j] = x[s].S ^ f.F;
          }
        }
      }
      __syncthreads();
    }
  }
#pragma unroll 8
  for (uint32_t i = threadIdx.x; i < n_slots * N; i += blockDim.x) ws[i] = sw[i];
}

// Words <-> one int8 per spin, [n_sets][n_temps][n_real][N]: a thread takes
// kSites consecutive sites of a word-lattice in all 32 realisations, the
// kSites bytes of each in one access (256 x 30 x 2 x L = 12 to bytes: 17.4 us
// with one site and single bytes).  kSites 4: N is a multiple of 4, the byte
// buffer 4-byte aligned.
template <int kSites>
__device__ __forceinline__ int64_t first_lat(const Geom &g, int64_t wl) {
  const int G = g.n_real / 32;
  const int64_t q = wl / g.n_temps;
  const int t = (int)(wl - q * g.n_temps), a = (int)(q / G), grp = (int)(q - (int64_t)a * G);
  return ((int64_t)a * g.n_temps + t) * g.n_real + 32 * grp;
}

template <int kSites, typename Bytes>
__global__ void unpack_msc_kernel(const uint32_t *__restrict__ w, Bytes *__restrict__ out, Geom g, uint32_t total,
                                  FastDiv fitems) {
  const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= total) return;
  const uint32_t wl = fdiv(k, fitems), i = (k - wl * fitems.d) * kSites, N = (uint32_t)g.N;
  uint32_t v[kSites];
#pragma unroll
  for (int s = 0; s < kSites; ++s) v[s] = w[(size_t)wl * N + cs_word(i + s, colour_of(g, i + s), N / 2)];
  Bytes *o = out + (size_t)first_lat<kSites>(g, wl) * (N / kSites) + i / kSites;
#pragma unroll 8
  for (int b = 0; b < 32; ++b) {
    uint32_t x = 0;
#pragma unroll
    for (int s = 0; s < kSites; ++s) x |= ((v[s] >> b & 1u) * 0xFEu | 1u) << (8 * s);  // 0x01 | 0xFE = -1
    o[(size_t)b * (N / kSites)] = (Bytes)x;
  }
}

template <int kSites, typename Bytes>
__global__ void pack_msc_kernel(const Bytes *__restrict__ in, uint32_t *__restrict__ w, Geom g, uint32_t total,
                                FastDiv fitems) {
  const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= total) return;
  const uint32_t wl = fdiv(k, fitems), i = (k - wl * fitems.d) * kSites, N = (uint32_t)g.N;
  const Bytes *p = in + (size_t)first_lat<kSites>(g, wl) * (N / kSites) + i / kSites;
  uint32_t v[kSites];
#pragma unroll
  for (int s = 0; s < kSites; ++s) v[s] = 0u;
#pragma unroll 8
  for (int b = 0; b < 32; ++b) {
    const uint32_t x = p[(size_t)b * (N / kSites)];
#pragma unroll
    for (int s = 0; s < kSites; ++s) v[s] |= (x >> (8 * s + 7) & 1u) << b;  // the sign
  }
#pragma unroll
  for (int s = 0; s < kSites; ++s) w[(size_t)wl * N + cs_word(i + s, colour_of(g, i + s), N / 2)] = v[s];
}

unsigned capped(int64_t n) {
  unsigned g = grid_for(n, 256);
  return g > (1u << 20) ? (1u << 20) : g;
}

}  // namespace

cudaError_t launch_init_msc(spin_lattice *h) {
  const Geom &g = h->g;
  const int64_t words = (int64_t)g.n_sets * (g.n_real / 32) * g.n_temps * g.N;
  if (!h->d.hot_start) return cudaMemsetAsync(h->spins, 0, (size_t)words * 4, h->stream);
  init_msc_kernel<<<capped(words / 4 + 1), 256, 0, h->stream>>>((uint32_t *)h->spins, g,
                                                                   make_round_keys(h->d.seed));
  return cudaGetLastError();
}

cudaError_t launch_couplings_msc(spin_lattice *h) {
  const Geom &g = h->g;
  couplings_msc_kernel<<<capped((int64_t)(g.n_real / 32) * g.dim * g.N / 4 + 1), 256, 0, h->stream>>>(
      (uint32_t *)h->couplings, g, make_round_keys(h->d.seed));
  return cudaGetLastError();
}

namespace {
using ResKern = decltype(&msc_res_kernel<3, false, false>);

// Sweeps of a call with the lattices in shared memory (msc_res_kernel): CTAs,
// threads and shared memory; grid 0 where the phase launches are better.
struct MscRes {
  unsigned grid = 0;
  int threads = 0;
  size_t smem = 0;
};

// The rule compares two estimates in us, fitted to calls of 2 to 16 sweeps of
// 1 to 2048 word-lattices, 3D L = 4 ... 20 and 2D L = 8 ... 94.  Here: start and
// loading (per word and thread, once per round of CTAs), then a sweep per
// round of CTAs; the phases: the larger of latency and words, and half the
// smaller.  Measured, phases against here, 4 and 16 sweeps: 3D L = 6, 512
// word-lattices x 4 slots, 28 / 116 against 17 / 44; L = 12, 480 word-lattices,
// 35 / 121 against 27 / 74; L = 16, the same, 46 / 170 against 42 / 115; L = 20, 64
// word-lattices, 22 / 92 against 85 / 261 (phases).
MscRes msc_res_plan(const spin_lattice *h, int64_t n_sweeps) {
  const Geom &g = h->g;
  MscRes p;
  const size_t smem = (size_t)(kSlots + (uint32_t)g.dim) * (size_t)g.N * 4;
  if (n_sweeps < 3 || smem > kResSmem) return p;
  const int sms = h->sms;
  const bool row = g.L % 8 == 0;
  const uint32_t quads = (uint32_t)((g.N / 2 + 3) / 4), items = row ? quads : 4 * quads;
  const uint32_t rounds = (items + kResThreads - 1) / kResThreads;
  const uint32_t T = (uint32_t)g.n_temps, TB = (T + kSlots - 1) / kSlots, st = (uint32_t)g.n_sets * (uint32_t)(g.n_real / 32);
  const int threads = std::max(128, (int)(((items + rounds - 1) / rounds + 31) / 32 * 32));  // 128: to load with
  const double n = (double)n_sweeps, per_sm = std::ceil((double)st * TB / sms), d = g.dim == 3 ? 1.0 : 0.75;
  const double frac = (double)items / kResThreads;
  const double sweep = row ? 1.6 + 1.2 * d * frac * std::min(kSlots, T) : 0.6 + 1.75 * d * frac;
  const double here = 7.0 + 0.17 * (double)smem / 4.0 / threads * per_sm +
                      n * sweep * std::max(1.0, per_sm * threads / 448.0);
  const double lat = row ? 2.0 + 1.1 * std::min(kSlots, T) : 3.3;
  const double words = (row ? 3.6e-6 : 4.8e-6) * d * (double)st * T * (double)g.N;
  if (here > 0.95 * (3.5 + n * (std::max(lat, words) + 0.5 * std::min(lat, words)))) return p;
  p.grid = st * TB;
  p.threads = threads;
  p.smem = std::min(std::max(smem, spread_smem(p.grid, sms)), kResSmem);
  return p;
}
}  // namespace

cudaError_t launch_sweeps_msc_ea(spin_lattice *h, const uint32_t *J, int64_t n_sweeps) {
  const Geom &g = h->g;
  const RoundKeys rk = make_round_keys(h->d.seed);
  const bool pair = h->msc_width == 64;
  const bool row_quads = g.L % 8 == 0;
  const uint32_t TB = ((uint32_t)g.n_temps + kSlots - 1) / kSlots;
  const uint32_t work = (uint32_t)g.n_sets * (uint32_t)(g.n_real / 32) * TB * (uint32_t)((g.N / 2 + 3) / 4);
  const FastDiv ftb = make_fastdiv(TB);
  using Kern = decltype(&msc_phase_kernel<3, false>);
  const Kern kerns[2][2][2] = {{{msc_site_phase_kernel<2, false>, msc_phase_kernel<2, false>},
                                {msc_site_phase_kernel<2, true>, msc_phase_kernel<2, true>}},
                               {{msc_site_phase_kernel<3, false>, msc_phase_kernel<3, false>},
                                {msc_site_phase_kernel<3, true>, msc_phase_kernel<3, true>}}};
  const Kern kern = kerns[g.dim == 3][pair][row_quads];
  const ResKern res_kerns[2][2][2] = {{{msc_res_kernel<2, false, false>, msc_res_kernel<2, false, true>},
                                       {msc_res_kernel<2, true, false>, msc_res_kernel<2, true, true>}},
                                      {{msc_res_kernel<3, false, false>, msc_res_kernel<3, false, true>},
                                       {msc_res_kernel<3, true, false>, msc_res_kernel<3, true, true>}}};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
  static OncePerDevice limits;
  if (!limits.done(dev)) {
    for (int k = 0; k < 8; ++k) {
      cudaError_t e = cudaFuncSetAttribute(kerns[k >> 2][k >> 1 & 1][k & 1],
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmem);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(res_kerns[k >> 2][k >> 1 & 1][k & 1], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kResSmem);
      if (e != cudaSuccess) return e;
    }
    limits.mark(dev);
  }
  const MscRes res = msc_res_plan(h, n_sweeps);
  if (res.grid) {
    const ResKern kern = res_kerns[g.dim == 3][pair][row_quads];
    cudaError_t e = cudaSuccess;
    for (int64_t k = 0; e == cudaSuccess && k < n_sweeps; k += kResSweeps)
      e = launch_dependent(kern, dim3(res.grid), dim3(res.threads), res.smem, h->stream, (uint32_t *)h->spins, J, g,
                           ftb, (const uint32_t *)h->d_thr, rk, (uint32_t)(h->sweeps_done + k),
                           (uint32_t)std::min<int64_t>(n_sweeps - k, kResSweeps));
    return e;
  }
  const int64_t threads = row_quads ? work : 4 * (int64_t)work;  // < 2^30: fewer than 2^27 words
  const int grid = (int)grid_for(threads, 256);
  // Up to two CTAs per SM one more on some SMs counts; beyond, three and four
  // at a time are faster.  10 sweeps in us with an exchange and E, M, Q after every
  // second, as they fall / spread: 2D L = 40, 33 slots, 0.9 CTAs per SM 156 / 143,
  // 1.7 206 / 178; 3D L = 16, 32 slots, 0.8 169 / 149, 1.9 197 / 197; L = 12, 33 slots, 2.0
  // 138 / 122; 2D L = 64, 4 slots, 1.1 140 / 144, 1.9 186 / 165.
  const size_t smem = grid <= 2 * h->sms ? spread_smem(grid, h->sms) : 0;
  for (int64_t k = 0; k < n_sweeps; ++k) {
    const uint32_t sweep = (uint32_t)(h->sweeps_done + k);
    for (int colour = 0; colour < 2; ++colour) {
      const cudaError_t e = launch_dependent(kern, dim3(grid), dim3(256), smem, h->stream,
                                             (uint32_t *)h->spins, J, g, work, ftb, (const uint32_t *)h->d_thr,
                                             rk, sweep, colour);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

cudaError_t launch_sweeps_msc2d(spin_lattice *h, int64_t n_sweeps);  // msc2d.cu

cudaError_t launch_sweeps_msc(spin_lattice *h, const uint32_t *J, int64_t n_sweeps) {
  if (h->d.model == SPIN_EA) return launch_sweeps_msc_ea(h, J, n_sweeps);
  return launch_sweeps_msc2d(h, n_sweeps);
}

cudaError_t launch_unpack_msc2d(spin_lattice *h, int8_t *out);      // msc2d.cu
cudaError_t launch_pack_msc2d(spin_lattice *h, const int8_t *in);   // msc2d.cu

cudaError_t launch_unpack_msc(spin_lattice *h, int8_t *out) {
  if (h->d.model != SPIN_EA) return launch_unpack_msc2d(h, out);
  const Geom &g = h->g;
  const uint32_t sites = (g.N & 3) == 0 && ((uintptr_t)out & 3u) == 0 ? 4 : 1;
  const uint32_t items = (uint32_t)(g.N / sites);
  const uint32_t total = (uint32_t)((int64_t)g.n_sets * (g.n_real / 32) * g.n_temps) * items;  // < 2^27
  if (sites == 4)
    unpack_msc_kernel<4><<<grid_for(total, 256), 256, 0, h->stream>>>((const uint32_t *)h->spins, (uint32_t *)out, g,
                                                                      total, make_fastdiv(items));
  else
    unpack_msc_kernel<1><<<grid_for(total, 256), 256, 0, h->stream>>>((const uint32_t *)h->spins, (uint8_t *)out, g,
                                                                      total, make_fastdiv(items));
  return cudaGetLastError();
}

cudaError_t launch_pack_msc(spin_lattice *h, const int8_t *in) {
  if (h->d.model != SPIN_EA) return launch_pack_msc2d(h, in);
  const Geom &g = h->g;
  const uint32_t sites = (g.N & 3) == 0 && ((uintptr_t)in & 3u) == 0 ? 4 : 1;
  const uint32_t items = (uint32_t)(g.N / sites);
  const uint32_t total = (uint32_t)((int64_t)g.n_sets * (g.n_real / 32) * g.n_temps) * items;  // < 2^27
  if (sites == 4)
    pack_msc_kernel<4><<<grid_for(total, 256), 256, 0, h->stream>>>((const uint32_t *)in, (uint32_t *)h->spins, g,
                                                                    total, make_fastdiv(items));
  else
    pack_msc_kernel<1><<<grid_for(total, 256), 256, 0, h->stream>>>((const uint8_t *)in, (uint32_t *)h->spins, g, total,
                                                                    make_fastdiv(items));
  return cudaGetLastError();
}

}  // namespace spin
