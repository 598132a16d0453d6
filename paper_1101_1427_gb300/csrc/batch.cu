// Batched persistent launch: many lattices of several handles, many sweeps,
// one kernel launch.  The paper maps independent replicas to thread blocks
// (Sec. 5) and tempering copies to extra blocks (Sec. 6) but returns to the
// host for every exchange; here measurement, exchange decisions and the
// exchange itself run inside the same persistent launch.
//
// Work units:
//   EA unit     = one realisation group (32 realisations) of an EA handle in
//                 the coded layout: all replica sets, all temperature slots.
//                 Its team of P CTAs splits the slots: CTA p owns slots
//                 [p n_T / P, (p+1) n_T / P) of every set, so a colour phase
//                 needs no synchronisation beyond __syncthreads.  Exchange
//                 steps read the energy of a neighbour's slot and write its
//                 words, so they are framed by two team barriers.
//   Ising unit  = one lattice of a 2D int8 ferromagnet handle; its team
//                 splits the rows and synchronises after each colour phase.
// Team barriers are counters in global memory; every wait is bounded in
// time (globaltimer) and sets the error word on expiry, after which all
// CTAs leave the kernel and spin_sync reports SPIN_ETIMEOUT.
//
// The kernel is launched cooperatively so that all CTAs are co-resident.
#include <algorithm>
#include <map>
#include <mutex>
#include <vector>

#include "bitslice.cuh"
#include "ea_cs.cuh"
#include "i8chunk.cuh"
#include "internal.h"
#include "msc2d_block.cuh"

namespace spin {

struct BatchUnit {
  int kind;        // 0 EA coded group, 1 Ising 2D int8 lattice, 2 Ising 2D coded lattice
  int team_first;  // first CTA of the team
  int team_size;   // CTAs in the team
  int L;
  uint32_t N;
  int n_T, n_sets;
  FastDiv fL;
  const uint32_t *thr;  // [n_T][4]
  int key;              // round keys of the handle
  const long long *ctr;  // handle's [sweeps_done, pt_steps_done] on the device
  uint32_t sweep0;      // ctr[0] when the launch starts
  uint32_t pt0;         // ctr[1] when the launch starts
  unsigned *bar;        // the team's barrier counter (zeroed before the launch)
  // EA
  uint32_t *w;          // EA: words of set 0, this group, slot 0; coded Ising: the lattice's words
  size_t set_stride;    // words between replica sets
  const uint32_t *J;    // couplings of this group [3][N]
  int grp, n_real;
  int rgrp;             // key of the group's uniforms: grp (w = 32) or grp / 2 (w = 64)
  const uint32_t *pt_tab;
  const int32_t *pt_off, *pt_len;
  const double *pt_dbeta;
  long long *E_series, *M_series, *Q_series, *accepted;
  int *labels;          // configuration labels of the handle's lattices (or NULL)
  long long n_lat;      // lattices of the handle (series row length)
  int *Escr;            // [n_sets][n_T][32] unsatisfied-bond counts
  // Ising
  int8_t *s;
  FastDiv fC;           // divides by the L / 8 chunks of 8 sites in a row
  long long lat_index;
  uint32_t lid;
  int slot;
};

constexpr int kMaxUnits = 96;
constexpr int kMaxHandles = 16;

// Everything a launch needs travels in the kernel's parameter space (under
// 32 KB), so a launch is one kernel node: capturable, nothing to upload.
struct BatchParams {
  int n_units;
  int measure_every, pt_every, extra;
  uint32_t staged_words;  // dynamic shared memory for couplings, in words
  uint32_t smem_words;    // all of it; more than staged_words: EA words stay resident
  int64_t n_sweeps;
  uint64_t timeout_ns;
  RoundKeys keys[kMaxHandles];
  BatchUnit units[kMaxUnits];
};
// kernel parameters are limited to 32764 bytes
static_assert(sizeof(BatchParams) <= 32764, "batch parameters exceed the kernel parameter space");

namespace {

constexpr int kPairThreads = 256;      // per CTA, two CTAs per SM
constexpr int kResidentThreads = 512;  // one CTA per SM that keeps words in shared memory
constexpr int kPl = 12;  // per-lane counter planes (counts < 4096)

__device__ __forceinline__ uint32_t ld_acquire(const unsigned *p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

struct Sync {
  unsigned *ctr;
  unsigned target;
  int size;
  int *err;
  uint64_t timeout_ns;
  int extra;  // arrivals that never come (fault injection for the timeout test)
};

// A team barrier in two halves: the arrival makes the CTA's writes before it
// visible to every CTA whose wait returns true; work that touches none of the
// team's data may come in between.  The wait returns false if the team (or the
// whole launch) has failed.
__device__ __forceinline__ void team_arrive(Sync &sy) {
  __syncthreads();
  sy.target += sy.size;
  // release: the CTA's writes (ordered before this by the barrier above)
  // become visible to every CTA that acquires the final count
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(sy.ctr) : "memory");
}

__device__ bool team_wait(const Sync &sy) {
  __shared__ int s_ok;
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned want = sy.target + (unsigned)sy.extra;
    const uint64_t t0 = globaltimer();
    while ((int)(ld_acquire(sy.ctr) - want) < 0) {
      if (*(volatile int *)sy.err) {
        ok = 0;
        break;
      }
      if (globaltimer() - t0 > sy.timeout_ns) {
        atomicExch(sy.err, 1);
        ok = 0;
        break;
      }
      __nanosleep(100);
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

__device__ __forceinline__ bool team_barrier(Sync &sy) {
  team_arrive(sy);
  return team_wait(sy);
}

// Harley-Seal counting of 1-bit planes: eight planes go through seven
// carry-save adders into (ones, twos, fours) and one plane of weight 8,
// which is rippled into the counter; flush() adds the remainders.
struct HsCount {
  uint32_t C[kPl];
  uint32_t ones, twos, fours;
  __device__ HsCount() : ones(0), twos(0), fours(0) {
#pragma unroll
    for (int k = 0; k < kPl; ++k) C[k] = 0;
  }
  __device__ __forceinline__ void add8(const uint32_t (&x)[8]) {
    uint32_t twosA, twosB, foursA, foursB, eights;
    csa(twosA, ones, ones, x[0], x[1]);
    csa(twosB, ones, ones, x[2], x[3]);
    csa(foursA, twos, twos, twosA, twosB);
    csa(twosA, ones, ones, x[4], x[5]);
    csa(twosB, ones, ones, x[6], x[7]);
    csa(foursB, twos, twos, twosA, twosB);
    csa(eights, fours, fours, foursA, foursB);
    ripple_at<3>(C, eights);
  }
  __device__ __forceinline__ void flush() {
    ripple_at<2>(C, fours);
    ripple_at<1>(C, twos);
    ripple_at<0>(C, ones);
    ones = twos = fours = 0;
  }
};

// counter planes += the sum of four 3-bit values (a_k0 + 2 a_k1 + 4 a_k2),
// formed first by a small adder tree (at most 24, five bits)
__device__ __forceinline__ void add_quad(uint32_t (&C)[kPl], const uint32_t (&a)[4][3]) {
  // s = a0 + a1 and t = a2 + a3 (4 bits each)
  uint32_t s[4], t[4];
  {
    uint32_t c = a[0][0] & a[1][0];
    s[0] = a[0][0] ^ a[1][0];
    csa(c, s[1], a[0][1], a[1][1], c);
    csa(s[3], s[2], a[0][2], a[1][2], c);
  }
  {
    uint32_t c = a[2][0] & a[3][0];
    t[0] = a[2][0] ^ a[3][0];
    csa(c, t[1], a[2][1], a[3][1], c);
    csa(t[3], t[2], a[2][2], a[3][2], c);
  }
  // v = s + t (5 bits)
  uint32_t v[5], c = s[0] & t[0];
  v[0] = s[0] ^ t[0];
  csa(c, v[1], s[1], t[1], c);
  csa(c, v[2], s[2], t[2], c);
  csa(v[4], v[3], s[3], t[3], c);
  // counter += v
  uint32_t carry = 0;
#pragma unroll
  for (int k = 0; k < kPl; ++k) {
    const uint32_t x = k < 5 ? v[k] : 0u;
    const uint32_t n = (C[k] & x) | (carry & (C[k] ^ x));
    C[k] = C[k] ^ x ^ carry;
    carry = n;
  }
}

// Sum of the per-lane counters of a warp; every lane returns the count of
// realisation bit `lane`.
__device__ __forceinline__ int warp_bit_counts(const uint32_t (&C)[kPl]) {
  constexpr int K = kPl + 5;
  uint32_t P[K];
#pragma unroll
  for (int k = 0; k < K; ++k) P[k] = k < kPl ? C[k] : 0u;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    uint32_t carry = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t a = P[k], b = __shfl_xor_sync(0xffffffffu, P[k], o);
      P[k] = a ^ b ^ carry;
      carry = (a & b) | (carry & (a ^ b));
    }
  }
  const int lane = threadIdx.x & 31;
  int cnt = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) cnt += (int)((P[k] >> lane) & 1u) << k;
  return cnt;
}

// One colour phase of one word-lattice by one warp (lanes strided over the
// quads of colour sites).  With kCount the post-update number of
// unsatisfied bonds of each updated (colour-1) site is added to C: every
// bond joins a colour-0 and a colour-1 site, so summing over colour-1 sites
// counts each bond once.
// Collects the post-update counts of the (up to) four sites of a quad and
// adds them to the counter in one go.
struct AddTo {
  uint32_t (&C)[kPl];
  uint32_t (&buf)[4][3];
  int &n;
  __device__ void operator()(uint32_t x0, uint32_t x1, uint32_t x2) const {
    buf[n][0] = x0;
    buf[n][1] = x1;
    buf[n][2] = x2;
    if (++n == 4) {
      add_quad(C, buf);
      n = 0;
    }
  }
};

// The counting passes of a CTA go over the chunks (128 sites: 32 quads, one per
// lane) of all its word-lattices in turn, an equal share of them per warp, so
// that ten word-lattices take eight warps 1.25 times and not twice as long as
// eight; a warp sums up its part of each word-lattice that it touches.
struct Share {
  uint32_t c, end;  // chunks of all word-lattices
};

__device__ __forceinline__ Share warp_share(uint32_t chunks, uint32_t warp, uint32_t warps) {
  Share s;
  s.c = chunks * warp / warps;
  s.end = chunks * (warp + 1) / warps;
  return s;
}

// One colour phase of the chunks [c0, c1) of one word-lattice (colour-split)
// by a warp.  With kCount the post-update number of
// unsatisfied bonds of each updated (colour-1) site is added to C: every
// bond joins a colour-0 and a colour-1 site, so summing over colour-1 sites
// counts each bond once.
template <bool kCount>
__device__ __forceinline__ void ea_phase_warp(uint32_t *__restrict__ s, const uint32_t *__restrict__ Jg,
                                              const BatchUnit &U, const RoundKeys &rk, uint32_t sweep,
                                              uint32_t lid, int colour, uint32_t t4, uint32_t t8,
                                              uint32_t t12, uint32_t c0, uint32_t c1, uint32_t (&C)[kPl]) {
  uint32_t buf[4][3];
  int n = 0;
  if ((U.L & 7) != 0) {  // whole warps: lanes take consecutive sites
    ea_sites_phase(s, Jg, colour, (uint32_t)U.L, U.N, U.fL, rk, sweep, lid, t4, t8, t12, c0, c1,
                   [&](const Flip &f, bool on) {
                     if (!kCount) return;
                     uint32_t a0 = 0, a1 = 0, a2 = 0;
                     if (on) ea_after(f, a0, a1, a2);
                     AddTo{C, buf, n}(a0, a1, a2);  // four sites per 128: the buffer is empty at the end
                   });
    return;
  }
  const uint32_t quads = U.N / 8;
  const uint32_t wctr = ctr_w(TAG_UPDATE, (uint32_t)colour, 0);
  const uint32_t end = min(32u * c1, quads);
  for (uint32_t j4 = 32u * c0 + (threadIdx.x & 31u); j4 < end; j4 += 32u) {
    const uint4 r = philox(make_uint4(j4, sweep, lid, wctr), rk);
    const EaQuadGeom q = ea_quad_geom<3>(j4, colour, (uint32_t)U.L, U.fL);
    ea_quad_update<3, kCount>(s, q, ea_quad_couplings<3>(Jg, q, colour, U.N), colour, U.N, r, t4, t8, t12,
                              AddTo{C, buf, n});
  }
}

// Counts per bit the words a[i] (or a[i] ^ b[i]) of i in [i0, i1), by a warp;
// the loads of sixteen words per lane are under way together.
__device__ __forceinline__ void count_words(HsCount &hc, const uint32_t *a, const uint32_t *b, uint32_t i0,
                                            uint32_t i1) {
  uint32_t i = i0 + (threadIdx.x & 31u);
  for (; i + 15 * 32 < i1; i += 16 * 32) {
    uint32_t x[8], y[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = a[i + 32 * k], y[k] = a[i + 32 * (k + 8)];
    if (b) {
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] ^= b[i + 32 * k], y[k] ^= b[i + 32 * (k + 8)];
    }
    hc.add8(x);
    hc.add8(y);
  }
  for (; i + 7 * 32 < i1; i += 8 * 32) {
    uint32_t x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = b ? (a[i + 32 * k] ^ b[i + 32 * k]) : a[i + 32 * k];
    hc.add8(x);
  }
  hc.flush();
  for (; i < i1; i += 32) ripple_at<0>(hc.C, b ? (a[i] ^ b[i]) : a[i]);
}

// What a CTA of kThreads threads does for its unit.
template <int kThreads>
struct Cta {
static constexpr int kWarps = kThreads / 32;

// Per-bit counts of the set bits of n_items word arrays of N words each
// (item k: a_k[i], or a_k[i] ^ b_k[i]), shared out among the warps in chunks
// of 256 words; cnt[k][b] receives item k's count for bit b.  Called by the
// whole CTA.
template <typename ItemFn>
static __device__ void cta_bit_counts(int n_items, uint32_t N, ItemFn item, int (*cnt)[32]) {
  __syncthreads();
  for (int k = threadIdx.x; k < n_items * 32; k += kThreads) (&cnt[0][0])[k] = 0;
  __syncthreads();
  const uint32_t per = (N + 255) / 256, lane = threadIdx.x & 31u;
  Share sh = warp_share(per * (uint32_t)n_items, threadIdx.x >> 5, kWarps);
  while (sh.c < sh.end) {
    const uint32_t k = sh.c / per, c0 = sh.c - k * per, c1 = min(per, c0 + (sh.end - sh.c));
    const uint32_t *a = nullptr, *b = nullptr;
    item((int)k, a, b);
    HsCount hc;
    count_words(hc, a, b, 256 * c0, min(256 * c1, N));
    atomicAdd(&cnt[k][lane], warp_bit_counts(hc.C));
    sh.c += c1 - c0;
  }
  __syncthreads();
}

// Bitwise exchange of the bits set in A between two word arrays of N words
// (N a multiple of 4, 16-byte aligned), by the whole CTA.
static __device__ __forceinline__ void cta_swap_bits(uint32_t *w0, uint32_t *w1, uint32_t N, uint32_t A) {
  uint4 *v0 = reinterpret_cast<uint4 *>(w0), *v1 = reinterpret_cast<uint4 *>(w1);
  const uint32_t n4 = N >> 2;
  uint32_t i = threadIdx.x;
  constexpr int kU = 4;  // pairs of 16-byte words under way per thread
  for (; i + (kU - 1) * kThreads < n4; i += kU * kThreads) {
    uint4 x[kU], y[kU];
#pragma unroll
    for (int k = 0; k < kU; ++k) x[k] = v0[i + k * kThreads], y[k] = v1[i + k * kThreads];
#pragma unroll
    for (int k = 0; k < kU; ++k) {
      const uint4 d = make_uint4((x[k].x ^ y[k].x) & A, (x[k].y ^ y[k].y) & A, (x[k].z ^ y[k].z) & A,
                                 (x[k].w ^ y[k].w) & A);
      v0[i + k * kThreads] = make_uint4(x[k].x ^ d.x, x[k].y ^ d.y, x[k].z ^ d.z, x[k].w ^ d.w);
      v1[i + k * kThreads] = make_uint4(y[k].x ^ d.x, y[k].y ^ d.y, y[k].z ^ d.z, y[k].w ^ d.w);
    }
  }
  for (; i < n4; i += kThreads) {
    const uint4 x0 = v0[i], x1 = v1[i];
    const uint4 d = make_uint4((x0.x ^ x1.x) & A, (x0.y ^ x1.y) & A, (x0.z ^ x1.z) & A, (x0.w ^ x1.w) & A);
    v0[i] = make_uint4(x0.x ^ d.x, x0.y ^ d.y, x0.z ^ d.z, x0.w ^ d.w);
    v1[i] = make_uint4(x1.x ^ d.x, x1.y ^ d.y, x1.z ^ d.z, x1.w ^ d.w);
  }
}

struct NoCount {
  __device__ void operator()(uint32_t, uint32_t, uint32_t) const {}
};

// ---------------------------------------------------------------- EA unit
// The word-lattices of a CTA, numbered g = t * n_sets + a: whole slots while
// the team has at most n_T CTAs, single word-lattices beyond that.
struct Owned {
  int g0, g1;
};

static __device__ __forceinline__ Owned ea_owned(const BatchUnit &U, int part) {
  const int P = U.team_size, W = U.n_T * U.n_sets;
  Owned o;
  o.g0 = P <= U.n_T ? (part * U.n_T / P) * U.n_sets : part * W / P;
  o.g1 = P <= U.n_T ? ((part + 1) * U.n_T / P) * U.n_sets : (part + 1) * W / P;
  return o;
}

// Owned word-lattices kept in shared memory for the whole launch: g = first ..
// first + n - 1 at base + k N.  Word-lattices that another CTA writes or reads
// are never among them: the owner of (a, t) exchanges it with (a, t + 1), so
// those with g < g0 + n_sets may be written by the CTA before (part > 0); and
// there are none when a team has more CTAs than slots, where the overlap reads
// another CTA's words.
struct Resident {
  uint32_t *base;
  int first, n;
};

static __device__ __forceinline__ Resident ea_resident(const BatchUnit &U, int part, uint32_t *base, uint32_t room) {
  const Owned o = ea_owned(U, part);
  Resident r;
  r.base = base;
  r.first = part > 0 ? min(o.g0 + U.n_sets, o.g1) : o.g0;
  r.n = U.team_size <= U.n_T ? min(o.g1 - r.first, (int)(room / U.N)) : 0;
  return r;
}

// Copies the resident word-lattices in (to_shared) or out, by the whole CTA.
static __device__ __forceinline__ void ea_resident_copy(const BatchUnit &U, const Resident &R, bool to_shared) {
  const uint32_t n4 = U.N / 4;
  for (int k = 0; k < R.n; ++k) {
    const int g = R.first + k, a = g % U.n_sets, t = g / U.n_sets;
    uint4 *home = reinterpret_cast<uint4 *>(U.w + a * U.set_stride + (size_t)t * U.N);
    uint4 *here = reinterpret_cast<uint4 *>(R.base + (size_t)k * U.N);
    for (uint32_t i = threadIdx.x; i < n4; i += blockDim.x) {
      if (to_shared) here[i] = home[i];
      else home[i] = here[i];
    }
  }
  __syncthreads();
}

static __device__ bool ea_sweep(const BatchUnit &U, const Resident &R, const uint32_t *Jsrc, int part, const RoundKeys &rk,
                         Sync &sy, uint32_t s_abs, bool measure, bool pt, long long meas_row,
                         uint32_t pt_step) {
  __shared__ int e_cnt[64][32];   // per owned word-lattice counts (energies, then M, then Q)
  __shared__ uint32_t masks[64];  // accept masks per owned word-lattice that starts a pair
  const int P = U.team_size;
  const Owned own = ea_owned(U, part);
  const int g0 = own.g0, g1 = own.g1;
  const int n_w = g1 - g0;  // <= 64
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // chunks of one colour of a word-lattice
  const uint32_t per = ((U.N / 2 + 3) / 4 + 31) / 32;
  const bool need_e = measure || pt;
  const uint32_t N = U.N;
  auto words = [&](int a, int t) -> uint32_t * {
    const int k = t * U.n_sets + a - R.first;
    return k >= 0 && k < R.n ? R.base + (size_t)k * N : U.w + a * U.set_stride + (size_t)t * N;
  };
  for (int colour = 0; colour < 2; ++colour) {
    if (colour == 1 && need_e)
      for (int k = threadIdx.x; k < n_w * 32; k += kThreads) (&e_cnt[0][0])[k] = 0;
    if (colour == 1) __syncthreads();
    if (!(colour == 1 && need_e) && (U.L & 7) == 0 && n_w >= 2) {
      // phases that count nothing: a thread takes one quad in a block of up
      // to four owned word-lattices, whose geometry and coupling words it
      // reads once (the same group for all of them)
      const uint32_t quads = N / 8;
      const uint32_t nb = (uint32_t)(n_w + 3) / 4, items = quads * nb;
      const uint32_t wctr = ctr_w(TAG_UPDATE, (uint32_t)colour, 0);
      for (uint32_t it = threadIdx.x; it < items; it += kThreads) {
        const uint32_t blk = it / quads, j4 = it - blk * quads;
        const EaQuadGeom q = ea_quad_geom<3>(j4, colour, (uint32_t)U.L, U.fL);
        const EaQuadJ c = ea_quad_couplings<3>(Jsrc, q, colour, N);
        const int w0 = 4 * (int)blk, w1 = w0 + 4 < n_w ? w0 + 4 : n_w;
#pragma unroll 1
        for (int wi = w0; wi < w1; ++wi) {
          const int g = g0 + wi, a = g % U.n_sets, t = g / U.n_sets;
          const uint4 r = philox(make_uint4(j4, s_abs, lattice_id((uint32_t)a, (uint32_t)U.rgrp, (uint32_t)t), wctr), rk);
          ea_quad_update<3, false>(words(a, t), q, c, colour, N, r, __ldg(U.thr + 4 * t + 1), __ldg(U.thr + 4 * t + 2),
                                   __ldg(U.thr + 4 * t + 3), NoCount());
        }
      }
      __syncthreads();
      continue;
    }
    Share sh = warp_share(per * (uint32_t)n_w, (uint32_t)warp, kWarps);
    while (sh.c < sh.end) {
      const int wi = (int)(sh.c / per);
      const uint32_t c0 = sh.c - (uint32_t)wi * per, c1 = min(per, c0 + (sh.end - sh.c));
      sh.c += c1 - c0;
      const int g = g0 + wi, a = g % U.n_sets, t = g / U.n_sets;
      uint32_t *s = words(a, t);
      const uint32_t lid = lattice_id((uint32_t)a, (uint32_t)U.rgrp, (uint32_t)t);
      const uint32_t t4 = __ldg(U.thr + 4 * t + 1), t8 = __ldg(U.thr + 4 * t + 2), t12 = __ldg(U.thr + 4 * t + 3);
      uint32_t C[kPl];
#pragma unroll
      for (int k = 0; k < kPl; ++k) C[k] = 0;
      if (colour == 1 && need_e) {
        ea_phase_warp<true>(s, Jsrc, U, rk, s_abs, lid, 1, t4, t8, t12, c0, c1, C);
        atomicAdd(&e_cnt[wi][lane], warp_bit_counts(C));
      } else {
        ea_phase_warp<false>(s, Jsrc, U, rk, s_abs, lid, colour, t4, t8, t12, c0, c1, C);
      }
    }
    __syncthreads();
  }
  if (need_e) {
    for (int k = threadIdx.x; k < n_w * 32; k += kThreads) {
      const int wi = k >> 5, b = k & 31;
      const int g = g0 + wi, a = g % U.n_sets, t = g / U.n_sets;
      const int unsat = e_cnt[wi][b];
      U.Escr[(a * U.n_T + t) * 32 + b] = unsat;
      if (measure && U.E_series) {
        const long long lat = ((long long)a * U.n_T + t) * U.n_real + 32 * U.grp + b;
        U.E_series[meas_row * U.n_lat + lat] = 2LL * unsat - 3LL * N;
      }
    }
  }
  const long long r0 = 32 * U.grp;
  if (measure && U.M_series) {  // magnetisation of every owned word-lattice
    cta_bit_counts(n_w, N, [&](int k, const uint32_t *&x, const uint32_t *&y) {
      x = words((g0 + k) % U.n_sets, (g0 + k) / U.n_sets);
      y = nullptr;
    }, e_cnt);
    for (int k = threadIdx.x; k < n_w * 32; k += kThreads) {
      const int g = g0 + (k >> 5), a = g % U.n_sets, t = g / U.n_sets;
      U.M_series[meas_row * U.n_lat + ((long long)a * U.n_T + t) * U.n_real + r0 + (k & 31)] =
          (long long)N - 2LL * e_cnt[k >> 5][k & 31];
    }
  }
  // overlap of sets 0 and 1 for every slot whose set-0 word-lattice is
  // owned; its set-1 word-lattice may belong to another CTA of the team
  const bool do_q = measure && U.Q_series && U.n_sets >= 2;
  const bool q_cross = P > U.n_T;
  const int gq0 = (g0 + U.n_sets - 1) / U.n_sets, gq1 = (g1 + U.n_sets - 1) / U.n_sets;  // slots
  auto overlap = [&]() {
    const int n_q = gq1 - gq0;
    if (n_q <= 0) {
      __syncthreads();
      return;
    }
    cta_bit_counts(n_q, N, [&](int k, const uint32_t *&x, const uint32_t *&y) {
      x = words(0, gq0 + k);
      y = words(1, gq0 + k);
    }, e_cnt);
    for (int k = threadIdx.x; k < n_q * 32; k += kThreads)
      U.Q_series[meas_row * (long long)U.n_T * U.n_real + (long long)(gq0 + (k >> 5)) * U.n_real + r0 +
                 (k & 31)] = (long long)N - 2LL * e_cnt[k >> 5][k & 31];
  };
  if (do_q && !q_cross) overlap();
  if (!pt && !(do_q && q_cross)) {
    __syncthreads();  // measurements read words the next sweep rewrites
    return true;
  }
  if (!team_barrier(sy)) return false;  // energies and words of all slots visible
  if (do_q && q_cross) {
    overlap();
    if (!team_barrier(sy)) return false;  // overlap reads done before any word changes
  }
  if (!pt) return true;
  // decisions for pairs (t, t+1) of set a, t = step parity (mod 2), made by
  // the owner of (a, t), which then exchanges the two word-lattices
  const int parity = (int)(pt_step & 1u);
  for (int k = warp; k < n_w; k += kWarps) {
    const int g = g0 + k, a = g % U.n_sets, t = g / U.n_sets;
    if (((t - parity) & 1) != 0 || t + 1 >= U.n_T) {
      if (lane == 0) masks[k] = 0u;
      continue;
    }
    const int r = 32 * U.grp + lane;
    const int e0 = U.Escr[(a * U.n_T + t) * 32 + lane], e1 = U.Escr[(a * U.n_T + t + 1) * 32 + lane];
    const long long dE = 2LL * (e1 - e0);
    const double db = U.pt_dbeta[t];
    bool acc;
    if (db * (double)dE >= 0.0) {
      acc = true;
    } else {
      const long long m = (dE < 0 ? -dE : dE) / 4;
      const uint32_t th = m < U.pt_len[t] ? __ldg(U.pt_tab + U.pt_off[t] + m) : 0u;
      const uint4 v = philox(make_uint4((uint32_t)r >> 2, pt_step, lattice_id((uint32_t)a, 0, (uint32_t)t),
                                        ctr_w(TAG_PT, 0, 0)), rk);
      acc = word_of(v, (uint32_t)r & 3u) < th;
    }
    if (U.labels && acc) {  // this lane alone owns realisation r of pair (t, t+1)
      const long long l0 = ((long long)a * U.n_T + t) * U.n_real + r, l1 = l0 + U.n_real;
      const int x = U.labels[l0];
      U.labels[l0] = U.labels[l1];
      U.labels[l1] = x;
    }
    const uint32_t A = __ballot_sync(0xffffffffu, acc);
    if (lane == 0) {
      masks[k] = A;
      if (U.accepted && A) atomicAdd((unsigned long long *)&U.accepted[a * U.n_T + t], (unsigned long long)__popc(A));
    }
  }
  __syncthreads();
  for (int k = 0; k < n_w; ++k) {
    const uint32_t A = masks[k];
    if (!A) continue;
    const int g = g0 + k, a = g % U.n_sets, t = g / U.n_sets;
    cta_swap_bits(words(a, t), words(a, t + 1), N, A);
  }
  return team_barrier(sy);  // exchanged words visible before the next sweep
}

// ---------------------------------------------------------------- Ising unit
// One colour phase over the rows [r0, r1) of a 2D int8 lattice: four chunks
// per thread and iteration, all their loads issued before any store.
template <int kCount>
static __device__ void ising_rows_phase(const BatchUnit &U, const RoundKeys &rk, uint32_t sweep, int colour, int r0,
                                 int r1, long long &anti, long long &down) {
  const int L = U.L;
  const uint32_t chunks = (uint32_t)L >> 3;
  const uint32_t thr4 = __ldg(U.thr + 4 * U.slot + 1), thr8 = __ldg(U.thr + 4 * U.slot + 2);
  const uint32_t wctr = ctr_w(TAG_UPDATE, (uint32_t)colour, 0);
  const uint32_t total = (uint32_t)(r1 - r0) * chunks;
  int8_t *base = U.s;
  constexpr int kU = 4;  // chunks per thread and iteration
  for (uint32_t k = threadIdx.x; k < total; k += kU * kThreads) {
    int y[kU];
    uint32_t m[kU];
    uint64_t C[kU], Uw[kU], Dw[kU], lb[kU], rb[kU];
#pragma unroll
    for (int j = 0; j < kU; ++j) {
      // a chunk beyond the range repeats chunk k and is not stored
      const uint32_t kj = k + j * kThreads < total ? k + j * kThreads : k;
      const uint32_t dy = fdiv(kj, U.fC);
      y[j] = r0 + (int)dy;
      m[j] = kj - dy * chunks;
      const int yu = y[j] == 0 ? L - 1 : y[j] - 1, yd = y[j] == L - 1 ? 0 : y[j] + 1;
      const int8_t *row = base + (int64_t)y[j] * L;
      C[j] = reinterpret_cast<const uint64_t *>(row)[m[j]];
      Uw[j] = reinterpret_cast<const uint64_t *>(base + (int64_t)yu * L)[m[j]];
      Dw[j] = reinterpret_cast<const uint64_t *>(base + (int64_t)yd * L)[m[j]];
      lb[j] = (uint8_t)row[m[j] == 0 ? L - 1 : 8 * m[j] - 1];
      rb[j] = (uint8_t)row[m[j] == chunks - 1 ? 0 : 8 * m[j] + 8];
    }
    // the generator blocks first, as independent chains
    uint4 q[kU];
#pragma unroll
    for (int j = 0; j < kU; ++j) q[j] = philox(make_uint4((uint32_t)y[j] * chunks + m[j], sweep, U.lid, wctr), rk);
#pragma unroll
    for (int j = 0; j < kU; ++j) {
      long long a2 = 0, d2 = 0;
      const uint64_t nw =
          ising_chunk<kCount>(C[j], Uw[j], Dw[j], lb[j], rb[j], q[j], (colour + y[j]) & 1, thr4, thr8, a2, d2);
      if (k + j * kThreads < total) {
        reinterpret_cast<uint64_t *>(base + (int64_t)y[j] * L)[m[j]] = nw;
        anti += a2;
        down += d2;
      }
    }
  }
}

// One sweep of the team's rows.  Measurements come out of the phases: the
// magnetisation from the sites each phase updated, the energy from the
// updated sites of colour 1, since every bond has exactly one such end.
static __device__ bool ising_sweep(const BatchUnit &U, int part, const RoundKeys &rk, Sync &sy, uint32_t s_abs,
                            bool measure, long long meas_row) {
  const int P = U.team_size;
  const int r0 = part * U.L / P, r1 = (part + 1) * U.L / P;
  const bool count = measure && (U.E_series || U.M_series);
  long long anti = 0, down = 0;
  for (int colour = 0; colour < 2; ++colour) {
    if (!count) ising_rows_phase<0>(U, rk, s_abs, colour, r0, r1, anti, down);
    else if (colour == 0) ising_rows_phase<1>(U, rk, s_abs, 0, r0, r1, anti, down);
    else ising_rows_phase<2>(U, rk, s_abs, 1, r0, r1, anti, down);
    if (colour == 1 && count) {
      anti = warp_sum(anti);
      down = warp_sum(down);
      if ((threadIdx.x & 31) == 0) {
        const long long N = (long long)U.N;
        const long long idx = meas_row * U.n_lat + U.lat_index;
        // the series entries were zeroed before the launch; part 0 adds the constants
        const bool first = part == 0 && threadIdx.x == 0;
        if (U.E_series)
          atomicAdd((unsigned long long *)&U.E_series[idx], (unsigned long long)(2 * anti - (first ? 2 * N : 0)));
        if (U.M_series)
          atomicAdd((unsigned long long *)&U.M_series[idx], (unsigned long long)(-2 * down + (first ? N : 0)));
      }
    }
    if (!team_barrier(sy)) return false;
  }
  return true;
}

// ---------------------------------------------------------------- coded Ising unit
// Acceptance masks of one block of 128 sites, drawn by one thread as in
// msc2d_phase_kernel (msc2d.cu).
struct Masks {
  uint4 m4, m8;
};

static __device__ __forceinline__ Masks msc2d_draw(const BatchUnit &U, const RoundKeys &rk, uint32_t sweep, int colour,
                                                   uint32_t gb, uint32_t thr4, uint32_t thr8) {
  const PhiloxX0 pre = philox_x0_setup(sweep, U.lid, rk);
  const uint32_t wctr = ctr_w(TAG_UPDATE, (uint32_t)colour, 0);
  const MaskBits b4(thr4), b8(thr8);
  uint32_t A[4] = {0u, 0u, 0u, 0u}, E[4] = {0u, 0u, 0u, 0u};
#pragma unroll 4
  for (int i = 31; i >= 0; --i) {
    const uint4 r = philox_x0(pre, philox_x0_shared(32u * gb + (uint32_t)i, wctr, rk), rk);
    b4.push(A[0], r.x);
    b4.push(A[1], r.y);
    b4.push(A[2], r.z);
    b4.push(A[3], r.w);
    b8.push(E[0], r.x);
    b8.push(E[1], r.y);
    b8.push(E[2], r.z);
    b8.push(E[3], r.w);
  }
  Masks m;
  m.m4 = make_uint4(b4.mask(A[0]), b4.mask(A[1]), b4.mask(A[2]), b4.mask(A[3]));
  m.m8 = make_uint4(b8.mask(E[0]), b8.mask(E[1]), b8.mask(E[2]), b8.mask(E[3]));
  return m;
}

// One colour phase over the blocks [fb, fb + nblk) of a 2D coded lattice, one
// thread per block; the masks of the thread's first block are there already.
template <int kCount>
static __device__ void msc2d_rows_phase(const BatchUnit &U, const RoundKeys &rk, uint32_t sweep, int colour,
                                        uint32_t fb, uint32_t nblk, uint32_t thr4, uint32_t thr8, Masks m,
                                        long long &anti, long long &down) {
  const int L = U.L, wpr = L / 64, bpr = L / 256;
  for (uint32_t k = threadIdx.x; k < nblk; k += kThreads) {
    const uint32_t gb = fb + k;
    if (k != threadIdx.x) m = msc2d_draw(U, rk, sweep, colour, gb, thr4, thr8);
    const uint32_t y = gb / (uint32_t)bpr, B = gb - y * (uint32_t)bpr;
    msc2d_block<kCount>(U.w, L, wpr, bpr, colour, (int)y, B, m.m4, m.m8, anti, down);
  }
}

// All sweeps of the team's rows of a coded lattice, measurements fused as in
// ising_sweep.  Each thread draws the masks of its first block of the next
// phase between the two halves of the team barrier, so that the barrier's
// latency is covered by the generator.
static __device__ void msc2d_run(const BatchUnit &U, int part, const RoundKeys &rk, Sync &sy, int64_t n_sweeps,
                                 int measure_every) {
  const int P = U.team_size, bpr = U.L / 256;
  const int r0 = part * U.L / P, r1 = (part + 1) * U.L / P;
  const uint32_t fb = (uint32_t)r0 * (uint32_t)bpr, nblk = (uint32_t)(r1 - r0) * (uint32_t)bpr;
  const uint32_t thr4 = __ldg(U.thr + 4 * U.slot + 1), thr8 = __ldg(U.thr + 4 * U.slot + 2);
  long long meas_row = 0;
  Masks m = {};
  if (threadIdx.x < nblk) m = msc2d_draw(U, rk, U.sweep0, 0, fb + threadIdx.x, thr4, thr8);
  for (int64_t k = 0; k < n_sweeps; ++k) {
    const uint32_t s_abs = U.sweep0 + (uint32_t)k;
    const bool measure = measure_every > 0 && ((s_abs + 1u) % (uint32_t)measure_every) == 0u;
    const bool count = measure && (U.E_series || U.M_series);
    long long anti = 0, down = 0;
    for (int colour = 0; colour < 2; ++colour) {
      if (!count) msc2d_rows_phase<0>(U, rk, s_abs, colour, fb, nblk, thr4, thr8, m, anti, down);
      else if (colour == 0) msc2d_rows_phase<1>(U, rk, s_abs, 0, fb, nblk, thr4, thr8, m, anti, down);
      else msc2d_rows_phase<2>(U, rk, s_abs, 1, fb, nblk, thr4, thr8, m, anti, down);
      if (colour == 1 && count) {
        anti = warp_sum(anti);
        down = warp_sum(down);
        if ((threadIdx.x & 31) == 0) {
          const long long N = (long long)U.N;
          const long long idx = meas_row * U.n_lat + U.lat_index;
          const bool first = part == 0 && threadIdx.x == 0;
          if (U.E_series)
            atomicAdd((unsigned long long *)&U.E_series[idx], (unsigned long long)(2 * anti - (first ? 2 * N : 0)));
          if (U.M_series)
            atomicAdd((unsigned long long *)&U.M_series[idx], (unsigned long long)(-2 * down + (first ? N : 0)));
        }
      }
      if (colour == 1 && k + 1 == n_sweeps) break;
      team_arrive(sy);
      if (threadIdx.x < nblk)
        m = msc2d_draw(U, rk, s_abs + (uint32_t)colour, colour ^ 1, fb + threadIdx.x, thr4, thr8);
      if (!team_wait(sy)) return;
    }
    if (measure) ++meas_row;
  }
}
};

template <int kThreads>
__global__ void __launch_bounds__(kThreads, 512 / kThreads) batch_kernel(const __grid_constant__ BatchParams prm,
                                                         int *err) {
  using C = Cta<kThreads>;
  __shared__ BatchUnit U;
  __shared__ RoundKeys rk;
  extern __shared__ __align__(16) uint32_t sJ[];  // an EA unit's couplings, when staged, then its resident words
  // CTA -> unit: teams are consecutive CTA ranges in unit order
  int lo = 0, hi = prm.n_units - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (prm.units[mid].team_first <= (int)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const int u = lo;
  if (threadIdx.x == 0) {
    U = prm.units[u];
    // the counters come from device memory, so that a captured launch
    // replayed later continues the handle's random streams
    U.sweep0 = (uint32_t)U.ctr[0];
    U.pt0 = (uint32_t)U.ctr[1];
    rk = prm.keys[U.key];
  }
  __syncthreads();
  const int part = (int)blockIdx.x - U.team_first;
  Sync sy{U.bar, 0u, U.team_size, err, prm.timeout_ns, prm.extra};
  // the couplings never change during a launch: stage them once if they fit
  const uint32_t *Jsrc = U.J;
  typename C::Resident R = {sJ, 0, 0};
  uint32_t used = 0;
  if (U.kind == 0 && 3u * U.N <= prm.staged_words) {
    for (uint32_t k = threadIdx.x; k < 3u * U.N / 4u; k += blockDim.x)
      reinterpret_cast<uint4 *>(sJ)[k] = __ldg(reinterpret_cast<const uint4 *>(U.J) + k);
    __syncthreads();
    Jsrc = sJ;
    used = 3u * U.N;
  }
  if (U.kind == 0 && prm.smem_words > prm.staged_words) {
    R = C::ea_resident(U, part, sJ + used, prm.smem_words - used);
    C::ea_resident_copy(U, R, true);
  }
  if (U.kind == 2) {
    C::msc2d_run(U, part, rk, sy, prm.n_sweeps, prm.measure_every);
    return;
  }
  long long meas_row = 0;
  uint32_t pt_step = U.pt0;
  for (int64_t k = 0; k < prm.n_sweeps; ++k) {
    const uint32_t s_abs = U.sweep0 + (uint32_t)k;
    const bool measure = prm.measure_every > 0 && ((s_abs + 1u) % (uint32_t)prm.measure_every) == 0u;
    const bool pt = prm.pt_every > 0 && ((s_abs + 1u) % (uint32_t)prm.pt_every) == 0u;
    const bool ok = U.kind == 0 ? C::ea_sweep(U, R, Jsrc, part, rk, sy, s_abs, measure, pt, meas_row, pt_step)
                                : C::ising_sweep(U, part, rk, sy, s_abs, measure, meas_row);
    if (!ok) break;  // (the resident words go home all the same)
    if (measure) ++meas_row;
    if (pt) ++pt_step;
  }
  if (R.n > 0) {
    __syncthreads();
    C::ea_resident_copy(U, R, false);
  }
}

// Work around a batched launch, per handle: zero the barrier counters and
// (outside a stream capture) load the device counters from the host's; after
// the launch, advance the device counters as the launch advanced the host's.
struct BatchCtl {
  int n;
  int set;  // prologue: write ctr from sweeps / pt
  int32_t pt_every;
  int64_t n_sweeps;
  int *err;
  long long *ctr[kMaxHandles];
  long long sweeps[kMaxHandles], pt[kMaxHandles];
  unsigned *bar[kMaxHandles];
  int n_bar[kMaxHandles];
  // series rows that Ising units accumulate with atomics: zeroed first
  long long *zero[2 * kMaxHandles];
  int64_t n_zero[2 * kMaxHandles];
};

__global__ void batch_prologue_kernel(const BatchCtl c) {
  for (int k = 0; k < c.n; ++k)
    for (int i = threadIdx.x; i < c.n_bar[k]; i += blockDim.x) c.bar[k][i] = 0u;
  for (int k = 0; k < 2 * kMaxHandles; ++k)
    for (int64_t i = threadIdx.x; i < c.n_zero[k]; i += blockDim.x) c.zero[k][i] = 0;
  if (threadIdx.x < (unsigned)c.n && c.set) {
    c.ctr[threadIdx.x][0] = c.sweeps[threadIdx.x];
    c.ctr[threadIdx.x][1] = c.pt[threadIdx.x];
  }
  if (threadIdx.x == 0 && c.err) *c.err = 0;
}

__global__ void batch_epilogue_kernel(const BatchCtl c) {
  if (threadIdx.x >= (unsigned)c.n) return;
  long long *ctr = c.ctr[threadIdx.x];
  const long long s = ctr[0];
  if (c.pt_every > 0) ctr[1] += (s + c.n_sweeps) / c.pt_every - s / c.pt_every;
  ctr[0] = s + c.n_sweeps;
}

}  // namespace

// ---------------------------------------------------------------- host side
struct Tuned {
  int ctas_per_sm;
  double ising_scale;
  double ea_n0;
};
static std::map<std::vector<long long>, Tuned> g_tuned;  // autotuner cache, by batch signature

static constexpr double kEaFixedUs = 13.0, kLatticeUs = 0.45, kQuadUs = 1.0e-3, kSiteUs = 2.0e-3;
static constexpr double kQuadUnstaged = 1.6, kSiteUnstaged = 1.1;

// Time of one sweep of a unit with a team of P CTAs, with measurement and
// exchange every sweep, in us (fitted to the times at which the units of the
// uneven batch end, two CTAs per SM): for EA units a fixed part (barriers,
// reductions) and, for the CTA with the most word-lattices n of N sites, a part
// per word-site, larger where the quads of a row do not fit (L % 8 != 0) or the
// couplings are not staged; 6.2 coded Ising sites per ns and CTA.  What counts
// is the largest share: a team of 9 for 32 slots is no faster than one of 8.
// The autotuner rescales the Ising share and adds ea_n0 sites per EA
// word-lattice.
static double unit_time(const BatchUnit &U, int P, double ising_scale, double ea_n0) {
  if (U.kind == 0) {
    const int W = U.n_T * U.n_sets;
    const int owned = P <= U.n_T ? (U.n_T + P - 1) / P * U.n_sets : (W + P - 1) / P;
    const bool unstaged = 3u * U.N > 12288u;
    const double per_site = U.L % 8 != 0 ? kSiteUs * (unstaged ? kSiteUnstaged : 1.0)
                                           : kQuadUs * (unstaged ? kQuadUnstaged : 1.0);
    return kEaFixedUs + owned * (kLatticeUs + per_site * ((double)U.N + ea_n0));
  }
  const double rows = (U.L + P - 1) / P;
  return 3.0 + (U.kind == 1 ? 0.45e-3 : 0.16e-3) * ising_scale * rows * U.L;
}

// The next larger team for which the unit's time falls (cap + 1: none).
static int next_team(const BatchUnit &U, int P, int cap) {
  if (U.kind != 0) return P + 1;
  const int W = U.n_T * U.n_sets;
  if (P < U.n_T) {
    const int m = (U.n_T + P - 1) / P;  // slots of the largest share, more than one
    return (U.n_T + m - 2) / (m - 1);
  }
  const int o = (W + P - 1) / P;
  return o > 1 ? (W + o - 2) / (o - 1) : cap + 1;
}

// The fewest CTAs of a unit (EA: each CTA owns at most 64 word-lattices).
static int least_team(const BatchUnit &U) {
  int p = 1;
  while (U.kind == 0 && U.n_sets * ((U.n_T + p - 1) / p) > 64) ++p;
  return p;
}

// Distributes `grid` CTAs over the units: every unit gets its minimum (EA:
// at most 64 owned word-lattices per CTA; Ising: 1), then the unit with the
// longest time gets its next larger team, as long as one fits, up to each
// unit's maximum (EA: one word-lattice per CTA; Ising: 8 rows, or 256 coded
// blocks, per CTA).  Returns the CTAs used.
static int assign_teams(BatchUnit *units, int n, int grid, double ising_scale, double ea_n0) {
  std::vector<int> P(n), cap(n);
  std::vector<double> time(n);
  int used = 0;
  for (int u = 0; u < n; ++u) {
    P[u] = least_team(units[u]);
    if (units[u].kind == 0) {
      cap[u] = units[u].n_T * units[u].n_sets;  // one word-lattice per CTA at most
    } else if (units[u].kind == 1) {
      cap[u] = std::max(1, units[u].L / 8);
    } else {  // at least 256 blocks (one per thread) per CTA
      cap[u] = std::max(1, units[u].L * (units[u].L / 256) / 256);
    }
    used += P[u];
    time[u] = unit_time(units[u], P[u], ising_scale, ea_n0);
  }
  for (;;) {
    int best = -1;
    for (int u = 0; u < n; ++u)
      if (time[u] >= 0.0 && (best < 0 || time[u] > time[best])) best = u;
    if (best < 0) break;
    const int next = next_team(units[best], P[best], cap[best]);
    if (next > cap[best] || used + next - P[best] > grid) {
      time[best] = -1.0;  // stays as it is
      continue;
    }
    used += next - P[best];
    P[best] = next;
    time[best] = unit_time(units[best], next, ising_scale, ea_n0);
  }
  int first = 0;
  for (int u = 0; u < n; ++u) {
    units[u].team_first = first;
    units[u].team_size = P[u];
    first += P[u];
  }
  return first;
}

}  // namespace spin

using namespace spin;

namespace spin {
int upload_thresholds_for_batch(spin_lattice *h, const double *betas);  // api.cu
int upload_pt_tables_for_batch(spin_lattice *h, const double *betas);   // api.cu
bool tables_cached_for_batch(const spin_lattice *h, const double *betas, bool pt);  // api.cu
}

// work units of a handle in a batched launch: EA realisation groups or Ising lattices
static int64_t units_of(const spin_lattice *h) {
  return h->d.model == SPIN_EA ? h->g.n_real / 32 : h->n_lat;
}

// Per-handle workspace of batched launches, allocated once (never inside a
// stream capture) and kept until spin_destroy, so that captured launches
// keep valid pointers.
static int ensure_batch_ws(spin_lattice *h) {
  if (h->d_ctr) return SPIN_OK;
  const size_t escr = h->d.model == SPIN_EA ? (size_t)units_of(h) * h->g.n_sets * h->g.n_temps * 32 : 0;
  if (cudaMalloc(&h->d_ctr, 2 * sizeof(int64_t)) != cudaSuccess) return SPIN_ENOMEM;
  if (cudaMalloc(&h->d_bar, (size_t)units_of(h) * sizeof(unsigned)) != cudaSuccess) return SPIN_ENOMEM;
  if (escr && cudaMalloc(&h->d_escr, escr * sizeof(int)) != cudaSuccess) return SPIN_ENOMEM;
  h->ctr_dev[0] = h->ctr_dev[1] = -1;
  return SPIN_OK;
}

static void fill_ctl(BatchCtl &c, const spin_batch_item *items, int n_items, int set, int64_t n_sweeps,
                     int32_t pt_every, int *err) {
  c = BatchCtl{};
  c.n = n_items;
  c.set = set;
  c.n_sweeps = n_sweeps;
  c.pt_every = pt_every;
  c.err = err;
  for (int k = 0; k < n_items; ++k) {
    spin_lattice *h = items[k].lat;
    c.ctr[k] = (long long *)h->d_ctr;
    c.sweeps[k] = h->sweeps_done;
    c.pt[k] = h->pt_steps_done;
    c.bar[k] = h->d_bar;
    c.n_bar[k] = (int)units_of(h);
  }
}

// Loads the device counters of a handle from its host counters (stream-ordered).
int spin::sync_device_counters(spin_lattice *h, cudaStream_t st) {
  if (!h->d_ctr) return SPIN_OK;
  spin_batch_item it = {};
  it.lat = h;
  BatchCtl c;
  fill_ctl(c, &it, 1, 1, 0, 0, nullptr);
  c.n_bar[0] = 0;
  batch_prologue_kernel<<<1, 32, 0, st>>>(c);
  if (cudaGetLastError() != cudaSuccess) return SPIN_ECUDA;
  h->ctr_dev[0] = h->sweeps_done;
  h->ctr_dev[1] = h->pt_steps_done;
  return SPIN_OK;
}

static int batch_build(const spin_batch_item *items, int n_items, BatchParams &prm) {
  prm.n_units = 0;
  for (int k = 0; k < n_items; ++k) {
    spin_lattice *h = items[k].lat;
    prm.keys[k] = make_round_keys(h->d.seed);
    const Geom &g = h->g;
    if (h->d.model == SPIN_EA) {
      const int G = g.n_real / 32;
      for (int grp = 0; grp < G; ++grp) {
        if (prm.n_units >= kMaxUnits) return SPIN_EINVAL;
        BatchUnit &U = prm.units[prm.n_units++];
        U = BatchUnit{};
        U.kind = 0;
        U.L = g.L;
        U.N = (uint32_t)g.N;
        U.n_T = g.n_temps;
        U.n_sets = g.n_sets;
        U.fL = g.fL;
        U.thr = h->d_thr;
        U.key = k;
        U.ctr = (const long long *)h->d_ctr;
        U.bar = h->d_bar + grp;
        U.set_stride = (size_t)G * g.n_temps * g.N;
        U.w = (uint32_t *)h->spins + (size_t)grp * g.n_temps * g.N;
        U.J = (const uint32_t *)items[k].couplings + (size_t)grp * 3 * g.N;
        U.grp = grp;
        U.rgrp = h->msc_width == 64 ? grp / 2 : grp;
        U.n_real = g.n_real;
        U.pt_tab = h->d_pt_thr;
        U.pt_off = h->d_pt_off;
        U.pt_len = h->d_pt_len;
        U.pt_dbeta = h->d_pt_dbeta;
        U.E_series = (long long *)items[k].E_series;
        U.M_series = (long long *)items[k].M_series;
        U.Q_series = (long long *)items[k].Q_series;
        U.accepted = (long long *)items[k].accepted;
        U.labels = (int *)items[k].labels;
        U.n_lat = h->n_lat;
        U.Escr = h->d_escr + (size_t)grp * g.n_sets * g.n_temps * 32;
      }
    } else {
      const bool coded = h->d.layout == SPIN_MSC1;
      for (int64_t lat = 0; lat < h->n_lat; ++lat) {
        if (prm.n_units >= kMaxUnits) return SPIN_EINVAL;
        BatchUnit &U = prm.units[prm.n_units++];
        U = BatchUnit{};
        U.kind = coded ? 2 : 1;
        if (coded) U.w = (uint32_t *)h->spins + lat * (g.N / 32);
        U.L = g.L;
        U.N = (uint32_t)g.N;
        U.n_T = g.n_temps;
        U.n_sets = g.n_sets;
        U.thr = h->d_thr;
        U.key = k;
        U.ctr = (const long long *)h->d_ctr;
        U.bar = h->d_bar + lat;
        if (!coded) U.s = (int8_t *)h->spins + lat * g.N;
        U.fC = make_fastdiv((uint32_t)(g.L / 8));
        U.E_series = (long long *)items[k].E_series;
        U.M_series = (long long *)items[k].M_series;
        U.n_lat = h->n_lat;
        U.lat_index = lat;
        U.lid = lattice_id_of(g, lat);
        U.slot = slot_of(g, lat);
      }
    }
  }
  return SPIN_OK;
}

static bool batch_item_ok(const spin_batch_item &it, int32_t pt_every) {
  const spin_lattice *h = it.lat;
  if (!h || !it.betas) return false;
  if (h->d.model == SPIN_EA)
    return h->d.layout == SPIN_MSC1 && h->d.dim == 3 && it.couplings != nullptr && h->g.L <= 32 &&
           h->d.n_sets <= 32;
  if (h->d.model == SPIN_ISING)
    return h->g.dim == 2 && it.Q_series == nullptr &&
           ((h->d.layout == SPIN_I8 && h->g.L % 16 == 0) || (h->d.layout == SPIN_MSC1 && h->g.L % 256 == 0)) &&
           h->order == SPIN_ORDER_CHECKERBOARD &&
           !(pt_every > 0 && h->d.n_temps > 1);
  return false;
}

// Dynamic shared memory of a CTA that has its SM to itself, beside 9 KB of
// counters and masks.
constexpr int kResidentSmem = 212 * 1024;

// One 512-thread CTA per SM with word-lattices in shared memory, against two
// of 256 threads that read them from L2: the update is bound by the latency of
// those loads at 16 warps per SM.  For batches of EA units alone whose
// word-lattices are small enough that most of a CTA's fit (32 KB at L = 20),
// and whose units are large enough for three CTAs and more each (a unit takes
// whole CTAs) but have no more CTAs than slots.  A batch whose least teams need
// more CTAs than there are SMs only fits two to an SM.  Otherwise the form with
// less work on its fullest SM: word-sites of the CTA with the most slots and
// what the barriers of one CTA leave idle (as much as 2100 of them), 0.87 (0.91
// from L = 18 on) of the time per word-site of two CTAs, of which one has the
// most slots and one an average share.  Us per 8 sweeps with E, M, Q and an
// exchange after each, one / two CTAs per SM, groups x slots of two sets:
//   L = 8   20 x 60 231 / 171, 40 x 32 234 / 205, 48 x 33 239 / 248
//   L = 10  12 x 32 202 / 178, 28 x 60 414 / 444
//   L = 12  28 x 16 251 / 227, 28 x 60 556 / 608, 40 x 32 512 / 483
//   L = 16  32 x 32 474 / 520, 40 x 32 655 / 624, 48 x 33 664 / 803
//   L = 20  28 x 16 678 / 609, 12 x 32 558 / 611, 40 x 60 3446 / 3028
// Of 112 shapes with 8 <= L <= 20 it takes the slower one by more than 3 % in
// five, 7 % at most.
static bool resident_preferred(const BatchParams &prm, int sms) {
  double total = 0.0;
  int least = 0;
  for (int u = 0; u < prm.n_units; ++u) {
    const BatchUnit &U = prm.units[u];
    if (U.kind != 0 || U.N > 8192u) return false;
    total += (double)U.n_sets * U.n_T * U.N;
    least += least_team(U);
  }
  if (least > sms) return false;
  double one = 0.0, two = 0.0;  // work of the fullest SM with one, with two CTAs
  for (int u = 0; u < prm.n_units; ++u) {
    const BatchUnit &U = prm.units[u];
    const int W = U.n_sets * U.n_T;
    const double share = sms * (double)W * U.N / total, slot = (double)U.n_sets * U.N;
    if (share < 3.0 || share > (double)U.n_T) return false;
    const int P1 = (int)share, P2 = std::min((int)(2.0 * share), W);
    const int m1 = (U.n_T + P1 - 1) / P1;
    const double m2 = P2 <= U.n_T ? (U.n_T + P2 - 1) / P2 : (double)((W + P2 - 1) / P2) / U.n_sets;
    one = std::max(one, (U.N <= 4096u ? 0.87 : 0.91) * (m1 * slot + 2100.0));
    two = std::max(two, (m2 + (double)U.n_T / P2) * slot);
  }
  return one < two;
}

static bool resident(const BatchParams &prm) { return prm.smem_words > prm.staged_words; }

static cudaError_t batch_launch(BatchParams &prm, int grid, cudaStream_t st, int *err) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(resident(prm) ? kResidentThreads : kPairThreads);
  cfg.dynamicSmemBytes = (size_t)prm.smem_words * 4;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return resident(prm) ? cudaLaunchKernelEx(&cfg, batch_kernel<kResidentThreads>, prm, err)
                       : cudaLaunchKernelEx(&cfg, batch_kernel<kPairThreads>, prm, err);
}

static cudaError_t batch_occupancy(const BatchParams &prm, int *per_sm) {
  const size_t smem = (size_t)prm.smem_words * 4;
  return resident(prm)
             ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, batch_kernel<kResidentThreads>, kResidentThreads, smem)
             : cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, batch_kernel<kPairThreads>, kPairThreads, smem);
}

// The launch parameters are built in function-static buffers and the tuning
// cache is shared: calls from several host threads are serialised.
static std::recursive_mutex g_batch_mutex;

extern "C" int spin_batch_run(const spin_batch_item *items, int n_items, int64_t n_sweeps,
                              int32_t measure_every, int32_t pt_every, void *stream_v) {
  NvtxRange nvtx_range("spin_batch_run");
  if (!items || n_items <= 0 || n_items > kMaxHandles || n_sweeps < 0 || measure_every < 0 || pt_every < 0)
    return SPIN_EINVAL;
  std::lock_guard<std::recursive_mutex> lock(g_batch_mutex);
  cudaStream_t st = (cudaStream_t)stream_v;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return SPIN_ECUDA;
  const bool capturing = cs != cudaStreamCaptureStatusNone;
  // inside a capture nothing may be uploaded or allocated, and the number of
  // series rows a launch writes must not depend on the count it starts from
  if (capturing && measure_every > 0 && n_sweeps % measure_every != 0) return SPIN_EINVAL;
  for (int k = 0; k < n_items; ++k) {
    if (!batch_item_ok(items[k], pt_every)) return SPIN_EINVAL;
    spin_lattice *h = items[k].lat;
    for (int q = 0; q < k; ++q)
      if (items[q].lat == h) return SPIN_EINVAL;
    if (h->sweeps_done + n_sweeps > (int64_t)0xFFFFFFFFll) return SPIN_EINVAL;
    const bool pt_tab = h->d.model == SPIN_EA && pt_every > 0;
    if (capturing) {
      if (!tables_cached_for_batch(h, items[k].betas, pt_tab) || !h->d_ctr ||
          h->ctr_dev[0] != h->sweeps_done || h->ctr_dev[1] != h->pt_steps_done)
        return SPIN_EINVAL;  // prepare with an uncaptured call first (n_sweeps = 0 will do)
      continue;
    }
    int rc = upload_thresholds_for_batch(h, items[k].betas);
    if (rc) return rc;
    if (pt_tab) {
      rc = upload_pt_tables_for_batch(h, items[k].betas);
      if (rc) return rc;
    }
    rc = ensure_batch_ws(h);
    if (rc) return rc;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return SPIN_ECUDA;
  static OncePerDevice limits;
  if (!limits.done(dev)) {
    if (cudaFuncSetAttribute(batch_kernel<kResidentThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kResidentSmem) != cudaSuccess ||
        cudaFuncSetAttribute(batch_kernel<kPairThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize, 12288 * 4) !=
            cudaSuccess)
      return SPIN_ECUDA;
    limits.mark(dev);
  }
  spin_lattice *h0 = items[0].lat;
  static BatchCtl ctl;
  fill_ctl(ctl, items, n_items, capturing ? 0 : 1, n_sweeps, pt_every, h0->d_err);
  if (n_sweeps == 0) {  // preparation only: tables, workspace and device counters
    if (!capturing) {
      batch_prologue_kernel<<<1, 256, 0, st>>>(ctl);
      if (cudaGetLastError() != cudaSuccess) return SPIN_ECUDA;
      for (int k = 0; k < n_items; ++k) {
        items[k].lat->ctr_dev[0] = items[k].lat->sweeps_done;
        items[k].lat->ctr_dev[1] = items[k].lat->pt_steps_done;
      }
    }
    return SPIN_OK;
  }
  static BatchParams prm;  // large; built on the host for each call
  int rc = batch_build(items, n_items, prm);
  if (rc) return rc;
  prm.n_sweeps = n_sweeps;
  prm.measure_every = measure_every;
  prm.pt_every = pt_every;
  prm.timeout_ns = h0->batch_timeout_ns ? h0->batch_timeout_ns : 2000000000ull;
  prm.extra = h0->batch_fault_extra;
  // couplings of EA units with 3N <= 12288 words (48 KiB) are staged in
  // shared memory for the whole launch
  prm.staged_words = 0;
  for (int u = 0; u < prm.n_units; ++u)
    if (prm.units[u].kind == 0 && 3u * prm.units[u].N <= 12288u)
      prm.staged_words = std::max(prm.staged_words, 3u * prm.units[u].N);
  // CTAs per SM: autotuned once per batch signature (see spin_batch_tune)
  std::vector<long long> sig;
  for (int u = 0; u < prm.n_units; ++u) {
    sig.push_back(prm.units[u].kind);
    sig.push_back(prm.units[u].L);
    sig.push_back(prm.units[u].n_T);
    sig.push_back(prm.units[u].n_sets);
  }
  const auto it = g_tuned.find(sig);
  const int asked = h0->batch_ctas_per_sm > 0 ? h0->batch_ctas_per_sm : it != g_tuned.end() ? it->second.ctas_per_sm : 0;
  // co-resident grid
  int sms = 0, per_sm = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return SPIN_ECUDA;
  prm.smem_words = asked <= 1 && resident_preferred(prm, sms) ? kResidentSmem / 4 : prm.staged_words;
  if (batch_occupancy(prm, &per_sm) != cudaSuccess || per_sm < 1) return SPIN_ECUDA;
  // Ising series rows are accumulated with atomics: the prologue zeroes the
  // rows of this call (a memset per series before: ten for five lattices)
  for (int k = 0; k < n_items; ++k) {
    spin_lattice *h = items[k].lat;
    if (h->d.model != SPIN_ISING || measure_every <= 0) continue;
    const int64_t n_meas = (h->sweeps_done + n_sweeps) / measure_every - h->sweeps_done / measure_every;
    ctl.zero[2 * k] = (long long *)items[k].E_series;
    ctl.zero[2 * k + 1] = (long long *)items[k].M_series;
    ctl.n_zero[2 * k] = items[k].E_series ? n_meas * h->n_lat : 0;
    ctl.n_zero[2 * k + 1] = items[k].M_series ? n_meas * h->n_lat : 0;
  }
  int bps = std::min(per_sm, h0->batch_ctas_per_sm > 0 ? h0->batch_ctas_per_sm : 2);  // (1 where words are resident)
  double scale = h0->batch_ising_scale > 0.0 ? h0->batch_ising_scale : 1.0;
  double n0 = h0->batch_ea_n0 > 0.0 ? h0->batch_ea_n0 - 1.0 : 0.0;
  if (it != g_tuned.end()) {
    if (h0->batch_ctas_per_sm <= 0) bps = std::min(per_sm, it->second.ctas_per_sm);
    if (h0->batch_ising_scale <= 0.0) scale = it->second.ising_scale;
    if (h0->batch_ea_n0 <= 0.0) n0 = it->second.ea_n0;
  }
  const int grid = assign_teams(prm.units, prm.n_units, sms * bps, scale, n0);
  if (grid > sms * per_sm) return SPIN_EINVAL;
  batch_prologue_kernel<<<1, 256, 0, st>>>(ctl);
  if (cudaGetLastError() != cudaSuccess) return SPIN_ECUDA;
  if (batch_launch(prm, grid, st, h0->d_err) != cudaSuccess) return SPIN_ECUDA;
  batch_epilogue_kernel<<<1, 32, 0, st>>>(ctl);
  if (cudaGetLastError() != cudaSuccess) return SPIN_ECUDA;
  for (int k = 0; k < n_items; ++k) {
    spin_lattice *h = items[k].lat;
    const int64_t before = h->sweeps_done;
    h->sweeps_done += n_sweeps;
    if (pt_every > 0)  // as spin_run: every exchange point advances the counter
      h->pt_steps_done += h->sweeps_done / pt_every - before / pt_every;
    h->ctr_dev[0] = h->sweeps_done;
    h->ctr_dev[1] = h->pt_steps_done;
  }
  return SPIN_OK;
}

// Autotuner: times one short batch per (CTAs per SM, Ising weight) candidate
// on copies of the spins (the handles' own state is untouched) and caches
// the fastest for this batch signature.
extern "C" int spin_batch_tune(const spin_batch_item *items, int n_items, int64_t n_sweeps,
                               int32_t measure_every, int32_t pt_every, void *stream_v,
                               int32_t *best_out) {
  NvtxRange nvtx_range("spin_batch_tune");
  std::lock_guard<std::recursive_mutex> lock(g_batch_mutex);
  if (!items || n_items <= 0 || n_items > kMaxHandles) return SPIN_EINVAL;
  cudaStream_t st = (cudaStream_t)stream_v;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel<kPairThreads>, kPairThreads, 0) !=
      cudaSuccess)
    return SPIN_ECUDA;
  // back up the spins and counters; series outputs are not written
  std::vector<spin_batch_item> tmp(items, items + n_items);
  std::vector<void *> backup(n_items, nullptr);
  std::vector<size_t> bytes(n_items);
  std::vector<int64_t> sw(n_items), ps(n_items);
  for (int k = 0; k < n_items; ++k) {
    spin_lattice *h = items[k].lat;
    bytes[k] = h->d.layout == SPIN_I8 ? (size_t)(h->n_lat * h->g.N)
               : h->d.model == SPIN_ISING ? (size_t)(h->n_lat * h->g.N / 8)
                                          : (size_t)h->g.n_sets * (h->g.n_real / 32) * h->g.n_temps * h->g.N * 4;
    if (cudaMalloc(&backup[k], bytes[k]) != cudaSuccess) return SPIN_ENOMEM;
    cudaMemcpyAsync(backup[k], h->spins, bytes[k], cudaMemcpyDeviceToDevice, st);
    sw[k] = h->sweeps_done;
    ps[k] = h->pt_steps_done;
    tmp[k].E_series = tmp[k].M_series = tmp[k].Q_series = tmp[k].accepted = nullptr;
    tmp[k].labels = nullptr;
  }
  // scratch series, so that the trials measure as the real runs will
  std::vector<void *> scratch;
  const int64_t n_meas = measure_every > 0 ? n_sweeps / measure_every + 1 : 0;
  for (int k = 0; k < n_items && n_meas > 0; ++k) {
    spin_lattice *h = items[k].lat;
    const size_t rows[3] = {(size_t)h->n_lat, (size_t)h->n_lat, (size_t)h->g.n_temps * h->g.n_real};
    int64_t **dst[3] = {&tmp[k].E_series, &tmp[k].M_series, &tmp[k].Q_series};
    const int64_t *src[3] = {items[k].E_series, items[k].M_series, items[k].Q_series};
    for (int q = 0; q < 3; ++q) {
      if (!src[q]) continue;
      void *buf = nullptr;
      if (cudaMalloc(&buf, 8 * rows[q] * (size_t)n_meas) != cudaSuccess) return SPIN_ENOMEM;
      scratch.push_back(buf);
      *dst[q] = (int64_t *)buf;
    }
  }
  spin_lattice *h0 = items[0].lat;
  const int saved_bps = h0->batch_ctas_per_sm;
  const double saved_scale = h0->batch_ising_scale, saved_n0 = h0->batch_ea_n0;
  float best_ms = 1e30f;
  Tuned best{1, 1.0, 0.0};
  // weights that can change the split: the Ising share only with Ising and
  // EA units together, the EA overhead only with EA units of several sizes
  bool has_ising = false, has_ea = false, ea_sizes = false;
  {
    BatchParams *p0 = new BatchParams;
    batch_build(items, n_items, *p0);
    uint32_t n_first = 0;
    for (int u = 0; u < p0->n_units; ++u) {
      if (p0->units[u].kind == 0) {
        if (has_ea && p0->units[u].N != n_first) ea_sizes = true;
        if (!has_ea) n_first = p0->units[u].N;
        has_ea = true;
      } else {
        has_ising = true;
      }
    }
    delete p0;
  }
  const std::vector<double> scales =
      has_ising && has_ea ? std::vector<double>{0.5, 1.0, 2.0} : std::vector<double>{1.0};
  const std::vector<double> n0s = ea_sizes ? std::vector<double>{0.0, 1024.0, 4096.0} : std::vector<double>{0.0};
  cudaEvent_t a, b;
  cudaEventCreate(&a);
  cudaEventCreate(&b);
  int rc = SPIN_OK;
  for (int c = 1; c <= std::min(per_sm, 4) && !rc; ++c)
    for (double sc : scales)
    for (double e0 : n0s) {
      h0->batch_ctas_per_sm = c;
      h0->batch_ising_scale = sc;
      h0->batch_ea_n0 = e0 + 1.0;  // held plus one: 0 means not set
      float ms = 1e30f;
      for (int rep = 0; rep < 2 && !rc; ++rep) {  // best of two
        cudaEventRecord(a, st);
        rc = spin_batch_run(tmp.data(), n_items, n_sweeps, measure_every, pt_every, stream_v);
        cudaEventRecord(b, st);
        if (rc) break;
        cudaEventSynchronize(b);
        float t = 0;
        cudaEventElapsedTime(&t, a, b);
        ms = std::min(ms, t);
        for (int k = 0; k < n_items; ++k) {
          items[k].lat->sweeps_done = sw[k];
          items[k].lat->pt_steps_done = ps[k];
        }
      }
      if (rc) break;
      if (ms < best_ms) {
        best_ms = ms;
        best = Tuned{c, sc, e0};
      }
    }
  h0->batch_ctas_per_sm = saved_bps;
  h0->batch_ising_scale = saved_scale;
  h0->batch_ea_n0 = saved_n0;
  for (int k = 0; k < n_items; ++k) {
    cudaMemcpyAsync(items[k].lat->spins, backup[k], bytes[k], cudaMemcpyDeviceToDevice, st);
    items[k].lat->sweeps_done = sw[k];
    items[k].lat->pt_steps_done = ps[k];
    if (sync_device_counters(items[k].lat, st) != SPIN_OK) rc = rc ? rc : SPIN_ECUDA;
  }
  cudaStreamSynchronize(st);
  for (int k = 0; k < n_items; ++k) cudaFree(backup[k]);
  for (void *p : scratch) cudaFree(p);
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  if (rc) return rc;
  std::vector<long long> sig;
  BatchParams *prm = new BatchParams;
  batch_build(items, n_items, *prm);
  for (int u = 0; u < prm->n_units; ++u) {
    sig.push_back(prm->units[u].kind);
    sig.push_back(prm->units[u].L);
    sig.push_back(prm->units[u].n_T);
    sig.push_back(prm->units[u].n_sets);
  }
  delete prm;
  g_tuned[sig] = best;
  if (best_out) *best_out = best.ctas_per_sm;
  return SPIN_OK;
}
