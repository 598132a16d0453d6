// Reductions (energy, magnetisation, overlap; Sec. 3.5 measurements by
// parallel reduction, double accumulation for continuous spins, Sec. 4)
// and the replica-exchange step (Eq. parallel_tempering, Sec. 6).
#include "bitslice.cuh"
#include "ea_cs.cuh"
#include "heis_reduce.cuh"
#include "internal.h"

namespace spin {

cudaError_t launch_measure_msc2d(spin_lattice *h, int64_t *E, int64_t *M);  // msc2d.cu

namespace {

__device__ __forceinline__ void add_ll(long long *p, long long v) {
  atomicAdd(reinterpret_cast<unsigned long long *>(p), (unsigned long long)v);
}

// ---------------------------------------------------------------- int8 lattices
// E = -sum_{i,d} J_{i,d} s_i s_{i+d}, M = sum_i s_i; integer sums, so the
// atomic accumulation order does not matter.  Any even L, with or without
// couplings; site indices are 32-bit (spin_init bounds the lattices) and the
// coordinates come from multiply-high divisions.
__global__ void measure_i8_kernel(const int8_t *__restrict__ s, const int8_t *__restrict__ J,
                                  Geom g, long long *__restrict__ E, long long *__restrict__ M) {
  griddep_wait();
  griddep_release();
  const int64_t lat = blockIdx.y;
  const int8_t *sl = s + lat * g.N;
  const int8_t *Jr = J ? J + (lat % g.n_real) * (int64_t)g.dim * g.N : nullptr;
  const uint32_t L = (uint32_t)g.L, LL = L * L, N = (uint32_t)g.N;
  long long e = 0, m = 0;
  for (uint64_t i64 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i64 < N;
       i64 += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)i64;
    const uint32_t row = fdiv(i, g.fL), x = i - row * L;
    const uint32_t z = g.dim == 3 ? fdiv(row, g.fL) : 0u, y = row - z * L;
    const int si = sl[i];
    const uint32_t ixp = x == L - 1 ? i - x : i + 1;
    const uint32_t iyp = y == L - 1 ? i - (L - 1) * L : i + L;
    int bonds = (Jr ? Jr[i] : 1) * sl[ixp] + (Jr ? Jr[g.N + i] : 1) * sl[iyp];
    if (g.dim == 3) {
      const uint32_t izp = z == L - 1 ? i - (L - 1) * LL : i + LL;
      bonds += (Jr ? Jr[2 * g.N + i] : 1) * sl[izp];
    }
    e -= si * bonds;
    m += si;
  }
  e = warp_sum(e);
  m = warp_sum(m);
  if ((threadIdx.x & 31) == 0) {
    if (E) add_ll(&E[lat], e);
    if (M) add_ll(&M[lat], m);
  }
}

// Ferromagnets with L % 8 == 0: a thread counts the 8-byte chunk m of a row
// through len planes (3D; row y of planes z0 .. ) or len rows (2D; rows
// y0 .. ), keeping the next plane's (row's) chunk for its next step, so each
// byte is fetched from memory about once: antiparallel bonds to x + 1, to
// y + 1 and, in 3D, to z + 1 by popcounts of (a ^ b) & 0x02.. (bit 1 of a
// +-1 byte is set for -1), E = 2 n_anti - dim N, M = N - 2 n_down.  Bound by
// memory: the per-site form above with its three divisions and byte loads
// took 1276 us for one 3D lattice of L = 512, where 134 MB need 20 us at the
// measured copy rate; a call of four sweeps and one measurement there went
// from 2067 to 859 us.  Grid: (tiles of chunks x rows, segments, lattices);
// the blocks of segment 0 and tile 0 add the constants.
template <int kDim>
__global__ void __launch_bounds__(256) measure_chunks_i8_kernel(const int8_t *__restrict__ s, int L, int tiles_x,
                                                                int len, long long *__restrict__ E,
                                                                long long *__restrict__ M) {
  __shared__ int red[8][2];
  griddep_wait();
  griddep_release();
  constexpr uint64_t kBit1 = 0x0202020202020202ull;
  const int chunks = L >> 3;
  const int tile_y = blockIdx.x / tiles_x, tile_x = blockIdx.x - tile_y * tiles_x;
  const int m = tile_x * blockDim.x + threadIdx.x;
  // 3D: row y of the planes z0 ..; 2D: the rows z0 .. of the one plane
  const int ty = tile_y * blockDim.y + threadIdx.y;
  const int y = kDim == 3 ? ty : 0;
  const int z0 = kDim == 3 ? blockIdx.y * len : ty * len;
  const int64_t LL = (int64_t)L * L, N = kDim == 3 ? LL * L : LL;
  const int64_t zs = kDim == 3 ? LL >> 3 : chunks;  // words from one step to the next
  const int64_t lat = blockIdx.z;
  int anti = 0, down = 0;
  if (m < chunks && y < L && z0 < L) {
    const int z1 = min(z0 + len, L);
    const uint64_t *col = reinterpret_cast<const uint64_t *>(s + lat * N + (int64_t)y * L) + m;
    const int64_t dd = (int64_t)((y == L - 1 ? 0 : y + 1) - y) * chunks;  // to row y + 1
    const int64_t dx = m == chunks - 1 ? 1 - chunks : 1;                  // to the next chunk of the row
    const uint64_t *cz = col + (int64_t)z0 * zs;
    uint64_t C = *cz;
#pragma unroll 4
    for (int z = z0; z < z1; ++z) {
      const uint64_t Bk = z == L - 1 ? col[0] : cz[zs];
      const uint64_t nb = *reinterpret_cast<const uint8_t *>(cz + dx);
      const uint64_t R = (C >> 8) | (nb << 56);
      anti += __popcll((C ^ R) & kBit1) + __popcll((C ^ Bk) & kBit1);
      if (kDim == 3) anti += __popcll((C ^ cz[dd]) & kBit1);
      down += __popcll(C & kBit1);
      C = Bk;
      cz += zs;
    }
  }
  anti = __reduce_add_sync(0xffffffffu, anti);
  down = __reduce_add_sync(0xffffffffu, down);
  const int tid = threadIdx.y * blockDim.x + threadIdx.x, warps = (blockDim.x * blockDim.y + 31) >> 5;
  if ((tid & 31) == 0) {
    red[tid >> 5][0] = anti;
    red[tid >> 5][1] = down;
  }
  __syncthreads();
  if (tid != 0) return;
  long long a = 0, d = 0;
  for (int k = 0; k < warps; ++k) a += red[k][0], d += red[k][1];
  const bool first = blockIdx.x == 0 && blockIdx.y == 0;
  if (E) add_ll(&E[lat], 2 * a - (first ? kDim * (long long)N : 0));
  if (M) add_ll(&M[lat], (first ? (long long)N : 0) - 2 * d);
}

// q_{t,r} = sum_i s_i^(0) s_i^(1) between sets 0 and 1.
__global__ void overlap_i8_kernel(const int8_t *__restrict__ s, Geom g, long long *__restrict__ Q) {
  griddep_wait();
  griddep_release();
  const int64_t tr = blockIdx.y;  // t * n_real + r
  const int64_t set_stride = (int64_t)g.n_temps * g.n_real * g.N;
  const int8_t *s0 = s + tr * g.N, *s1 = s0 + set_stride;
  long long q = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.N;
       i += (int64_t)gridDim.x * blockDim.x)
    q += s0[i] * s1[i];
  q = warp_sum(q);
  if ((threadIdx.x & 31) == 0) add_ll(&Q[tr], q);
}

// ---------------------------------------------------------------- EA, coded words
// Per word-lattice (a, g, t) and realisation bit b: the number of
// unsatisfied bonds, of down spins and (set 0 only) of spins that differ
// from set 1, counted with carry-save adders.  Each word-lattice gets one
// block (of 64 threads, so that all of them are resident at once, or of 256
// where they are few) or, for large lattices, several; a thread takes at most
// kRowItems groups of four sites: quads of four consecutive colour indices of
// one row when L % 8 == 0, else four sites a block apart (so that the
// loads of a warp are contiguous).  Per group the four unsatisfied-bond sums
// (weight 1) and carries (weight 2) of E, and the four words of M and of Q
// (weight 1), go through carry-save adders into running planes of weight 1,
// 2, 4 (and 8 for E); only what carries out of those is rippled into the
// counter.  Then one butterfly per counter over the warp, and the warps of a
// word-lattice add their counts through shared memory.
constexpr int kRowThreads = 64;        // many word-lattices: all their blocks resident at once
constexpr int kRowThreadsFew = 256;    // few: more warps in flight
constexpr int kRowItems = 16;
constexpr int kRP = 8;   // per-thread planes: at most 16 groups x 4 sites x 3 bonds = 192 < 256
constexpr int kRW = 13;  // per-warp planes: at most 32 x 192 = 6144 < 8192

// Running count of weight-1 words: planes o1, o2, o4 and the counter above.
struct CsaCount {
  uint32_t C[kRP];
  uint32_t o1, o2, o4;
  __device__ CsaCount() : o1(0), o2(0), o4(0) {
#pragma unroll
    for (int k = 0; k < kRP; ++k) C[k] = 0;
  }
  __device__ __forceinline__ void add4(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3) {
    uint32_t t1, t2, f;
    csa(t1, o1, o1, x0, x1);
    csa(t2, o1, o1, x2, x3);
    csa(f, o2, o2, t1, t2);
    const uint32_t e = o4 & f;
    o4 ^= f;
    ripple_at<3>(C, e);
  }
  __device__ __forceinline__ void flush() {
    ripple_at<2>(C, o4);
    ripple_at<1>(C, o2);
    ripple_at<0>(C, o1);
    o1 = o2 = o4 = 0;
  }
};

// The same for four weight-1 words s and four weight-2 words c at a time.
struct CsaCount2 {
  uint32_t C[kRP];
  uint32_t o1, o2, o4, o8;
  __device__ CsaCount2() : o1(0), o2(0), o4(0), o8(0) {
#pragma unroll
    for (int k = 0; k < kRP; ++k) C[k] = 0;
  }
  __device__ __forceinline__ void add(const uint32_t (&sv)[4], const uint32_t (&cv)[4]) {
    uint32_t t1, t2, f1, f2, f3, e1, x;
    csa(t1, o1, o1, sv[0], sv[1]);
    csa(t2, o1, o1, sv[2], sv[3]);
    csa(f1, o2, o2, t1, t2);
    csa(f2, o2, o2, cv[0], cv[1]);
    csa(f3, o2, o2, cv[2], cv[3]);
    csa(e1, o4, o4, f1, f2);
    const uint32_t e2 = o4 & f3;
    o4 ^= f3;
    csa(x, o8, o8, e1, e2);
    ripple_at<4>(C, x);
  }
  __device__ __forceinline__ void flush() {
    ripple_at<3>(C, o8);
    ripple_at<2>(C, o4);
    ripple_at<1>(C, o2);
    ripple_at<0>(C, o1);
    o1 = o2 = o4 = o8 = 0;
  }
};

// Sum of the warp's counters; lane b returns the count of bit b.
__device__ __forceinline__ int warp_count(const uint32_t (&C)[kRP]) {
  uint32_t P[kRW];
#pragma unroll
  for (int k = 0; k < kRW; ++k) P[k] = k < kRP ? C[k] : 0u;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    uint32_t carry = 0;
#pragma unroll
    for (int k = 0; k < kRW; ++k) {
      const uint32_t a = P[k], b = __shfl_xor_sync(0xffffffffu, P[k], o);
      P[k] = a ^ b ^ carry;
      carry = (a & b) | (carry & (a ^ b));
    }
  }
  const int lane = threadIdx.x & 31;
  int cnt = 0;
#pragma unroll
  for (int k = 0; k < kRW; ++k) cnt += (int)((P[k] >> lane) & 1u) << k;
  return cnt;
}

// grid: (blocks per word-lattice, word-lattices), kThreads threads; the
// register bound lets 14 blocks share an SM.
template <int kDim, bool kQuads, int kThreads>
__global__ void __launch_bounds__(kThreads, 896 / kThreads) measure_msc_rows_kernel(const uint32_t *__restrict__ w,
                                                               const uint32_t *__restrict__ J, Geom g,
                                                               long long *__restrict__ E,
                                                               long long *__restrict__ M,
                                                               long long *__restrict__ Q) {
  griddep_wait();
  griddep_release();
  constexpr int kWarps = kThreads / 32;
  __shared__ int cnt[3][kWarps][32];
  const uint32_t G = (uint32_t)g.n_real / 32, T = (uint32_t)g.n_temps;
  const uint32_t wl = blockIdx.y, lt = threadIdx.x;
  const uint32_t t = wl % T, grp = (wl / T) % G, a = wl / (T * G);
  const uint32_t L = (uint32_t)g.L, N = (uint32_t)g.N, half = N / 2, quads = half / 4, LH = L / 2;
  const uint32_t *s = w + (size_t)wl * N;
  const uint32_t *Jg = J + (size_t)grp * kDim * N;
  const bool do_q = Q && a == 0 && g.n_sets >= 2;
  const uint32_t *s1 = s + (size_t)G * T * N;  // set 1, same (g, t)
  CsaCount2 ce;
  CsaCount cm, cq;
  if (kQuads) {
  for (uint32_t q = blockIdx.x * kThreads + lt; q < 2 * quads; q += gridDim.x * kThreads) {
    const uint32_t c = q >= quads ? 1u : 0u;
      const uint32_t j0 = 4 * (q - c * quads);
      const uint32_t co = c * half, oc = (c ^ 1u) * half;
      const CsSite st = kDim == 3 ? cs_site(j0, (int)c, L, g.fL) : cs_site2(j0, (int)c, L, g.fL);
      const uint32_t p = st.i & 1u, jr = st.rb >> 1;
      const uint4 S = ldv4(s + co + j0), O = ldv4(s + oc + j0);
      // x + 1: the other colour at the same index (p = 0) or the next (p = 1)
      const uint32_t jx = j0 + 4 == jr + LH ? jr : j0 + 4;
      const uint32_t Ox = p ? s[oc + jx] : 0u;
      const uint4 YP = ldv4(s + oc + (st.yp >> 1));
      const uint4 ZP = kDim == 3 ? ldv4(s + oc + (st.zp >> 1)) : make_uint4(0, 0, 0, 0);
      const uint4 JX = ldv4(Jg + co + j0), JY = ldv4(Jg + N + co + j0);
      const uint4 JZ = kDim == 3 ? ldv4(Jg + 2 * N + co + j0) : make_uint4(0, 0, 0, 0);
      const uint32_t sv[4] = {S.x, S.y, S.z, S.w}, ov[4] = {O.x, O.y, O.z, O.w};
      const uint32_t yv[4] = {YP.x, YP.y, YP.z, YP.w}, zv[4] = {ZP.x, ZP.y, ZP.z, ZP.w};
      const uint32_t jxv[4] = {JX.x, JX.y, JX.z, JX.w}, jyv[4] = {JY.x, JY.y, JY.z, JY.w};
      const uint32_t jzv[4] = {JZ.x, JZ.y, JZ.z, JZ.w};
      // the bonds (i, i + e_d) of every site count each bond once
      uint32_t sum[4], car[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t xp = p ? (k < 3 ? ov[k + 1] : Ox) : ov[k];
        const uint32_t u0 = sv[k] ^ xp ^ jxv[k], u1 = sv[k] ^ yv[k] ^ jyv[k];
        const uint32_t u2 = kDim == 3 ? sv[k] ^ zv[k] ^ jzv[k] : 0u;
        sum[k] = u0 ^ u1 ^ u2;
        car[k] = (u0 & u1) | (u2 & (u0 ^ u1));
      }
      ce.add(sum, car);
      if (M) cm.add4(sv[0], sv[1], sv[2], sv[3]);
      if (do_q) {
        const uint4 S1 = ldv4(s1 + co + j0);
        cq.add4(S.x ^ S1.x, S.y ^ S1.y, S.z ^ S1.z, S.w ^ S1.w);
      }
    }
  } else {
    // storage index k: colour c = k / half, colour index j = k % half; the
    // last group of a thread may be short
    for (uint32_t k0 = blockIdx.x * 4 * kThreads + lt; k0 < N; k0 += gridDim.x * 4 * kThreads) {
      uint32_t sum[4], car[4], S[4], D[4];
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i) {
        const uint32_t k = k0 + i * kThreads;
        sum[i] = car[i] = S[i] = D[i] = 0u;
        if (k >= N) continue;
        const uint32_t c = k >= half ? 1u : 0u, oc = (c ^ 1u) * half;
        const CsSite st = kDim == 3 ? cs_site(k - c * half, (int)c, L, g.fL) : cs_site2(k - c * half, (int)c, L, g.fL);
        S[i] = s[k];
        const uint32_t u0 = S[i] ^ s[oc + (st.xp >> 1)] ^ Jg[k], u1 = S[i] ^ s[oc + (st.yp >> 1)] ^ Jg[N + k];
        const uint32_t u2 = kDim == 3 ? S[i] ^ s[oc + (st.zp >> 1)] ^ Jg[2 * N + k] : 0u;
        sum[i] = u0 ^ u1 ^ u2;
        car[i] = (u0 & u1) | (u2 & (u0 ^ u1));
        if (do_q) D[i] = S[i] ^ s1[k];
      }
      ce.add(sum, car);
      if (M) cm.add4(S[0], S[1], S[2], S[3]);
      if (do_q) cq.add4(D[0], D[1], D[2], D[3]);
    }
  }
  ce.flush();
  cm.flush();
  cq.flush();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  cnt[0][warp][lane] = warp_count(ce.C);
  if (M) cnt[1][warp][lane] = warp_count(cm.C);
  if (Q) cnt[2][warp][lane] = warp_count(cq.C);
  __syncthreads();
  if (warp != 0) return;
  // lane b of warp 0 adds the warps' counts of bit b
  long long e = 0, m = 0, d = 0;
#pragma unroll
  for (int k = 0; k < kWarps; ++k) {
    e += cnt[0][k][lane];
    if (M) m += cnt[1][k][lane];
    if (do_q) d += cnt[2][k][lane];
  }
  const int64_t lat = ((int64_t)a * T + t) * g.n_real + 32 * grp + lane;
  // E = 2 unsat - kDim N, M = N - 2 down, Q = N - 2 diff: part 0 adds the
  // constants; with one part per word-lattice the counts are stored
  const long long n0 = blockIdx.x == 0 ? (long long)N : 0;
  const bool direct = gridDim.x == 1;
  auto put = [direct](long long *ptr, long long v) {
    if (direct) *ptr = v;
    else add_ll(ptr, v);
  };
  if (E) put(&E[lat], 2 * e - kDim * n0);
  if (M) put(&M[lat], n0 - 2 * m);
  if (do_q) put(&Q[(int64_t)t * g.n_real + 32 * grp + lane], n0 - 2 * d);
}

// ---------------------------------------------------------------- Heisenberg
// Per-block partial sums in double, then a fixed-order second pass, so the
// result does not depend on scheduling.
template <int kC>
__global__ void measure_heis_kernel(const float4 *__restrict__ s, Geom g,
                                    double *__restrict__ partial) {
  griddep_wait();
  griddep_release();
  const int64_t lat = blockIdx.y;
  heis_block_partials<kC>(s + lat * g.N, (uint32_t)g.L, g.fL, g.dim, (uint32_t)g.N, blockIdx.x, gridDim.x,
                          partial + lat * kHeisParts * 4);
}

__global__ void finish_heis_kernel(const double *__restrict__ partial, int64_t n_lat,
                                   double *__restrict__ Ef, double *__restrict__ Mf) {
  griddep_wait();
  griddep_release();
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k < 4 * n_lat) heis_finish_component(partial, k, Ef, Mf);
}

// ---------------------------------------------------------------- replica exchange
// Thread per (set a, realisation r, pair t) of the step's parity.
__global__ void pt_decide_kernel(const long long *__restrict__ E, Geom g,
                                 PtTables tables, RoundKeys rk, uint32_t step,
                                 uint8_t *__restrict__ decision, long long *__restrict__ accepted,
                                 int *__restrict__ labels) {
  griddep_wait();
  griddep_release();
  const int parity = (int)(step & 1u);
  const int n_pairs = (g.n_temps - parity) / 2;  // pairs (t, t+1), t = parity + 2k
  const int64_t total = (int64_t)g.n_sets * n_pairs * g.n_real;
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= total) return;
  const int r = (int)(k % g.n_real);
  const int pk = (int)((k / g.n_real) % n_pairs);
  const int a = (int)(k / ((int64_t)g.n_real * n_pairs));
  const int t = parity + 2 * pk;
  const int64_t lat0 = ((int64_t)a * g.n_temps + t) * g.n_real + r;
  const int64_t lat1 = lat0 + g.n_real;
  const bool acc = pt_accept(pt_pair(tables, a, t, r, step, rk), E[lat0], E[lat1]);
  decision[lat0] = acc ? 1 : 0;
  if (labels && acc) {  // one thread per pair: no other thread touches these two
    const int l0 = labels[lat0];
    labels[lat0] = labels[lat1];
    labels[lat1] = l0;
  }
  if (!accepted) return;
  if ((g.n_real & 31) == 0) {
    // the 32 lanes of a warp share (a, t): one atomic per warp
    const uint32_t votes = __ballot_sync(0xffffffffu, acc);
    if ((threadIdx.x & 31) == 0 && votes) add_ll(&accepted[a * g.n_temps + t], __popc(votes));
  } else if (acc) {
    add_ll(&accepted[a * g.n_temps + t], 1);
  }
}

// Exchange of whole lattices (int8, or coded 2D lattices): 16 bytes per
// thread step when the lattice size is a multiple of 16 bytes (the spins
// buffer is 16-byte aligned, so every lattice then is), single bytes
// otherwise (e.g. 6^3 = 216-byte int8 lattices).
__global__ void pt_swap_bytes_kernel(uint8_t *__restrict__ s, const uint8_t *__restrict__ decision,
                                     Geom g, int parity, int64_t lat_bytes) {
  griddep_wait();
  griddep_release();
  const int64_t lat0 = blockIdx.y;
  const int t = (int)slot_of32(g, (uint32_t)lat0);
  if (((t - parity) & 1) || t + 1 >= g.n_temps || !decision[lat0]) return;
  uint8_t *b0 = s + lat0 * lat_bytes, *b1 = s + (lat0 + g.n_real) * lat_bytes;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  if ((lat_bytes & 15) == 0) {
    uint4 *p0 = reinterpret_cast<uint4 *>(b0), *p1 = reinterpret_cast<uint4 *>(b1);
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < lat_bytes / 16; k += step) {
      const uint4 a = p0[k], b = p1[k];
      p0[k] = b;
      p1[k] = a;
    }
  } else {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < lat_bytes; k += step) {
      const uint8_t a = b0[k], b = b1[k];
      b0[k] = b;
      b1[k] = a;
    }
  }
}

// Bitwise exchange of coded EA words: per (a, g, pair) the accepted
// realisations form a mask A (one warp ballot over their decisions);
// x = (w_t ^ w_{t+1}) & A exchanges those bits, 16 bytes at a time (N is a
// multiple of 8 and every word-lattice starts 32-byte aligned).
__global__ void pt_swap_msc_kernel(uint32_t *__restrict__ w, const uint8_t *__restrict__ decision,
                                   Geom g, int parity) {
  griddep_wait();
  griddep_release();
  const int G = g.n_real / 32;
  const int64_t wl = blockIdx.y;  // (a, grp, t)
  const int t = (int)(wl % g.n_temps);
  if (((t - parity) & 1) || t + 1 >= g.n_temps) return;
  const int grp = (int)((wl / g.n_temps) % G);
  const int a = (int)(wl / ((int64_t)g.n_temps * G));
  const int64_t lat0 = ((int64_t)a * g.n_temps + t) * g.n_real + 32 * grp;
  const uint32_t mask = __ballot_sync(0xffffffffu, decision[lat0 + (threadIdx.x & 31)] != 0);
  if (!mask) return;
  uint4 *w0 = reinterpret_cast<uint4 *>(w + wl * g.N), *w1 = reinterpret_cast<uint4 *>(w + (wl + 1) * g.N);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.N / 4;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint4 a0 = w0[i], a1 = w1[i];
    const uint4 x = make_uint4((a0.x ^ a1.x) & mask, (a0.y ^ a1.y) & mask, (a0.z ^ a1.z) & mask,
                               (a0.w ^ a1.w) & mask);
    w0[i] = make_uint4(a0.x ^ x.x, a0.y ^ x.y, a0.z ^ x.z, a0.w ^ x.w);
    w1[i] = make_uint4(a1.x ^ x.x, a1.y ^ x.y, a1.z ^ x.z, a1.w ^ x.w);
  }
}

unsigned capped(int64_t n, unsigned cap) {
  unsigned g = grid_for(n, 256);
  return g > cap ? cap : g;
}

}  // namespace

cudaError_t launch_measure(spin_lattice *h, const void *J, int64_t *E, int64_t *M, int64_t *Q,
                           double *Ef, double *Mf) {
  const Geom &g = h->g;
  cudaStream_t st = h->stream;
  const int64_t nl = h->n_lat;
  if (h->d.model == SPIN_HEISENBERG) {
    if (!Ef && !Mf) return cudaSuccess;
    double *partial = (double *)h->d_scratch64;
    const int c = heis_measure_cluster(g.N);
    const dim3 grid((unsigned)(kHeisParts * c), (unsigned)nl);
    const auto kern = c == 8   ? measure_heis_kernel<8>
                      : c == 4 ? measure_heis_kernel<4>
                      : c == 2 ? measure_heis_kernel<2>
                               : measure_heis_kernel<1>;
    const cudaError_t e = launch_clusters(kern, grid, dim3(256), c, 0, st, (const float4 *)h->spins, g, partial);
    if (e != cudaSuccess) return e;
    return launch_dependent(finish_heis_kernel, dim3(grid_for(4 * nl, 128)), dim3(128), 0, st,
                            (const double *)partial, nl, Ef, Mf);
  }
  if (h->d.layout == SPIN_MSC1 && h->d.model == SPIN_ISING) {
    if (Q) cudaMemsetAsync(Q, 0, sizeof(int64_t) * g.n_temps * g.n_real, st);
    return launch_measure_msc2d(h, E, M);
  }
  // EA coded words: parts of kRowThreads (or kRowThreadsFew) threads per
  // word-lattice, at most kRowItems groups of four sites per thread; with one
  // part per word-lattice the counts are stored, not added, and need no zeroing.
  // More threads for few word-lattices of more than 512 sites, and where one part
  // of them holds the lattice and kRowThreads need several.  4 sweeps in us with E,
  // M, Q after each, 64 / 256 threads, L x word-lattices: 2D 20 x 1024 54 / 63, 28 x
  // 768 61 / 61, 28 x 1280 76 / 88, 3D 12 x 768 101 / 96, 12 x 1024 116 / 114, 16 x 1280
  // 174 / 169, 12 x 2048 165 / 208, 18 x 2048 529 / 507, 26 x 1024 764 / 779.
  // A lattice of several parts has as many as give two CTAs to an SM (E, M and Q
  // alone of 28 x 4 in 2 parts 21.6, in 22 parts 9.1), and so has a lattice of one
  // part where its latency outweighs the zeroing: 4 sweeps with an exchange
  // after each, one / several parts, 20 x 4 69 / 47, 20 x 96 109 / 87, 16 x 96 66 / 73;
  // with E, M, Q after each 22 x 96 125 / 113, 20 x 96 100 / 104, 24 x 96 89 / 113.
  const int64_t n_wl = (int64_t)g.n_sets * (g.n_real / 32) * g.n_temps;
  const bool one = g.N <= 4 * kRowThreadsFew * kRowItems;
  const bool few = g.N > 512 && (g.N > 4096 && one ? true : n_wl < (g.N > 1024 && one ? 8 : 5) * h->sms);
  const int threads = few ? kRowThreadsFew : kRowThreads;
  int64_t parts = (g.N / 4 + threads * kRowItems - 1) / (threads * kRowItems);
  if (parts > 1 || (g.N > 4096 && !M && !Q) || (g.N > 8192 && g.L % 8 != 0))
    parts = std::max(parts, std::min((g.N / 4 + threads - 1) / threads, 2 * h->sms / n_wl));
  const unsigned gx = (unsigned)parts;
  const bool coded_direct = h->d.layout == SPIN_MSC1 && gx == 1;
  if (!coded_direct) {
    if (E) cudaMemsetAsync(E, 0, sizeof(int64_t) * nl, st);
    if (M) cudaMemsetAsync(M, 0, sizeof(int64_t) * nl, st);
    if (Q) cudaMemsetAsync(Q, 0, sizeof(int64_t) * g.n_temps * g.n_real, st);
  }
  cudaError_t e = cudaSuccess;
  if (h->d.layout == SPIN_I8) {
    if ((E || M) && !J && g.L % 8 == 0) {
      // full warps (the block is 256 threads); len steps per thread: few
      // enough blocks that their atomics do not queue, enough to fill the GPU
      const int chunks = g.L / 8;
      int bx = 1;
      while (bx < chunks && bx < 64) bx *= 2;
      const int by = 256 / bx, tiles_x = (chunks + bx - 1) / bx;
      int len = 16;
      while (len > 1 && nl * (g.N / 8) / len < 152 * 1024) len /= 2;
      const int segs = (g.L + len - 1) / len;
      const dim3 grid((unsigned)(tiles_x * (((g.dim == 3 ? g.L : segs) + by - 1) / by)),
                      g.dim == 3 ? (unsigned)segs : 1u, (unsigned)nl);
      e = launch_dependent(g.dim == 3 ? measure_chunks_i8_kernel<3> : measure_chunks_i8_kernel<2>, grid,
                           dim3(bx, by), 0, st, (const int8_t *)h->spins, g.L, tiles_x, len, (long long *)E,
                           (long long *)M);
    } else if (E || M) {
      e = launch_dependent(measure_i8_kernel, dim3(capped(g.N, 1024), (unsigned)nl), dim3(256), 0, st,
                           (const int8_t *)h->spins, (const int8_t *)J, g, (long long *)E, (long long *)M);
    }
    if (e == cudaSuccess && Q && g.n_sets >= 2)
      e = launch_dependent(overlap_i8_kernel, dim3(capped(g.N, 1024), (unsigned)(g.n_temps * g.n_real)),
                           dim3(256), 0, st, (const int8_t *)h->spins, g, (long long *)Q);
    return e;
  }
  const bool quads = g.L % 8 == 0;
  using Kern = decltype(&measure_msc_rows_kernel<3, true, kRowThreads>);
  const Kern kerns[2][2][2] = {
      {{measure_msc_rows_kernel<2, false, kRowThreads>, measure_msc_rows_kernel<2, false, kRowThreadsFew>},
       {measure_msc_rows_kernel<2, true, kRowThreads>, measure_msc_rows_kernel<2, true, kRowThreadsFew>}},
      {{measure_msc_rows_kernel<3, false, kRowThreads>, measure_msc_rows_kernel<3, false, kRowThreadsFew>},
       {measure_msc_rows_kernel<3, true, kRowThreads>, measure_msc_rows_kernel<3, true, kRowThreadsFew>}}};
  const Kern kern = kerns[g.dim == 3][quads][few];
  return launch_dependent(kern, dim3(gx, (unsigned)n_wl), dim3((unsigned)threads), 0, st,
                          (const uint32_t *)h->spins, (const uint32_t *)J, g, (long long *)E, (long long *)M,
                          (g.n_sets >= 2) ? (long long *)Q : nullptr);
}

cudaError_t launch_pt_swap(spin_lattice *h, const void *J, int64_t *accepted, int32_t *labels,
                           const int64_t *energies, void *planes) {
  const Geom &g = h->g;
  cudaStream_t st = h->stream;
  if (!energies) {
    cudaError_t e = planes ? planes_measure(h, h->d_energy, nullptr)
                           : launch_measure(h, J, h->d_energy, nullptr, nullptr, nullptr, nullptr);
    if (e != cudaSuccess) return e;
    energies = h->d_energy;
  }
  const uint32_t step = (uint32_t)h->pt_steps_done;
  const int parity = (int)(step & 1u);
  const int n_pairs = (g.n_temps - parity) / 2;
  uint8_t *decision = (uint8_t *)(h->d_energy + 2 * h->n_lat);
  if (n_pairs <= 0) return cudaSuccess;
  const int64_t total = (int64_t)g.n_sets * n_pairs * g.n_real;
  cudaError_t e = launch_dependent(pt_decide_kernel, dim3(grid_for(total, 256)), dim3(256), 0, st,
                                   (const long long *)energies, g, pt_tables(h), make_round_keys(h->d.seed), step,
                                   decision,
                                   (long long *)accepted, (int *)labels);
  if (e != cudaSuccess) return e;
  if (h->d.layout == SPIN_MSC1 && h->d.model == SPIN_EA) {
    const int64_t n_wl = (int64_t)g.n_sets * (g.n_real / 32) * g.n_temps;
    return launch_dependent(pt_swap_msc_kernel, dim3(capped(g.N / 4, 64), (unsigned)n_wl), dim3(256), 0, st,
                            (uint32_t *)h->spins, (const uint8_t *)decision, g, parity);
  } else {
    int64_t lat_bytes = g.N;  // int8
    if (h->d.layout == SPIN_MSC1) lat_bytes = g.N / 8;
    if (planes) lat_bytes = (int64_t)planes_lattice_bytes(h);
    const int64_t units = (lat_bytes & 15) == 0 ? lat_bytes / 16 : lat_bytes;
    return launch_dependent(pt_swap_bytes_kernel, dim3(capped(units, 1024), (unsigned)h->n_lat), dim3(256), 0, st,
                            (uint8_t *)(planes ? planes : h->spins), (const uint8_t *)decision, g, parity,
                            lat_bytes);
  }
}

}  // namespace spin
