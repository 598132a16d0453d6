// Longer calls on int8 ferromagnets (L % 8 == 0): the lattices are packed into
// bit planes (planes.cuh) in a handle-owned buffer, swept, measured and
// exchanged there, and unpacked at the end.  The random words and decisions
// are those of every int8 kernel, so the results are the same bit for bit.
//
// The byte kernels spend 22 to 25 lane instructions per flip, most of them on
// bytes; on planes the generator and its two or three comparisons per word
// are nearly all that is left.  Measured against them (us per call of the
// byte kernels -> here): one 3D L = 512, 4 sweeps and a measurement, 859 ->
// 530; three L = 1000, 20 sweeps and 2 measurements, 164 -> 111; 20 x L = 512,
// 20 sweeps and 2 exchanges, 135 -> 113 (packed once instead of per exchange).
#include <algorithm>

#include "internal.h"
#include "planes.cuh"

namespace spin {
int upload_pt_tables_for_batch(spin_lattice *h, const double *betas);  // api.cu
namespace {

// One colour phase, one thread per block and kN lattices, in the manner of
// msc2d_phase_kernel (msc2d.cu): the thread draws the block's calls, last one
// first, and shifts the comparisons into its masks (MaskBits) before
// griddep_wait(), since they depend on no spin; only the update waits for the
// previous phase.  Blocks with fewer bits than their colour's longest draw a
// few calls they do not use, so that a warp's loops end together.
template <int kDim, bool kNarrow, int kN>
__global__ void __launch_bounds__(256) planes_phase_kernel(uint4 *__restrict__ w, Planes m, Geom g, uint32_t n_lat,
                                                           const uint32_t *__restrict__ thr, RoundKeys rk,
                                                           uint32_t sweep, int colour) {
  griddep_release();
  const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= m.blocks) return;
  const PlaneBlock k = plane_block<kNarrow>(m, b);
  const uint32_t lat0 = blockIdx.y * kN;
  constexpr int kT = kDim;  // thresholds: dE = 4, 8 and, in 3D, 12
  PhiloxX0 pre[kN];
  uint32_t t[kN][kT], A[kN][kT][4];
#pragma unroll
  for (int n = 0; n < kN; ++n) {
    const uint32_t lat = min(lat0 + n, n_lat - 1);  // (a last group that is not full draws one lattice twice)
    const uint32_t slot = slot_of32(g, lat);
    pre[n] = philox_x0_setup(sweep, lattice_id32(g, lat), rk);
#pragma unroll
    for (int e = 0; e < kT; ++e) {
      t[n][e] = __ldg(thr + 4 * slot + 1 + e);
#pragma unroll
      for (int q = 0; q < 4; ++q) A[n][e][q] = 0u;
    }
  }
  const uint32_t wctr = ctr_w(TAG_UPDATE, (uint32_t)colour, 0);
#pragma unroll(kN == 1 ? 4 : 2)
  for (int i = (int)(kNarrow ? m.R * m.nb : m.w) - 1; i >= 0; --i) {
    const PhiloxX0Shared sh = philox_x0_shared(k.j4 + (uint32_t)i, wctr, rk);
#pragma unroll
    for (int n = 0; n < kN; ++n) {
      const uint4 r = philox_x0(pre[n], sh, rk);
#pragma unroll
      for (int e = 0; e < kT; ++e) {
        const MaskBits mb(t[n][e]);
        mb.push(A[n][e][0], r.x);
        mb.push(A[n][e][1], r.y);
        mb.push(A[n][e][2], r.z);
        mb.push(A[n][e][3], r.w);
      }
    }
  }
  griddep_wait();
  const uint32_t valid = low_bits(k.bits);
#pragma unroll
  for (int n = 0; n < kN; ++n) {
    if (lat0 + n >= n_lat) break;
    uint4 *S = w + ((size_t)(lat0 + n) * 2 + colour) * m.blocks;
    const uint4 *O = w + ((size_t)(lat0 + n) * 2 + (colour ^ 1)) * m.blocks;
    PlaneNbrs<kDim> nb;
    plane_nbrs<kDim, kNarrow>(m, O, b, k, colour, nb);
    uint32_t s[4];
    put4(s, S[b]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t m4 = MaskBits(t[n][0]).mask(A[n][0][q]), m8 = MaskBits(t[n][1]).mask(A[n][1][q]);
      const uint32_t m12 = kDim == 3 ? MaskBits(t[n][kT - 1]).mask(A[n][kT - 1][q]) : 0u;
      s[q] ^= plane_flips<kDim>(s[q], nb, q, m4, m8, m12) & valid;
    }
    S[b] = make_uint4(s[0], s[1], s[2], s[3]);
  }
}

// int8 <-> planes, one warp per block place (both colours): lane l holds the
// 8-byte chunk of call l of the block (the chunks of a block are contiguous
// in the row-major lattice), whose byte 2 q + p is the site of colour
// (p + y + z) & 1 in plane q, and one ballot per byte position builds a word.
__device__ __forceinline__ size_t chunk_index(const Planes &m, const PlaneBlock &k, uint32_t lat, int lane) {
  return (size_t)lat * ((size_t)m.L * (m.dim == 3 ? m.L : 1) * m.nb) + k.j4 + lane;
}

template <bool kNarrow, bool kPack>
__global__ void __launch_bounds__(256) planes_bytes_kernel(uint64_t *__restrict__ bytes, uint4 *__restrict__ w,
                                                           Planes m, uint32_t total, FastDiv fblocks) {
  griddep_wait();
  griddep_release();
  const int lane = threadIdx.x & 31;
  constexpr int kPer = 2;  // blocks a warp has in flight
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t first = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kPer; first < total; first += nwarps * kPer) {
    PlaneBlock k[kPer];
    uint32_t lat[kPer], b[kPer], par[kPer];
    uint64_t v[kPer];
    uint4 w0[kPer], w1[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      if (first + u >= total) break;  // uniform across the warp
      lat[u] = fdiv(first + u, fblocks);
      b[u] = first + u - lat[u] * m.blocks;
      k[u] = plane_block<kNarrow>(m, b[u]);
      // parity of the lane's row
      par[u] = kNarrow ? (k[u].par + (uint32_t)lane / m.nb) & 1u : k[u].par;
      if (kPack) {
        v[u] = (uint32_t)lane < k[u].bits ? bytes[chunk_index(m, k[u], lat[u], lane)] : 0ull;
      } else {
        w0[u] = w[(size_t)lat[u] * 2 * m.blocks + b[u]];
        w1[u] = w[((size_t)lat[u] * 2 + 1) * m.blocks + b[u]];
      }
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      if (first + u >= total) break;
      const bool mine = (uint32_t)lane < k[u].bits;
      if (kPack) {
        const uint2 x = chunk_words(v[u], par[u]);
        uint32_t word[8];
#pragma unroll
        for (int o = 0; o < 8; ++o)  // bit 1 of a +-1 byte is set for -1
          word[o] = __ballot_sync(0xffffffffu, mine && ((o < 4 ? x.x : x.y) >> (8 * (o & 3) + 1) & 1u));
        if (lane < 2)
          w[((size_t)lat[u] * 2 + lane) * m.blocks + b[u]] =
              lane ? make_uint4(word[1], word[3], word[5], word[7]) : make_uint4(word[0], word[2], word[4], word[6]);
      } else if (mine) {
        bytes[chunk_index(m, k[u], lat[u], lane)] = chunk_of(w0[u], w1[u], lane, par[u]);
      }
    }
  }
}

// Packing pieces of rows that start on 16-byte boundaries (nb and w even), one
// thread per block place: it reads its chunks two at a time, last ones first,
// and shifts the sign of every byte into its word (a funnel shift each, no
// ballot).  One 3D lattice of L = 512 packed in 72 us by warps, bound by the
// ballots, and in 41 here (134 MB: 20 us at the copy rate); unpacked this way
// its strided 16-byte stores took 91 us against 65 by warps.
__global__ void __launch_bounds__(256) planes_pack_thread_kernel(const uint4 *__restrict__ bytes,
                                                                 uint4 *__restrict__ w, Planes m, uint32_t total,
                                                                 FastDiv fblocks) {
  griddep_wait();
  griddep_release();
  const uint32_t id = blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= total) return;
  const uint32_t lat = fdiv(id, fblocks), b = id - lat * m.blocks;
  const PlaneBlock k = plane_block<false>(m, b);
  const uint4 *p = bytes + chunk_index(m, k, lat, 0) / 2;
  uint32_t a[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};  // by byte position of the chunk
  auto push = [&a](uint32_t x, int o) {
#pragma unroll
    for (int i = 0; i < 4; ++i) a[o + i] = __funnelshift_l(x << (24 - 8 * i), a[o + i], 1);
  };
#pragma unroll 8
  for (int i = (int)k.bits / 2 - 1; i >= 0; --i) {
    const uint4 v = __ldcs(p + i);
    push(v.z, 0);
    push(v.w, 4);
    push(v.x, 0);
    push(v.y, 4);
  }
  // byte 2 q + o of a chunk is the site of colour o ^ par in plane q
  const uint4 e = make_uint4(a[0], a[2], a[4], a[6]), o = make_uint4(a[1], a[3], a[5], a[7]);
  uint4 *w0 = w + (size_t)lat * 2 * m.blocks + b, *w1 = w0 + m.blocks;
  *w0 = k.par ? o : e;
  *w1 = k.par ? e : o;
}

// Energy and magnetisation: every bond joins the two colours, so the
// antiparallel neighbours of the colour-0 sites count each once;
// E = 2 n_anti - dim N, M = N - 2 n_down.  Adds to outputs the host zeroed.
template <int kDim, bool kNarrow>
__global__ void __launch_bounds__(256) planes_measure_kernel(const uint4 *__restrict__ w, Planes m, long long N,
                                                             long long *__restrict__ E, long long *__restrict__ M) {
  __shared__ int red[8][2];
  griddep_wait();
  griddep_release();
  const uint32_t lat = blockIdx.y;
  const uint4 *S = w + (size_t)lat * 2 * m.blocks, *O = S + m.blocks;
  int anti = 0, down = 0;
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < m.blocks; b += gridDim.x * blockDim.x) {
    const PlaneBlock k = plane_block<kNarrow>(m, b);
    PlaneNbrs<kDim> nb;
    plane_nbrs<kDim, kNarrow>(m, O, b, k, 0, nb);
    uint32_t s[4];
    put4(s, S[b]);
    const uint32_t valid = low_bits(k.bits);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      anti += __popc((s[q] ^ nb.u[q]) & valid) + __popc((s[q] ^ nb.d[q]) & valid) + __popc(s[q] ^ nb.o[q]) +
              __popc((s[q] ^ nb.s[q]) & valid);
      if (kDim == 3) anti += __popc(s[q] ^ nb.f[q]) + __popc(s[q] ^ nb.b[q]);
      down += __popc(s[q]) + __popc(nb.o[q]);
    }
  }
  anti = __reduce_add_sync(0xffffffffu, anti);
  down = __reduce_add_sync(0xffffffffu, down);
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5][0] = anti;
    red[threadIdx.x >> 5][1] = down;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  long long a = 0, d = 0;
  for (int i = 0; i < 8; ++i) a += red[i][0], d += red[i][1];
  const bool first = blockIdx.x == 0;
  if (E) atomicAdd((unsigned long long *)&E[lat], (unsigned long long)(2 * a - (first ? kDim * N : 0)));
  if (M) atomicAdd((unsigned long long *)&M[lat], (unsigned long long)((first ? N : 0) - 2 * d));
}

bool narrow(const Planes &m) { return m.nb <= 16; }

template <int kN>
auto phase_kernel(const Planes &m) {
  return m.dim == 3 ? (narrow(m) ? planes_phase_kernel<3, true, kN> : planes_phase_kernel<3, false, kN>)
                    : (narrow(m) ? planes_phase_kernel<2, true, kN> : planes_phase_kernel<2, false, kN>);
}

cudaError_t transcode(spin_lattice *h, bool pack) {
  const Planes m = make_planes(h->g.dim, h->g.L);
  const uint32_t total = (uint32_t)(h->n_lat * m.blocks);  // < 2^32: a block has at least 8 sites
  // (enough blocks for a thread each to fill the GPU)
  if (pack && !narrow(m) && m.nb % 2 == 0 && m.w % 2 == 0 && total >= (1u << 16))
    return launch_dependent(planes_pack_thread_kernel, dim3(grid_for(total, 256)), dim3(256), 0, h->stream,
                            (const uint4 *)h->spins, (uint4 *)h->d_pingpong, m, total, make_fastdiv(m.blocks));
  const auto kern = pack ? (narrow(m) ? planes_bytes_kernel<true, true> : planes_bytes_kernel<false, true>)
                         : (narrow(m) ? planes_bytes_kernel<true, false> : planes_bytes_kernel<false, false>);
  unsigned grid = grid_for(total, 16);  // 8 warps of 2 blocks
  if (grid > 152 * 64) grid = 152 * 64;
  return launch_dependent(kern, dim3(grid), dim3(256), 0, h->stream, (uint64_t *)h->spins, (uint4 *)h->d_pingpong, m, total,
                          make_fastdiv(m.blocks));
}

cudaError_t planes_sweeps(spin_lattice *h, int64_t n_sweeps) {
  const Planes m = make_planes(h->g.dim, h->g.L);
  const RoundKeys rk = make_round_keys(h->d.seed);
  const int kn = lattices_per_thread(h->n_lat, h->n_lat * m.blocks);
  const auto kern = kn == 3 ? phase_kernel<3>(m) : kn == 2 ? phase_kernel<2>(m) : phase_kernel<1>(m);
  const dim3 grid((m.blocks + 255) / 256, (unsigned)((h->n_lat + kn - 1) / kn));
  for (int64_t k = 0; k < n_sweeps; ++k)
    for (int colour = 0; colour < 2; ++colour) {
      const cudaError_t e = launch_dependent(kern, grid, dim3(256), 0, h->stream, (uint4 *)h->d_pingpong, m, h->g,
                                             (uint32_t)h->n_lat, (const uint32_t *)h->d_thr, rk,
                                             (uint32_t)(h->sweeps_done + k), colour);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

// Sweeps, measurements and exchanges of a call.  Its first launch takes the
// caller's bytes and its last one leaves them there; in between the lattices
// alternate between two buffers of planes.  An exchange is decided and carried
// out by the launch that follows it, the call's last one on the bytes.
int run_resident(spin_lattice *h, const double *betas, int64_t n_sweeps, int32_t measure_every, int32_t pt_every,
                 int64_t *E_series, int64_t *M_series, int64_t *accepted, int32_t *labels) {
  const int64_t nl = h->n_lat;
  const bool measuring = measure_every > 0 && (E_series || M_series);
  int64_t done = 0, rows = 0, tape_at = 0, tape_left = 0;
  int64_t *energies[2] = {h->d_energy, h->d_energy + nl};
  int which = 0;
  bool pending = false;  // an exchange with energies[which ^ 1] is due
  int rc = SPIN_OK, cur = 0;
  while (done < n_sweeps && rc == SPIN_OK) {
    const int64_t at = h->sweeps_done;
    if (tape_left == 0) {
      cudaError_t e;
      tape_left = planes_res_draw(h, at, n_sweeps - done, &e);
      tape_at = 0;
      if (e != cudaSuccess) return SPIN_ECUDA;
    }
    int64_t next = n_sweeps - done;
    if (pt_every > 0) next = std::min(next, pt_every - at % pt_every);
    next = std::min(next, tape_left);
    const bool exchange = pt_every > 0 && (at + next) % pt_every == 0;
    PlanesResCall call = {};
    call.every = call.first = 1;
    if (measuring) {
      call.E = E_series ? E_series + rows * nl : nullptr;
      call.M = M_series ? M_series + rows * nl : nullptr;
      call.every = measure_every;
      call.first = (int)(measure_every - at % measure_every);
      rows += (at + next) / measure_every - at / measure_every;
    }
    if (exchange) {
      call.E_last = energies[which];
      rc = upload_pt_tables_for_batch(h, betas);  // refused: the sweeps up to the exchange still run
    }
    call.bytes_in = done == 0;
    call.bytes_out = rc != SPIN_OK || done + next == n_sweeps;
    if (pending) {
      call.E_prev = energies[which ^ 1];
      call.step = (uint32_t)(h->pt_steps_done - 1);
      call.accepted = accepted;
      call.labels = labels;
    }
    if (planes_res_sweeps(h, tape_at, next, cur, call) != cudaSuccess) return SPIN_ECUDA;
    cur ^= 1;
    pending = false;
    h->sweeps_done += next;
    done += next;
    tape_at += next;
    tape_left -= next;
    if (exchange && rc == SPIN_OK) {
      pending = true;
      which ^= 1;
      h->pt_steps_done += 1;
    }
  }
  if (pending) {
    h->pt_steps_done -= 1;
    const cudaError_t e = launch_pt_swap(h, nullptr, accepted, labels, energies[which ^ 1]);
    h->pt_steps_done += 1;
    if (e != cudaSuccess) return SPIN_ECUDA;
  }
  return rc;
}

// The same with a launch per colour phase, in one buffer.
int run_phases(spin_lattice *h, const double *betas, int64_t n_sweeps, int32_t measure_every, int32_t pt_every,
               int64_t *E_series, int64_t *M_series, int64_t *accepted, int32_t *labels) {
  const int64_t nl = h->n_lat;
  const bool measuring = measure_every > 0 && (E_series || M_series);
  int64_t done = 0, rows = 0;
  int rc = SPIN_OK;
  while (done < n_sweeps && rc == SPIN_OK) {
    const int64_t at = h->sweeps_done;
    int64_t next = n_sweeps - done;
    if (measuring) next = std::min(next, measure_every - at % measure_every);
    if (pt_every > 0) next = std::min(next, pt_every - at % pt_every);
    if (planes_sweeps(h, next) != cudaSuccess) return SPIN_ECUDA;
    h->sweeps_done += next;
    done += next;
    const int64_t now = h->sweeps_done;
    const int64_t *energies = nullptr;  // energies measured at this sweep, if any
    if (measuring && now % measure_every == 0) {
      if (planes_measure(h, E_series ? E_series + rows * nl : nullptr, M_series ? M_series + rows * nl : nullptr) !=
          cudaSuccess)
        return SPIN_ECUDA;
      if (E_series) energies = E_series + rows * nl;
      ++rows;
    }
    if (pt_every > 0 && now % pt_every == 0) {
      rc = upload_pt_tables_for_batch(h, betas);
      if (rc == SPIN_OK && launch_pt_swap(h, nullptr, accepted, labels, energies, h->d_pingpong) != cudaSuccess)
        return SPIN_ECUDA;
      if (rc == SPIN_OK) h->pt_steps_done += 1;
    }
  }
  return rc;
}

}  // namespace

bool planes_supported(const spin_lattice *h) {
  return h->d.model == SPIN_ISING && h->d.layout == SPIN_I8 && h->g.L % 8 == 0;
}

size_t planes_lattice_bytes(const spin_lattice *h) {
  return (size_t)make_planes(h->g.dim, h->g.L).blocks * 2 * sizeof(uint4);
}

namespace {
// Whether one CTA per lattice with the masks drawn ahead (planes_res.cu) is the
// fastest form of long calls, by the number of lattices.  What ends it is the
// size of the masks: with few sweeps of them in a half of the buffer a call is
// many short launches.  Us per call of 32 sweeps, here / phases / the kernel
// with the lattice as bytes, at sweeps per half in brackets: 2D L = 8 x 38912
// 314 / 2579 / 334 (7), x 65520 637 / 4282 / 558 (4); L = 32 x 9728 282 / 1744 /
// 330 (7), x 19456 737 / 3299 / 655 (3); L = 64 x 4864 564 / 842 / 673 (3); L = 96
// x 2432 627 / 727 / 873 (2); L = 112 x 1216 383 / 421 / 593 (4); L = 128 x 608 243 /
// 249 / 347 (7), x 1024 413 / 382 / 606 (4), x 1216 560 / 479 / 693 (3); 3D L = 16 x
// 4864 594 / 998 / 816 (2); L = 24 x 304 124 / 169 / 179 (8), x 608 260 / 300 / 356
// (4); L = 32 x 152 150 / 150 / 418 (10), x 200 206 / 177 / 572 (7), x 304 285 / 256
// / 629 (5).  Two sizes have a byte kernel whose warps are just full and a word
// per thread of few warps here: 2D L = 16 x 1216 18 / 247 / 15, x 9728 99 / 1763 /
// 86; 3D L = 8 x 304 15 / 121 / 14 and 41 / 359 / 40 for 100 sweeps, x 2432 63 / 224 /
// 55.
//
// A measurement costs next to nothing here and about 8 us there (0.6 with the
// lattice as bytes in one CTA), an exchange one launch here and four to five small
// ones there: calls with many of them end later.  33 sweeps, an exchange every 8:
// 2D L = 16 x 9728 137 / 1948 / 215, L = 8 x 65520 891 / 5028 / 1204, L = 32 x 19456
// 806 / 3630 / 976, 3D L = 8 x 2432 77 / 292 / 197.  30 sweeps, here / phases,
// nothing, E and M every 10, 5, 1 sweeps: 2D L = 128 x 2048 821 / 699, 825 / 761, 828
// / 837, 847 / 1392; 3D L = 32 x 200 190 / 167, 192 / 201, 193 / 232, 202 / 444, x 304
// 279 / 241, 281 / 272, 283 / 305, 291 / 514, x 452 489 / 353, 492 / 382, 495 / 417,
// 508 / 696.
bool resident_pays(const spin_lattice *h, int32_t measure_every, int32_t pt_every) {
  if (!h->res_words) return false;
  const int64_t N = h->g.N, sweeps = h->res_tape_sweeps;
  const int words = h->res_words;
  auto within = [](int32_t every, int most) { return every > 0 && every <= most; };
  const int32_t swaps = h->g.n_temps > 1 ? pt_every : 0;
  if (words <= 192) {
    if (within(swaps, 10) || within(measure_every, 2)) return sweeps >= 2;
    if (h->g.dim == 2 && N == 256 && h->n_lat > 1024) return false;
    if (h->g.dim == 3 && N == 512 && h->n_lat > 304) return false;
    return sweeps >= (words <= 4 ? 6 : words <= 16 ? 4 : 2);
  }
  if (sweeps >= (words <= 288 ? 4 : 8)) return true;
  const int often = h->g.dim == 2 ? 5 : words <= 288 ? 4 : sweeps >= 4 ? 10 : 2;
  return sweeps >= 2 && (within(swaps, often) || within(measure_every, often));
}

// The conversions of a call cost about what planes save in a few sweeps of the
// byte kernels.  Us per call, planes / bytes.  Against the fused pass, 4
// sweeps: one 2D L = 144 21 / 33, 20 x L = 512 30 / 49, three L = 8000 619 / 893;
// 2 sweeps 13 / 17, 21 / 25, 381 / 446: the line could lie lower.
constexpr int64_t kFusedMinSweeps = 4;
// Against the colour phases in three dimensions, 2 sweeps: one L = 40 14 / 26,
// three L = 264 198 / 202, one L = 512 293 / 409.
constexpr int64_t kPhases3MinSweeps = 2;
// In two dimensions small lattices wait for launches in either form, 3.5 us per
// sweep (one L = 136 ... 760, 60 sweeps: 220 / 205), and the conversions are
// lost: the least sweeps by the sites of all lattices (one L = 840: 6 sweeps 27 /
// 27; one L = 1000: 3 17 / 16, 4 21 / 22; three: 2 16 / 15, 3 19 / 22; 20 x L = 184:
// 8 38 / 36, 20 80 / 106; 20 x L = 440: 2 19 / 18, 3 22 / 27; one L = 2008: 2 18 / 18).
int64_t phases2_min_sweeps(int64_t sites) {
  return sites >= 3500000 ? 2 : sites >= 2400000 ? 3 : sites >= 900000 ? 4
         : sites >= 700000  ? 6 : sites >= 550000  ? 16 : INT64_MAX;
}
}  // namespace

PlanesForm planes_form(const spin_lattice *h, int64_t n, int32_t measure_every, int32_t pt_every) {
  if (!planes_supported(h) || h->order != SPIN_ORDER_CHECKERBOARD || n < 1) return PlanesForm::none;
  auto phases_from = [n](int64_t least) { return n >= least ? PlanesForm::phases : PlanesForm::none; };
  const int64_t N = h->g.N;
  if (h->variant == 4) return phases_from(kFusedMinSweeps);
  const bool crowded = 2 * h->n_lat > h->sms;
  if (h->variant == 3) {
    // The launch that draws the masks ahead costs what the sweeps must win back
    // from the kernel with the lattice as bytes, about 0.14 us + 0.13 ns per site
    // and sweep, and 12 us per exchange (us per call of 4 / 8 / 16 / 64 sweeps,
    // bytes against planes: L = 16 5.1 / 5.5 / 8.1 / 24 against 7.3 / 7.6 / 7.7 /
    // 16, L = 64 5.5 / 8.7 / 14 / 51 against 8.1 / 8.9 / 10 / 20, L = 128 14 / 25
    // / 45 / 171 against 8.7 / 9.7 / 12 / 25); a little more where other lattices'
    // CTAs are in the way (120 x L = 128: 3 sweeps 11 against 14; 152 x L = 80: 8
    // sweeps 12 against 14; 450 x L = 32: 24 sweeps 15 against 19), unless the
    // byte kernel's do not all fit at once (200 x 3D L = 24: 4 sweeps 27 against 19).
    const double wins = (double)n * (0.14 + 0.00013 * (double)N) +
                        (pt_every > 0 ? 12.0 * (double)(n / pt_every) : 0.0);
    const bool in_the_way = crowded && N >= 1024 && (N < 6400 || h->n_lat <= h->sms);
    if (resident_pays(h, measure_every, pt_every))
      return wins >= (in_the_way ? 8.0 : 5.5) ? PlanesForm::resident : PlanesForm::none;
    // too many for the masks: the byte kernel up to L = 72 (2D) and 16 (3D), the
    // phases above (us per call of 4 / 32 sweeps, bytes against phases: 9728 x
    // L = 64 200 / 1338 against 262 / 1751, 4864 x L = 80 205 / 1326 against 146 /
    // 852, x L = 128 410 / 2777 against 294 / 1760, x 3D L = 24 421 / 2847
    // against 410 / 2601; with E and M after every sweep the bytes again, 30 sweeps
    // of 2048 x 3D L = 24 1502 against 1699)
    return h->auto_form && N >= 6400 && (measure_every < 1 || measure_every > 2) ? phases_from(3) : PlanesForm::none;
  }
  if (!h->auto_form) return PlanesForm::none;
  if (h->variant == 1) return phases_from(kFusedMinSweeps);
  if (h->g.dim == 2) return phases_from(phases2_min_sweeps(h->n_lat * N));
  // (3D L = 32: 84 lattices, 4 sweeps 25 by phases against 19, 120 27 against 31, 6
  // sweeps 36 against 33, 4 with E and M after each 57 against 32)
  if (resident_pays(h, measure_every, pt_every) &&
      n >= (3 * h->n_lat > 2 * h->sms && measure_every < 1 && pt_every < 1 ? 6 : kPhases3MinSweeps))
    return PlanesForm::resident;
  return phases_from(kPhases3MinSweeps);
}

PlanesForm planes_ready(spin_lattice *h, PlanesForm form, int64_t n_sweeps) {
  if (form == PlanesForm::none || h->sweeps_done + n_sweeps > (int64_t)0xFFFFFFFFll)  // (refused by the other paths)
    return PlanesForm::none;
  if (form == PlanesForm::resident) {
    if (planes_res_reserve(h, n_sweeps)) return form;
    if (h->variant == 3) return PlanesForm::none;
  }
  const size_t bytes = (size_t)h->n_lat * planes_lattice_bytes(h);
  return working_buffer(h, bytes, false) == cudaSuccess ? PlanesForm::phases : PlanesForm::none;
}

int planes_run(spin_lattice *h, PlanesForm form, const double *betas, int64_t n_sweeps, int32_t measure_every,
               int32_t pt_every, int64_t *E_series, int64_t *M_series, int64_t *accepted, int32_t *labels) {
  if (form == PlanesForm::resident)
    return run_resident(h, betas, n_sweeps, measure_every, pt_every, E_series, M_series, accepted, labels);
  if (transcode(h, true) != cudaSuccess) return SPIN_ECUDA;
  const int rc = run_phases(h, betas, n_sweeps, measure_every, pt_every, E_series, M_series, accepted, labels);
  if (rc == SPIN_ECUDA) return rc;
  // also after a refused exchange: the sweeps up to it stand
  return transcode(h, false) == cudaSuccess ? rc : SPIN_ECUDA;
}

cudaError_t planes_measure(spin_lattice *h, int64_t *E, int64_t *M) {
  if (!E && !M) return cudaSuccess;
  const Planes m = make_planes(h->g.dim, h->g.L);
  if (E) cudaMemsetAsync(E, 0, sizeof(int64_t) * h->n_lat, h->stream);
  if (M) cudaMemsetAsync(M, 0, sizeof(int64_t) * h->n_lat, h->stream);
  const auto kern = m.dim == 3 ? (narrow(m) ? planes_measure_kernel<3, true> : planes_measure_kernel<3, false>)
                               : (narrow(m) ? planes_measure_kernel<2, true> : planes_measure_kernel<2, false>);
  unsigned gx = grid_for(m.blocks, 256);
  if (gx > 1024) gx = 1024;
  return launch_dependent(kern, dim3(gx, (unsigned)h->n_lat), dim3(256), 0, h->stream, (const uint4 *)h->d_pingpong, m,
                          (long long)h->g.N, (long long *)E, (long long *)M);
}

}  // namespace spin
