// 2D Ising ferromagnet with synchronous multi-spin coding (Sec. 5: several
// spins of one lattice per word).  Per lattice the spins are stored as
// [2 colours][L rows][L/64 words]; in row y the colour-c sites are
// x = 2k + ((c + y) & 1), k = 0 .. L/2-1, grouped in blocks of 128 k's with
// k = 128 B + 4 l + q stored in bit l of word 4 B + q (bit set <=> s = -1).
//
// Every site keeps its own uniform (sites of one lattice must not share
// random numbers), drawn exactly as in the int8 layout: for k = 128 B + 4 l + q
// the colour index is j = y L/2 + k, so the Philox call j >> 2 = y L/8 + 32 B
// + l serves bit l of the four words 4 B + q, word q of the call for word q.
// The comparisons with the two thresholds become acceptance masks; the
// neighbour count and the flip decision are bit-sliced.
#include "internal.h"
#include "msc2d_block.cuh"

namespace spin {
namespace {

struct Msc2d {
  int L;
  int wpr;   // words per row and colour = L / 64
  int bpr;   // blocks per row = L / 256
  int64_t lat_words;  // 2 * L * wpr
};

__device__ __forceinline__ int64_t row_word(const Msc2d &m, int64_t lat, int c, int y) {
  return lat * m.lat_words + ((int64_t)c * m.L + y) * m.wpr;
}

// One colour phase, one thread per block of 128 sites and kN lattices: the
// thread draws the block's 32 Philox calls, last call first, shifts every
// word's two comparisons into the block's masks (MaskBits), and updates the
// block from registers.  The kN lattices share the part of each call that
// depends only on the site.  Bound by the wide multiplies (16.7 to 18 per
// call, at about 26 per clock and SM with the rest of the generator around
// them), the ALU pipe close behind.
//
// The masks depend on no spin, so they are drawn before griddep_wait(): the
// generator of a phase fills the SMs while the previous phase drains, and
// only the update waits for it.  Measured per phase, against one warp per 32
// blocks with ballots for masks, all of it after the wait (us): 3 x L = 16384
// 300 -> 242, 16 x L = 1024 9.1 -> 5.4, 20 x L = 512 7.5 -> 2.4, one L = 1024
// 5.8 -> 2.0.  Grid: (blocks of a lattice / 256, groups of kN lattices).
template <int kN>
__global__ void __launch_bounds__(256) msc2d_phase_kernel(uint32_t *__restrict__ w, Msc2d m, Geom g,
                                                                 uint32_t n_lat, uint32_t per_lat,
                                                                 const uint32_t *__restrict__ thr, RoundKeys rk,
                                                                 uint32_t sweep, int colour) {
  griddep_release();
  const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= per_lat) return;
  const uint32_t lat0 = blockIdx.y * kN;
  PhiloxX0 pre[kN];
  uint32_t thr4[kN], thr8[kN], A[kN][4], E[kN][4];
#pragma unroll
  for (int n = 0; n < kN; ++n) {
    const uint32_t lat = min(lat0 + n, n_lat - 1);  // (a last group that is not full draws one lattice twice)
    const uint32_t t = slot_of32(g, lat);
    pre[n] = philox_x0_setup(sweep, lattice_id32(g, lat), rk);
    thr4[n] = __ldg(thr + 4 * t + 1);
    thr8[n] = __ldg(thr + 4 * t + 2);
#pragma unroll
    for (int q = 0; q < 4; ++q) A[n][q] = E[n][q] = 0u;
  }
  const uint32_t wctr = ctr_w(TAG_UPDATE, (uint32_t)colour, 0);
#pragma unroll(kN == 1 ? 4 : 2)
  for (int i = 31; i >= 0; --i) {
    const PhiloxX0Shared sh = philox_x0_shared(32u * b + (uint32_t)i, wctr, rk);
#pragma unroll
    for (int n = 0; n < kN; ++n) {
      const uint4 r = philox_x0(pre[n], sh, rk);
      const MaskBits m4(thr4[n]), m8(thr8[n]);
      m4.push(A[n][0], r.x);
      m4.push(A[n][1], r.y);
      m4.push(A[n][2], r.z);
      m4.push(A[n][3], r.w);
      m8.push(E[n][0], r.x);
      m8.push(E[n][1], r.y);
      m8.push(E[n][2], r.z);
      m8.push(E[n][3], r.w);
    }
  }
  griddep_wait();  // the masks depend on no spin
  const uint32_t y = b / (uint32_t)m.bpr, B = b - y * (uint32_t)m.bpr;
  long long unused_a = 0, unused_d = 0;
#pragma unroll
  for (int n = 0; n < kN; ++n) {
    if (lat0 + n >= n_lat) break;
    const MaskBits m4(thr4[n]), m8(thr8[n]);
    msc2d_block<0>(w + (int64_t)(lat0 + n) * m.lat_words, m.L, m.wpr, m.bpr, colour, (int)y, B,
                   make_uint4(m4.mask(A[n][0]), m4.mask(A[n][1]), m4.mask(A[n][2]), m4.mask(A[n][3])),
                   make_uint4(m8.mask(E[n][0]), m8.mask(E[n][1]), m8.mask(E[n][2]), m8.mask(E[n][3])), unused_a,
                   unused_d);
  }
}

// Hot start: bit 0 of the INIT word of each site, as in the int8 layout.
__global__ void msc2d_init_kernel(uint32_t *__restrict__ w, Msc2d m, Geom g, int64_t n_lat,
                                  RoundKeys rk, int hot) {
  const int64_t total = n_lat * m.lat_words;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total;
       k += (int64_t)gridDim.x * blockDim.x) {
    if (!hot) {
      w[k] = 0u;
      continue;
    }
    const int64_t lat = k / m.lat_words;
    const int64_t rem = k - lat * m.lat_words;
    const int c = (int)(rem / ((int64_t)m.L * m.wpr));
    const int y = (int)((rem / m.wpr) % m.L);
    const int wi = (int)(rem % m.wpr);
    const int B = wi >> 2, q = wi & 3;
    const int p = (c + y) & 1;
    const uint32_t lid = lattice_id_of(g, lat);
    uint32_t v = 0;
    for (int l = 0; l < 32; ++l) {
      const int k2 = 128 * B + 4 * l + q;
      const int64_t i = (int64_t)y * m.L + 2 * k2 + p;
      const uint4 r = philox(make_uint4((uint32_t)(i >> 2), 0u, lid, ctr_w(TAG_INIT, 0, 0)), rk);
      v |= (word_of(r, (uint32_t)(i & 3)) & 1u) << l;
    }
    w[k] = v;
  }
}

// Layout conversion site by site, for byte buffers at any address.
__global__ void msc2d_unpack_kernel(const uint32_t *__restrict__ w, int8_t *__restrict__ out,
                                    Msc2d m, int64_t n_lat) {
  const int64_t N = (int64_t)m.L * m.L;
  const int64_t total = n_lat * N;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t lat = k / N, i = k - lat * N;
    const int y = (int)(i / m.L), x = (int)(i % m.L);
    const int c = (x + y) & 1, kk = x >> 1;
    const int B = kk >> 7, l = (kk >> 2) & 31, q = kk & 3;
    const uint32_t v = w[row_word(m, lat, c, y) + 4 * B + q];
    out[k] = ((v >> l) & 1u) ? (int8_t)-1 : (int8_t)1;
  }
}

__global__ void msc2d_pack_kernel(const int8_t *__restrict__ in, uint32_t *__restrict__ w,
                                  Msc2d m, int64_t n_lat) {
  const int64_t total = n_lat * m.lat_words;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t lat = k / m.lat_words;
    const int64_t rem = k - lat * m.lat_words;
    const int c = (int)(rem / ((int64_t)m.L * m.wpr));
    const int y = (int)((rem / m.wpr) % m.L);
    const int wi = (int)(rem % m.wpr);
    const int B = wi >> 2, q = wi & 3;
    const int p = (c + y) & 1;
    uint32_t v = 0;
    for (int l = 0; l < 32; ++l) {
      const int x = 2 * (128 * B + 4 * l + q) + p;
      v |= (in[lat * (int64_t)m.L * m.L + (int64_t)y * m.L + x] < 0 ? 1u : 0u) << l;
    }
    w[k] = v;
  }
}

// int8 <-> coded transcoding, one warp per 256-site block (lattice, row y,
// block B) and both colours: lane l holds the eight bytes x = 256 B + 8 l ..
// + 7 of the row, i.e. the sites k = 128 B + 4 l + q of both colours
// (x = 2k + p, p = (c + y) & 1), so byte o = 2q + p of every lane is bit l of
// coded word 4 B + q of colour c, and one warp ballot per byte position o
// builds that word.  Loads and stores of the int8 rows are 256 contiguous
// bytes per warp; a warp takes kTcBlocks blocks at a time, all loads first,
// so that several are in flight.  Block indices are < 2^31 (spin_init checks
// n_lat L L / 256 < 2^31); fper divides by the blocks per lattice, fbpr by
// the blocks per row.
constexpr int kTcBlocks = 4;

struct TcBlock {
  uint32_t lat;
  int y, B;
};

__device__ __forceinline__ TcBlock tc_block(uint32_t blk, const FastDiv &fper, const FastDiv &fbpr) {
  TcBlock t;
  t.lat = fdiv(blk, fper);
  const uint32_t rem = blk - t.lat * fper.d;
  t.y = (int)fdiv(rem, fbpr);
  t.B = (int)(rem - (uint32_t)t.y * fbpr.d);
  return t;
}

__device__ __forceinline__ int64_t tc_row_byte(const Msc2d &m, const TcBlock &t) {
  return ((int64_t)t.lat * m.L + t.y) * (int64_t)m.L + 256 * t.B;
}

__global__ void msc2d_pack_warp_kernel(const int8_t *__restrict__ in, uint32_t *__restrict__ w, Msc2d m,
                                       uint32_t n_blocks, FastDiv fper, FastDiv fbpr) {
  const int lane = threadIdx.x & 31;
  const uint32_t warp0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t first = warp0 * kTcBlocks; first < n_blocks; first += nwarps * kTcBlocks) {
    uint2 v[kTcBlocks];
#pragma unroll
    for (int u = 0; u < kTcBlocks; ++u) {
      v[u] = make_uint2(0u, 0u);
      if (first + u < n_blocks) {
        const TcBlock t = tc_block(first + u, fper, fbpr);
        v[u] = reinterpret_cast<const uint2 *>(in + tc_row_byte(m, t))[lane];
      }
    }
#pragma unroll
    for (int u = 0; u < kTcBlocks; ++u) {
      if (first + u >= n_blocks) break;  // uniform across the warp
      const TcBlock t = tc_block(first + u, fper, fbpr);
      uint32_t word = 0;
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        const uint32_t half = o < 4 ? v[u].x : v[u].y;
        const uint32_t bal = __ballot_sync(0xffffffffu, (half >> (8 * (o & 3) + 1)) & 1u);  // bit 1 <=> -1
        if (lane == o) word = bal;
      }
      if (lane < 8) {
        const int q = lane >> 1, c = (lane & 1) ^ (t.y & 1);  // byte parity p = (c + y) & 1
        w[row_word(m, t.lat, c, t.y) + 4 * t.B + q] = word;
      }
    }
  }
}

__global__ void msc2d_unpack_warp_kernel(const uint32_t *__restrict__ w, int8_t *__restrict__ out, Msc2d m,
                                         uint32_t n_blocks, FastDiv fper, FastDiv fbpr) {
  const int lane = threadIdx.x & 31;
  const uint32_t warp0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t first = warp0 * kTcBlocks; first < n_blocks; first += nwarps * kTcBlocks) {
    // lanes 0..7 fetch the eight words of each block, every lane then takes its bit of each
    uint32_t mine[kTcBlocks];
#pragma unroll
    for (int u = 0; u < kTcBlocks; ++u) {
      mine[u] = 0u;
      if (lane < 8 && first + u < n_blocks) {
        const TcBlock t = tc_block(first + u, fper, fbpr);
        const int q = lane >> 1, c = (lane & 1) ^ (t.y & 1);
        mine[u] = w[row_word(m, t.lat, c, t.y) + 4 * t.B + q];
      }
    }
#pragma unroll
    for (int u = 0; u < kTcBlocks; ++u) {
      if (first + u >= n_blocks) break;  // uniform across the warp
      const TcBlock t = tc_block(first + u, fper, fbpr);
      uint32_t lo = 0, hi = 0;
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        const uint32_t word = __shfl_sync(0xffffffffu, mine[u], o);
        const uint32_t byte = ((word >> lane) & 1u) ? 0xFFu : 0x01u;
        if (o < 4) lo |= byte << (8 * o);
        else hi |= byte << (8 * (o - 4));
      }
      reinterpret_cast<uint2 *>(out + tc_row_byte(m, t))[lane] = make_uint2(lo, hi);
    }
  }
}

Msc2d geom2d(const spin_lattice *h) {
  Msc2d m;
  m.L = h->g.L;
  m.wpr = m.L / 64;
  m.bpr = m.L / 256;
  m.lat_words = 2 * (int64_t)m.L * m.wpr;
  return m;
}

unsigned capped2(int64_t n) {
  unsigned g = grid_for(n, 256);
  return g > (1u << 20) ? (1u << 20) : g;
}

}  // namespace

cudaError_t launch_init_msc2d(spin_lattice *h) {
  const Msc2d m = geom2d(h);
  msc2d_init_kernel<<<capped2(h->n_lat * m.lat_words), 256, 0, h->stream>>>(
      (uint32_t *)h->spins, m, h->g, h->n_lat, make_round_keys(h->d.seed), h->d.hot_start);
  return cudaGetLastError();
}

// Lattices per thread: the count with the best rate (1547, 1631, 1665
// flips/ns for 1, 2, 3 when the GPU and every group are full) after the idle
// places of the last group, among those that leave 2^15 threads, about half
// the threads of the GPU at this kernel's registers (20 x L = 512, 20480
// blocks, us per phase for 1, 2, 3: 2.42, 2.79, 3.16; 16 x L = 1024, 65536
// blocks: 5.62, 5.42, 5.98; 12 x L = 2048, 196608 blocks: 16.5, 15.6, 15.4).
int lattices_per_thread(int64_t n_lat, int64_t blocks) {
  const double rate[4] = {0.0, 1547.0, 1631.0, 1665.0};
  int best = 1;
  double most = 0.0;
  for (int k = 1; k <= 3; ++k) {
    if (k > 1 && blocks / k < (1 << 15)) break;
    const double r = rate[k] * (double)n_lat / (double)((n_lat + k - 1) / k * k);
    if (r > most) most = r, best = k;
  }
  return best;
}

cudaError_t launch_sweeps_msc2d(spin_lattice *h, int64_t n_sweeps) {
  const Msc2d m = geom2d(h);
  const RoundKeys rk = make_round_keys(h->d.seed);
  const uint32_t per_lat = (uint32_t)(m.L * m.bpr);
  const int kn = lattices_per_thread(h->n_lat, h->n_lat * per_lat);
  const auto kern = kn == 3 ? msc2d_phase_kernel<3> : kn == 2 ? msc2d_phase_kernel<2> : msc2d_phase_kernel<1>;
  const dim3 grid((per_lat + 255) / 256, (unsigned)((h->n_lat + kn - 1) / kn));
  for (int64_t k = 0; k < n_sweeps; ++k) {
    const uint32_t sweep = (uint32_t)(h->sweeps_done + k);
    for (int colour = 0; colour < 2; ++colour) {
      const cudaError_t e =
          launch_dependent(kern, grid, dim3(256), 0, h->stream, (uint32_t *)h->spins, m, h->g, (uint32_t)h->n_lat, per_lat,
                           (const uint32_t *)h->d_thr, rk, sweep, colour);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

// Whether int8 lattices may ask for the coded form of their sweeps (variant 4,
// planes.cu).
bool coded_i8_supported(const spin_lattice *h) {
  return h->d.model == SPIN_ISING && h->d.layout == SPIN_I8 && h->d.dim == 2 && h->g.L % 256 == 0 &&
         h->n_lat * (int64_t)h->g.L * (h->g.L / 256) < ((int64_t)1 << 31);
}

namespace {
// Conversion of all lattices of the handle between bytes and the words w.
// The warp kernels read and write 8 bytes per lane; a byte buffer that is
// not 8-byte aligned takes the per-site kernels (16 x L = 1024: pack 17.6 us
// and unpack 90 us per site, 7 and 5 us by warps).
cudaError_t transcode(spin_lattice *h, const int8_t *in, int8_t *out, uint32_t *words) {
  const Msc2d m = geom2d(h);
  const uint32_t n_blocks = (uint32_t)(h->n_lat * (int64_t)m.L * m.bpr);  // < 2^31, checked by spin_init
  const FastDiv fper = make_fastdiv((uint32_t)(m.L * m.bpr)), fbpr = make_fastdiv((uint32_t)m.bpr);
  // one group of kTcBlocks blocks per warp, 8 warps per CTA
  const unsigned grid = (unsigned)(((int64_t)n_blocks + 8 * kTcBlocks - 1) / (8 * kTcBlocks));
  const bool aligned = ((uintptr_t)(in ? (const void *)in : (const void *)out) & 7u) == 0;
  if (in && aligned)
    msc2d_pack_warp_kernel<<<grid, 256, 0, h->stream>>>(in, words, m, n_blocks, fper, fbpr);
  else if (in)
    msc2d_pack_kernel<<<capped2(h->n_lat * m.lat_words), 256, 0, h->stream>>>(in, words, m, h->n_lat);
  else if (aligned)
    msc2d_unpack_warp_kernel<<<grid, 256, 0, h->stream>>>(words, out, m, n_blocks, fper, fbpr);
  else
    msc2d_unpack_kernel<<<capped2(h->n_lat * h->g.N), 256, 0, h->stream>>>(words, out, m, h->n_lat);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_unpack_msc2d(spin_lattice *h, int8_t *out) {
  return transcode(h, nullptr, out, (uint32_t *)h->spins);
}

cudaError_t launch_pack_msc2d(spin_lattice *h, const int8_t *in) {
  return transcode(h, in, nullptr, (uint32_t *)h->spins);
}

// Energy and magnetisation of the 2D coded lattices: every bond joins a
// colour-0 and a colour-1 site, so counting the antiparallel neighbours of
// the colour-0 words counts each bond once; E = 2 n_anti - 2N, M = N - 2 n_down.
__global__ void msc2d_measure_kernel(const uint32_t *__restrict__ w, Msc2d m, int64_t n_lat,
                                     long long *__restrict__ E, long long *__restrict__ M) {
  const int64_t lat = blockIdx.y;
  const uint32_t blocks = (uint32_t)m.L * (uint32_t)m.bpr;  // blocks of 4 colour-0 words per lattice
  griddep_wait();
  griddep_release();
  const uint32_t *wl = w + lat * m.lat_words;
  int anti = 0, down = 0;  // (at most 64 blocks of 512 bonds per thread, L < 2^16)
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < blocks; k += gridDim.x * blockDim.x) {
    const uint32_t y = k / (uint32_t)m.bpr, B = k - y * (uint32_t)m.bpr;
    const uint32_t yu = y == 0 ? (uint32_t)m.L - 1 : y - 1, yd = y == (uint32_t)m.L - 1 ? 0 : y + 1;
    const uint32_t *O = wl + ((int64_t)m.L + y) * m.wpr;  // colour 1, row y
    const uint4 s = *reinterpret_cast<const uint4 *>(wl + (int64_t)y * m.wpr + 4 * B);
    const uint4 o = *reinterpret_cast<const uint4 *>(O + 4 * B);
    const uint4 u = *reinterpret_cast<const uint4 *>(wl + ((int64_t)m.L + yu) * m.wpr + 4 * B);
    const uint4 d = *reinterpret_cast<const uint4 *>(wl + ((int64_t)m.L + yd) * m.wpr + 4 * B);
    // second horizontal neighbour of the colour-0 sites: k - 1 (y even) or k + 1 (y odd)
    uint4 sh;
    if ((y & 1u) == 0) {
      const uint32_t Bp = B == 0 ? (uint32_t)m.bpr - 1 : B - 1;
      sh = make_uint4((o.w << 1) | (O[4 * Bp + 3] >> 31), o.x, o.y, o.z);
    } else {
      const uint32_t Bn = B == (uint32_t)m.bpr - 1 ? 0 : B + 1;
      sh = make_uint4(o.y, o.z, o.w, (o.x >> 1) | (O[4 * Bn] << 31));
    }
    anti += __popc(s.x ^ u.x) + __popc(s.x ^ d.x) + __popc(s.x ^ o.x) + __popc(s.x ^ sh.x) +
            __popc(s.y ^ u.y) + __popc(s.y ^ d.y) + __popc(s.y ^ o.y) + __popc(s.y ^ sh.y) +
            __popc(s.z ^ u.z) + __popc(s.z ^ d.z) + __popc(s.z ^ o.z) + __popc(s.z ^ sh.z) +
            __popc(s.w ^ u.w) + __popc(s.w ^ d.w) + __popc(s.w ^ o.w) + __popc(s.w ^ sh.w);
    down += __popc(s.x) + __popc(s.y) + __popc(s.z) + __popc(s.w) + __popc(o.x) + __popc(o.y) + __popc(o.z) +
            __popc(o.w);
  }
  // one pair of atomics per CTA: per warp, their queue at the lattice's two
  // sums took most of the time (3 x L = 16384: 126 us)
  __shared__ int red[8][2];
  anti = __reduce_add_sync(0xffffffffu, anti);
  down = __reduce_add_sync(0xffffffffu, down);
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5][0] = anti;
    red[threadIdx.x >> 5][1] = down;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  long long a = 0, d = 0;
  for (int k = 0; k < 8; ++k) a += red[k][0], d += red[k][1];
  const long long N = (long long)m.L * m.L;
  const bool first = blockIdx.x == 0;
  atomicAdd((unsigned long long *)&E[lat], (unsigned long long)(2 * a - (first ? 2 * N : 0)));
  atomicAdd((unsigned long long *)&M[lat], (unsigned long long)((first ? N : 0) - 2 * d));
}

cudaError_t launch_measure_msc2d(spin_lattice *h, int64_t *E, int64_t *M) {
  const Msc2d m = geom2d(h);
  long long *e = (long long *)E, *mm = (long long *)M;
  // both outputs are required by the kernel; route a missing one to scratch
  if (!e) e = (long long *)h->d_energy;
  if (!mm) mm = (long long *)h->d_energy + h->n_lat;
  cudaMemsetAsync(e, 0, sizeof(long long) * h->n_lat, h->stream);
  cudaMemsetAsync(mm, 0, sizeof(long long) * h->n_lat, h->stream);
  const int64_t blocks = (int64_t)m.L * m.bpr;  // one thread per block of 4 colour-0 words
  unsigned gx = grid_for(blocks, 256 * 4);  // a few blocks per thread, where there are enough
  if (gx > 1024u) gx = 1024u;
  return launch_dependent(msc2d_measure_kernel, dim3(gx, (unsigned)h->n_lat), dim3(256), 0, h->stream,
                          (const uint32_t *)h->spins, m, h->n_lat, e, mm);
}

}  // namespace spin
