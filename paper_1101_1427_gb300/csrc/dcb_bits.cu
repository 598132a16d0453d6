// Double checkerboard of the 2D int8 ferromagnet (Sec. 3.2, 3.4) with the
// tile as bits in registers.
//
// dcb_tile_kernel (dcb.cu) keeps a tile as bytes in shared memory, one thread
// per 8-byte chunk, with a CTA barrier per fine colour.  Here a thread owns
// kR rows of a T x T tile as bit planes and gives them all hits: per colour
// four words, plane q holding the sites k = 4 n + q of the rows (site
// x = 2 k + p, p = (colour + y) & 1), bit r T/8 + n for row r -- the layout
// of the coded 2D lattices on a tile.  The T / kR lanes of a tile fetch the
// rows above and below theirs by warp shuffles.  A Philox call serves one bit
// of the four planes, so the thread draws its calls last bit first and shifts
// the comparisons into its masks (MaskBits); three hits are drawn together,
// since the calls of a chunk at successive sweep numbers share their first
// rounds (PhiloxX1).  Tile halos do not change during a launch and stay in
// registers too.
//
// Bound by the wide multiplies (16 per call, 26 per clock and SM) once the
// GPU is full; 22 lane instructions per flip in the byte form, 13.5 here.
// One L = 8192 lattice, 100 hits (us, both coarse colours, byte form -> here):
// T = 8 6415 -> 4514, T = 16 6434 -> 4084, T = 32 6366 -> 4157, T = 64
// 6262 -> 4460; three L = 4096: 4825 -> 3518, 4833 -> 3496, 4784 -> 3557,
// 4764 -> 3527 (T = 16: 3072 warps for 3040 places at 96 registers, so that
// 32 of them make a second wave); one hit on three L = 4096: T = 16 121 -> 69.
#include "internal.h"

namespace spin {
namespace {

template <int kT, int kR>
struct BitTile {
  static constexpr int kNb = kT / 8;  // bits (calls) per row and plane
  static constexpr int kRows = kR;    // rows per thread (even)
  static constexpr int kLanes = kT / kRows;                    // lanes per tile
  static constexpr int kBits = kRows * kNb;
  static constexpr uint32_t rows_mask(int first, int step, uint32_t pattern) {
    uint32_t v = 0;
    for (int r = first; r < kRows; r += step) v |= pattern << (r * kNb);
    return v;
  }
  static constexpr uint32_t kRow = (1u << kNb) - 1u;                            // one row
  static constexpr uint32_t kOdd = rows_mask(1, 2, kRow);                       // rows with y odd
  static constexpr uint32_t kStart = rows_mask(0, 1, 1u);                       // first bit of every row
  static constexpr uint32_t kEnd = rows_mask(0, 1, 1u << (kNb - 1));            // last bit of every row
  static constexpr uint32_t kAll = kBits == 32 ? 0xffffffffu : (1u << (kBits & 31)) - 1u;
};

// Bit 1 of a +-1 byte is set for -1.
__device__ __forceinline__ uint32_t down_bit(uint64_t chunk, int byte) {
  return (uint32_t)(chunk >> (8 * byte + 1)) & 1u;
}

// Updates colour c of the thread's rows: s its planes, o the other colour's,
// ud the rows beyond the tile (row above in the first row's bits, row below
// in the last row's), lr the sites beside it (left neighbours of the rows
// with p = 0 in their first bit, right neighbours of the others in the last).
template <int kT, int kR>
__device__ __forceinline__ void update_bits(uint32_t (&s)[4], const uint32_t (&o)[4], const uint32_t (&ud)[4],
                                            uint32_t lr, int c, bool top, bool bottom, const uint32_t (&m4)[4],
                                            const uint32_t (&m8)[4]) {
  using G = BitTile<kT, kR>;
  constexpr int kLast = (G::kRows - 1) * G::kNb;
  const uint32_t p1 = c ? G::kAll & ~G::kOdd : G::kOdd;  // rows whose second neighbour is k + 1
  const uint32_t left = (o[3] << 1 & ~G::kStart) | (lr & G::kStart);
  const uint32_t right = (o[0] >> 1 & ~G::kEnd) | (lr & G::kEnd);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t above = ud[q] & G::kRow, below = ud[q] & (G::kRow << kLast);
    if (G::kLanes > 1) {
      const uint32_t a = __shfl_up_sync(0xffffffffu, o[q], 1, G::kLanes) >> kLast;
      const uint32_t b = __shfl_down_sync(0xffffffffu, o[q], 1, G::kLanes) << kLast;
      above = top ? above : a;
      below = bottom ? below : b;
    }
    const uint32_t u = (o[q] << G::kNb) | above, d = (o[q] >> G::kNb) | below;
    const uint32_t km = q == 0 ? left : o[q == 0 ? 0 : q - 1], kp = q == 3 ? right : o[q == 3 ? 3 : q + 1];
    const uint32_t sh = (km & ~p1) | (kp & p1);
    const uint32_t a0 = s[q] ^ u, a1 = s[q] ^ d, a2 = s[q] ^ o[q], a3 = s[q] ^ sh;
    const uint32_t s1 = a0 ^ a1, c1 = a0 & a1, s2 = a2 ^ a3, c2 = a2 & a3;
    const uint32_t ge2 = c1 | c2 | (s1 & s2), b0 = s1 ^ s2;
    // n antiparallel neighbours: n >= 2 flips, n = 1 flips iff r < thr4, n = 0 iff r < thr8
    s[q] ^= (ge2 | (b0 & m4[q]) | (~b0 & m8[q])) & G::kAll;
  }
}

template <int kT, int kR, int kS>
__device__ __forceinline__ void hits(uint32_t (&s)[2][4], const uint32_t (&ud)[2][4], const uint32_t (&lr)[2],
                                     bool top, bool bottom, uint32_t j0, uint32_t row_chunks, uint32_t lid,
                                     uint32_t sweep, const MaskBits &b4, const MaskBits &b8, const RoundKeys &rk) {
  using G = BitTile<kT, kR>;
  uint32_t A[2][kS][4], E[2][kS][4];
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int h = 0; h < kS; ++h)
#pragma unroll
      for (int q = 0; q < 4; ++q) A[c][h][q] = E[c][h][q] = 0u;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const uint32_t wctr = ctr_w(TAG_UPDATE, (uint32_t)c, 0);
#pragma unroll 1
    for (int r = G::kRows - 1; r >= 0; --r) {
#pragma unroll(G::kNb > 1 ? 2 : 1)
      for (int n = G::kNb - 1; n >= 0; --n) {
        const PhiloxX1 pre = philox_x1_setup(j0 + (uint32_t)r * row_chunks + (uint32_t)n, lid, wctr, rk);
#pragma unroll
        for (int h = 0; h < kS; ++h) {
          const uint4 w = philox_x1(pre, sweep + (uint32_t)h, rk);
          b4.push(A[c][h][0], w.x);
          b4.push(A[c][h][1], w.y);
          b4.push(A[c][h][2], w.z);
          b4.push(A[c][h][3], w.w);
          b8.push(E[c][h][0], w.x);
          b8.push(E[c][h][1], w.y);
          b8.push(E[c][h][2], w.z);
          b8.push(E[c][h][3], w.w);
        }
      }
    }
  }
#pragma unroll
  for (int h = 0; h < kS; ++h)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      uint32_t m4[4], m8[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) m4[q] = b4.mask(A[c][h][q]), m8[q] = b8.mask(E[c][h][q]);
      update_bits<kT, kR>(s[c], s[c ^ 1], ud[c], lr[c], c, top, bottom, m4, m8);
    }
}

constexpr int kBitThreads = 64;  // small CTAs, for even shares of a launch that is one or two waves

template <int kT, int kR, int kS>
__global__ void __launch_bounds__(kBitThreads) dcb_bits_kernel(int8_t *__restrict__ spins, int L, int coarse,
                                                               uint32_t sweep0, int k,
                                                               const uint32_t *__restrict__ thr, Geom g,
                                                               RoundKeys rk) {
  using G = BitTile<kT, kR>;
  griddep_wait();
  griddep_release();
  const int half = (L / kT) >> 1, n_tiles = (L / kT) * half;
  const uint32_t id = blockIdx.x * kBitThreads + threadIdx.x;
  const bool active = id / G::kLanes < (uint32_t)n_tiles;  // (whole tiles: the shuffles below need every lane)
  const int t = active ? (int)(id / G::kLanes) : 0, lane = (int)(id % G::kLanes);
  const bool top = lane == 0, bottom = lane == G::kLanes - 1;
  const int by = t / half, bx = 2 * (t % half) + ((by + coarse) & 1);
  const int64_t lat = blockIdx.y;
  const int x0 = bx * kT, y0 = by * kT + lane * G::kRows;
  int8_t *base = spins + lat * (int64_t)L * L + x0;
  const int xl = x0 == 0 ? L - 1 : -1, xr = x0 + kT == L ? kT - L : kT;  // the columns beside the tile
  uint32_t s[2][4], ud[2][4], lr[2] = {0u, 0u};
#pragma unroll
  for (int q = 0; q < 4; ++q) s[0][q] = s[1][q] = ud[0][q] = ud[1][q] = 0u;
  // rows -1 .. kRows; y0 is even, so row r has the parity of r
#pragma unroll
  for (int r = -1; r <= G::kRows; ++r) {
    const bool beyond = r < 0 || r == G::kRows;
    if (beyond && !(r < 0 ? top : bottom)) continue;
    const int y = y0 + r, yw = y < 0 ? L - 1 : y == L ? 0 : y;
    const int8_t *row = base + (int64_t)yw * L;
#pragma unroll
    for (int n = 0; n < G::kNb; ++n) {
      const uint64_t v = reinterpret_cast<const uint64_t *>(row)[n];
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        const int c = (b + r) & 1;  // byte 2 q + p belongs to colour (p + y) & 1
        // a halo site of colour c neighbours the sites of the other colour
        if (!beyond)
          s[c][b >> 1] |= down_bit(v, b) << (r * G::kNb + n);
        else
          ud[c ^ 1][b >> 1] |= down_bit(v, b) << ((r < 0 ? 0 : G::kRows - 1) * G::kNb + n);
      }
    }
    if (!beyond) {
      const uint32_t vl = ((uint32_t)(uint8_t)row[xl] >> 1) & 1u, vr = ((uint32_t)(uint8_t)row[xr] >> 1) & 1u;
      // p = 0 for colour r & 1, p = 1 for the other
      lr[r & 1] |= vl << (r * G::kNb);
      lr[(r & 1) ^ 1] |= vr << (r * G::kNb + G::kNb - 1);
    }
  }
  const uint32_t slot = slot_of32(g, (uint32_t)lat);
  const MaskBits b4(__ldg(thr + 4 * slot + 1)), b8(__ldg(thr + 4 * slot + 2));
  const uint32_t lid = lattice_id32(g, (uint32_t)lat), row_chunks = (uint32_t)L >> 3;
  const uint32_t j0 = (uint32_t)y0 * row_chunks + (uint32_t)(x0 >> 3);
  int h = 0;
  for (; h + kS <= k; h += kS)
    hits<kT, kR, kS>(s, ud, lr, top, bottom, j0, row_chunks, lid, sweep0 + (uint32_t)h, b4, b8, rk);
  for (; h < k; ++h) hits<kT, kR, 1>(s, ud, lr, top, bottom, j0, row_chunks, lid, sweep0 + (uint32_t)h, b4, b8, rk);
  if (!active) return;
#pragma unroll
  for (int r = 0; r < G::kRows; ++r)
#pragma unroll
    for (int n = 0; n < G::kNb; ++n) {
      uint64_t v = 0x0101010101010101ull;
#pragma unroll
      for (int b = 0; b < 8; ++b)
        v |= (uint64_t)((s[(b + r) & 1][b >> 1] >> (r * G::kNb + n)) & 1u ? 0xFEu : 0u) << (8 * b);
      reinterpret_cast<uint64_t *>(base + (int64_t)(y0 + r) * L)[n] = v;
    }
}

template <int kT, int kR>
cudaError_t launch_t(spin_lattice *h, int coarse, uint32_t sweep0) {
  constexpr int kS = 3;
  const int B = h->g.L / kT;
  const int64_t threads = (int64_t)B * B / 2 * BitTile<kT, kR>::kLanes;
  const dim3 grid((unsigned)((threads + kBitThreads - 1) / kBitThreads), (unsigned)h->n_lat);
  // even shares of grids that fit at once (us for 100 hits on three L = 1440, as
  // the CTAs fall / spread: T = 8 619 / 537, T = 16 668 / 584)
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
  static OncePerDevice limit;
  if (!limit.done(dev)) {
    const cudaError_t e = cudaFuncSetAttribute(dcb_bits_kernel<kT, kR, kS>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)spread_smem(1, 1));
    if (e != cudaSuccess) return e;
    limit.mark(dev);
  }
  const size_t smem = spread_smem((int64_t)grid.x * grid.y, h->sms);
  return launch_dependent(dcb_bits_kernel<kT, kR, kS>, grid, dim3(kBitThreads), smem, h->stream, (int8_t *)h->spins,
                          h->g.L, coarse, sweep0, h->order_hits, (const uint32_t *)h->d_thr, h->g,
                          make_round_keys(h->d.seed));
}

}  // namespace

// Sites of a coarse colour / 256.  The byte form spreads a tile over more
// threads and stays for fewer sites, and for T = 128, whose tiles span warps.
// Us for 100 hits at 6144 / 8192 / 24576 / 36864 / 98304 units, T = 16:
// byte form 387 / 444 / 1275 / 1869 / 4833, 4 rows per thread 413 / 413 /
// 1116 / 1468 / 3711, 16 rows 784 / 783 / 1210 / 1505 / 3496; T = 8 (8 rows)
// at 2048 / 6144 / 8192: byte form 158 / 391 / 453, here 229 / 366 / 367.
// T = 64: 2 rows beat 4 up to 98304 units (3527 against 3727); byte form and
// here at 9600 / 11616 / 13824 / 16224 units 514 / 499, 629 / 732, 743 / 732, 858 /
// 734.
namespace {
int64_t units(const spin_lattice *h) { return h->n_lat * (h->g.N / 512); }
}  // namespace

bool dcb_bits_preferred(const spin_lattice *h) {
  const int64_t least = h->order_tile == 8 ? 6144 : h->order_tile == 64 ? 13500 : 8192;
  return h->g.dim == 2 && h->order_tile <= 64 && units(h) >= least;
}

cudaError_t launch_dcb_bits(spin_lattice *h, int coarse, uint32_t sweep0) {
  const bool wide = units(h) >= 49152;  // rows enough per thread to fill its words
  switch (h->order_tile) {
    case 8:
      return launch_t<8, 8>(h, coarse, sweep0);
    case 16:
      return wide ? launch_t<16, 16>(h, coarse, sweep0) : launch_t<16, 4>(h, coarse, sweep0);
    case 32:
      return wide ? launch_t<32, 8>(h, coarse, sweep0) : launch_t<32, 2>(h, coarse, sweep0);
    default:
      return launch_t<64, 2>(h, coarse, sweep0);
  }
}

}  // namespace spin
