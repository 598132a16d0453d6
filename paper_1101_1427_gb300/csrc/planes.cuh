// Ising ferromagnets on the square and the cubic lattice as bit planes, for
// any L % 8 == 0: the working form of int8 lattices in longer calls.
//
// The sites of colour c in row (y, z) are x = 2 k + p, p = (c + y + z) & 1;
// plane q of the row holds the sites k = 4 n + q, n < L/8, so that bit n of
// the four planes is one Philox call (colour index >> 2 = row L/8 + n).  A
// block is up to 32 bits of the four planes of one colour, one uint4: either
// one of bpr pieces of w bits of a row (L > 128), or R whole rows of L/8 bits
// (L <= 128).  Pieces and row groups are of equal size, only the last may be
// smaller; bits beyond a block's own are 0.  A lattice is [2 colours][blocks]
// of uint4, block ((z nby + g) bpr + B) for piece B of row group g.  With
// L % 256 == 0 in two dimensions this is the public coded layout.
#pragma once
#include "common.cuh"

namespace spin {

struct Planes {
  int dim, L;
  uint32_t nb;      // bits (calls) per row
  uint32_t bpr, w;  // pieces per row, bits per piece
  uint32_t R, nby;  // rows per block, blocks per column of L rows
  uint32_t zstep;   // blocks per plane z
  uint32_t blocks;  // blocks per colour
  FastDiv fbpr, fnby;
};

inline Planes make_planes(int dim, int L) {
  Planes g;
  g.dim = dim;
  g.L = L;
  g.nb = (uint32_t)L / 8;
  g.bpr = (g.nb + 31) / 32;
  g.w = (g.nb + g.bpr - 1) / g.bpr;
  const uint32_t most = g.nb <= 16 ? 32 / g.nb : 1;  // rows that fit a word
  g.nby = ((uint32_t)L + most - 1) / most;
  g.R = ((uint32_t)L + g.nby - 1) / g.nby;
  g.nby = ((uint32_t)L + g.R - 1) / g.R;
  g.zstep = g.nby * g.bpr;
  g.blocks = g.zstep * (dim == 3 ? (uint32_t)L : 1u);
  g.fbpr = make_fastdiv(g.bpr);
  g.fnby = make_fastdiv(g.nby);
  return g;
}

// Block b of a colour: its place, its first call and its bits.
struct PlaneBlock {
  uint32_t z, g, B;
  uint32_t bits;  // calls of the block
  uint32_t j4;    // Philox counter word 0 of bit 0
  uint32_t par;   // parity of y + z of its first row
};

template <bool kNarrow>
__device__ __forceinline__ PlaneBlock plane_block(const Planes &m, uint32_t b) {
  PlaneBlock k;
  const uint32_t gz = kNarrow ? b : fdiv(b, m.fbpr);
  k.B = kNarrow ? 0u : b - gz * m.bpr;
  k.z = m.dim == 3 ? fdiv(gz, m.fnby) : 0u;
  k.g = gz - k.z * m.nby;
  const uint32_t y = k.g * m.R, row = k.z * (uint32_t)m.L + y;
  k.j4 = row * m.nb + k.B * m.w;
  k.bits = kNarrow ? min(m.R, (uint32_t)m.L - y) * m.nb : min(m.w, m.nb - k.B * m.w);
  k.par = (y + k.z) & 1u;
  return k;
}

__device__ __forceinline__ uint32_t low_bits(uint32_t n) { return n >= 32 ? 0xffffffffu : (1u << n) - 1u; }

// The 8-byte chunk v of a call's sites as two words whose byte 2 q + c (of the
// eight) is the site of colour c in plane q; par: parity of y + z of its row.
__device__ __forceinline__ uint2 chunk_words(uint64_t v, uint32_t par) {
  uint32_t lo = (uint32_t)v, hi = (uint32_t)(v >> 32);
  if (par) {
    lo = __byte_perm(lo, 0u, 0x2301);
    hi = __byte_perm(hi, 0u, 0x2301);
  }
  return make_uint2(lo, hi);
}

// The chunk of bit `lane` of a block's planes w0, w1 (colours 0 and 1).
__device__ __forceinline__ uint64_t chunk_of(const uint4 &w0, const uint4 &w1, int lane, uint32_t par) {
  const uint32_t a[8] = {w0.x, w1.x, w0.y, w1.y, w0.z, w1.z, w0.w, w1.w};
  uint32_t lo = 0x01010101u, hi = 0x01010101u;
#pragma unroll
  for (int o = 0; o < 8; ++o) {
    const uint32_t f = (a[o] >> lane & 1u) * (0xFEu << (8 * (o & 3)));  // 0x01 | 0xFE = -1
    if (o < 4) lo |= f;
    else hi |= f;
  }
  if (par) {
    lo = __byte_perm(lo, 0u, 0x2301);
    hi = __byte_perm(hi, 0u, 0x2301);
  }
  return ((uint64_t)hi << 32) | lo;
}

// The neighbours of the sites of block k of colour c in the other colour's
// blocks O: per plane the sites above and below (y -+ 1), the two beside
// (x -+ 1; which is which does not matter) and, in 3D, in front and behind.
template <int kDim>
struct PlaneNbrs {
  uint32_t u[4], d[4], o[4], s[4], f[4], b[4];
};

__device__ __forceinline__ void put4(uint32_t (&v)[4], const uint4 &a) {
  v[0] = a.x;
  v[1] = a.y;
  v[2] = a.z;
  v[3] = a.w;
}

template <int kDim, bool kNarrow>
__device__ __forceinline__ void plane_nbrs(const Planes &m, const uint4 *__restrict__ O, uint32_t b,
                                           const PlaneBlock &k, int c, PlaneNbrs<kDim> &n) {
  put4(n.o, O[b]);
  const uint32_t gu = k.g == 0 ? m.nby - 1 : k.g - 1, gd = k.g == m.nby - 1 ? 0u : k.g + 1;
  put4(n.u, O[b + (gu - k.g) * m.bpr]);
  put4(n.d, O[b + (gd - k.g) * m.bpr]);
  if (kDim == 3) {
    put4(n.f, O[k.z == 0 ? b + m.blocks - m.zstep : b - m.zstep]);
    put4(n.b, O[k.z == (uint32_t)m.L - 1 ? b + m.zstep - m.blocks : b + m.zstep]);
  }
  if (kNarrow) {
    const uint32_t nb = m.nb, last = k.bits - nb;
    const uint32_t last_u = (min(m.R, (uint32_t)m.L - gu * m.R) - 1) * nb, row = low_bits(nb);
    // one bit per row: the first, the last; rows of odd parity
    uint32_t start = 0, odd = 0;
    for (uint32_t r = 0; r < m.R; ++r) {
      start |= 1u << (r * nb);
      if (((r + k.par + (uint32_t)c) & 1u) != 0) odd |= row << (r * nb);
    }
    const uint32_t end = start << (nb - 1);
    const uint32_t left = (n.o[3] << 1 & ~start) | (n.o[3] >> (nb - 1) & start);
    const uint32_t right = (n.o[0] >> 1 & ~end) | (n.o[0] << (nb - 1) & end);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      n.u[q] = (n.o[q] << nb) | (n.u[q] >> last_u);
      n.d[q] = (n.o[q] >> nb) | ((n.d[q] & row) << last);
      n.s[q] = ((q == 0 ? left : n.o[q == 0 ? 0 : q - 1]) & ~odd) | ((q == 3 ? right : n.o[q == 3 ? 3 : q + 1]) & odd);
    }
  } else if (((k.par + (uint32_t)c) & 1u) == 0) {  // p = 0: the second neighbour is k - 1
    const uint32_t Bp = k.B == 0 ? m.bpr - 1 : k.B - 1, wp = min(m.w, m.nb - Bp * m.w);
    n.s[0] = (n.o[3] << 1) | (O[b + (Bp - k.B)].w >> (wp - 1));
    n.s[1] = n.o[0];
    n.s[2] = n.o[1];
    n.s[3] = n.o[2];
  } else {
    const uint32_t Bn = k.B == m.bpr - 1 ? 0u : k.B + 1;
    n.s[0] = n.o[1];
    n.s[1] = n.o[2];
    n.s[2] = n.o[3];
    n.s[3] = (n.o[0] >> 1) | (O[b + (Bn - k.B)].x << (k.bits - 1));
  }
}

// One plane of the Metropolis update: s its sites, the antiparallel
// neighbours counted bit-sliced.  2D: dE = 8 - 4 n, n >= 2 flips, n = 1, 0
// flip by m4, m8; 3D: dE = 12 - 4 n, n >= 3 flips, n = 2, 1, 0 by m4, m8, m12.
template <int kDim>
__device__ __forceinline__ uint32_t plane_flips(uint32_t s, const PlaneNbrs<kDim> &n, int q, uint32_t m4,
                                                uint32_t m8, uint32_t m12) {
  const uint32_t a0 = s ^ n.u[q], a1 = s ^ n.d[q], a2 = s ^ n.o[q], a3 = s ^ n.s[q];
  if (kDim == 2) {
    const uint32_t s1 = a0 ^ a1, s2 = a2 ^ a3, b0 = s1 ^ s2;
    const uint32_t ge2 = (a0 & a1) | (a2 & a3) | (s1 & s2);
    return ge2 | (b0 & m4) | (~b0 & m8);
  }
  const uint32_t a4 = s ^ n.f[q], a5 = s ^ n.b[q];
  const uint32_t x0 = a0 ^ a1, x1 = a3 ^ a4;
  const uint32_t s1 = x0 ^ a2, c1 = (a0 & a1) | (x0 & a2);
  const uint32_t s2 = x1 ^ a5, c2 = (a3 & a4) | (x1 & a5);
  const uint32_t b0 = s1 ^ s2, c3 = s1 & s2;
  const uint32_t any2 = c1 | c2 | c3;
  const uint32_t ge3 = (c1 & c2) | (c1 & c3) | (c2 & c3) | (any2 & b0);
  return ge3 | (any2 & m4) | (~any2 & ((b0 & m8) | (~b0 & m12)));
}

}  // namespace spin
