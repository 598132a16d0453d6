// Heisenberg energy and magnetisation in FP64 (Sec. 4: double accumulation
// for continuous spins), shared by spin_measure and the allocation-free
// reduction so that the two give bit-identical sums.
//
// E = -sum_<ij> s_i . s_j with each bond counted once as (i, i + e_d), and
// M = sum_i s_i, over one lattice of L^dim float4 spins (x fastest, periodic).
// A thread sums its sites in grid-stride order, then warp, block, cluster and
// (in the finishing step) the partials are added in FP64 in a fixed order.
//
// This GPU adds about 2 doubles per clock and SM against 128 floats, and the
// 25 FP64 additions, products and conversions of a site bound the kernel
// (one lattice of L = 128: 251 us on 64 CTAs, 125 us on 512).  So a thread
// keeps its sums as exact three-term expansions of floats (Sum3): each
// product is split without error into its rounded value and the remainder
// (one FMA), and each addition passes its rounding error (Knuth's two-sum)
// to the next term.  The expansion carries 72 bits, more than a double, and
// becomes a double once per thread: about 36 us, and a call of 20 sweeps and one
// measurement at L = 128 went from 601 to 384 us.  Sums whose spins are far from
// unit length, where an FP32 product could overflow or vanish, are formed in FP64.
//
// A lattice has kHeisParts partials whatever its size; large lattices take a
// cluster of 2, 4 or 8 CTAs per partial, whose sums rank 0 adds in rank order,
// so that up to 512 CTAs share the work.  The rule depends on the lattice size
// alone, so that the sums do not depend on how many lattices a call takes.  It
// keeps 16 sites and more per thread, since the FP64 additions of the tree cost a
// thread as much as several sites: with 8 CTAs per partial, 8 lattices of L = 64
// took 123 us and 4 of L = 80 68 us, with one 37 and 39; one of L = 80 26 against
// 33, of L = 100 30 against 55.
#pragma once
#include <cooperative_groups.h>
#include <stdint.h>

#include "common.cuh"

namespace spin {

constexpr int kHeisParts = 64;  // partials per lattice

// CTAs per partial of a lattice of N sites.
inline int heis_measure_cluster(int64_t N) {
  return N >= (1 << 21) ? 8 : N >= (1 << 20) ? 4 : N >= (1 << 19) ? 2 : 1;
}

// The exact sum a + b = s + e (Knuth; no assumption on magnitudes).
__device__ __forceinline__ float two_sum(float a, float b, float &e) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}

// Three-term running sum: rounding errors of s go to c, those of c to d.
struct Sum3 {
  float s, c, d;
  __device__ __forceinline__ Sum3() : s(0.0f), c(0.0f), d(0.0f) {}
  __device__ __forceinline__ void low(float v) {
    float f;
    c = two_sum(c, v, f);
    d = __fadd_rn(d, f);
  }
  __device__ __forceinline__ void add(float v) {
    float e;
    s = two_sum(s, v, e);
    low(e);
  }
  __device__ __forceinline__ void add_product(float a, float b) {
    const float p = __fmul_rn(a, b);
    add(p);
    low(__fmaf_rn(a, b, -p));
  }
  __device__ __forceinline__ void add(const Sum3 &o) {
    add(o.s);
    low(o.c);
    d = __fadd_rn(d, o.d);
  }
  __device__ __forceinline__ double value() const { return (double)s + ((double)c + (double)d); }
};

// The site and its forward neighbours (bz = 0 in 2D).
struct HeisBonds {
  float4 a, bx, by, bz;
};

__device__ __forceinline__ HeisBonds heis_bonds(const float4 *__restrict__ sl, uint32_t i, uint32_t L,
                                                const FastDiv &fL, int dim) {
  const uint32_t row = fdiv(i, fL), x = i - row * L;
  const uint32_t z = dim == 3 ? fdiv(row, fL) : 0u, y = row - z * L;
  HeisBonds h;
  h.a = sl[i];
  h.bx = sl[x == L - 1 ? i - x : i + 1];
  h.by = sl[y == L - 1 ? i - (L - 1) * L : i + L];
  h.bz = dim == 3 ? sl[z == L - 1 ? i - (L - 1) * L * L : i + L * L] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  return h;
}

// One CTA's share of the partials [E, Mx, My, Mz] (out4[4 p .. 4 p + 3] for
// partial p) of lattice `sl` (N = L^dim < 2^31 sites): CTA b of nb visits
// sites b * blockDim.x + tid, then strides by nb * blockDim.x; the kC CTAs of
// a cluster share partial b / kC.  blockDim.x is a multiple of 32, <= 1024.
template <int kC>
__device__ __forceinline__ void heis_block_partials(const float4 *__restrict__ sl, uint32_t L, const FastDiv &fL,
                                                    int dim, uint32_t N, uint32_t b, uint32_t nb,
                                                    double *__restrict__ out4) {
  if (kC == 1 && b * (uint64_t)blockDim.x >= N) {  // no site
    if (threadIdx.x < 4) out4[4 * b + threadIdx.x] = 0.0;
    return;
  }
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  // rank 0's shared memory may be written once that CTA is known to run: every
  // CTA says so here and waits for it before the store, behind its sites
  if (kC > 1) cl.barrier_arrive();
  Sum3 ex, ey, ez, sx, sy, sz;
  float norm2 = 0.0f, count = 0.0f;
  const uint64_t first = b * (uint64_t)blockDim.x + threadIdx.x, stride = (uint64_t)nb * blockDim.x;
#pragma unroll 2
  for (uint64_t i = first; i < N; i += stride) {
    const HeisBonds h = heis_bonds(sl, (uint32_t)i, L, fL, dim);
    ex.add_product(h.a.x, h.bx.x);
    ey.add_product(h.a.y, h.bx.y);
    ez.add_product(h.a.z, h.bx.z);
    ex.add_product(h.a.x, h.by.x);
    ey.add_product(h.a.y, h.by.y);
    ez.add_product(h.a.z, h.by.z);
    if (dim == 3) {
      ex.add_product(h.a.x, h.bz.x);
      ey.add_product(h.a.y, h.bz.y);
      ez.add_product(h.a.z, h.bz.z);
    }
    sx.add(h.a.x);
    sy.add(h.a.y);
    sz.add(h.a.z);
    norm2 += h.a.x * h.a.x + h.a.y * h.a.y + h.a.z * h.a.z;
    count += 1.0f;
  }
  // (the three sums of E become one before they become a double, threads convert
  // what they have summed only, and CTAs without a site left above: a conversion
  // is 5 FP64 operations, which lattices of a site per thread or less do not win
  // back.  Us per measurement with all six sums converted by every thread, with
  // FP64 sums per site, and here: 250 x 2D L = 128 429 / 332 / 336, 150 x L = 92
  // 198 / 170 / 115, 2000 x 3D L = 8 1529 / 1415 / 145)
  double e = 0.0, mx = 0.0, my = 0.0, mz = 0.0;
  if (count > 0.0f) {
    ex.add(ey);
    ex.add(ez);
    e = -ex.value();
    if (count > 1.0f) {
      mx = sx.value();
      my = sy.value();
      mz = sz.value();
    } else {  // one site: its components
      mx = (double)sx.s;
      my = (double)sy.s;
      mz = (double)sz.s;
    }
  }
  // unit spins: norm2 = count; the whole block decides, as one site's spin
  // enters the products of its neighbours' threads too (a spin that another
  // block reads is caught there: an overflow makes e non-finite)
  const bool odd = !(norm2 >= 0.25f * count && norm2 <= 4.0f * count) || !(fabs(e) < 1e30);
  if (__syncthreads_or(odd)) {
    e = mx = my = mz = 0.0;
    for (uint64_t i = first; i < N; i += stride) {
      const HeisBonds h = heis_bonds(sl, (uint32_t)i, L, fL, dim);
      const double ax = h.a.x, ay = h.a.y, az = h.a.z;
      if (dim == 3) {
        e -= ax * ((double)h.bx.x + (double)h.by.x + (double)h.bz.x) +
             ay * ((double)h.bx.y + (double)h.by.y + (double)h.bz.y) +
             az * ((double)h.bx.z + (double)h.by.z + (double)h.bz.z);
      } else {
        e -= ax * ((double)h.bx.x + (double)h.by.x) + ay * ((double)h.bx.y + (double)h.by.y) +
             az * ((double)h.bx.z + (double)h.by.z);
      }
      mx += ax;
      my += ay;
      mz += az;
    }
  }
  __shared__ double red[4][32];
  e = warp_sum(e);
  mx = warp_sum(mx);
  my = warp_sum(my);
  mz = warp_sum(mz);
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    red[0][wid] = e;
    red[1][wid] = mx;
    red[2][wid] = my;
    red[3][wid] = mz;
  }
  __syncthreads();
  if (kC == 1) {
    if (threadIdx.x < 4) {
      double acc = 0.0;
      for (int k = 0; k < (int)(blockDim.x >> 5); ++k) acc += red[threadIdx.x][k];
      out4[4 * b + threadIdx.x] = acc;
    }
    return;
  }
  // the CTAs of the cluster leave their sums in rank 0's shared memory
  __shared__ double all[kC][4];
  cl.barrier_wait();
  if (threadIdx.x < 4) {
    double acc = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) acc += red[threadIdx.x][k];
    cl.map_shared_rank(&all[0][0], 0)[4 * cl.block_rank() + threadIdx.x] = acc;
  }
  cl.sync();
  if (cl.block_rank() == 0 && threadIdx.x < 4) {
    double acc = 0.0;
    for (int k = 0; k < kC; ++k) acc += all[k][threadIdx.x];
    out4[4 * (b / kC) + threadIdx.x] = acc;
  }
}

// Component c = k % 4 of lattice k / 4 (k the thread): adds its kHeisParts
// partials (layout [lat][partial][4]) in order and stores E (Ef[lat]) or a
// component of M (Mf[3 lat ..]); NULL skips.
__device__ __forceinline__ void heis_finish_component(const double *__restrict__ part, int64_t k,
                                                      double *__restrict__ Ef, double *__restrict__ Mf) {
  const int64_t lat = k >> 2;
  const int c = (int)(k & 3);
  double acc = 0.0;
#pragma unroll 16
  for (int b = 0; b < kHeisParts; ++b) acc += part[(lat * kHeisParts + b) * 4 + c];
  if (c == 0) {
    if (Ef) Ef[lat] = acc;
  } else if (Mf) {
    Mf[3 * lat + c - 1] = acc;
  }
}

}  // namespace spin
