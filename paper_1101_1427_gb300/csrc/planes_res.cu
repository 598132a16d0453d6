// Sweeps of small int8 ferromagnets: the lattice as bit planes (planes.cuh) in
// one CTA's shared memory, the acceptance masks drawn ahead by the whole GPU.
//
// A sweep of a small lattice is a serial chain of colour phases, and one SM
// cannot draw its random words as fast as it can run that chain: the kernel
// this replaces (int8 in shared memory, words drawn in each phase) took 1.33
// us per sweep of L = 64 with a measurement, 0.78 us without, 19 SMs of 20
// idle.  The masks (r < thr per site, sweep and threshold) depend on no spin,
// so a first kernel writes them for many sweeps to a tape in global memory,
// every SM working, and a second one, one CTA per lattice and one thread per
// word and colour, only reads its words from the tape (fetched several phases
// ahead) and does the bit-sliced update with one barrier per phase.  Energies and magnetisations are counted in place, and an
// exchange step is folded into the start of the next launch: each CTA decides
// its pair from the energies the last launch left and loads its partner's
// planes instead of its own where the exchange is accepted.  One L = 64, 1000
// sweeps with E and M after each 1335 -> 256 us; 20 x L = 64, 100 sweeps and 10
// exchanges 181 -> 55 us; 20 x 3D L = 16, 256 sweeps 234 -> 63 us.
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "planes.cuh"

namespace spin {
namespace {

constexpr int kTapeSweeps = 2;  // sweeps drawn together: their calls share the first rounds (PhiloxX1)

// Masks of n_sweeps sweeps from sweep0 on.  Thread: block b of a lattice and
// colour, kTapeSweeps sweeps; tape[((s * 2 + c) * n_lat + lat) * kT + e][b] is
// the mask of dE = 4 (e + 1), one uint4 per block.  Bound by the wide
// multiplies, as msc2d_phase_kernel.  Writes its half of the tape without
// waiting: the launch that read it last was complete before the launch before
// this one passed its own wait (planes_res_kernel releases its dependents
// only after that).  It waits at its end, so that whatever follows it also follows that
// launch.
template <int kT>
__global__ void __launch_bounds__(128) planes_tape_kernel(uint4 *__restrict__ tape, Planes m, Geom g, uint32_t n_lat,
                                                          FastDiv flat, FastDiv fblocks,
                                                          const uint32_t *__restrict__ thr, RoundKeys rk,
                                                          uint32_t sweep0, uint32_t n_sweeps) {
  griddep_release();
  const uint32_t id = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t lc = fdiv(id, fblocks), b = id - lc * m.blocks;  // (sweep group, colour, lattice)
  const uint32_t sc = fdiv(lc, flat), lat = lc - sc * n_lat;
  const uint32_t c = sc & 1u, s0 = (sc >> 1) * kTapeSweeps;
  if (s0 < n_sweeps) {
    const PlaneBlock k = plane_block<true>(m, b);
    const uint32_t slot = slot_of32(g, lat), lid = lattice_id32(g, lat), wctr = ctr_w(TAG_UPDATE, c, 0);
    uint32_t t[kT], A[kTapeSweeps][kT][4];
#pragma unroll
    for (int e = 0; e < kT; ++e) t[e] = __ldg(thr + 4 * slot + 1 + e);
#pragma unroll
    for (int u = 0; u < kTapeSweeps; ++u)
#pragma unroll
      for (int e = 0; e < kT; ++e)
#pragma unroll
        for (int q = 0; q < 4; ++q) A[u][e][q] = 0u;
#pragma unroll 2
    for (int i = (int)k.bits - 1; i >= 0; --i) {
      const PhiloxX1 pre = philox_x1_setup(k.j4 + (uint32_t)i, lid, wctr, rk);
#pragma unroll
      for (int u = 0; u < kTapeSweeps; ++u) {
        const uint4 r = philox_x1(pre, sweep0 + s0 + (uint32_t)u, rk);
#pragma unroll
        for (int e = 0; e < kT; ++e) {
          const MaskBits mb(t[e]);
          mb.push(A[u][e][0], r.x);
          mb.push(A[u][e][1], r.y);
          mb.push(A[u][e][2], r.z);
          mb.push(A[u][e][3], r.w);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kTapeSweeps; ++u)
      if (s0 + u < n_sweeps)
#pragma unroll
        for (int e = 0; e < kT; ++e) {
          const MaskBits mb(t[e]);
          tape[(((size_t)(2 * (s0 + u) + c) * n_lat + lat) * kT + e) * m.blocks + b] =
              make_uint4(mb.mask(A[u][e][0]), mb.mask(A[u][e][1]), mb.mask(A[u][e][2]), mb.mask(A[u][e][3]));
        }
  }
  griddep_wait();
}

struct ResSeries {
  long long *E, *M;  // rows of n_lat for the sweeps first, first + every, ... (1-based in the launch)
  int every, first;
  long long *E_last;        // energies after the last sweep (NULL: not wanted)
  const long long *E_prev;  // energies for an exchange before the first sweep (NULL: none)
  uint32_t step;            // its exchange step
  long long *accepted;
  int *labels;
};

constexpr int kResThreads = 512;  // most words of a colour
constexpr int kResRows = 32;  // measurement rows kept in shared memory before they are written

// n_sweeps sweeps of every lattice with the masks on the tape, from bytes_in
// (the first launch of a call) or the planes `src` (own or, after an accepted
// exchange, the partner's) to bytes_out (the last launch) or the planes `dst`.
// Thread i holds word i (4 block + plane) of both colours in registers and
// publishes them in shared memory for its neighbours.  Grid: lattices; at
// least `words` threads.  Bound by latency: about 61 instructions per phase, a
// measurement included, in a chain of shared-memory loads, logic and a barrier
// (0.10 us per phase of L = 64, 0.13 us of L = 128 and of L = 64 measured after
// every sweep).
// kLong: long launches run a copy of the loop that does not look for the end (1000
// sweeps of one L = 64 measured after each 265 -> 254 us; not in 3D, where the two
// copies need over 96 registers).
template <int kDim, bool kPadded, bool kLong>
__global__ void __launch_bounds__(kResThreads, 1) planes_res_kernel(const uint64_t *bytes_in, uint64_t *bytes_out,
                                                                 const uint32_t *__restrict__ src,
                                                                 uint32_t *__restrict__ dst,
                                                                 const uint32_t *__restrict__ tape, Planes m, Geom g,
                                                                 int n_sweeps, ResSeries ser, PtTables pt,
                                                                 RoundKeys rk) {
  constexpr int kT = kDim;
  constexpr int kAhead = 8;                         // phases fetched ahead (even)
  __shared__ __align__(16) uint32_t sw[2 * kResThreads];  // [2 colours][words]
  __shared__ int cnt[kResRows + 1][2];
  __shared__ bool exchanged;
  const uint32_t lat = blockIdx.x, n_lat = gridDim.x, words = 4 * m.blocks, wd = min(threadIdx.x, words - 1);
  const bool mine = threadIdx.x < words;
  const long long N = (long long)g.N;
  // the lattice's pair in the exchange due before the first sweep: (t0, t0 + 1)
  uint32_t partner = lat, l0 = lat, l1 = lat;
  int a = 0, t0 = 0;
  PtPair pair = {};
  if (ser.E_prev) {
    const uint32_t qt = fdiv(lat, g.freal), r = lat - qt * (uint32_t)g.n_real;
    a = (int)fdiv(qt, g.ftemps);
    const int t = (int)qt - a * g.n_temps, parity = (int)(ser.step & 1u);
    const bool lower = ((t - parity) & 1) == 0;
    t0 = lower ? t : t - 1;
    if (t0 >= parity && t0 + 1 < g.n_temps) {
      l0 = lower ? lat : lat - (uint32_t)g.n_real;
      l1 = l0 + (uint32_t)g.n_real;
      partner = lower ? l1 : l0;
      if (threadIdx.x == 0) pair = pt_pair(pt, a, t0, (int)r, ser.step, rk);
    }
  }
  for (int i = threadIdx.x; i < 2 * (kResRows + 1); i += blockDim.x) (&cnt[0][0])[i] = 0;
  // the word's neighbours, shifts and masks (plane_nbrs for one plane)
  const uint32_t nb = m.nb, row = low_bits(nb), b = wd >> 2, q = wd & 3u;
  const PlaneBlock k = plane_block<true>(m, b);
  const uint32_t gu = k.g == 0 ? m.nby - 1 : k.g - 1, gd = k.g == m.nby - 1 ? 0u : k.g + 1;
  const uint32_t iu = wd + 4 * (gu - k.g), id = wd + 4 * (gd - k.g);
  const uint32_t il = 4 * b + ((q + 3) & 3u), ir = 4 * b + ((q + 1) & 3u);
  const uint32_t jf = kDim == 3 ? 4 * (k.z == 0 ? b + m.blocks - m.zstep : b - m.zstep) + q : 0u;
  const uint32_t jb = kDim == 3 ? 4 * (k.z == (uint32_t)m.L - 1 ? b + m.zstep - m.blocks : b + m.zstep) + q : 0u;
  const uint32_t last = k.bits - nb, last_u = (min(m.R, (uint32_t)m.L - gu * m.R) - 1) * nb;
  uint32_t startm = 0, odd = 0;  // first bit of every row; rows whose colour-0 sites have p = 1
  for (uint32_t r = 0; r < m.R; ++r) {
    startm |= 1u << (r * nb);
    if (((r + k.par) & 1u) != 0) odd |= row << (r * nb);
  }
  // (only the first and the last plane shift, between the ends of a row)
  const uint32_t endm = q == 3 ? startm << (nb - 1) : 0u;
  startm = q == 0 ? startm : 0u;
  const uint32_t shl = q == 0 ? 1u : 0u, shr = q == 3 ? 1u : 0u, valid = mine ? low_bits(k.bits) : 0u;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const size_t chunk0 = (size_t)lat * (size_t)(N / 8);  // the lattice's first 8-byte chunk
  griddep_wait();
  griddep_release();
  // the tape: phase p at ((p n_lat + lat) kT + e) words + word; kPadded: it is
  // longer than its sweeps by the phases fetched ahead
  const int phases = 2 * n_sweeps;
  const size_t phase_step = (size_t)n_lat * kT * words;
  const uint32_t *tp = tape + (size_t)lat * kT * words + wd;
  uint32_t mk[kAhead][kT];
  auto fetch = [&](uint32_t (&v)[kT], bool there) {  // the next phase's masks, if there is one
    if (!kPadded && !there) return;
#pragma unroll
    for (int e = 0; e < kT; ++e) v[e] = tp[e * words];
    tp += phase_step;
  };
  uint32_t s[2] = {0u, 0u};
  if (bytes_in) {  // one warp per block, as planes_bytes_kernel
#pragma unroll 4
    for (uint32_t bb = warp; bb < m.blocks; bb += warps) {
      const PlaneBlock kk = plane_block<true>(m, bb);
      const bool in = (uint32_t)lane < kk.bits;
      const uint2 x = chunk_words(in ? bytes_in[chunk0 + kk.j4 + lane] : 0ull, (kk.par + (uint32_t)lane / nb) & 1u);
      uint32_t word[8];
#pragma unroll
      for (int o = 0; o < 8; ++o)  // bit 1 of a +-1 byte is set for -1
        word[o] = __ballot_sync(0xffffffffu, in && ((o < 4 ? x.x : x.y) >> (8 * (o & 3) + 1) & 1u));
      if (lane == 0) {
        reinterpret_cast<uint4 *>(sw)[bb] = make_uint4(word[0], word[2], word[4], word[6]);
        reinterpret_cast<uint4 *>(sw)[m.blocks + bb] = make_uint4(word[1], word[3], word[5], word[7]);
      }
    }
#pragma unroll
    for (int d = 0; d < kAhead; ++d) fetch(mk[d], d < phases);
    __syncthreads();
    if (mine) s[0] = sw[wd], s[1] = sw[words + wd];
  } else {
    // own planes and the partner's, both fetched before the decision is known
    const uint32_t *own = src + (size_t)lat * 2 * words + wd, *other = src + (size_t)partner * 2 * words + wd;
    const uint32_t w0 = own[0], w1 = own[words], x0 = other[0], x1 = other[words];
#pragma unroll
    for (int d = 0; d < kAhead; ++d) fetch(mk[d], d < phases);
    if (threadIdx.x == 0) {
      bool acc = false;
      if (partner != lat) {
        acc = pt_accept(pair, ser.E_prev[l0], ser.E_prev[l1]);
        if (acc && lat == l0) {
          if (ser.accepted) atomicAdd((unsigned long long *)&ser.accepted[a * g.n_temps + t0], 1ull);
          if (ser.labels) {
            const int x = ser.labels[l0];
            ser.labels[l0] = ser.labels[l1];
            ser.labels[l1] = x;
          }
        }
      }
      exchanged = acc;
    }
    __syncthreads();
    if (mine) {
      sw[wd] = s[0] = exchanged ? x0 : w0;
      sw[words + wd] = s[1] = exchanged ? x1 : w1;
    }
    __syncthreads();
  }
  int next = ser.first - 1, rows = 0, written = 0;  // next: sweep (0-based) of the next measurement
  auto write_rows = [&]() {  // rows counted since the last write (the caller has a barrier before)
    if ((int)threadIdx.x < rows) {
      const int i = threadIdx.x;
      if (ser.E) ser.E[(size_t)(written + i) * n_lat + lat] = 2ll * cnt[i][0] - kDim * N;
      if (ser.M) ser.M[(size_t)(written + i) * n_lat + lat] = N - 2ll * cnt[i][1];
      cnt[i][0] = cnt[i][1] = 0;
    }
    written += rows;
    rows = 0;
    __syncthreads();
  };
  // kAhead phases from `base` on; kLast: the last ones, with no more to fetch
  auto run = [&](int base, auto last_phases) {
    constexpr bool kLast = decltype(last_phases)::value;
#pragma unroll
    for (int d = 0; d < kAhead; ++d) {
      const int p = base + d;
      if (kLast && p >= phases) break;  // (after a whole sweep: phases is even)
      const int c = d & 1;
      const uint32_t *O = sw + (c ^ 1) * words;
      const uint32_t o = s[c ^ 1], km = O[il], kp = O[ir];
      PlaneNbrs<kDim> n;
      n.u[0] = (o << nb) | (O[iu] >> last_u);
      n.d[0] = (o >> nb) | ((O[id] & row) << last);
      n.f[0] = kDim == 3 ? O[jf] : 0u;
      n.b[0] = kDim == 3 ? O[jb] : 0u;
      n.o[0] = o;
      const uint32_t left = (km << shl & ~startm) | (km >> (nb - 1) & startm);
      const uint32_t right = (kp >> shr & ~endm) | (kp << (nb - 1) & endm);
      const uint32_t od = c ? ~odd : odd;
      n.s[0] = (left & ~od) | (right & od);
      const uint32_t v = s[c] ^ (plane_flips<kDim>(s[c], n, 0, mk[d][0], mk[d][1], mk[d][kT - 1]) & valid);
      s[c] = v;
      if (mine) sw[c * words + wd] = v;
      fetch(mk[d], !kLast || p + kAhead < phases);
      if (c == 1) {
        const int sweep = p >> 1;
        const bool row_now = (ser.E || ser.M) && sweep == next, last_now = ser.E_last && sweep == n_sweeps - 1;
        if (row_now || last_now) {
          int anti = __popc((v ^ n.u[0]) & valid) + __popc((v ^ n.d[0]) & valid) + __popc((v ^ o) & valid) +
                     __popc((v ^ n.s[0]) & valid);
          if (kDim == 3) anti += __popc((v ^ n.f[0]) & valid) + __popc((v ^ n.b[0]) & valid);
          // a warp's counts, at most 32 x 32 x 6, side by side
          const uint32_t both =
              __reduce_add_sync(0xffffffffu, (uint32_t)anti + ((uint32_t)(__popc(v) + __popc(o)) << 16));
          if (lane == 0) {
            if (row_now) {
              atomicAdd(&cnt[rows][0], (int)(both & 0xffffu));
              atomicAdd(&cnt[rows][1], (int)(both >> 16));
            }
            if (last_now) atomicAdd(&cnt[kResRows][0], (int)(both & 0xffffu));
          }
          if (row_now) {
            ++rows;
            next += ser.every;
          }
        }
        __syncthreads();
        if (rows == kResRows) write_rows();
      } else {
        __syncthreads();
      }
    }
  };
  int base = 0;
  if (kLong)
    for (; base + 2 * kAhead <= phases; base += kAhead) run(base, std::false_type());
  for (; base < phases; base += kAhead) run(base, std::true_type());
  if (rows) write_rows();
  if (ser.E_last && threadIdx.x == 0) ser.E_last[lat] = 2ll * cnt[kResRows][0] - kDim * N;
  if (bytes_out) {
    for (uint32_t bb = warp; bb < m.blocks; bb += warps) {
      const PlaneBlock kk = plane_block<true>(m, bb);
      if ((uint32_t)lane >= kk.bits) continue;
      const uint4 w0 = reinterpret_cast<uint4 *>(sw)[bb], w1 = reinterpret_cast<uint4 *>(sw)[m.blocks + bb];
      bytes_out[chunk0 + kk.j4 + lane] = chunk_of(w0, w1, lane, (kk.par + (uint32_t)lane / nb) & 1u);
    }
  } else {
    uint32_t *dl = dst + (size_t)lat * 2 * words;
    for (uint32_t i = threadIdx.x; i < 2 * words; i += blockDim.x) dl[i] = sw[i];
  }
}

constexpr size_t kTapeMax = 18u << 20;  // bytes of the sweeps of one half of the tape, at most
// Sweeps by which a half is longer than what it holds, so that no phase looks
// whether there is another to fetch (3 to 8 % of the time per phase in 3D), where a
// half holds kTapePadFrom sweeps or more: 9 MB for both halves at most.
constexpr int kTapePad = 4;
constexpr int kTapePadFrom = 16;
constexpr int kResSpread = 200 * 1024;
constexpr int kTapeSpread = 20 * 1024;

// Dynamic shared memory asked for (not used) to place CTAs: the sweeps' and the
// masks'.  The few CTAs of the sweeps spread over the SMs: a launch that starts
// while the masks' CTAs drain would otherwise find its places on a few SMs (20
// x L = 64, 256 sweeps: 145 us against 55 for one lattice), and beside one of
// them there is room for one CTA of the next masks only, which may run at the
// same time.  From more than half as many lattices as SMs on, a CTA that asks
// for most of an SM waits until it is empty of masks (us per call of 8 / 16 / 32
// / 100 sweeps, asking for 200 KB / lattices per SM, against here: 152 x 2D L =
// 64 9.3 / 33 / 35 / 61 and 9.2 / 12 / 18 / 56, 304 x 2D L = 16 18 / 21 / 30 /
// 44 and 7 / 7 / 9 / 22, 152 x 2D L = 128 33 / 36 / 80 / 181 and 18 / 33 / 59 /
// 174): there no such masks and half of the share do better, or the whole where a
// CTA has 96 threads and more, four of which on an SM are in one another's way (159 x
// L = 80, 60 sweeps 52 against 56), and nothing at all for the CTAs of 256 threads
// and more, of which few fit anyway (but longer launches of 3D L = 24 up to a
// lattice per SM keep the share: 120, 100 sweeps 165 against 182, 8 sweeps 27
// against 20).
// Launches that do not follow their masks at once (`at` > 0: between exchanges)
// ask for the large share again.
struct Places {
  size_t sweeps, masks;
};
Places places(const spin_lattice *h, const Planes &m, int64_t at, int64_t n_sweeps) {
  const int64_t per_sm = (h->n_lat + h->sms - 1) / h->sms;
  const size_t share = per_sm <= 8 ? (size_t)(kResSpread / per_sm) : 0;
  const bool crowded = 2 * h->n_lat > h->sms, small = m.blocks < 24, large = m.blocks >= 64;
  Places p = {share, kTapeSpread};
  if (!crowded || share == 0) return p;
  if (!large) p.masks = 0;
  if (at == 0 && small) p.sweeps = share / 2;
  if (at == 0 && large) p.sweeps = per_sm == 1 && m.dim == 3 && n_sweeps >= 24 ? share : 0;
  return p;
}

constexpr int64_t kResMinTape = 512;
constexpr int64_t kResMaxSweeps = 4096;  // per launch, so that none runs for long

}  // namespace

namespace {
size_t tape_sweep_bytes(const spin_lattice *h, const Planes &m) {
  return (size_t)2 * h->n_lat * m.dim * m.blocks * sizeof(uint4);
}
auto res_kernel(const spin_lattice *h, int64_t n_sweeps) {
  const bool pad = h->res_tape_pad != 0;
  if (h->g.dim == 3) return pad ? planes_res_kernel<3, true, false> : planes_res_kernel<3, false, false>;
  if (n_sweeps >= 32) return pad ? planes_res_kernel<2, true, true> : planes_res_kernel<2, false, true>;
  return pad ? planes_res_kernel<2, true, false> : planes_res_kernel<2, false, false>;
}
// The working buffer: two buffers of planes, then the two halves of the tape.
size_t planes_pair_bytes(const spin_lattice *h) { return 2 * (size_t)h->n_lat * planes_lattice_bytes(h); }
size_t tape_half_bytes(const spin_lattice *h) {
  return (h->pingpong_bytes - planes_pair_bytes(h)) / 2 / sizeof(uint4) * sizeof(uint4);
}
uint4 *tape_of(const spin_lattice *h) {
  return (uint4 *)((uint8_t *)h->d_pingpong + planes_pair_bytes(h) + (size_t)h->tape_half * tape_half_bytes(h));
}
}  // namespace

void planes_init(spin_lattice *h) {
  if (!planes_supported(h)) return;
  const Planes m = make_planes(h->g.dim, h->g.L);
  if (m.nb > 16 || 4 * m.blocks > kResThreads) return;
  h->res_words = (int)(4 * m.blocks);
  h->res_tape_sweeps = (int64_t)(kTapeMax / tape_sweep_bytes(h, m));
  h->res_tape_pad = h->res_tape_sweeps >= kTapePadFrom ? kTapePad : 0;
}

// The working buffer for calls of n sweeps; false: no memory, or a capture
// that must not allocate.
bool planes_res_reserve(spin_lattice *h, int64_t n_sweeps) {
  const Planes m = make_planes(h->g.dim, h->g.L);
  const size_t per = tape_sweep_bytes(h, m);
  // (calls of growing length make few buffers: a power of two, at least 512)
  int64_t sweeps = kResMinTape;
  while (sweeps < n_sweeps && sweeps < kResMaxSweeps) sweeps *= 2;
  sweeps = std::min(sweeps, h->res_tape_sweeps);
  if (sweeps < kTapeSweeps) return false;
  const size_t need = planes_pair_bytes(h) + 2 * (size_t)(sweeps + h->res_tape_pad) * per;
  if (working_buffer(h, need, false) != cudaSuccess) return false;
  if (!h->res_smem_set) {
    h->res_smem_set = true;
    for (int64_t n : {1, 32})  // short and long launches
      h->res_smem_set =
          h->res_smem_set && cudaFuncSetAttribute(res_kernel(h, n), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                  kResSpread) == cudaSuccess;
  }
  return h->res_smem_set;
}

// The tape for the next sweeps; returns how many it covers (at most n).
int64_t planes_res_draw(spin_lattice *h, int64_t sweep0, int64_t n, cudaError_t *err) {
  const Planes m = make_planes(h->g.dim, h->g.L);
  int64_t cover = (int64_t)(tape_half_bytes(h) / tape_sweep_bytes(h, m)) - h->res_tape_pad;
  cover = std::min(cover, kResMaxSweeps);
  // (whole groups of sweeps that are drawn together, but for the call's last ones)
  cover = n <= cover ? n : cover / kTapeSweeps * kTapeSweeps;
  h->tape_half ^= 1;
  const int64_t groups = (cover + kTapeSweeps - 1) / kTapeSweeps;
  const int64_t threads = groups * 2 * h->n_lat * m.blocks;  // < 2^31: 16 bytes of tape each
  *err = launch_dependent(m.dim == 3 ? planes_tape_kernel<3> : planes_tape_kernel<2>, dim3(grid_for(threads, 128)),
                          dim3(128), places(h, m, 0, cover).masks, h->stream, tape_of(h), m, h->g, (uint32_t)h->n_lat,
                          make_fastdiv((uint32_t)h->n_lat), make_fastdiv(m.blocks), (const uint32_t *)h->d_thr,
                          make_round_keys(h->d.seed), (uint32_t)sweep0, (uint32_t)cover);
  return cover;
}

// n sweeps from tape sweep `at` on, planes buffer `from` (0 or 1) to the other.
cudaError_t planes_res_sweeps(spin_lattice *h, int64_t at, int64_t n, int from, const PlanesResCall &call) {
  const Planes m = make_planes(h->g.dim, h->g.L);
  const size_t buf = (size_t)h->n_lat * (planes_lattice_bytes(h) / 4);
  uint32_t *p = (uint32_t *)h->d_pingpong;
  const uint4 *tape = tape_of(h) + (size_t)at * (tape_sweep_bytes(h, m) / sizeof(uint4));
  ResSeries s;
  s.E = (long long *)call.E;
  s.M = (long long *)call.M;
  s.every = call.every;
  s.first = call.first;
  s.E_last = (long long *)call.E_last;
  s.E_prev = (const long long *)call.E_prev;
  s.step = call.step;
  s.accepted = (long long *)call.accepted;
  s.labels = call.labels;
  return launch_dependent(res_kernel(h, n), dim3((unsigned)h->n_lat),
                          dim3((4 * m.blocks + 31) / 32 * 32), places(h, m, at, n).sweeps, h->stream,
                          (const uint64_t *)(call.bytes_in ? h->spins : nullptr),
                          (uint64_t *)(call.bytes_out ? h->spins : nullptr), (const uint32_t *)(p + (size_t)from * buf),
                          p + (size_t)(from ^ 1) * buf, (const uint32_t *)tape, m, h->g, (int)n, s, pt_tables(h),
                          make_round_keys(h->d.seed));
}

}  // namespace spin
