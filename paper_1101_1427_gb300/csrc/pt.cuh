// The decision of one replica exchange (Eq. parallel_tempering), shared by the
// exchange kernel and the resident sweeps.
#pragma once
#include "common.cuh"

namespace spin {

// Device tables of the exchange step (see spin_pt_swap): the decision table of
// pair t is tab[off[t]], len[t] entries; dbeta[t] = beta_{t+1} - beta_t.
struct PtTables {
  const double *dbeta;
  const uint32_t *tab;
  const int32_t *off, *len;
};

// What the exchange of slots t and t + 1 of set a, realisation r, at exchange
// step `step` needs besides the energies; the tables were complete before any
// launch that reads them was enqueued.
struct PtPair {
  double db;
  const uint32_t *tab;
  int len;
  uint32_t word;
};

__device__ __forceinline__ PtPair pt_pair(const PtTables &p, int a, int t, int r, uint32_t step, const RoundKeys &rk) {
  PtPair x;
  x.db = p.dbeta[t];
  x.tab = p.tab + p.off[t];
  x.len = p.len[t];
  const uint4 w = philox(make_uint4((uint32_t)r >> 2, step, lattice_id(a, 0, t), ctr_w(TAG_PT, 0, 0)), rk);
  x.word = word_of(w, (uint32_t)r & 3u);
  return x;
}

// Delta = dbeta_t (E1 - E0) for energies E0, E1 of slots t, t + 1; accept iff
// Delta >= 0 or the PT word is below the tabulated threshold of exp(Delta).
__device__ __forceinline__ bool pt_accept(const PtPair &x, long long E0, long long E1) {
  const long long dE = E1 - E0;
  if (x.db * (double)dE >= 0.0) return true;
  const long long m = (dE < 0 ? -dE : dE) / 4;
  return x.word < (m < x.len ? x.tab[m] : 0u);
}

}  // namespace spin
