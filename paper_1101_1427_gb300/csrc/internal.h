// Host-side handle and the launchers each translation unit provides.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/spin.h"
#include "common.cuh"
#include "per_device.h"
#include "pt.cuh"

// NVTX range over one ABI call, so that a profiler's timeline shows which
// entry point enqueued which kernels (no cost when no tool is attached).
struct NvtxRange {
  explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange &) = delete;
  NvtxRange &operator=(const NvtxRange &) = delete;
};

namespace spin {
// Decomposition of the resident 3D Heisenberg sweeps (heis_res.cu).
struct HeisResPlan {
  int Py, Pz;   // pencils per lattice along y and z
  int grid;     // CTAs: n_lat Py Pz, one per SM at most
  size_t smem;  // dynamic shared memory per CTA
};
}  // namespace spin

struct spin_lattice {
  spin_desc d;
  spin::Geom g;
  cudaStream_t stream;
  void *spins;           // caller-owned
  void *couplings;       // caller-owned (may be NULL)
  int64_t n_lat;         // n_sets * n_temps * n_real lattices
  int sms;               // of the device
  int64_t sweeps_done;
  int64_t pt_steps_done;
  int variant;           // int8 sweep: 0 phases, 1 fused, 3 resident, 4 coded
  int default_variant;   // as spin_init chose it
  int auto_form;         // no variant was asked for: longer int8 calls may take the bit planes
  int msc_width;         // EA coded: realisations sharing one uniform (32 or 64)
  int order;             // spin_update_order
  int order_tile;        // double checkerboard: tile edge T
  int order_hits;        // double checkerboard: hits k per compound move

  // handle-owned device workspaces
  uint32_t *d_thr;       // [n_temps][4] Metropolis thresholds, index dE/4
  std::vector<double> betas_cached;
  int thr_valid;
  uint32_t *d_pt_thr;    // concatenated replica-exchange tables
  int32_t *d_pt_off;     // [n_temps]: offset of pair t's table
  int32_t *d_pt_len;     // [n_temps]: its length (entries beyond are 0)
  double *d_pt_dbeta;    // [n_temps]: beta_{t+1} - beta_t
  std::vector<double> pt_betas_cached;
  int64_t *d_energy;     // [n_lat] scratch energies for the exchange step
  int64_t *d_scratch64;  // small reduction scratch
  int *d_err;            // device error word
  void *d_pingpong;      // working buffer of the sweeps that need one (lazy)
  size_t pingpong_bytes;
  bool pingpong_captured;   // a captured call has used it: it outlives its replacement
  void *d_retired[8];       // replaced working buffers that captured calls used
  int n_retired;
  int res_words;            // words of a colour in that form, its threads (0: not for these lattices)
  int64_t res_tape_sweeps;  // sweeps of masks that are drawn together at most
  int res_tape_pad;         // sweeps by which their buffer is longer
  bool res_smem_set;        // the resident planes kernel may ask for its shared memory on this device
  int tape_half;         // half of the tape in it that was drawn last (planes_res.cu)
  // batched launches (options set with spin_set_batch_options)
  uint64_t batch_timeout_ns;  // bound on every team-barrier wait (0: 2 s)
  int batch_ctas_per_sm;      // 0: autotuned / default
  double batch_ising_scale;   // 0: autotuned / default; weight of Ising units in the CTA split
  double batch_ea_n0;         // 0: autotuned / default; else 1 + fixed cost per EA word-lattice, in sites
  int batch_fault_extra;      // arrivals a barrier waits for that never come (tests)
  // batched-launch workspace, allocated by the first uncaptured batch call
  int64_t *d_ctr;             // [sweeps_done, pt_steps_done] as the batch kernel reads them
  unsigned *d_bar;            // one team-barrier counter per work unit of this handle
  int *d_escr;                // EA: [group][n_sets][n_temps][32] energy scratch
  int64_t ctr_dev[2];         // what d_ctr holds once the enqueued work is done (-1: unknown)
  // resident 3D Heisenberg sweeps (heis_res.cu), allocated on first use
  unsigned *d_res_flags;      // one published-phase counter per CTA
  int res_flags_n;
  uint32_t res_base;          // phases the counters have advanced by in earlier launches
  spin::HeisResPlan res_plan[2];  // per variant (full accuracy, fast math)
  int res_plan_state[2];          // 0: not made yet, 1: usable, -1: the lattices do not fit
};

namespace spin {

// api.cu: the handle's working buffer, made or made longer where it holds fewer
// than `bytes`; with in_capture false never inside a stream capture.  A buffer
// that a captured call has used is kept until spin_destroy when a longer one
// takes its place, since the graph may be replayed at any time; a handle
// lengthens its buffer a few times at most (the masks of planes_res.cu four
// times, the planes and the fused pass once each).
cudaError_t working_buffer(spin_lattice *h, size_t bytes, bool in_capture);

// ising_i8.cu
cudaError_t launch_init_i8(spin_lattice *h);
cudaError_t launch_couplings_i8(spin_lattice *h);
cudaError_t launch_sweeps_i8(spin_lattice *h, const int8_t *J, int64_t n_sweeps);

// msc.cu
cudaError_t launch_init_msc(spin_lattice *h);
cudaError_t launch_couplings_msc(spin_lattice *h);
cudaError_t launch_sweeps_msc(spin_lattice *h, const uint32_t *J, int64_t n_sweeps);
cudaError_t launch_unpack_msc(spin_lattice *h, int8_t *out);
cudaError_t launch_pack_msc(spin_lattice *h, const int8_t *in);

// heis.cu
cudaError_t launch_init_heis(spin_lattice *h);
cudaError_t launch_sweeps_heis(spin_lattice *h, int64_t n_sweeps);

// heis_res.cu: 3D lattices resident in the SMs' shared memory for a whole
// call, one pencil of rows per CTA (L = 64 or 128, where they fit); the
// plan (HeisResPlan, above the handle) is made once per handle and variant
bool heis_resident_plan(const spin_lattice *h, HeisResPlan *plan);
// sweeps sweep0 .. sweep0 + n_sweeps - 1 (no renormalisation inside)
cudaError_t launch_sweeps_heis_resident(spin_lattice *h, const HeisResPlan &plan, int64_t sweep0, int64_t n_sweeps);

// measure.cu
cudaError_t launch_measure(spin_lattice *h, const void *J, int64_t *E, int64_t *M, int64_t *Q,
                           double *Ef, double *Mf);
// energies: the lattices' current energies if the caller has them (device,
// [n_lat]), else NULL to compute them
// labels: configuration labels moved with accepted exchanges (device, [n_lat], or NULL)
// planes: the lattices are bit planes in this buffer (planes.cu), not NULL
cudaError_t launch_pt_swap(spin_lattice *h, const void *J, int64_t *accepted, int32_t *labels,
                           const int64_t *energies, void *planes = nullptr);

// Launches kernel k as a programmatic dependent of the previous work in
// stream s (the kernel must call griddep_wait() before touching memory), in
// clusters of `cluster` CTAs along x.
template <typename... KArgs, typename... Args>
cudaError_t launch_clusters(void (*k)(KArgs...), dim3 grid, dim3 block, int cluster, size_t smem, cudaStream_t s,
                            Args... args) {
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k, static_cast<KArgs>(args)...);
}

// The same without clusters.
template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                             Args... args) {
  return launch_clusters(k, grid, block, 1, smem, s, args...);
}

inline PtTables pt_tables(const spin_lattice *h) {
  PtTables p;
  p.dbeta = h->d_pt_dbeta;
  p.tab = h->d_pt_thr;
  p.off = h->d_pt_off;
  p.len = h->d_pt_len;
  return p;
}

// planes.cu: longer calls of int8 ferromagnets on bit planes in the handle's
// working buffer
bool planes_supported(const spin_lattice *h);
size_t planes_lattice_bytes(const spin_lattice *h);
cudaError_t planes_measure(spin_lattice *h, int64_t *E, int64_t *M);
// the form that serves a call of n sweeps best: none (bytes), a launch per colour
// phase, or one CTA per lattice with the masks drawn ahead
enum class PlanesForm { none, phases, resident };
PlanesForm planes_form(const spin_lattice *h, int64_t n_sweeps, int32_t measure_every, int32_t pt_every);
// makes the buffers ready; what can run in the place of that form (none: no
// memory, or a capture that must not allocate)
PlanesForm planes_ready(spin_lattice *h, PlanesForm form, int64_t n_sweeps);
// the call (SPIN_* status), spin_run without Q; counters advanced
int planes_run(spin_lattice *h, PlanesForm form, const double *betas, int64_t n_sweeps, int32_t measure_every,
               int32_t pt_every, int64_t *E_series, int64_t *M_series, int64_t *accepted, int32_t *labels);

// planes_res.cu: the same for lattices small enough for one CTA each
struct PlanesResCall {
  int64_t *E, *M;         // series rows (NULL: none) after sweeps first, first + every, ... (1-based)
  int every, first;
  int64_t *E_last;        // energies after the last sweep (NULL: not wanted)
  const int64_t *E_prev;  // energies that decide exchange `step` before the first sweep (NULL: none)
  uint32_t step;
  int64_t *accepted;
  int32_t *labels;
  bool bytes_in, bytes_out;  // from or to the caller's bytes instead of the planes
};
void planes_init(spin_lattice *h);  // res_words, res_tape_sweeps
bool planes_res_reserve(spin_lattice *h, int64_t n_sweeps);
int64_t planes_res_draw(spin_lattice *h, int64_t sweep0, int64_t n, cudaError_t *err);
cudaError_t planes_res_sweeps(spin_lattice *h, int64_t at, int64_t n, int from, const PlanesResCall &call);

// msc2d.cu: lattices per thread of the coded phase kernels
int lattices_per_thread(int64_t n_lat, int64_t blocks);

// rng.cu
cudaError_t launch_rng_fill(uint64_t seed, uint32_t w, uint32_t lattice_id, uint32_t sweep,
                            uint64_t count, uint32_t *out, cudaStream_t s);
cudaError_t launch_rng_probe(uint64_t seed, uint32_t threads, uint32_t calls, uint32_t *out,
                             cudaStream_t s);

// probe.cu (returns a SPIN_* status)
int launch_pipe_probe(int op, int blocks_per_sm, uint32_t iters, long long *clocks, uint32_t *sink,
                      int *sms, cudaStream_t s);

// heis.cu (double checkerboard of the 2D Heisenberg model)
cudaError_t launch_heis_dcb_tiles(spin_lattice *h, int coarse, uint32_t sweep0);
cudaError_t launch_heis_renorm(spin_lattice *h);

// ising_i8.cu: whole-lattice-in-shared-memory sweeps of small 2D and 3D
// int8 ferromagnets (variant 3)
constexpr int kResidentMaxL = 128;  // 2D
constexpr int kResident3MaxL = 24;  // 3D (four chunks per thread of 512)
bool resident_supported(int dim, int L);
// n sweeps; with E or M (device, rows of n_lat) also measures after the
// sweeps first, first + every, ... (1-based in the call) into rows 0, 1, ...
cudaError_t launch_resident(spin_lattice *h, int64_t n_sweeps, int64_t *E, int64_t *M, int every, int first);

// dcb.cu
bool dcb_supported(const spin_lattice *h, int tile);
cudaError_t launch_sweeps_dcb(spin_lattice *h, int64_t n_sweeps);

// dcb_bits.cu: one coarse colour of the 2D int8 double checkerboard with the
// tiles as bits in registers, and the rule for when that is the faster form
bool dcb_bits_preferred(const spin_lattice *h);
cudaError_t launch_dcb_bits(spin_lattice *h, int coarse, uint32_t sweep0);

// batch.cu: load the batch kernel's device counters from the host counters
int sync_device_counters(spin_lattice *h, cudaStream_t st);

// Dynamic shared memory that a grid asks for so that at most ceil(ctas / sms) of
// its CTAs fit on an SM (to 16 of them): a kernel that starts while another one
// still runs fills the free places first, and several of its CTAs would share one
// SM while others idle.  An SM has 228 KB, 1 KB of it per CTA the system's.
inline size_t spread_smem(int64_t ctas, int sms) {
  const int64_t per_sm = (ctas + sms - 1) / sms;
  return per_sm <= 16 ? (size_t)(228 * 1024 / (per_sm + 1) - 1024 + 128) : 0;
}

inline unsigned grid_for(int64_t n, int block) {
  int64_t g = (n + block - 1) / block;
  return (unsigned)(g < 1 ? 1 : g);
}

}  // namespace spin
