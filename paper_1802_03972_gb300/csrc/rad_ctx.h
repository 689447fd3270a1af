// Host-side definition of a radiation context (opaque in the C ABI).
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "rad.h"
#include "rad_impl.h"

namespace radimpl {
// The most that calls of up to n particles need: floats of partials, partials_f and
// partials_l (low 0: no call may take the low band).
struct CallLimits {
  long long n = 0, part = 0, fine = 0, low = 0;
};
}  // namespace radimpl

struct rad_ctx {
  int n_omega = 0, n_dir = 0, n_bins = 0;
  rad_ff ff{};
  int prec = RAD_PREC_MIXED;
  cudaStream_t stream = nullptr;
  rad_tile tile{};
  // device buffers
  double* d_omega = nullptr;
  double* d_om_turns = nullptr;
  float* d_om_tab = nullptr;
  double* d_dirs = nullptr;
  float* d_dir_tab = nullptr;
  double* d_ref = nullptr;
  int* d_status = nullptr;
  unsigned long long* d_counter = nullptr;
  radimpl::JobStatic* d_js = nullptr;
  double* d_spec = nullptr;      // [3][n_bins] readout staging for host outputs
  float* d_state = nullptr;      // MIXED: [16][n_bins]
  // FP64: [12][n_bins]; in the same allocation, the partial sums of a call cut
  // into up to f64_chunks particle chunks, [f64_chunks][8][n_bins], and the
  // arrival counters of its blocks (self-resetting)
  double* d_state64 = nullptr;
  double* d_part64 = nullptr;
  unsigned* d_cnt64 = nullptr;
  int f64_chunks = 1;
  // in-situ coupling (rad_push_step): three step slots of r, beta, w and beta_dot
  double* d_push = nullptr;      // [3][7 n_push] doubles: r (3n), beta (3n), w (n) per slot
  double* d_push_bdot = nullptr; // [3 n_push]
  long long n_push = 0;          // particle count of the held steps (0: none)
  int push_held = 0;             // steps held (0, 1, 2)
  int push_slot[2] = {0, 1};     // slots of the older / newer held step
  double push_t[3] = {0, 0, 0}, push_dt[3] = {0, 0, 0};
  float* d_state_p = nullptr;    // literal mode: [8][n_bins]
  float* d_f2 = nullptr;         // literal mode: [n_omega] f(omega)^2
  double* d_stage = nullptr;     // staging for host particle arrays
  size_t stage_cap = 0;
  radimpl::JobStatic h_js{};     // host mirror of d_js
  // kernel timing (rad_profile_*): event triples around pre-pass / accumulate
  bool prof_on = false;
  std::vector<cudaEvent_t> prof_ev;  // 3 per timed call
  size_t prof_used = 0;
  unsigned long long* d_prof_clk = nullptr;  // [2] cycles, ns of the accumulate CTAs
  int n_low = 0;                 // low-band alternatives of the grid (host copies)
  double low_full = 0.0;         // cost of the full tiling, in full tiles
  radimpl::LowSet low[radimpl::kLowSets]{};
  long long generation = 0;      // bumped whenever d_js changes
  unsigned last_low = 0;         // low_ok of the last call: with none its plan was not written
  size_t tab_floats = 0;         // of d_om_tab: om_tab, then the low band's tables
  // Some call's low-band buffers did not fit the device: calls take the bin tiles, as
  // they do without the band, until rad_reset.
  bool low_nomem = false;
  bool js_stale = false;         // h_js names buffers that d_js does not (yet)
  radimpl::CallLimits limit;     // n > 0: calls have at most so many particles, and their buffers stay within this
  int fail_alloc = 0;            // test support: the so-many-th buffer allocation from now fails ...
  int fail_times = 0;            // ... and this many in all
  uint64_t grid_hash = 0;        // FNV-1a of the frequencies and unit directions
  int device = -1;               // the CUDA device current at rad_create
  rad_status last_err = RAD_OK;
  bool failed = false;
};

namespace radimpl {

// A named NVTX range for the enclosing scope (host side; shows the library's
// calls on a profiler timeline, a no-op when no tool is attached).
struct TraceRange {
  explicit TraceRange(const char* name) { nvtxRangePushA(name); }
  ~TraceRange() { nvtxRangePop(); }
  TraceRange(const TraceRange&) = delete;
  TraceRange& operator=(const TraceRange&) = delete;
};

rad_status fail(rad_ctx* c, rad_status s);
// RAD_OK when the context's device is the calling thread's current device;
// otherwise RAD_EINVAL (its memory, stream and kernels belong to that device).
rad_status check_device(rad_ctx* c);
rad_status cuda_check(rad_ctx* c, cudaError_t e);
int default_omega_tile(int variant, int n_omega);
bool valid_omega_tile(int variant, int wt);
// n_low: the context's low-band alternatives, used with the default tiling
void fill_tiles(JobStatic& js, int variant, int wt, int n_low);
int resident_ctas(int variant);
// fine_tail: the job's last tiles are fine-chunked (TailPlan), which allows longer items.
int auto_chunk_for(int variant, long long n, int n_tiles, bool fine_tail);
int auto_chunk(const rad_ctx* c, int variant, long long n, int n_tiles);
// Device bytes of a MIXED context with these buffer capacities (js): its tables and
// accumulators, and its calls' records, sort buffers and partial sums.
size_t context_bytes(const rad_ctx* c, const JobStatic& js);
// Capacity for n particles and for so many floats of the coarse tiles', the fine
// tiles' (TailPlan::fine_floats) and the low band's partial sums.
rad_status ensure_capacity(rad_ctx* c, long long n, long long part_floats, long long fine_floats = 0,
                           long long low_floats = 0);
// How a call of n particles is cut into work items.
struct CallPlan {
  int ck = 0, n_chunks = 0;
  TailPlan tail;
  unsigned low_ok = 0;  // the alternatives that pay for this call (bits)
  LowCall low[kLowSets];  // (of those)
  long long hi_items = 0, low_items = 0;
  // of partials, partials_f and partials_l, the most over the alternatives
  long long part_floats = 0, fine_floats = 0, low_floats = 0;
  // items of the bin tiles (run: chunks per item), the most over the alternatives
  long long items(const JobStatic& js, int run) const;
  void fill(JobCall& K, const JobStatic& js, int run) const;
};
CallPlan plan_call(const rad_ctx* c, const JobStatic& js, int variant, long long n);
// Sizes, default tile, low-band alternatives and tiles of a context of this grid (host only).
void plan_grid(rad_ctx* c, const double* omega, int n_omega, int n_dir, int prec, bool literal);
// With the default tile (band: with the low band, where the grid has alternatives).
CallLimits call_limits(const rad_ctx* c, long long n, bool band);
// Bytes of the context when its buffers have grown to the limits.
size_t context_bytes_at(const rad_ctx* c, const CallLimits& limits);
// A call's evaluated updates as a share of its particles x bins when it takes
// alternative `set` of the low band (-1: none): tiles and nodes against all tiles.
double evaluated_share(const rad_ctx* c, int set);
// Whether a call of n particles may take the low band (with the default tile).
bool low_possible(const rad_ctx* c, long long n);
// Makes room for a planned call.  The low band is taken only where its buffers fit:
// without memory for them the call is planned again without it.
rad_status reserve_call(rad_ctx* c, const JobStatic& js, int variant, long long n, CallPlan& plan);
rad_status enqueue_accumulate(rad_ctx* c, long long n, const double* r, const double* beta,
                              const double* bdot, const double* w, double t, double dt);
rad_status upload_static(rad_ctx* c);

}  // namespace radimpl
