// Kernels around the accumulate kernel (which lives in rad_accumulate.cu):
// the per-particle FP64 pre-pass, the readout of the spectra, the plain FP64
// kernel and the state merge (Pausch et al. 2018, Eq. 1, Eq. 12, Eq. 13).
//
// pre-pass (one thread per particle, FP64): moves positions to a per-call
// reference point r_ref (the first particle), so that
//    t - n.r/c = tau_ref(n) + dtau,   tau_ref = t - n.r_ref/c,   dtau = -n.(r - r_ref)/c,
// and writes a compact 80-byte FP32 record per particle (array of structures):
// (r - r_ref)/c and beta as float-float pairs, beta_dot, 1/gamma^2 = 1 - |beta|^2
// (FP64 before rounding), w dt and sqrt(w) dt.  FP64 is used here once per
// particle, never per (particle, direction, frequency).
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>

#include "rad_device.cuh"
#include "rad_impl.h"

namespace radimpl {

namespace {

using dev::kC;
using dev::kInvC;
// Physical prefactor q_e^2 / (16 pi^3 eps0 c) of Eq. 1, from the SI constants.
constexpr double kQe = 1.602176634e-19;
constexpr double kEps0 = 8.8541878128e-12;
constexpr double kPi = 3.14159265358979323846;

// ------------------------------------------------------------------ prepass
// Record layout (floats): 0-2 (r - r_ref)/c hi, 3-5 lo, 6-8 beta hi, 9-11 beta
// lo, 12-14 beta_dot, 15 1/gamma^2, 16 w dt, 17 sqrt(w) dt, 18 w - 1, 19 unused.
// Record of particle k with positions relative to rr; false for invalid data
// (the record then has zero weights and a harmless finite beta).
__device__ __forceinline__ bool make_record(const JobStatic& J, const JobCall& K, long long k,
                                            const double rr[3], float v[kRecFields]) {
  const long long n = K.n;
  const double x = K.r[k], y = K.r[n + k], z = K.r[2 * n + k];
  const double bx = K.beta[k], by = K.beta[n + k], bz = K.beta[2 * n + k];
  const double ax = K.bdot[k], ay = K.bdot[n + k], az = K.bdot[2 * n + k];
  const double w = K.w[k];
  const double g2 = 1.0 - (bx * bx + by * by + bz * bz);
  const bool valid = isfinite(x) && isfinite(y) && isfinite(z) && isfinite(bx) && isfinite(by) &&
                     isfinite(bz) && isfinite(ax) && isfinite(ay) && isfinite(az) && isfinite(w) &&
                     w > 0.0 && g2 > 0.0 && isfinite(K.dt) && isfinite(K.t);
  if (valid && !J.skip) {
    dev::split_ff((x - rr[0]) * kInvC, v[0], v[3]);
    dev::split_ff((y - rr[1]) * kInvC, v[1], v[4]);
    dev::split_ff((z - rr[2]) * kInvC, v[2], v[5]);
    dev::split_ff(bx, v[6], v[9]);
    dev::split_ff(by, v[7], v[10]);
    dev::split_ff(bz, v[8], v[11]);
    v[12] = __double2float_rn(ax);
    v[13] = __double2float_rn(ay);
    v[14] = __double2float_rn(az);
    v[15] = __double2float_rn(g2);
    v[16] = __double2float_rn(w * K.dt);
    // FP32 square root (the field is FP32; ~1e-7 relative): FP64's is slow on this GPU
    v[17] = sqrtf(__double2float_rn(w)) * __double2float_rn(K.dt);
    v[18] = __double2float_rn(w - 1.0);
  } else {
#pragma unroll
    for (int f = 0; f < 19; ++f) v[f] = 0.0f;
    v[8] = 0.5f;   // a harmless finite beta (zero weights)
    v[15] = 0.75f;
  }
  v[19] = 0.0f;
  return valid;
}

__device__ __forceinline__ void store_record(float* dst_rec, const float v[kRecFields]) {
  float4* dst = reinterpret_cast<float4*>(dst_rec);
#pragma unroll
  for (int q = 0; q < kRecFields / 4; ++q)
    dst[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}

// ---- low band (see LowSet)
// Integers in the order of the floats.
__device__ __forceinline__ int ordered(float x) {
  const int i = __float_as_int(x);
  return i < 0 ? i ^ 0x7fffffff : i;
}
__device__ __forceinline__ float from_ordered(int i) { return __int_as_float(i < 0 ? i ^ 0x7fffffff : i); }

// Coordinate of a record along a frame axis (seconds).  Explicit roundings: the
// extents, the histogram and the scatter must agree bit for bit.
__device__ __forceinline__ float frame_coord(const double ax[3], const float* v) {
  return __fmaf_rn((float)ax[0], v[0], __fmaf_rn((float)ax[1], v[1], __fmul_rn((float)ax[2], v[2])));
}

// A block's share of the call's extents along the frame (256 threads).
__device__ __forceinline__ void call_extents(const JobStatic& J, const float* v, bool live) {
  __shared__ int s_ext[6];
  if (threadIdx.x < 6) s_ext[threadIdx.x] = threadIdx.x & 1 ? INT_MIN : INT_MAX;
  __syncthreads();
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int o = live ? ordered(frame_coord(a == 0 ? J.fr1 : (a == 1 ? J.fr2 : J.axis), v)) : 0;
    const int lo = __reduce_min_sync(0xffffffffu, live ? o : INT_MAX);
    const int hi = __reduce_max_sync(0xffffffffu, live ? o : INT_MIN);
    if ((threadIdx.x & 31) == 0) {
      atomicMin(&s_ext[2 * a], lo);
      atomicMax(&s_ext[2 * a + 1], hi);
    }
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    if (threadIdx.x & 1) atomicMax(&J.ext[threadIdx.x], s_ext[threadIdx.x]);
    else atomicMin(&J.ext[threadIdx.x], s_ext[threadIdx.x]);
  }
}

// The call's plan: the first alternative whose cells are wide enough.  A cell's
// retarded times reach, from its centre, at most the grid's largest transverse
// share of the bunch's half-widths plus half the cell's width.
__device__ __forceinline__ LowPlan low_plan(const JobStatic& J, const JobCall& K) {
  LowPlan p = {-1, 0, 0.0f, 0.0f, 0.0f, 0.0f};
  if (!K.low_ok || (J.wide_flag != nullptr && *J.wide_flag != 0)) return p;
  float lo[3], hi[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (J.ext[2 * a] > J.ext[2 * a + 1]) return p;  // no valid particle
    lo[a] = from_ordered(J.ext[2 * a]);
    hi[a] = from_ordered(J.ext[2 * a + 1]);
  }
  const float side = __fmaf_rn(J.cone1, __fmul_rn(0.5f, __fsub_rn(hi[0], lo[0])),
                               __fmul_rn(J.cone2, __fmul_rn(0.5f, __fsub_rn(hi[1], lo[1]))));
  for (int s = 0; s < J.n_low; ++s) {
    if (!(K.low_ok >> s & 1u)) continue;
    const float h = __fmul_rn(2.0f, __fsub_rn(__fmul_rn(0.998f, J.low[s].H), __fmul_rn(1.001f, side)));
    if (!(h > 0.0f)) continue;
    const float cells = __fadd_rn(__fdiv_rn(__fsub_rn(hi[2], lo[2]), h), 1.0f);
    if (!(cells < (float)K.low[s].max_cells) || !(cells * kLowCellMin <= (float)K.n)) continue;
    p.set = s;
    p.cells = min((int)cells + 1, kLowMaxCells);
    p.s0 = lo[2];
    p.h = h;
    p.c1 = __fmul_rn(0.5f, __fadd_rn(lo[0], hi[0]));
    p.c2 = __fmul_rn(0.5f, __fadd_rn(lo[1], hi[1]));
    return p;
  }
  return p;
}

__device__ __forceinline__ int low_cell(const JobStatic& J, const LowPlan& p, const float* v) {
  const float q = floorf(__fdiv_rn(__fsub_rn(frame_coord(J.axis, v), p.s0), p.h));
  return max(0, min(p.cells - 1, (int)q));
}

__global__ void __launch_bounds__(256) prepass_kernel(const __grid_constant__ LaunchArgs a) {
  dev::pdl_trigger();
  dev::pdl_wait();  // (of the stream's last kernel: a call's chain may follow another's)
  const int j = dev::find_job_block(a, blockIdx.x);
  const JobStatic& J = a.js[j];
  const JobCall K = a.use_inline ? a.inline_call : a.jc[j];
  const long long n = K.n;
  // Reference point: the first particle (origin if it is not finite).
  double rr[3] = {K.r[0], K.r[n], K.r[2 * n]};
  if (!(isfinite(rr[0]) && isfinite(rr[1]) && isfinite(rr[2]))) rr[0] = rr[1] = rr[2] = 0.0;
  const long long k = (long long)(blockIdx.x - K.block_begin) * blockDim.x + threadIdx.x;
  if (k == 0) {
    J.ref[0] = rr[0];
    J.ref[1] = rr[1];
    J.ref[2] = rr[2];
    J.ref[3] = K.t;
  }
  float v[kRecFields];
  const bool valid = k < n && make_record(J, K, k, rr, v);
  if (K.low_ok) call_extents(J, v, valid && !J.skip);
  if (k >= n) return;
  if (!valid) atomicOr(J.status, ST_BAD_PARTICLE);
  // A particle that some direction of the grid may see beyond the fast phase
  // range makes the call wide (one atomic per warp that has one).  The bound
  // on |n . (r - r_ref)| over the grid: |axis . dr| + sin(largest angle from
  // the axis) |dr across the axis|.
  // A call of one sorted group or less gains nothing from sorting: never wide.
  // In FP32 on the record's (r - r_ref) / c (hi parts, seconds): the flag only
  // steers a call to the sorted path, and a call wrongly left unsorted still
  // runs correctly (its far tiles take the FP64 phase path).
  bool far = false;
  if (J.wide_flag && valid && !J.skip && n > kGroup && n < (1LL << 31)) {
    const float along = fmaf((float)J.axis[0], v[0], fmaf((float)J.axis[1], v[1], (float)J.axis[2] * v[2]));
    const float r2 = fmaf(v[0], v[0], fmaf(v[1], v[1], v[2] * v[2]));
    const float across = sqrtf(fmaxf(r2 - along * along, 0.0f));
    far = fabsf(along) + (float)J.cone_sin * across > 0.999f * J.tau_fast;
  }
  const unsigned far_lanes = __ballot_sync(__activemask(), far);
  if (far && (threadIdx.x & 31) == __ffs(far_lanes) - 1) {
    atomicOr(J.wide_flag, 1);
    if (a.any_wide && a.any_wide != J.wide_flag) atomicOr(a.any_wide, 1);
  }
  if (!dev::bounds_ok(k < J.n_cap, J.status)) return;
  store_record(J.rec + (size_t)k * kRecFields, v);
}

// ------------------------------------------------------------- wide calls
__device__ __forceinline__ bool call_is_wide(const JobStatic& J) {
  return J.wide_flag != nullptr && *J.wide_flag != 0;
}

// Bucket of particle k along the sort axis, centred on the call's reference.
// Explicit roundings: the histogram and the scatter kernels must agree bit for
// bit, whatever either compilation contracts into fused multiply-adds.
__device__ __forceinline__ int sort_bucket(const JobStatic& J, const JobCall& K, long long k) {
  const long long n = K.n;
  const double dx = __dsub_rn(K.r[k], J.ref[0]);
  const double dy = __dsub_rn(K.r[n + k], J.ref[1]);
  const double dz = __dsub_rn(K.r[2 * n + k], J.ref[2]);
  const double s = __fma_rn(J.axis[0], dx, __fma_rn(J.axis[1], dy, __dmul_rn(J.axis[2], dz)));
  const double q = __ddiv_rn(s, J.bucket_w);
  constexpr double kHalf = 0.5 * kSortBuckets;
  if (!(q > -kHalf)) return 0;  // also NaN
  if (!(q < kHalf)) return kSortBuckets - 1;
  return min(kSortBuckets - 1, (int)floor(q + kHalf));
}

constexpr int kFewBuckets = 512;

// Job of a sort-histogram block (jobs ordered by sort_block_begin).
__device__ __forceinline__ int find_job_sort_block(const LaunchArgs& a, int block) {
  if (a.n_jobs == 1) return 0;
  int lo = 0, hi = a.n_jobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.jc[mid].sort_block_begin <= block) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// The bucket of particle k: along the sort axis (wide calls), or its cell (low
// band; from the pre-pass's record).
struct Buckets {
  LowPlan plan;
  int n;  // buckets in use (0: the call is not sorted)
};
__device__ __forceinline__ int bucket_of(const JobStatic& J, const JobCall& K, const Buckets& b, long long k) {
  return b.plan.set >= 0 ? low_cell(J, b.plan, J.rec + (size_t)k * kRecFields) : sort_bucket(J, K, k);
}

// One block's share of the sort: bucket counts of kSortBlock particles.
__device__ __forceinline__ void hist_block(const JobStatic& J, const JobCall& K, const Buckets& B, long long blk,
                                           int* hist) {
  for (int b = threadIdx.x; b < B.n; b += blockDim.x) hist[b] = 0;
  __syncthreads();
  const long long k0 = blk * kSortBlock;
  for (int i = threadIdx.x; i < kSortBlock; i += blockDim.x)
    if (k0 + i < K.n) atomicAdd(&hist[bucket_of(J, K, B, k0 + i)], 1);
  __syncthreads();
  int* out = J.sort_counts + (size_t)blk * kSortBuckets;
  for (int b = threadIdx.x; b < B.n; b += blockDim.x) out[b] = hist[b];
}

// Per kSortBlock particles: bucket counts.
constexpr int kHistThreads = 1024;
__global__ void __launch_bounds__(kHistThreads) wide_hist_kernel(const __grid_constant__ LaunchArgs a) {
  dev::pdl_trigger();
  dev::pdl_wait();
  const int j = find_job_sort_block(a, blockIdx.x);
  const JobStatic& J = a.js[j];
  const JobCall& K = a.use_inline ? a.inline_call : a.jc[j];
  Buckets B;
  B.plan = low_plan(J, K);
  B.n = call_is_wide(J) ? kSortBuckets : B.plan.cells;
  if (B.n == 0) return;
  __shared__ int hist[kSortBuckets];
  hist_block(J, K, B, blockIdx.x - K.sort_block_begin, hist);
}

// By 1024 threads: per bucket, the prefix of the counts over the histogram blocks (in
// place), and the first sorted position of every bucket.
__device__ __forceinline__ void scan_job(const JobStatic& J, const JobCall& K, int n_b, int* tot, int* wsum) {
  const int nblk = (int)((K.n + kSortBlock - 1) / kSortBlock);
  // few buckets (cells): a warp per bucket, its lanes over the blocks
  const bool few = n_b <= kFewBuckets;
  if (few) {
    for (int b = threadIdx.x; b < kSortBuckets; b += 1024) tot[b] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int b = threadIdx.x >> 5; b < n_b; b += 32) {
      int run = 0;
      int* c = J.sort_counts + b;
      for (int blk0 = 0; blk0 < nblk; blk0 += 128) {
        int v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int blk = blk0 + 32 * u + lane;
          v[u] = blk < nblk ? c[(size_t)blk * kSortBuckets] : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int blk = blk0 + 32 * u + lane;
          int x = v[u];
          for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
          }
          if (blk < nblk) c[(size_t)blk * kSortBuckets] = run + x - v[u];
          run += __shfl_sync(0xffffffffu, x, 31);
        }
      }
      if (lane == 0) tot[b] = run;
    }
  }
  for (int b = few ? kSortBuckets : threadIdx.x; b < kSortBuckets; b += 1024) {
    int run = 0;
    int* c = J.sort_counts + b;
    int blk = b < n_b ? 0 : nblk;
    // eight independent loads in flight per step, then their prefix
    for (; blk + 8 <= nblk; blk += 8) {
      int v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = c[(size_t)(blk + u) * kSortBuckets];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        c[(size_t)(blk + u) * kSortBuckets] = run;
        run += v[u];
      }
    }
    for (; blk < nblk; ++blk) {
      const int v = c[(size_t)blk * kSortBuckets];
      c[(size_t)blk * kSortBuckets] = run;
      run += v;
    }
    tot[b] = run;
  }
  __syncthreads();
  static_assert(kSortBuckets == 4 * 1024, "four buckets per thread");
  const int t = threadIdx.x, lane = t & 31;
  const int v0 = tot[4 * t], v1 = tot[4 * t + 1], v2 = tot[4 * t + 2], v3 = tot[4 * t + 3];
  const int s = v0 + v1 + v2 + v3;
  int x = s;
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) wsum[t >> 5] = x;
  __syncthreads();
  if (t < 32) {
    int w = wsum[t];
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, off);
      if (t >= off) w += y;
    }
    wsum[t] = w;
  }
  __syncthreads();
  const int excl = x - s + ((t >> 5) ? wsum[(t >> 5) - 1] : 0);
  J.bucket_base[4 * t] = excl;
  J.bucket_base[4 * t + 1] = excl + v0;
  J.bucket_base[4 * t + 2] = excl + v0 + v1;
  J.bucket_base[4 * t + 3] = excl + v0 + v1 + v2;
}

// One block per job: scan_job.  Also settles
// the call's low-band plan for the kernels after it, and clears the extents
// for the next call.
__global__ void __launch_bounds__(1024) wide_scan_kernel(const __grid_constant__ LaunchArgs a) {
  dev::pdl_trigger();
  dev::pdl_wait();
  const JobStatic& J = a.js[blockIdx.x];
  const JobCall& K = a.use_inline ? a.inline_call : a.jc[blockIdx.x];
  __shared__ LowPlan s_plan;
  if (K.low_ok) {
    if (threadIdx.x == 0) {
      s_plan = low_plan(J, K);
      *J.plan = s_plan;
      if (s_plan.set >= 0) atomicOr(a.any_wide + 1, 1);
      for (int e = 0; e < 6; ++e) J.ext[e] = e & 1 ? INT_MIN : INT_MAX;
    }
  } else if (threadIdx.x == 0) {
    s_plan.cells = 0;
  }
  __syncthreads();
  const int n_b = call_is_wide(J) ? kSortBuckets : s_plan.cells;
  if (n_b == 0) return;
  __shared__ int tot[kSortBuckets];
  __shared__ int wsum[32];
  scan_job(J, K, n_b, tot, wsum);
}

// Per kSortBlock particles: the sorted position of every particle, stable
// (particles of one bucket keep their order), so the order is a function of
// the input alone.  The block computes the buckets into shared memory; then, with
// few buckets (cells), kRankWarps warps hand out the positions of an equal share
// of the particles each, in particle order, after counting the shares (the sort
// of 1e5 particles took 25 us here with one); with many, one warp does all.
constexpr int kScatterThreads = 512, kRankWarps = 8;
// cnt: the next position of every bucket; with few buckets, of every warp's share.
__device__ __forceinline__ void scatter_block(const JobStatic& J, const JobCall& K, const Buckets& B, long long blk,
                                              int* cnt, int* bkt) {
  static_assert(kRankWarps * kFewBuckets <= kSortBuckets, "the shares' counters");
  const bool few = B.n <= kFewBuckets;
  const int warps = few ? kRankWarps : 1, share = kSortBlock / warps;
  const long long k0 = blk * kSortBlock;
  const int* pre = J.sort_counts + (size_t)blk * kSortBuckets;
  for (int i = threadIdx.x; i < kSortBlock; i += blockDim.x)
    bkt[i] = k0 + i < K.n ? bucket_of(J, K, B, k0 + i) : -1;
  if (few) {
    for (int i = threadIdx.x; i < kRankWarps * kFewBuckets; i += blockDim.x) cnt[i] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < kSortBlock; i += blockDim.x)
      if (bkt[i] >= 0) atomicAdd(&cnt[(i / share) * kFewBuckets + bkt[i]], 1);
    __syncthreads();
  }
  for (int b = threadIdx.x; b < B.n; b += blockDim.x) {
    int at = J.bucket_base[b] + pre[b];
    if (!few) cnt[b] = at;
    for (int w = 0; few && w < kRankWarps; ++w) {
      const int v = cnt[w * kFewBuckets + b];
      cnt[w * kFewBuckets + b] = at;
      at += v;
    }
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5;
  if (warp >= warps) return;
  const int lane = threadIdx.x & 31;
  int* next = cnt + warp * kFewBuckets;
  const unsigned below = (1u << lane) - 1u;
  for (int it = 0; it < share / 32; ++it) {
    const int i = warp * share + it * 32 + lane;
    const long long k = k0 + i;
    const bool in = k < K.n;
    const int b = bkt[i];
    const unsigned peers = __match_any_sync(0xffffffffu, b);
    const int pos = in ? next[b] + __popc(peers & below) : 0;
    __syncwarp();
    if (in) {
      // positions are in [0, n) by construction; an inconsistency is reported
      // (the context then fails) instead of written
      if (pos >= 0 && pos < K.n) J.perm[pos] = (int)k;
      else atomicOr(J.status, ST_BOUNDS);
      if (lane == 31 - __clz(peers)) next[b] += __popc(peers);
    }
    __syncwarp();
  }
}

__global__ void __launch_bounds__(kScatterThreads) wide_scatter_kernel(const __grid_constant__ LaunchArgs a) {
  dev::pdl_trigger();
  dev::pdl_wait();
  const int j = find_job_sort_block(a, blockIdx.x);
  const JobStatic& J = a.js[j];
  const JobCall& K = a.use_inline ? a.inline_call : a.jc[j];
  Buckets B;
  B.plan.set = -1;
  B.plan.cells = 0;
  if (K.low_ok) B.plan = *J.plan;
  B.n = call_is_wide(J) ? kSortBuckets : B.plan.cells;
  if (B.n == 0) return;
  __shared__ int cnt[kSortBuckets];
  __shared__ int bkt[kSortBlock];
  scatter_block(J, K, B, blockIdx.x - K.sort_block_begin, cnt, bkt);
}

// Wide calls: the record at sorted position p, its group beginning at p0.
__device__ __forceinline__ void wide_record(const JobStatic& J, const JobCall& K, long long p0, long long p) {
  if (p >= K.n) return;
  const long long n = K.n;
  int k = J.perm[p], k0 = J.perm[p0];
  if (k < 0 || k >= n || k0 < 0 || k0 >= n) {  // never, for a consistent sort
    atomicOr(J.status, ST_BOUNDS);
    k = k0 = 0;
  }
  double R[3] = {K.r[k0], K.r[n + k0], K.r[2 * n + k0]};
  if (!(isfinite(R[0]) && isfinite(R[1]) && isfinite(R[2]))) {
    R[0] = J.ref[0];
    R[1] = J.ref[1];
    R[2] = J.ref[2];
  }
  float v[kRecFields];
  make_record(J, K, k, R, v);  // invalid data was reported by the pre-pass
  if (!dev::bounds_ok(p < J.n_cap, J.status)) return;
  store_record(J.rec + (size_t)p * kRecFields, v);
  if (p == p0) {
    double* g = J.gref + 3 * (p0 / kGroup);
    g[0] = R[0] - J.ref[0];
    g[1] = R[1] - J.ref[1];
    g[2] = R[2] - J.ref[2];
  }
}

// Wide calls: records in sorted order, positions relative to the first particle of
// each kGroup-particle group (its reference point); the group references
// relative to the call's reference go to gref.  Low band: the pre-pass's records
// in cell order.
__global__ void __launch_bounds__(256) wide_records_kernel(const __grid_constant__ LaunchArgs a) {
  dev::pdl_trigger();
  dev::pdl_wait();
  const int j = dev::find_job_block(a, blockIdx.x);
  const JobStatic& J = a.js[j];
  const JobCall& K = a.use_inline ? a.inline_call : a.jc[j];
  if (!call_is_wide(J)) {
    if (!K.low_ok || J.plan->set < 0) return;
    // five threads per record, 16 bytes each
    constexpr int kQ = kRecFields / 4;
    const long long b0 = (long long)(blockIdx.x - K.block_begin) * 256;
    const int count = (int)min(256LL, K.n - b0);
    for (int i = threadIdx.x; i < count * kQ; i += 256) {
      const long long p = b0 + i / kQ;
      int k = J.perm[p];
      if (k < 0 || k >= K.n) {  // never, for a consistent sort
        atomicOr(J.status, ST_BOUNDS);
        k = 0;
      }
      reinterpret_cast<float4*>(J.rec_s)[p * kQ + i % kQ] = reinterpret_cast<const float4*>(J.rec)[(size_t)k * kQ + i % kQ];
    }
    return;
  }
  const long long p0 = (long long)(blockIdx.x - K.block_begin) * kGroup;
  static_assert(kGroup == 256, "one block per group");
  wide_record(J, K, p0, p0 + threadIdx.x);
}

// The whole sort of a wide call of up to kSmallSort particles by one cluster of
// blocks, kSortBlock particles each: the four kernels' phases with the
// cluster's barrier between them.  A call that is not wide pays one empty
// launch instead of four (8 steps of 1777 particles, 96 x 25 bins: 318 -> 273 us).
constexpr int kClusterMax = 8;  // portable cluster size
constexpr long long kSmallSort = kClusterMax * kSortBlock;
static_assert(kSmallSort <= kLowMin, "calls that may take the low band use the four kernels");
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__global__ void __launch_bounds__(1024) wide_small_kernel(const __grid_constant__ LaunchArgs a) {
  dev::pdl_trigger();
  dev::pdl_wait();
  const JobStatic& J = a.js[0];
  if (!call_is_wide(J)) return;  // (the same for every block of the cluster)
  const JobCall& K = a.inline_call;
  __shared__ int cnt[kSortBuckets];
  __shared__ int bkt[kSortBlock];
  Buckets B;
  B.plan.set = -1;
  B.n = kSortBuckets;
  hist_block(J, K, B, blockIdx.x, cnt);
  cluster_barrier();
  if (blockIdx.x == 0) scan_job(J, K, B.n, cnt, bkt);
  cluster_barrier();
  scatter_block(J, K, B, blockIdx.x, cnt, bkt);
  cluster_barrier();
  for (long long p = (long long)blockIdx.x * 1024 + threadIdx.x; p < K.n; p += (long long)gridDim.x * 1024)
    wide_record(J, K, p / kGroup * kGroup, p);
}

// An alternative's tables (LowSet): the nodes' frequency factors, and per bin of the
// band its taps' weights (of the window) and first node.
__global__ void __launch_bounds__(128) low_tables_kernel(const LowSet* __restrict__ sets,
                                                         const double* __restrict__ om_turns) {
  const LowSet& L = sets[blockIdx.y];
  constexpr double k2Pi = 6.283185307179586476925286766559;
  if (blockIdx.x == 0 && threadIdx.x < kLowNodes) {
    const int i = threadIdx.x;
    const double nu = (i - kLowTaps / 2) * L.dnu;
    const float hi = __double2float_rn(nu);
    L.nodes[i] = hi;
    L.nodes[kLowNodes + i] = __double2float_rn(k2Pi * (double)hi);
    L.nodes[2 * kLowNodes + i] = __double2float_rn(k2Pi * (nu - (double)hi));
  }
  const int j = blockIdx.x * 128 + threadIdx.x;
  if (j >= L.js) return;
  const double s = om_turns[j] / L.dnu;  // in node spacings, from frequency 0
  const int base = min((int)floor(s), kLowReach);
  float* w = L.wts + (size_t)j * kLowWt;
  // taps at base - kLowTaps/2 + 1 .. base + kLowTaps/2; node 0 is -kLowTaps/2
  for (int t = 0; t < kLowTaps; ++t) {
    const double u = (s - (base - kLowTaps / 2 + 1 + t)) / (0.5 * kLowTaps);
    w[t] = fabs(u) < 1.0 ? __double2float_rn(exp(kLowBeta * (sqrt(1.0 - u * u) - 1.0))) : 0.0f;
  }
  w[kLowTaps] = __int_as_float(base + 1);
  w[kLowTaps + 1] = 0.0f;
}

// ------------------------------------------------------------------ readout
__device__ double sinc(double x) { return x == 0.0 ? 1.0 : sin(x) / x; }

// Amplitude form factor of Table 1, normalised to f(0) = 1.
__device__ double form_factor(int kind, double width, double omega) {
  const double x = omega * width * (0.5 * kInvC);
  switch (kind) {
    case RAD_FF_CIC: return sinc(x);
    case RAD_FF_TSC: { const double s = sinc(x); return s * s; }
    case RAD_FF_QSC: { const double s = sinc(x); return s * s * s; }
    case RAD_FF_GAUSS: { const double g = omega * width * kInvC; return exp(-0.5 * g * g); }
    default: return 1.0;
  }
}

// With RAD_FF_3D, box shapes are axis-aligned 3-D products: f = prod_d f_1(omega n_d).
__device__ double form_factor_3d(int kind, double width, double omega, const double* n) {
  return form_factor(kind, width, omega * n[0]) * form_factor(kind, width, omega * n[1]) *
         form_factor(kind, width, omega * n[2]);
}
__device__ __forceinline__ bool per_direction(int kind, int flags) {
  return (flags & RAD_FF_3D) && kind != RAD_FF_POINT && kind != RAD_FF_GAUSS;
}

// float to double on the integer pipe (the conversion shares the narrow FP64
// pipe): exponent rebias and shift; zero, and with the instruction what is
// subnormal, infinite or NaN.
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x), mag = b & 0x7fffffffu;
  if (mag - 0x00800000u >= 0x7f000000u && mag != 0u) return (double)x;
  return __hiloint2double((int)((b & 0x80000000u) | (mag ? (mag >> 3) + 0x38000000u : 0u)), (int)(b << 29));
}

// Readout, FP64: coherent k0 f^2 |U|^2, incoherent k0 (1 - f^2) |V|^2.  Bound by
// the FP64 pipe (1.7 lanes/clk/SM), not by the 88 bytes per bin: so a thread
// takes up to kReadBins bins of one frequency (bins t, t + stride, ..., the stride
// a multiple of the frequencies) and computes the shape's factor once for
// them, and the state's floats are widened on the integer pipe.  131072 bins, the
// whole call: 40 -> 30 us for a 1-D shape, 57 for a 3-D box (three sines per
// bin), 81 -> 59 for two species (kReadBins 2: 32 and 65; 8: 31 and 59).
constexpr int kReadBins = 4;

__global__ void __launch_bounds__(128) readout_kernel(
    const float* __restrict__ state, const double* __restrict__ state64, int mixed, int n_omega, int n_bins,
    long long stride, const double* __restrict__ omega, const double* __restrict__ dirs, int kind, int flags,
    double width, double k0, double* coh, double* inc, double* tot) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= stride || t >= n_bins) return;
  const bool by_dir = per_direction(kind, flags);
  const int o = (int)(t % n_omega);
  const double om = omega[o];
  double f = by_dir ? 0.0 : form_factor(kind, width, om);
#pragma unroll 1
  for (long long at = t; at < n_bins; at += stride) {
    const int bin = (int)at;
    double u2 = 0.0, v2 = 0.0;
    if (mixed) {
      float a[2 * kComps];
#pragma unroll
      for (int c = 0; c < 2 * kComps; ++c) a[c] = state[(size_t)c * n_bins + bin];
#pragma unroll
      for (int c = 0; c < kComps; ++c) {
        const double x = widen(a[c]) - widen(a[kComps + c]);
        if (c < 4) u2 += x * x;
        else v2 += x * x;
      }
    } else {
#pragma unroll
      for (int c = 0; c < 12; ++c) {
        const double x = state64[(size_t)c * n_bins + bin];
        if (c < 6) u2 += x * x;
        else v2 += x * x;
      }
    }
    if (by_dir) f = form_factor_3d(kind, width, om, dirs + 3 * (size_t)(bin / n_omega));
    const double f2 = f * f;
    const double ic = k0 * f2 * u2, ii = k0 * (1.0 - f2) * v2;
    if (coh) coh[bin] = ic;
    if (inc) inc[bin] = ii;
    if (tot) tot[bin] = ic + ii;
  }
}

template <bool MIXED>
__global__ void __launch_bounds__(128) readout_species_kernel(
    const __grid_constant__ SpeciesArgs a, int n_omega, int n_bins, long long stride,
    const double* __restrict__ omega, const double* __restrict__ dirs, double k0, double* coh, double* inc,
    double* tot) {
  constexpr int NU = MIXED ? 4 : 6;  // real components of U (and of V)
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < a.n_species) a.gathered[t] = *a.status[t];
  // (a failed species' sums are incomplete: nothing is written, the host reports it)
  for (int s = 0; s < a.n_species; ++s)
    if (*a.status[s] & (ST_TIMEOUT | ST_BOUNDS)) return;
  if (t >= stride || t >= n_bins) return;
  const double om = omega[(int)(t % n_omega)];
  double u[kReadBins][NU] = {}, ii[kReadBins] = {};  // (stride: at most kReadBins bins per thread)
  for (int s = 0; s < a.n_species; ++s) {
    const bool by_dir = per_direction(a.kind[s], a.flags[s]);
    double f = by_dir ? 0.0 : form_factor(a.kind[s], a.width[s], om);
    const float* st = a.state[s];
    const double* st64 = a.state64[s];
#pragma unroll
    for (int k = 0; k < kReadBins; ++k) {
      const long long at = t + k * stride;
      if (at >= n_bins) break;
      const int bin = (int)at;
      if (by_dir) f = form_factor_3d(a.kind[s], a.width[s], om, dirs + 3 * (size_t)(bin / n_omega));
      double v2 = 0.0;
#pragma unroll
      for (int c = 0; c < 2 * NU; ++c) {
        double x;
        if (MIXED) x = widen(st[(size_t)c * n_bins + bin]) - widen(st[(size_t)(kComps + c) * n_bins + bin]);
        else x = st64[(size_t)c * n_bins + bin];
        if (c < NU) u[k][c < NU ? c : 0] += f * x;  // amplitudes add across species before |.|^2
        else v2 += x * x;
      }
      ii[k] += (1.0 - f * f) * v2;
    }
  }
#pragma unroll
  for (int k = 0; k < kReadBins; ++k) {
    const long long bin = t + k * stride;
    if (bin >= n_bins) break;
    double u2 = 0.0;
#pragma unroll
    for (int c = 0; c < NU; ++c) u2 += u[k][c] * u[k][c];
    const double ic = k0 * u2, i2 = k0 * ii[k];
    if (coh) coh[bin] = ic;
    if (inc) inc[bin] = i2;
    if (tot) tot[bin] = ic + i2;
  }
}

// ----------------------------------------------------------- plain FP64 K5
// Eq. 1 and Eq. 13 in FP64 throughout, one thread per (direction, frequency)
// bin and particle chunk.
//
// Bound: the FP64 pipe, 1.68 lanes/clk/SM on this GPU, so the design counts
// FP64 instructions.  What does not depend on the frequency (the retarded time
// tau = t - n.r/c and the weighted amplitude, ~50 instructions) is computed once
// per (particle, direction) of the block's bins and shared through shared
// memory; A is perpendicular to n, so its two transverse components carry it (8
// multiply-adds per update instead of 12).  The phase is formed in turns, where
// the reduction modulo 1 is exact and needs no 2/pi tables at phases of 1e6
// radians, and sin/cos take a 256-entry table of the circle (built per block
// from its first octant by sincospi and symmetry) and the Taylor series about
// the entry: 27 FP64 instructions per update.  The rounding of omega/2pi is carried
// (f_lo), as is that of the product (fma), so the phase error is that of tau.
// The particles are cut into chunks when the bins alone are too few blocks.
//
// 4001 particles, 512 x 16 bins: 14.5 ms before (64 blocks, amplitude and a
// large-argument sincos per update), 1.90 ms (1.7e10 updates/s) now.
constexpr int kF64Threads = 128;
constexpr int kF64Records = 512;  // (particle, direction) records staged at once

struct F64Rec {
  double tau, u1, u2, v1, v2, pad;
};

__global__ void __launch_bounds__(kF64Threads) fp64_kernel(
    const double* __restrict__ omega, const double* __restrict__ dirs, int n_omega, int n_dir,
    long long n, long long ck, const double* __restrict__ r, const double* __restrict__ beta,
    const double* __restrict__ bdot, const double* __restrict__ w, double t, double dt,
    double* __restrict__ state, double* __restrict__ part, unsigned* __restrict__ cnt, int* status) {
  __shared__ double2 circle[256];
  __shared__ F64Rec rec[kF64Records];
  __shared__ double dtab[kF64Threads][9];  // n, e1, e2 of the block's directions
  __shared__ unsigned s_prev;
  const int n_bins = n_omega * n_dir;
  const int bin0 = blockIdx.x * kF64Threads;
  const int bin = bin0 + threadIdx.x;
  const bool live = bin < n_bins;
  const int d0 = bin0 / n_omega;
  const int nd = min(bin0 + kF64Threads - 1, n_bins - 1) / n_omega - d0 + 1;  // <= kF64Threads
  const int my_dl = (live ? bin : n_bins - 1) / n_omega - d0;
  const int KT = kF64Records / nd;

  // e^{2 pi i j / 256}: the first octant, then its mirror images.
  if (threadIdx.x <= 32) {
    double s, c;
    sincospi((double)threadIdx.x * (1.0 / 128.0), &s, &c);
    circle[threadIdx.x] = make_double2(c, s);
  }
  if (threadIdx.x < nd) {
    const double* q = dirs + 3 * (size_t)(d0 + threadIdx.x);
    const double x = q[0], y = q[1], z = q[2];
    int ax = 0;
    if (fabs(y) < fabs(x)) ax = 1;
    if (fabs(z) < fabs(ax ? y : x)) ax = 2;
    const double an = ax == 0 ? x : (ax == 1 ? y : z);
    double e0 = (ax == 0) - an * x, e1 = (ax == 1) - an * y, e2 = (ax == 2) - an * z;
    const double il = 1.0 / sqrt(e0 * e0 + e1 * e1 + e2 * e2);
    e0 *= il;
    e1 *= il;
    e2 *= il;
    double* o = dtab[threadIdx.x];
    o[0] = x, o[1] = y, o[2] = z, o[3] = e0, o[4] = e1, o[5] = e2;
    o[6] = y * e2 - z * e1, o[7] = z * e0 - x * e2, o[8] = x * e1 - y * e0;
  }
  __syncthreads();
  for (int j = threadIdx.x; j < 256; j += kF64Threads) {
    if (j <= 32) continue;
    const int o = j & 63, q = j >> 6;           // quadrant q, angle o / 256 of a turn within it
    const int b = o <= 32 ? o : 64 - o;
    double2 v = circle[b];
    if (o > 32) v = make_double2(v.y, v.x);
    if (q & 1) v = make_double2(-v.y, v.x);
    if (q & 2) v = make_double2(-v.x, -v.y);
    circle[j] = v;
  }

  const double om = omega[(live ? bin : n_bins - 1) - (d0 + my_dl) * n_omega];
  // omega / 2pi as f + f_lo
  constexpr double kInv2Pi = 0.15915494309189535, kInv2PiLo = -9.839338337591243e-18;
  const double f = om * kInv2Pi;
  const double f_lo = fma(om, kInv2PiLo, fma(om, kInv2Pi, -f));

  const long long k_begin = (long long)blockIdx.y * ck, k_end = min(n, k_begin + ck);
  double u1r = 0, u1i = 0, u2r = 0, u2i = 0, v1r = 0, v1i = 0, v2r = 0, v2i = 0;
  bool bad = false;
  for (long long k0 = k_begin; k0 < k_end; k0 += KT) {
    const int kn = (int)min((long long)KT, k_end - k0);
    __syncthreads();  // the circle is complete, the last records are used up
    for (int i = threadIdx.x; i < kn * nd; i += kF64Threads) {
      const int dl = i / kn;
      const long long k = k0 + (i - dl * kn);
      const double* D = dtab[dl];
      const double nx = D[0], ny = D[1], nz = D[2];
      const double rx = r[k], ry = r[n + k], rz = r[2 * n + k];
      const double bx = beta[k], by = beta[n + k], bz = beta[2 * n + k];
      const double ax = bdot[k], ay = bdot[n + k], az = bdot[2 * n + k];
      const double wk = w[k];
      const double g2 = 1.0 - (bx * bx + by * by + bz * bz);
      F64Rec o = {0, 0, 0, 0, 0, 0};
      if (!(wk > 0.0) || !(g2 > 0.0) || !isfinite(wk) || !isfinite(ax + ay + az) ||
          !isfinite(rx + ry + rz)) {
        bad = true;
      } else {
        // e_i . (n x ((n - beta) x bdot)) = (e_i . (n - beta)) (n . bdot) - (e_i . bdot) (n . (n - beta))
        const double ux = nx - bx, uy = ny - by, uz = nz - bz;
        const double cx = uy * az - uz * ay, cy = uz * ax - ux * az, cz = ux * ay - uy * ax;
        const double mx = ny * cz - nz * cy, my = nz * cx - nx * cz, mz = nx * cy - ny * cx;
        const double dd = 1.0 - (bx * nx + by * ny + bz * nz);
        const double id2 = 1.0 / (dd * dd);
        const double a1 = (D[3] * mx + D[4] * my + D[5] * mz) * id2;
        const double a2 = (D[6] * mx + D[7] * my + D[8] * mz) * id2;
        const double ww = wk * dt, sw = sqrt(wk) * dt;
        o.tau = t - (nx * rx + ny * ry + nz * rz) * kInvC;
        o.u1 = ww * a1;
        o.u2 = ww * a2;
        o.v1 = sw * a1;
        o.v2 = sw * a2;
      }
      rec[dl * KT + (i - dl * kn)] = o;
    }
    __syncthreads();
    const F64Rec* q = rec + my_dl * KT;
#pragma unroll 2
    for (int i = 0; i < kn; ++i) {
      const double tau = q[i].tau;
      // turns = hi + lo; m: hi in 256ths, rounded by the magic addition (its
      // low bits are the table index); z: the rest, |z| <= 1/512 turn
      // and lo, which is below 2^-12 + 2^-11 turn at the branch's 2^42 turns
      constexpr double kMagic = 6755399441055744.0;  // 1.5 * 2^52
      const double hi = f * tau;
      const double lo = fma(f_lo, tau, fma(f, tau, -hi));
      const double m = fma(hi, 256.0, kMagic);
      // Phases past 2^42 turns leave the magic range: reduce them first.
      double z;
      int j;
      if ((__double2hiint(hi) & 0x7fffffff) < 0x42900000) {  // |hi| < 2^42, on the integer pipe
        z = fma(m - kMagic, -1.0 / 256.0, hi) + lo;
        j = __double2loint(m) & 255;
      } else {
        const double h1 = (hi - rint(hi)) + (lo - rint(lo)), m1 = fma(h1, 256.0, kMagic);
        z = fma(m1 - kMagic, -1.0 / 256.0, h1);
        j = __double2loint(m1) & 255;
      }
      // sin and cos - 1 of w = 2 pi z by their Taylor series, the powers of
      // 2 pi in the coefficients (next terms: w^7/5040 <= 9e-18, 8e-17 with the
      // largest lo, and w^8/40320).
      const double z2 = z * z;
      const double sz = fma(z * z2, fma(z2, 81.605249276075054, -41.341702240399760), z * 6.283185307179586477);
      const double cz = z2 * fma(z2, fma(z2, -85.456817206693728, 64.939394022668291), -19.739208802178717);
      const double2 cs = circle[j];
      const double c = fma(-cs.y, sz, fma(cs.x, cz, cs.x));
      const double s = fma(cs.x, sz, fma(cs.y, cz, cs.y));
      u1r = fma(q[i].u1, c, u1r);
      u1i = fma(q[i].u1, s, u1i);
      u2r = fma(q[i].u2, c, u2r);
      u2i = fma(q[i].u2, s, u2i);
      v1r = fma(q[i].v1, c, v1r);
      v1i = fma(q[i].v1, s, v1i);
      v2r = fma(q[i].v2, c, v2r);
      v2i = fma(q[i].v2, s, v2i);
    }
  }
  if (bad) atomicOr(status, ST_BAD_PARTICLE);
  double S[8] = {u1r, u1i, u2r, u2i, v1r, v1i, v2r, v2i};
  // Several chunks: the last block of these bins adds the chunks' sums in order.
  if (gridDim.y > 1) {
    if (live)
#pragma unroll
      for (int c = 0; c < 8; ++c) part[((size_t)blockIdx.y * 8 + c) * n_bins + bin] = S[c];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      s_prev = atomicAdd(&cnt[blockIdx.x], 1u);
      if (s_prev == gridDim.y - 1) cnt[blockIdx.x] = 0u;  // ready for the next call
      __threadfence();
    }
    __syncthreads();
    if (s_prev != gridDim.y - 1) return;
#pragma unroll
    for (int c = 0; c < 8; ++c) S[c] = 0.0;
    if (live)
      for (int ch = 0; ch < (int)gridDim.y; ++ch)
#pragma unroll
        for (int c = 0; c < 8; ++c) S[c] += __ldcg(&part[((size_t)ch * 8 + c) * n_bins + bin]);
  }
  if (!live) return;
  const double* D = dtab[my_dl];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      state[(size_t)(2 * c + p) * n_bins + bin] += S[p] * D[3 + c] + S[2 + p] * D[6 + c];
      state[(size_t)(6 + 2 * c + p) * n_bins + bin] += S[4 + p] * D[3 + c] + S[6 + p] * D[6 + c];
    }
  }
}

// Literal spectrum K0 |P|^2 from the compensated P.e1, P.e2 sums.
__global__ void readout_literal_kernel(const float* __restrict__ state_p, int n_bins, double k0,
                                       double* out) {
  const int bin = blockIdx.x * blockDim.x + threadIdx.x;
  if (bin >= n_bins) return;
  double p2 = 0.0;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const double x = (double)state_p[(size_t)c * n_bins + bin] -
                     (double)state_p[(size_t)(4 + c) * n_bins + bin];
    p2 += x * x;
  }
  out[bin] = k0 * p2;
}

// Adds another accumulator array into state with compensation.  Both hold
// n_comps sums followed by their n_comps compensations per bin.
__global__ void state_add_kernel(float* __restrict__ state, const float* __restrict__ other,
                                 int n_bins, int n_comps) {
  const int bin = blockIdx.x * blockDim.x + threadIdx.x;
  if (bin >= n_bins) return;
  // other holds (sum, comp) pairs; add its value sum - comp with compensation.
  for (int c = 0; c < n_comps; ++c) {
    const float x = __fsub_rn(other[(size_t)c * n_bins + bin], other[(size_t)(n_comps + c) * n_bins + bin]);
    float* sum = &state[(size_t)c * n_bins + bin];
    float* cmp = &state[(size_t)(n_comps + c) * n_bins + bin];
    const float y = __fsub_rn(x, *cmp);
    const float tt = __fadd_rn(*sum, y);
    *cmp = __fsub_rn(__fsub_rn(tt, *sum), y);
    *sum = tt;
  }
}

__global__ void state64_add_kernel(double* __restrict__ state, const double* __restrict__ other,
                                   int n_bins) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 12 * n_bins) return;
  state[i] += other[i];
}

std::atomic<long long> g_launches{0};

}  // namespace

void count_launches(int n) { g_launches.fetch_add(n); }

cudaError_t launch_prepass(const LaunchArgs& a, int total_blocks, cudaStream_t s) {
  if (total_blocks <= 0) return cudaSuccess;
  count_launches(1);
  return launch_pdl(prepass_kernel, total_blocks, 256, 0, s, a);
}

cudaError_t launch_wide(const LaunchArgs& a, int sort_blocks, int prepass_blocks, cudaStream_t s) {
  if (sort_blocks <= 0 || prepass_blocks <= 0) return cudaSuccess;
  if (a.use_inline && a.inline_call.n <= kSmallSort && !a.inline_call.low_ok) {
    count_launches(1);
    return launch_pdl(wide_small_kernel, sort_blocks, 1024, 0, s, a, sort_blocks);
  }
  cudaError_t e = launch_pdl(wide_hist_kernel, sort_blocks, kHistThreads, 0, s, a);
  if (e == cudaSuccess) e = launch_pdl(wide_scan_kernel, a.n_jobs, 1024, 0, s, a);
  if (e == cudaSuccess) e = launch_pdl(wide_scatter_kernel, sort_blocks, kScatterThreads, 0, s, a);
  if (e == cudaSuccess) e = launch_pdl(wide_records_kernel, prepass_blocks, 256, 0, s, a);
  count_launches(kWideLaunches);
  return e;
}

void wide_geometry(const double* nd, int n_dir, float tau_fast, double axis[3], double* cone_sin,
                   double* bucket_w) {
  double m[3] = {0.0, 0.0, 0.0};
  for (int d = 0; d < n_dir; ++d)
    for (int i = 0; i < 3; ++i) m[i] += nd[3 * d + i];
  double len = sqrt(m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
  // A grid spread over all directions has no useful mean: sort along z.
  if (!(len > 0.5 * n_dir)) {
    m[0] = m[1] = 0.0;
    m[2] = len = 1.0;
  }
  for (int i = 0; i < 3; ++i) axis[i] = m[i] / len;
  double cos_min = 1.0;
  for (int d = 0; d < n_dir; ++d)
    cos_min = std::min(cos_min, axis[0] * nd[3 * d] + axis[1] * nd[3 * d + 1] + axis[2] * nd[3 * d + 2]);
  *cone_sin = cos_min <= 0.0 ? 1.0 : sqrt(std::max(0.0, 1.0 - cos_min * cos_min));
  // A group of sorted particles spans about two buckets along the axis: an
  // eighth of the fast range keeps it well inside.
  *bucket_w = (double)tau_fast * kC / 8.0;
}

void low_geometry(const double* nd, int n_dir, JobStatic& js) {
  const double* n = js.axis;
  int ax = 0;
  if (fabs(n[1]) < fabs(n[ax])) ax = 1;
  if (fabs(n[2]) < fabs(n[ax])) ax = 2;
  double len = 0.0;
  for (int i = 0; i < 3; ++i) {
    js.fr1[i] = (i == ax) - n[ax] * n[i];
    len += js.fr1[i] * js.fr1[i];
  }
  for (int i = 0; i < 3; ++i) js.fr1[i] /= sqrt(len);
  for (int i = 0; i < 3; ++i)
    js.fr2[i] = n[(i + 1) % 3] * js.fr1[(i + 2) % 3] - n[(i + 2) % 3] * js.fr1[(i + 1) % 3];
  double c1 = 0.0, c2 = 0.0;
  for (int d = 0; d < n_dir; ++d) {
    const double* q = nd + 3 * (size_t)d;
    c1 = std::max(c1, fabs(q[0] * js.fr1[0] + q[1] * js.fr1[1] + q[2] * js.fr1[2]));
    c2 = std::max(c2, fabs(q[0] * js.fr2[0] + q[1] * js.fr2[1] + q[2] * js.fr2[2]));
  }
  js.cone1 = (float)c1;
  js.cone2 = (float)c2;
}

cudaError_t launch_low_tables(const JobStatic& js, int n, cudaStream_t s) {
  low_tables_kernel<<<dim3((unsigned)((js.n_omega + 127) / 128), (unsigned)n), 128, 0, s>>>(js.low, js.om_turns);
  count_launches(1);
  return cudaGetLastError();
}

// Bins between a readout thread's bins: all of them for grids of less than a
// thread per lane of the GPU, else about a kReadBins-th, in whole frequency rows.
static long long readout_stride(int n_omega, int n_bins) {
  constexpr int kEnough = 152 * 128;
  const int per = std::max(1, std::min(kReadBins, n_bins / kEnough));
  const long long rows = ((n_bins + per - 1) / per + n_omega - 1) / n_omega;
  return rows * n_omega;
}

cudaError_t launch_readout(const float* state, int mixed, const double* state64, int n_omega,
                           int n_bins, const double* omega, const double* dirs, rad_ff ff,
                           double* coh, double* inc, double* tot, cudaStream_t s) {
  const double k0 = kQe * kQe / (16.0 * kPi * kPi * kPi * kEps0 * kC);
  const long long stride = readout_stride(n_omega, n_bins);
  readout_kernel<<<(unsigned)((stride + 127) / 128), 128, 0, s>>>(state, state64, mixed, n_omega, n_bins, stride,
                                                                   omega, dirs, ff.kind, ff.flags, ff.width, k0,
                                                                   coh, inc, tot);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_readout_species(const SpeciesArgs& a, int n_omega, int n_bins,
                                   const double* omega, const double* dirs, double* coh,
                                   double* inc, double* tot, cudaStream_t s) {
  const double k0 = kQe * kQe / (16.0 * kPi * kPi * kPi * kEps0 * kC);
  const long long stride = readout_stride(n_omega, n_bins);
  const unsigned blocks = (unsigned)((stride + 127) / 128);
  if (a.mixed)
    readout_species_kernel<true><<<blocks, 128, 0, s>>>(a, n_omega, n_bins, stride, omega, dirs, k0, coh, inc, tot);
  else
    readout_species_kernel<false><<<blocks, 128, 0, s>>>(a, n_omega, n_bins, stride, omega, dirs, k0, coh, inc, tot);
  count_launches(1);
  return cudaGetLastError();
}

// Chunks of an FP64 call: about kF64BlocksPerSm blocks per SM when the bins
// alone give fewer (the pipe is shared, so finer blocks only even out the SMs'
// shares), never below kF64MinChunk particles (a block's table and records).
constexpr int kF64BlocksPerSm = 8;
constexpr int kF64MinChunk = 64;

int fp64_max_chunks(int n_bins, int sms) {
  const int blocks = (n_bins + kF64Threads - 1) / kF64Threads;
  return std::max(1, kF64BlocksPerSm * sms / blocks);
}
int fp64_blocks(int n_bins) { return (n_bins + kF64Threads - 1) / kF64Threads; }

cudaError_t launch_fp64(const double* omega, const double* dirs, int n_omega, int n_dir,
                        long long n, const double* r, const double* beta, const double* bdot,
                        const double* w, double t, double dt, double* state64, double* part,
                        unsigned* cnt, int max_chunks, int* status, cudaStream_t s) {
  const int n_bins = n_omega * n_dir;
  const long long ck = std::max<long long>(kF64MinChunk, (n + max_chunks - 1) / max_chunks);
  const dim3 grid((unsigned)fp64_blocks(n_bins), (unsigned)((n + ck - 1) / ck));
  fp64_kernel<<<grid, kF64Threads, 0, s>>>(omega, dirs, n_omega, n_dir, n, ck, r, beta, bdot, w, t,
                                           dt, state64, part, cnt, status);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_state_add(float* state, const float* other, int n_bins, int n_comps,
                             cudaStream_t s) {
  state_add_kernel<<<(n_bins + 255) / 256, 256, 0, s>>>(state, other, n_bins, n_comps);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_readout_literal(const float* state_p, int n_bins, double* out, cudaStream_t s) {
  const double k0 = kQe * kQe / (16.0 * kPi * kPi * kPi * kEps0 * kC);
  readout_literal_kernel<<<(n_bins + 255) / 256, 256, 0, s>>>(state_p, n_bins, k0, out);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_state64_add(double* state, const double* other, int n_bins, cudaStream_t s) {
  state64_add_kernel<<<(12 * n_bins + 255) / 256, 256, 0, s>>>(state, other, n_bins);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace radimpl

extern "C" int64_t rad_kernel_launch_count(void) { return radimpl::g_launches.load(); }
