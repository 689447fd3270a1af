// The accumulate kernel of the far-field radiation sum (Pausch et al. 2018,
// Eq. 1 and the in-situ inner sum of Eq. 13).
//
// Persistent: one CTA per resident slot takes dynamic work items (job, bin
// tile, particle chunk).  A bin tile is NT directions x WT frequencies; the
// chunk's particle records (80 B each, written by the pre-pass) stream through
// shared memory in tiles of THREADS / NT particles, fetched by a TMA bulk copy
// (cp.async.bulk + mbarrier, time-bounded wait) one tile ahead of use.
//
// Stage 1, one (particle, direction) record per thread, FP32: the retarded-time
// offset dtau = -n.(r - r_ref)/c as a float-float pair (TwoProduct with fma,
// TwoSum), and the transverse amplitude components a_i = e_i . A in a basis
// (e1, e2) perpendicular to n.  n . A = 0 (Eq. 1), so these two carry |A|^2;
// with u = n - beta, n x (u x bdot) = u (n.bdot) - bdot D,
// D = 1 - beta.n = (1/gamma^2 + b1^2 + b2^2) / (1 + beta.n) and e_i.u = -b_i,
// a_i = -(b_i (n.bdot) + (e_i.bdot) D) / D^2, free of cancellation at high
// gamma.  Records are double-buffered, one barrier per particle tile.
//
// Stage 2, per (particle, direction, frequency), the "amplitude update": the
// phase in turns p = (omega/2pi) dtau is reduced exactly by one fused multiply-
// add against 1.5 * 2^23 (no FRND, which shares the MUFU pipe), the float-float
// cross terms are added in radians, and sin/cos come from the MUFU (2 per
// update).  The weighted sums U_i += w dt a_i e^{i phi}, V_i += sqrt(w) dt a_i
// e^{i phi} are then formed in one of two ways:
//  * FP32 variants: 8 packed FMAs (f32x2) per update into register accumulators,
//    two frequencies per packed lane pair;
//  * tensor-core variants: per warp, each 16-frequency x 8-particle block of
//    e^{i phi} (two or four blocks per warp) is the A operand of mma.sync
//    m16n8k8 TF32 and the 4 weighted amplitudes of the 8 particles are B.  Both are split into TF32 hi and lo
//    parts (hi = the top 19 bits, lo = the exact rest), B's hi and lo side by
//    side in the 8 N-columns, so two MMAs per cos/sin give all of
//    hi.hi + hi.lo + lo.hi + lo.lo with FP32 accumulation.  This takes the
//    accumulation FMAs off the FP32 pipe, which together with the phase
//    arithmetic and MUFU issue is what limits the FP32 variants.
// Wide calls (particles spread beyond the fast phase range about the call's
// reference point, sorted by the wide-call kernels) run in a second pass of
// the same launch, an instantiation of its own (WIDE): their records are relative to
// the first particle of each 256-particle group, so stage 1 and the update loop
// are unchanged, and each tile's sums are rotated by e^{i omega tau_group}
// before they join the chunk sums.
// Sums are two-level (per particle tile, then per chunk).  Each chunk's sums go to
// a buffer of partials; a second kernel (reduce_kernel) adds them in chunk
// order, multiplies by e^{i omega tau_ref(n)} (reduced in FP64) and adds the
// result into the resident state with compensated (Kahan) FP32 sums.  No float
// atomics: results are deterministic for a given chunking.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "rad_device.cuh"
#include "rad_impl.h"
#include "rad_stage.cuh"

namespace radimpl {

namespace {

using namespace dev;


template <int THREADS, bool TC, bool LIT = false, int PASSES = 1, bool XT = false>
struct Smem {
  static constexpr size_t raw_bytes = (size_t)THREADS * kRecFields * sizeof(float);
  static constexpr size_t rec_bytes = (size_t)THREADS * (XT ? 84 : TC ? 40 : (LIT ? 64 : 48));
  static constexpr size_t l2_bytes = TC ? (size_t)THREADS * 16 * sizeof(float) * PASSES : 0;
  // XT: the tile's direction rows (12 floats each; at most THREADS / 8 directions)
  static constexpr size_t dir_bytes = XT ? (size_t)(THREADS / 8) * 12 * sizeof(float) : 0;
  static constexpr size_t bytes = raw_bytes + 2 * rec_bytes + l2_bytes + dir_bytes;
};

struct TileGeom {
  int WT, NT, KT, d0, o0;
};

__device__ __forceinline__ TileGeom tile_geom(const JobStatic& J, int tile, int threads) {
  TileGeom g;
  int s = 0;
  while (s + 1 < J.n_seg && tile >= J.seg[s + 1].tile0) ++s;
  const TileSeg& sg = J.seg[s];
  g.WT = sg.wt;
  g.NT = sg.nt;
  g.KT = threads / g.NT;
  tile -= sg.tile0;
  const int tile_d = tile / sg.tiles_om;
  g.d0 = tile_d * g.NT;
  g.o0 = sg.o0 + (tile - tile_d * sg.tiles_om) * g.WT;
  return g;
}

// A work item: its tile, its particle chunks (run of them from `chunk`), and
// the chunking of that tile.  fine: the tile's index among the tiles of its
// fine-chunked level (TailPlan), -1 for the coarse tiles.  (The level itself
// follows from the tile and the call; the item, live across the whole particle
// loop, holds no more.)
struct ItemRef {
  int tile, chunk, run, ck, n_chunks, fine;
};

// The item in shared memory, for what is used after its first barrier: the hot
// loops are short of registers.
struct ItemShared {
  ItemRef it;
  int n_item;         // the item's particles
  long long k_begin;  // its first particle
};

// q = a / b, r = a - q b; 64-bit division only where 32 bits do not hold a.
__device__ __forceinline__ void div_rem(long long a, int b, int& q, int& r) {
  if (a < (1LL << 32)) {
    const unsigned u = (unsigned)a, v = u / (unsigned)b;
    q = (int)v;
    r = (int)(u - v * (unsigned)b);
  } else {
    q = (int)(a / b);
    r = (int)(a - (long long)q * b);
  }
}

// Item `local` of a job: the coarse tiles' items tile-major, then level 0's
// fine tiles' items, then level 1's, each tile-major.  FINE = false: the
// FP32 variants, whose jobs are never fine-chunked (every item coarse).
template <bool FINE>
__device__ __forceinline__ ItemRef decode_item(const JobStatic& J, const JobCall& K,
                                               long long local) {
  static_assert(kTailLevels == 2, "two fine levels");
  ItemRef it;
  const int first0 = FINE ? J.n_tiles - K.tail_tiles[0] - K.tail_tiles[1] : J.n_tiles;
  const int per_tile = K.run == 1 ? K.n_chunks : (K.n_chunks + K.run - 1) / K.run;
  const long long coarse = (long long)first0 * per_tile;
  const long long fine0 = (long long)K.tail_tiles[0] * K.n_chunks_f[0];
  if (!FINE || local < coarse) {
    div_rem(local, per_tile, it.tile, it.chunk);
    it.chunk *= K.run;
    it.run = min(K.run, K.n_chunks - it.chunk);
    it.ck = K.ck;
    it.n_chunks = K.n_chunks;
    it.fine = -1;
  } else if (local - coarse < fine0) {
    div_rem(local - coarse, K.n_chunks_f[0], it.fine, it.chunk);
    it.tile = first0 + it.fine;
    it.run = 1;
    it.ck = K.ck_f[0];
    it.n_chunks = K.n_chunks_f[0];
  } else {
    div_rem(local - coarse - fine0, K.n_chunks_f[1], it.fine, it.chunk);
    it.tile = first0 + K.tail_tiles[0] + it.fine;
    it.run = 1;
    it.ck = K.ck_f[1];
    it.n_chunks = K.n_chunks_f[1];
  }
  return it;
}

// Where an item's partial sums live: component comp of chunk ch at
// base[ch * chunk_stride + comp * comp_stride + bin offset].  Coarse tiles:
// J.partials [chunk][comp][bin], the bins those of the tiled frequencies (all, or
// the ones above the low band: rows of part_row per direction, so an
// alternative with few tiles and many chunks needs no room for the band's bins:
// a context of 4096 x 256 bins with 3e5 particles holds 0.81 GB instead of
// 3.23); fine tiles: their
// level's region of J.partials_f, [chunk][comp][level tiles][NT WT], level 1's
// after level 0's, the offset the bin's index within the tile.  room: the
// floats from the start of the item's buffer or region.
struct PartMap {
  float* base;
  size_t chunk_stride, comp_stride;
  long long room;
};
__device__ __forceinline__ PartMap part_map(const JobStatic& J, const JobCall& K, const ItemRef& it,
                                            const TileGeom& g) {
  PartMap m;
  if (it.fine < 0) {
    m.base = J.partials;
    m.comp_stride = (size_t)J.part_bins;
    m.room = J.part_cap;
  } else {
    const long long tb = (long long)g.NT * g.WT;
    const bool l1 = it.tile >= J.n_tiles - K.tail_tiles[1];
    const long long foff = l1 ? (long long)K.tail_tiles[0] * K.n_chunks_f[0] * kComps * tb : 0;
    m.base = J.partials_f + foff + (long long)it.fine * tb;
    m.comp_stride = (size_t)(l1 ? K.tail_tiles[1] : K.tail_tiles[0]) * tb;
    m.room = J.fine_cap - foff;
  }
  m.chunk_stride = (size_t)kComps * m.comp_stride;
  return m;
}
// Compensated (Kahan) add of x into sum with compensation cmp.
__device__ __forceinline__ void kahan_add(float* sum, float* cmp, float x) {
  const float y = __fsub_rn(x, *cmp);
  const float tt = __fadd_rn(*sum, y);
  *cmp = __fsub_rn(__fsub_rn(tt, *sum), y);
  *sum = tt;
}

// Whether an item's chunks fit the partial-sum buffer it writes.
__device__ __forceinline__ bool part_fits(const JobStatic& J, const ItemRef& it, const PartMap& m) {
  return m.room >= (long long)it.n_chunks * (long long)m.chunk_stride;
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Reference time of a wide call's particle group (the group holding particle
// kt) seen from direction d: -n . (r_group - r_ref) / c.
__device__ __forceinline__ double group_tau(const JobStatic& J, long long kt, int d) {
  const double* D = J.gref + 3 * (kt / kGroup);
  const double* nd = J.dirs + 3 * d;
  return -(nd[0] * D[0] + nd[1] * D[1] + nd[2] * D[2]) * kInvC;
}

// Loads kn raw particle records; thread 0 only.
__device__ __forceinline__ void issue_tile(const JobStatic& J, long long k0, int kn, float* raw,
                                           uint64_t* bar) {
  // (skipped in a debug build when out of range: the block's bounded wait then gives up)
  if (!bounds_ok(k0 + kn <= J.n_cap, J.status)) return;
  tma_load_1d(raw, J.rec + (size_t)k0 * kRecFields, (uint32_t)kn * kRecFields * sizeof(float), bar);
}

// Loads the tile at position `next` of the item, if there is one: it ends with
// its chunk (c_end: the current chunk's end).
__device__ __forceinline__ void issue_next(const JobStatic& J, const ItemShared& si, int next, int c_end,
                                           int KT, float* raw, uint64_t* bar) {
  if (next >= si.n_item) return;
  const int end = next == c_end ? min(c_end + si.it.ck, si.n_item) : c_end;
  issue_tile(J, si.k_begin + next, min(KT, end - next), raw, bar);
}

// ------------------------------------------------------------ FP32 variant
// LIT: also the paper's literal sum P_i += sqrt(w) dt a_i g e^{i phi} with
// g = sqrt(1 + (w - 1) f(omega)^2), i.e. F_k(omega) dt a_i (Eq. 13 with Eq. 12).
template <int THREADS, int W, int UNROLL, bool LIT = false, bool WIDE = false>
__device__ __forceinline__ bool process_item_fma(const JobStatic& J, const JobCall& K,
                                                 const ItemRef& item0, const ItemShared& si,
                                                 unsigned char* __restrict__ smem, uint64_t* bar,
                                                 uint32_t& phase) {
  const int tile = item0.tile;
  constexpr int NP = W / 2;
  constexpr int REC = LIT ? 4 : 3;                 // float4 per record
  constexpr int NC = kComps + (LIT ? 4 : 0);       // accumulated components per frequency
  using S = Smem<THREADS, false, LIT>;
  float* raw = reinterpret_cast<float*>(smem);
  const TileGeom g = tile_geom(J, tile, THREADS);
  const int lanes_per_dir = g.WT / W;
  const int my_dl = threadIdx.x / lanes_per_dir;
  const int my_d_raw = g.d0 + my_dl;
  const int my_d = min(my_d_raw, J.n_dir - 1);
  const int om_first = g.o0 + (threadIdx.x - my_dl * lanes_per_dir) * W;
  const int n_om = J.n_omega;
  const int s1_dl = threadIdx.x / g.KT, s1_kk = threadIdx.x - s1_dl * g.KT;
  const int s1_d = min(g.d0 + s1_dl, J.n_dir - 1);
  // WIDE: a wide call, whose records are relative to their group's reference point.
  constexpr bool wide = WIDE;

  float2 omh[NP], wh[NP], wl[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const int i0 = min(om_first + 2 * p, n_om - 1), i1 = min(om_first + 2 * p + 1, n_om - 1);
    omh[p] = make_float2(__ldg(J.om_tab + i0), __ldg(J.om_tab + i1));
    wh[p] = make_float2(__ldg(J.om_tab + n_om + i0), __ldg(J.om_tab + n_om + i1));
    wl[p] = make_float2(__ldg(J.om_tab + 2 * n_om + i0), __ldg(J.om_tab + 2 * n_om + i1));
  }
  float2 f2[NP];
  if (LIT) {
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const int i0 = min(om_first + 2 * p, n_om - 1), i1 = min(om_first + 2 * p + 1, n_om - 1);
      f2[p] = make_float2(__ldg(J.f2_tab + i0), __ldg(J.f2_tab + i1));
    }
  }
  float2 acc1[NP][NC], acc2[NP][NC];
#pragma unroll
  for (int p = 0; p < NP; ++p)
#pragma unroll
    for (int c = 0; c < NC; ++c) acc1[p][c] = acc2[p][c] = make_float2(0.f, 0.f);
  const float2 kOne = make_float2(1.0f, 1.0f);

  // The item's particles are walked in tiles of at most KT that end with their
  // chunk (c_end; positions from the item's first particle).
  int pos = 0, c_end;
  {
    const long long k_begin = (long long)item0.chunk * item0.ck;
    c_end = (int)min((long long)item0.ck, K.n - k_begin);
    if (threadIdx.x == 0) issue_tile(J, k_begin, min(g.KT, c_end), raw, bar);
  }
  const int nb = J.n_bins;
  do {
    const int kn = min(g.KT, c_end - pos);
    float4* rec = reinterpret_cast<float4*>(smem + S::raw_bytes + (size_t)phase * S::rec_bytes);
    const bool landed = mbar_wait(bar, phase);
    phase ^= 1u;
    bool slow = false;
    if (landed && s1_kk < kn) {
      float th, tl, a[4];
      slow = !compute_record(raw + s1_kk * kRecFields, J.dir_tab, J.n_dir, s1_d, J.tau_fast, th,
                             tl, a);
      float4* out = rec + (s1_kk * g.NT + s1_dl) * REC;
      out[0] = make_float4(th, th, tl, tl);
      out[1] = make_float4(a[0], a[0], a[1], a[1]);
      out[2] = make_float4(a[2], a[2], a[3], a[3]);
      if (LIT) {
        const float wm1 = raw[s1_kk * kRecFields + 18];
        out[REC - 1] = make_float4(wm1, wm1, 0.f, 0.f);
      }
    }
    const int flags = __syncthreads_or((slow ? 1 : 0) | (landed ? 0 : 2));
    if (flags & 2) {
      // The copy did not land within the bound: record it, wait (bounded) once
      // more for that copy, and leave.
      if (threadIdx.x == 0) {
        atomicOr(J.status, ST_TIMEOUT);
        mbar_wait(bar, phase ^ 1u);
      }
      return false;
    }
    if (threadIdx.x == 0) issue_next(J, si, pos + kn, c_end, g.KT, raw, bar);
    const float4* rc = rec + my_dl * REC;
    if (!(flags & 1)) {
      // kend particles at a record stride of nt; a full tile of one direction
      // instantiates it with both known at compile time.
      auto fast_loop = [&](const int kend, const int nt) {
#pragma unroll UNROLL
      for (int kk = 0; kk < kend; ++kk) {
        const float4 r0 = rc[kk * nt * REC + 0];
        const float4 r1 = rc[kk * nt * REC + 1];
        const float4 r2 = rc[kk * nt * REC + 2];
        const float2 th = make_float2(r0.x, r0.y), tl = make_float2(r0.z, r0.w);
        const float2 aw1 = make_float2(r1.x, r1.y), aw2 = make_float2(r1.z, r1.w);
        const float2 av1 = make_float2(r2.x, r2.y), av2 = make_float2(r2.z, r2.w);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          const float2 ph = phase2(omh[p], wh[p], wl[p], th, tl);
          const float2 cc = make_float2(cos_approx(ph.x), cos_approx(ph.y));
          const float2 ss = make_float2(sin_approx(ph.x), sin_approx(ph.y));
          acc1[p][0] = __ffma2_rn(aw1, cc, acc1[p][0]);
          acc1[p][1] = __ffma2_rn(aw1, ss, acc1[p][1]);
          acc1[p][2] = __ffma2_rn(aw2, cc, acc1[p][2]);
          acc1[p][3] = __ffma2_rn(aw2, ss, acc1[p][3]);
          acc1[p][4] = __ffma2_rn(av1, cc, acc1[p][4]);
          acc1[p][5] = __ffma2_rn(av1, ss, acc1[p][5]);
          acc1[p][6] = __ffma2_rn(av2, cc, acc1[p][6]);
          acc1[p][7] = __ffma2_rn(av2, ss, acc1[p][7]);
          if (LIT) {
            const float4 r3 = rc[kk * nt * REC + REC - 1];
            const float2 g2 = __ffma2_rn(make_float2(r3.x, r3.y), f2[p], kOne);
            const float2 gg = make_float2(sqrt_approx(g2.x), sqrt_approx(g2.y));
            const float2 pv1 = __fmul2_rn(av1, gg), pv2 = __fmul2_rn(av2, gg);
            acc1[p][NC - 4] = __ffma2_rn(pv1, cc, acc1[p][NC - 4]);
            acc1[p][NC - 3] = __ffma2_rn(pv1, ss, acc1[p][NC - 3]);
            acc1[p][NC - 2] = __ffma2_rn(pv2, cc, acc1[p][NC - 2]);
            acc1[p][NC - 1] = __ffma2_rn(pv2, ss, acc1[p][NC - 1]);
          }
        }
      }
      };
      if (g.NT == 1 && kn == THREADS) fast_loop(THREADS, 1);
      else fast_loop(kn, g.NT);
    } else {
      // Wide path: some |dtau| exceed the fast range in this tile; the phase of
      // every update is formed in FP64.
      if (threadIdx.x == 0) atomicOr(J.status, ST_SLOW_PHASE);
      double tau_g = 0.0;
      if constexpr (wide) tau_g = group_tau(J, si.k_begin + pos, my_d);
      double omt[W];
#pragma unroll
      for (int i = 0; i < W; ++i) omt[i] = J.om_turns[min(om_first + i, n_om - 1)];
      for (int kk = 0; kk < kn; ++kk) {
        const float4 r0 = rc[kk * g.NT * REC + 0];
        const float4 r1 = rc[kk * g.NT * REC + 1];
        const float4 r2 = rc[kk * g.NT * REC + 2];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          const float2 ph = make_float2(phase_wide(omt[2 * p], r0.x, r0.z, tau_g),
                                        phase_wide(omt[2 * p + 1], r0.x, r0.z, tau_g));
          const float2 cc = make_float2(cos_approx(ph.x), cos_approx(ph.y));
          const float2 ss = make_float2(sin_approx(ph.x), sin_approx(ph.y));
          acc1[p][0] = __ffma2_rn(make_float2(r1.x, r1.y), cc, acc1[p][0]);
          acc1[p][1] = __ffma2_rn(make_float2(r1.x, r1.y), ss, acc1[p][1]);
          acc1[p][2] = __ffma2_rn(make_float2(r1.z, r1.w), cc, acc1[p][2]);
          acc1[p][3] = __ffma2_rn(make_float2(r1.z, r1.w), ss, acc1[p][3]);
          acc1[p][4] = __ffma2_rn(make_float2(r2.x, r2.y), cc, acc1[p][4]);
          acc1[p][5] = __ffma2_rn(make_float2(r2.x, r2.y), ss, acc1[p][5]);
          acc1[p][6] = __ffma2_rn(make_float2(r2.z, r2.w), cc, acc1[p][6]);
          acc1[p][7] = __ffma2_rn(make_float2(r2.z, r2.w), ss, acc1[p][7]);
          if (LIT) {
            const float4 r3 = rc[kk * g.NT * REC + REC - 1];
            const float2 g2 = __ffma2_rn(make_float2(r3.x, r3.y), f2[p], kOne);
            const float2 gg = make_float2(sqrt_approx(g2.x), sqrt_approx(g2.y));
            const float2 pv1 = __fmul2_rn(make_float2(r2.x, r2.y), gg);
            const float2 pv2 = __fmul2_rn(make_float2(r2.z, r2.w), gg);
            acc1[p][NC - 4] = __ffma2_rn(pv1, cc, acc1[p][NC - 4]);
            acc1[p][NC - 3] = __ffma2_rn(pv1, ss, acc1[p][NC - 3]);
            acc1[p][NC - 2] = __ffma2_rn(pv2, cc, acc1[p][NC - 2]);
            acc1[p][NC - 1] = __ffma2_rn(pv2, ss, acc1[p][NC - 1]);
          }
        }
      }
    }
    // Wide call, fast path: the tile's sums are relative to its group's
    // reference; rotate them by e^{i omega tau_g} (the FP64 path above already
    // has tau_g in every phase).
    if constexpr (wide) {
      if (!(flags & 1)) {
        const double tau_g = group_tau(J, si.k_begin + pos, my_d);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          float2 cs, sn;
          group_rotation(J.om_turns[min(om_first + 2 * p, n_om - 1)], tau_g, cs.x, sn.x);
          group_rotation(J.om_turns[min(om_first + 2 * p + 1, n_om - 1)], tau_g, cs.y, sn.y);
#pragma unroll
          for (int c = 0; c < NC; c += 2) {
            const float2 re = acc1[p][c], im = acc1[p][c + 1];
            acc1[p][c] = __ffma2_rn(re, cs, __fmul2_rn(make_float2(-im.x, -im.y), sn));
            acc1[p][c + 1] = __ffma2_rn(re, sn, __fmul2_rn(im, cs));
          }
        }
      }
    }
    // Two-level summation: the tile's sums join the chunk sums.
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        acc2[p][c] = __fadd2_rn(acc2[p][c], acc1[p][c]);
        acc1[p][c] = make_float2(0.f, 0.f);
      }
    pos += kn;
    if (pos < c_end) continue;
    const int chunk = si.it.chunk + (pos - 1) / si.it.ck;
    // The chunk's partial sums.  (FP32 variants never take fine-chunked tiles,
    // TailPlan: their items write the coarse partials directly, which keeps the
    // fine tiles' bookkeeping out of this loop's registers.)
    float* part = J.partials + (size_t)chunk * kComps * nb;
    float* part_p = LIT ? J.partials_p + (size_t)chunk * 4 * nb : nullptr;
    const size_t cs = nb, off = (size_t)my_d * n_om + om_first;
    if (my_d_raw < J.n_dir) {
#pragma unroll
      for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int o = om_first + 2 * p + e;
          if (o < n_om && bounds_ok((chunk + 1) * (long long)(kComps * cs) <= J.part_cap && si.it.fine < 0, J.status)) {
#pragma unroll
            for (int c = 0; c < kComps; ++c)
              part[(size_t)c * cs + off + 2 * p + e] = e ? acc2[p][c].y : acc2[p][c].x;
            if (LIT) {
#pragma unroll
              for (int c = 0; c < 4; ++c)
                part_p[(size_t)c * cs + off + 2 * p + e] = e ? acc2[p][NC - 4 + c].y : acc2[p][NC - 4 + c].x;
            }
          }
        }
    }
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
      for (int c = 0; c < NC; ++c) acc2[p][c] = make_float2(0.f, 0.f);
    c_end = min(c_end + si.it.ck, si.n_item);
  } while (pos < si.n_item);
  return true;
}

// ------------------------------------------------------ tensor-core variant
// Warp layout: warp w handles direction d0 + w / (WT/(16 NB)) and 16 NB
// frequencies (NB 16-row MMA blocks) starting at o0 + 16 NB (w % (WT/(16 NB))).
// XT: the phases' cross terms 2pi (omega_lo th + omega_hi tl) come from one
// more MMA per block (below), and the phase arithmetic is packed over particle
// pairs instead of frequency pairs.
template <int THREADS, int PASSES, int NB, bool WIDE = false, bool XT = false>
__device__ __forceinline__ bool process_item_tc(const JobStatic& J, const JobCall& K,
                                                const ItemRef& item0, const ItemShared& si,
                                                unsigned char* __restrict__ smem, uint64_t* bar,
                                                uint32_t& phase) {
  const int tile = item0.tile;
  // NB: 16-frequency blocks per warp; GQ: second-level float4 groups per pass
  constexpr int GQ = 2 * NB;
  using S = Smem<THREADS, true, false, PASSES * NB / 2, XT>;
  float* raw = reinterpret_cast<float*>(smem);
  const TileGeom g = tile_geom(J, tile, THREADS);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = lane >> 2, c = lane & 3;
  // The tile's frequencies are swept in PASSES passes of PW over the same
  // staged particle records (one stage 1 and one barrier per tile and pass set).
  const int PW = g.WT / PASSES;
  const int warps_per_dir = PW / (16 * NB);
  const int my_dl = warp / warps_per_dir;
  const int my_d_raw = g.d0 + my_dl;
  const int my_d = min(my_d_raw, J.n_dir - 1);
  const int o_warp0 = g.o0 + (warp - my_dl * warps_per_dir) * 16 * NB;
  const int n_om = J.n_omega;
  const int s1_dl = threadIdx.x / g.KT, s1_kk = threadIdx.x - s1_dl * g.KT;
  const int s1_d = min(g.d0 + s1_dl, J.n_dir - 1);
  // WIDE: a wide call, whose records are relative to their group's reference point.
  constexpr bool wide = WIDE;

  // The item's particles are walked in tiles of at most KT that end with their
  // chunk (c_end; positions from the item's first particle).
  int pos = 0, c_end;
  {
    const long long k_begin = (long long)item0.chunk * item0.ck;
    c_end = (int)min((long long)item0.ck, K.n - k_begin);
    if (threadIdx.x == 0) issue_tile(J, k_begin, min(g.KT, c_end), raw, bar);
  }
  // XT: the tile's direction rows, staged once per item for stage 1 (the
  // previous item's last reads of them precede its closing barriers).
  float* sdir = reinterpret_cast<float*>(smem + S::raw_bytes + 2 * S::rec_bytes + S::l2_bytes);
  if constexpr (XT) {
    for (int t = threadIdx.x; t < 12 * g.NT; t += THREADS) {
      const int dl = t / 12, k = t - dl * 12;
      sdir[t] = __ldg(J.dir_tab + (size_t)k * J.n_dir + min(g.d0 + dl, J.n_dir - 1));
    }
  }

  float2 omh[NB], wh[NB], wl[NB];
  // XT: omega/2pi (hi) of rows r and r + 8 of each block, each in both halves
  // of a pair, and the A fragment of the cross-term product.  That product has
  // eight terms t (A columns, B rows), with x ~ x_hi + x_lo split into TF32
  // values:  t = 0..7: wl_hi th_hi, wl_hi th_lo, wl_lo th_hi, wh_hi tl_hi,
  // wh_hi tl_lo, wh_lo tl_hi, wl_lo th_lo, wh_lo tl_lo  (wh, wl: 2pi omega hi
  // and lo in radians; th, tl: the particle's dtau hi and lo), which sum to
  // wl th + wh tl.
  float2 omr[NB], omr8[NB];
  uint32_t xa[NB][4];
  auto load_omega = [&](int o_warp) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int i0 = min(o_warp + 16 * b + r, n_om - 1), i1 = min(o_warp + 16 * b + r + 8, n_om - 1);
      if constexpr (XT) {
        const float h0 = __ldg(J.om_tab + i0), h1 = __ldg(J.om_tab + i1);
        omr[b] = make_float2(h0, h0);
        omr8[b] = make_float2(h1, h1);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int i = h ? i1 : i0;
          uint32_t whh, whl, wlh, wll;
          split_tf32(__ldg(J.om_tab + n_om + i), whh, whl);
          split_tf32(__ldg(J.om_tab + 2 * n_om + i), wlh, wll);
          // a0/a1: column c of rows r / r + 8; a2/a3: column c + 4.
          xa[b][h] = c == 3 ? whh : (c == 2 ? wll : wlh);
          xa[b][2 + h] = c == 0 ? whh : (c == 2 ? wll : whl);
        }
      } else {
        omh[b] = make_float2(__ldg(J.om_tab + i0), __ldg(J.om_tab + i1));
        wh[b] = make_float2(__ldg(J.om_tab + n_om + i0), __ldg(J.om_tab + n_om + i1));
        wl[b] = make_float2(__ldg(J.om_tab + 2 * n_om + i0), __ldg(J.om_tab + 2 * n_om + i1));
      }
    }
  };
  load_omega(o_warp0);
  float dre[NB][4], dim[NB][4];
  // second-level sums of pass p: group q (q = b for the real parts of block b,
  // NB + b for the imaginary parts) of this thread at l2[(p * GQ + q) * THREADS + threadIdx.x]
  float4* l2 = reinterpret_cast<float4*>(smem + S::raw_bytes + 2 * S::rec_bytes);
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int e = 0; e < 4; ++e) dre[b][e] = dim[b][e] = 0.0f;

#pragma unroll
  for (int v = 0; v < GQ * PASSES; ++v) l2[v * THREADS + threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (XT) __syncthreads();
  do {
    const int kn = min(g.KT, c_end - pos);
    unsigned char* recb = smem + S::raw_bytes + (size_t)phase * S::rec_bytes;
    float2* tau2 = reinterpret_cast<float2*>(recb);                     // [NT][KT]
    float* ampb = reinterpret_cast<float*>(recb + (size_t)THREADS * 8);  // [NT][KT][8]
    // XT records: dtau hi [NT][KT]; the cross-term B rows [NT][KT][8] as four
    // pairs (terms c, c + 4), pair c of particle p at position c ^ 2 ((p >> 2) & 1)
    // (lane c reads its pair with one 8-byte load); the amplitudes' hi/lo parts
    // [NT][KT][12], 8 used.  The swizzle and the 12-word stride keep both the
    // stage-1 stores and the loop's loads free of bank conflicts.
    float* xth = reinterpret_cast<float*>(recb);
    float* xrt = reinterpret_cast<float*>(recb + (size_t)THREADS * 4);
    float* xam = reinterpret_cast<float*>(recb + (size_t)THREADS * 36);
    const bool landed = mbar_wait(bar, phase);
    phase ^= 1u;
    bool slow = false;
    if (landed) {
      float th = 0.f, tl = 0.f, a[4] = {0.f, 0.f, 0.f, 0.f};
      if (s1_kk < kn) {
        if constexpr (XT)
          slow = !compute_record(raw + s1_kk * kRecFields, dir_row_staged(sdir + 12 * s1_dl),
                                 J.tau_fast, th, tl, a);
        else
          slow = !compute_record(raw + s1_kk * kRecFields, J.dir_tab, J.n_dir, s1_d, J.tau_fast,
                                 th, tl, a);
      }
      // Particles past kn are zero padding of the last 8-particle MMA step.
      if constexpr (XT) {
        store_record_xt(th, tl, a, s1_kk, xth + s1_dl * g.KT, xrt + (size_t)s1_dl * g.KT * 8,
                        xam + (size_t)s1_dl * g.KT * 12);
      } else {
        const int slot = s1_dl * g.KT + s1_kk;
        const uint32_t h0 = tf32_hi(a[0]), h1 = tf32_hi(a[1]), h2 = tf32_hi(a[2]), h3 = tf32_hi(a[3]);
        tau2[slot] = make_float2(th, tl);
        float4* ap = reinterpret_cast<float4*>(ampb + (size_t)slot * 8);
        ap[0] = make_float4(__uint_as_float(h0), __uint_as_float(h1), __uint_as_float(h2),
                            __uint_as_float(h3));
        ap[1] = make_float4(a[0] - __uint_as_float(h0), a[1] - __uint_as_float(h1),
                            a[2] - __uint_as_float(h2), a[3] - __uint_as_float(h3));
      }
    }
    const int flags = __syncthreads_or((slow ? 1 : 0) | (landed ? 0 : 2));
    if (flags & 2) {
      if (threadIdx.x == 0) {
        atomicOr(J.status, ST_TIMEOUT);
        mbar_wait(bar, phase ^ 1u);
      }
      return false;
    }
    if (threadIdx.x == 0) issue_next(J, si, pos + kn, c_end, g.KT, raw, bar);
    const float2* tw = tau2 + my_dl * g.KT;
    const float* aw = ampb + (size_t)my_dl * g.KT * 8;
    const float* xtw = xth + my_dl * g.KT;
    const float* xrw = xrt + (size_t)my_dl * g.KT * 8;
    const float* xaw = xam + (size_t)my_dl * g.KT * 12;
    // this lane's cross-term pair within particle kk + r's row (kk % 8 == 0)
    const int xr_off = 2 * (c ^ ((r >> 1) & 2));
    // XT, the 8-particle step at kk: the main product's k = c and k = c + 4 are
    // particles kk + 2c and kk + 2c + 1 (the columns of the cross-term result
    // this lane holds).
    auto xamp = [&](int kk) {
      return make_uint2(__float_as_uint(xaw[(kk + 2 * c) * 12 + r]),
                        __float_as_uint(xaw[(kk + 2 * c + 1) * 12 + r]));
    };
    const int kn8 = (kn + 7) & ~7;
#pragma unroll 1
    for (int ps = 0; ps < PASSES; ++ps) {
      const int o_warp = o_warp0 + ps * PW;
      if (PASSES > 1) load_omega(o_warp);
      if (!(flags & 1)) {
        // Unrolled 2x with two 16-frequency blocks per warp, 16x with four (LWFA step: 8x 6.88 ms, 16x 6.82).
        constexpr int kUnroll = NB >= 4 ? 16 : 2;
        auto fast_loop = [&](const int kend) {
#pragma unroll kUnroll
          for (int kk = 0; kk < kend; kk += 8) {
            if constexpr (XT) {
              const float2 th2 = *reinterpret_cast<const float2*>(xtw + kk + 2 * c);
              const uint2 rt = *reinterpret_cast<const uint2*>(xrw + (size_t)(kk + r) * 8 + xr_off);
              const uint2 bb = xamp(kk);
              // cr: rows r, r + 8 x particles kk + 2c, kk + 2c + 1.  All blocks'
              // products first: one block's wait covers the next (0.1-1.3 % of a call).
              float cr[NB][4];
#pragma unroll
              for (int b = 0; b < NB; ++b)
                mma_tf32_zero(cr[b], xa[b][0], xa[b][1], xa[b][2], xa[b][3], rt.x, rt.y);
#pragma unroll
              for (int b = 0; b < NB; ++b) {
                const float2 p0 = phase2x(omr[b], th2, make_float2(cr[b][0], cr[b][1]));
                const float2 p8 = phase2x(omr8[b], th2, make_float2(cr[b][2], cr[b][3]));
                tc_block(make_float2(p0.x, p8.x), make_float2(p0.y, p8.y), bb.x, bb.y, dre[b],
                         dim[b]);
              }
              continue;
            }
            const float2 tA = tw[kk + c], tB = tw[kk + c + 4];
            const uint32_t b0 = __float_as_uint(aw[(kk + c) * 8 + r]);
            const uint32_t b1 = __float_as_uint(aw[(kk + c + 4) * 8 + r]);
            const float2 thA = make_float2(tA.x, tA.x), tlA = make_float2(tA.y, tA.y);
            const float2 thB = make_float2(tB.x, tB.x), tlB = make_float2(tB.y, tB.y);
#pragma unroll
            for (int b = 0; b < NB; ++b) {
              const float2 pA = phase2(omh[b], wh[b], wl[b], thA, tlA);
              const float2 pB = phase2(omh[b], wh[b], wl[b], thB, tlB);
              tc_block(pA, pB, b0, b1, dre[b], dim[b]);
            }
          }
        };
        // Full tiles of one and two directions take the loop with its trip count
        // known at compile time (LWFA step, two directions: 4880 -> 4726 us);
        // ragged and narrower tiles the runtime bound.
        if (kn8 == THREADS) fast_loop(THREADS);
        else if (kn8 == THREADS / 2) fast_loop(THREADS / 2);
        else fast_loop(kn8);
      } else {
        if (threadIdx.x == 0) atomicOr(J.status, ST_SLOW_PHASE);
        double tau_g = 0.0;
        if constexpr (wide) tau_g = group_tau(J, si.k_begin + pos, my_d);
        double omt[NB][2];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          omt[b][0] = J.om_turns[min(o_warp + 16 * b + r, n_om - 1)];
          omt[b][1] = J.om_turns[min(o_warp + 16 * b + r + 8, n_om - 1)];
        }
        for (int kk = 0; kk < kn8; kk += 8) {
          float2 tA, tB;
          uint32_t b0, b1;
          if constexpr (XT) {
            // particles kk + 2c and kk + 2c + 1; tl = tl_hi + tl_lo (terms 3, 7:
            // pair 3, at position 3 ^ 2 ((p >> 2) & 1))
            const int pa = kk + 2 * c;
            auto tl_of = [&](int p) {
              const float* q = xrw + (size_t)p * 8 + 2 * (3 ^ (((p >> 2) & 1) << 1));
              return q[0] + q[1];
            };
            tA = make_float2(xtw[pa], tl_of(pa));
            tB = make_float2(xtw[pa + 1], tl_of(pa + 1));
            const uint2 bb = xamp(kk);
            b0 = bb.x;
            b1 = bb.y;
          } else {
            tA = tw[kk + c];
            tB = tw[kk + c + 4];
            b0 = __float_as_uint(aw[(kk + c) * 8 + r]);
            b1 = __float_as_uint(aw[(kk + c + 4) * 8 + r]);
          }
#pragma unroll
          for (int b = 0; b < NB; ++b) {
            const float2 pA = make_float2(phase_wide(omt[b][0], tA.x, tA.y, tau_g),
                                          phase_wide(omt[b][1], tA.x, tA.y, tau_g));
            const float2 pB = make_float2(phase_wide(omt[b][0], tB.x, tB.y, tau_g),
                                          phase_wide(omt[b][1], tB.x, tB.y, tau_g));
            tc_block(pA, pB, b0, b1, dre[b], dim[b]);
          }
        }
      }
      // Wide call, fast path: rotate the tile's sums by e^{i omega tau_g}.  The
      // warp's 16 NB frequencies are shared out: lane L reduces the phases of
      // frequencies L and L + 32 of the warp's range in FP64 (FP64 is narrow on
      // this GPU), and each lane takes the factors of its rows r and r + 8 of
      // every block from their owners by shuffles.
      if constexpr (wide) {
        if (!(flags & 1)) {
          const double tau_g = group_tau(J, si.k_begin + pos, my_d);
          float cA, sA, cB = 1.0f, sB = 0.0f;
          group_rotation(J.om_turns[min(o_warp + lane, n_om - 1)], tau_g, cA, sA);
          if constexpr (NB > 2)
            group_rotation(J.om_turns[min(o_warp + lane + 32, n_om - 1)], tau_g, cB, sB);
#pragma unroll
          for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int src = (16 * b + r + 8 * h) & 31;
              const float cs = __shfl_sync(0xffffffffu, b < 2 ? cA : cB, src);
              const float sn = __shfl_sync(0xffffffffu, b < 2 ? sA : sB, src);
#pragma unroll
              for (int e = 2 * h; e < 2 * h + 2; ++e) {
                const float re = dre[b][e], im = dim[b][e];
                dre[b][e] = fmaf(re, cs, -im * sn);
                dim[b][e] = fmaf(re, sn, im * cs);
              }
            }
        }
      }
      // Second level: after every particle tile the tile sums join the chunk
      // sums in shared memory, so the MMA accumulators never sum more than one
      // tile.  Longer runs would be faster (LWFA workload, variant 9: a flush
      // every second tile 0.2 % and every fourth 0.5 % less time per step) but
      // the MMA's FP32 accumulation error grows with the run's length: at every
      // fourth tile a 5000-particle workload read 1.3e-5 of row error against
      // the oracle (gate 1e-5), about four times that of a flush every tile.
      float4* l2p = l2 + ps * GQ * THREADS + threadIdx.x;
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const float4 x = l2p[b * THREADS], y = l2p[(NB + b) * THREADS];
        const float2 x01 = __fadd2_rn(make_float2(x.x, x.y), make_float2(dre[b][0], dre[b][1]));
        const float2 x23 = __fadd2_rn(make_float2(x.z, x.w), make_float2(dre[b][2], dre[b][3]));
        const float2 y01 = __fadd2_rn(make_float2(y.x, y.y), make_float2(dim[b][0], dim[b][1]));
        const float2 y23 = __fadd2_rn(make_float2(y.z, y.w), make_float2(dim[b][2], dim[b][3]));
        l2p[b * THREADS] = make_float4(x01.x, x01.y, x23.x, x23.y);
        l2p[(NB + b) * THREADS] = make_float4(y01.x, y01.y, y23.x, y23.y);
#pragma unroll
        for (int e = 0; e < 4; ++e) dre[b][e] = dim[b][e] = 0.0f;
      }
    }
    pos += kn;
    if (pos < c_end) continue;
    // The chunk's partial sums.  The D fragment holds rows (r, r+8) and columns
    // (2c, 2c+1); columns 0-3 are the hi parts of (U.e1, U.e2, V.e1, V.e2),
    // columns 4-7 the lo parts: lane c (c < 2) adds lane c+2's values.  One base
    // pointer per column and part, the rows at constant offsets.
    {
      const int chunk = si.it.chunk + (pos - 1) / si.it.ck;
      const PartMap pm = part_map(J, K, si.it, g);
      float* part = pm.base + (size_t)chunk * pm.chunk_stride;
      const size_t cs = pm.comp_stride;
      // (32 bits, enough for 2^31 bins: in 64 the loop above spills differently, and 20000
      // particles, 250 x 40 bins take 159.0 us instead of 156.9; the wide pass the other
      // way round, 2064 us instead of 2035 for 1e5 particles over 2 mm, 512 x 64 bins)
      using Off = std::conditional_t<WIDE, size_t, unsigned>;
      const Off off = si.it.fine < 0 ? (Off)my_d * (Off)J.part_row + (Off)o_warp0
                                     : (Off)(my_dl * g.WT + (o_warp0 - g.o0));
      float* q = part + off + r + (size_t)(4 * c) * cs;
      const int left = n_om - o_warp0 - r;  // rows past the grid are not written
      const bool mine = c < 2 && my_d_raw < J.n_dir &&
                        bounds_ok(chunk < si.it.n_chunks && part_fits(J, si.it, pm), J.status);
#pragma unroll 1
      for (int ps = 0; ps < PASSES; ++ps)
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const float4 re4 = l2[(ps * GQ + b) * THREADS + threadIdx.x];
          const float4 im4 = l2[(ps * GQ + NB + b) * THREADS + threadIdx.x];
          const float re[4] = {re4.x, re4.y, re4.z, re4.w}, im[4] = {im4.x, im4.y, im4.z, im4.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float vr = re[e] + __shfl_xor_sync(0xffffffffu, re[e], 2);
            const float vi = im[e] + __shfl_xor_sync(0xffffffffu, im[e], 2);
            const int row = ps * PW + 16 * b + ((e >> 1) << 3);
            if (mine && row < left) {  // amplitude column 2c + (e & 1)
              q[(size_t)(2 * (e & 1)) * cs + row] = vr;
              q[(size_t)(2 * (e & 1) + 1) * cs + row] = vi;
            }
          }
        }
    }
    c_end = min(c_end + si.it.ck, si.n_item);
    if (pos < si.n_item)
#pragma unroll
      for (int v = 0; v < GQ * PASSES; ++v) l2[v * THREADS + threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
  } while (pos < si.n_item);
  return true;
}

// ------------------------------------------------------------------ low band
// One item of a call's low band (LowSet): 8 directions, one per warp, and a chunk
// of the cell-sorted particles.  A warp's 64 frequencies are the nodes; its
// records are relative to the cell's centre and weighted by the interpolation's
// particle-side factor.  Warps share only the raw particles (two buffers of
// kLowTile, one barrier each): every warp computes its own direction's
// records.  At a cell's end the warp interpolates its node sums to the
// band's bins, rotates them by e^{i omega tau_c} (tau_c the centre's time) and
// adds them to the chunk's sums.  Bound: MUFU, as the direct bins, for 64
// frequencies instead of js; the interpolation is 10 taps x 8 sums per bin and
// cell.  LWFA step (1e5 particles, 512 x 256 bins, 256 bins from nodes): 6.79 ->
// 4.73 ms; 1e6 particles, 1024 x 256 bins (512 from nodes) 132.2 -> 76.4 ms.
constexpr int kLowTile = 128;
constexpr int kLowDirs = 8;

struct LowTile {
  long long pos;  // first particle (sorted)
  int kn, cell;
  int last;       // ends its cell or the chunk
};

// The tile from pos in `cell`, whose particles end at cell_end.
__device__ __forceinline__ LowTile low_tile(long long pos, long long cell_end, int cell) {
  LowTile t;
  t.pos = pos;
  t.kn = (int)min((long long)kLowTile, cell_end - pos);
  t.cell = cell;
  t.last = pos + t.kn == cell_end;
  return t;
}

// Particle-side factor of the interpolation, 1 / (the window's Fourier transform
// at x / (2 kLowOversample), x = tau / H): a polynomial in x^2 fitted to
// quadratures of the transform (relative error 1e-7 in FP32 on |x| <= 1).  Only
// records of invalid particles, of zero weight, lie outside: kept finite.
__device__ __forceinline__ float low_factor(float x) {
  const float y = fminf(x * x, 1.0f);
  float p = 0.00316812399f;
  p = fmaf(p, y, -0.00347217099f);
  p = fmaf(p, y, 0.0177691517f);
  p = fmaf(p, y, 0.0227779421f);
  p = fmaf(p, y, 0.0826435269f);
  p = fmaf(p, y, 0.189933115f);
  p = fmaf(p, y, 0.381905146f);
  p = fmaf(p, y, 0.599662798f);
  p = fmaf(p, y, 0.657055849f);
  return fmaf(p, y, 0.376632672f);
}

template <int THREADS>
__device__ __forceinline__ bool process_item_low(const JobStatic& J, const JobCall& K, const LowPlan& P,
                                                 const LowSet& L, int tile, int chunk, LowTile* desc,
                                                 unsigned char* __restrict__ smem, uint64_t* bars,
                                                 uint32_t& phases) {
  constexpr int NB = kLowNodes / 16, GQ = 2 * NB;
  static_assert(THREADS / 32 == kLowDirs, "one direction per warp");
  using S = Smem<THREADS, true, false, NB / 2, true>;
  static_assert(2 * kLowTile * kRecFields * sizeof(float) <= S::raw_bytes, "two raw tiles");
  static_assert(kLowDirs * kLowNodes * kComps * sizeof(float) <= S::rec_bytes, "node sums");
  float* raw = reinterpret_cast<float*>(smem);
  unsigned char* recb = smem + S::raw_bytes;
  float4* l2 = reinterpret_cast<float4*>(smem + S::raw_bytes + 2 * S::rec_bytes);
  float* sdir = reinterpret_cast<float*>(smem + S::raw_bytes + 2 * S::rec_bytes + S::l2_bytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = lane >> 2, c = lane & 3;
  float* ns = reinterpret_cast<float*>(smem + S::raw_bytes + S::rec_bytes) + warp * kLowNodes * kComps;
  float* xth = reinterpret_cast<float*>(recb) + warp * 32;
  float* xrt = reinterpret_cast<float*>(recb + (size_t)THREADS * 4) + warp * 32 * 8;
  float* xam = reinterpret_cast<float*>(recb + (size_t)THREADS * 36) + warp * 32 * 12;
  const int my_d = min(tile * kLowDirs + warp, J.n_dir - 1);
  const bool live = tile * kLowDirs + warp < J.n_dir;
  const int ck = K.low[P.set].ck_lo;
  const long long k0 = (long long)chunk * ck, k1 = min(k0 + ck, K.n);

  for (int t = lane; t < 12; t += 32) sdir[warp * 12 + t] = __ldg(J.dir_tab + (size_t)t * J.n_dir + my_d);
  auto issue = [&](const LowTile& t, int buf) {
    if (!bounds_ok(t.pos + t.kn <= J.rec_s_cap, J.status)) return;
    tma_load_1d(raw + (size_t)buf * kLowTile * kRecFields, J.rec_s + (size_t)t.pos * kRecFields,
                (uint32_t)t.kn * kRecFields * sizeof(float), &bars[buf]);
  };
  // first sorted position after the cell's particles, within the chunk
  auto cell_end = [&](int cell) {
    return cell + 1 < P.cells ? min((long long)J.bucket_base[cell + 1], k1) : k1;
  };
  if (threadIdx.x == 0) {
    int lo = 0, hi = P.cells - 1;  // the last cell that begins at or before k0
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (J.bucket_base[mid] <= k0) lo = mid;
      else hi = mid - 1;
    }
    desc[0] = low_tile(k0, cell_end(lo), lo);
    issue(desc[0], 0);
  }
  // the nodes' frequency factors, as load_omega's
  float2 omr[NB], omr8[NB];
  uint32_t xa[NB][4];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = 16 * b + r + 8 * h;
      const float h0 = __ldg(L.nodes + i);
      (h ? omr8 : omr)[b] = make_float2(h0, h0);
      uint32_t whh, whl, wlh, wll;
      split_tf32(__ldg(L.nodes + kLowNodes + i), whh, whl);
      split_tf32(__ldg(L.nodes + 2 * kLowNodes + i), wlh, wll);
      xa[b][h] = c == 3 ? whh : (c == 2 ? wll : wlh);
      xa[b][2 + h] = c == 0 ? whh : (c == 2 ? wll : whl);
    }
  }
  float dre[NB][4], dim[NB][4];
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int e = 0; e < 4; ++e) dre[b][e] = dim[b][e] = 0.0f;
#pragma unroll
  for (int v = 0; v < GQ; ++v) l2[v * THREADS + threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
  const int xr_off = 2 * (c ^ ((r >> 1) & 2));
  float* part = J.partials_l + (size_t)chunk * kComps * J.n_dir * L.js + (size_t)my_d * L.js;
  const size_t cs = (size_t)J.n_dir * L.js;
  const bool slot = bounds_ok((chunk + 1) * (long long)(kComps * cs) <= J.low_cap, J.status);
  bool first = true;  // the chunk's first cell starts its sums
  int cell = -1;
  float tch = 0.0f, tcl = 0.0f;
  const float inv_h = 1.0f / L.H;
  __syncthreads();
  for (int buf = 0;; buf ^= 1) {
    const LowTile t = desc[buf];
    // the next tile, into the other buffer (used up before the last barrier)
    const long long next = t.pos + t.kn;
    if (threadIdx.x == 0 && next < k1) {
      int nc = t.cell;
      long long ce = cell_end(nc);
      while (ce <= next) ce = cell_end(++nc);  // (past empty cells)
      desc[buf ^ 1] = low_tile(next, ce, nc);
      issue(desc[buf ^ 1], buf ^ 1);
    }
    if (t.cell != cell) {
      cell = t.cell;
      const double sc = (double)P.s0 + ((double)cell + 0.5) * (double)P.h;
      const double* nd = J.dirs + 3 * (size_t)my_d;
      double tc = 0.0;
#pragma unroll
      for (int i = 0; i < 3; ++i)
        tc -= nd[i] * ((double)P.c1 * J.fr1[i] + (double)P.c2 * J.fr2[i] + sc * J.axis[i]);
      split_ff(tc, tch, tcl);
    }
    const bool landed = mbar_wait(&bars[buf], (phases >> buf) & 1u);
    phases ^= 1u << buf;
    if (landed) {
      for (int s0 = 0; s0 < t.kn; s0 += 32) {
        const int kn = min(32, t.kn - s0);
        float th = 0.f, tl = 0.f, a[4] = {0.f, 0.f, 0.f, 0.f};
        if (lane < kn) {
          compute_record(raw + ((size_t)buf * kLowTile + s0 + lane) * kRecFields,
                         dir_row_staged(sdir + 12 * warp), J.tau_fast, th, tl, a);
          // relative to the cell's centre (TwoDiff)
          const float d = __fsub_rn(th, tch), bb = __fsub_rn(d, th);
          const float e = __fsub_rn(__fsub_rn(th, __fsub_rn(d, bb)), __fadd_rn(tch, bb));
          const float lo = __fadd_rn(e, __fsub_rn(tl, tcl));
          th = __fadd_rn(d, lo);
          tl = __fsub_rn(lo, __fsub_rn(th, d));
          const float f = low_factor(th * inv_h);
#pragma unroll
          for (int i = 0; i < 4; ++i) a[i] *= f;
        }
        store_record_xt(th, tl, a, lane, xth, xrt, xam);
        __syncwarp();
        const int kn8 = (kn + 7) & ~7;
        if (kn8 == 32) {
#pragma unroll
          for (int kk = 0; kk < 32; kk += 8)
            xt_step<NB>(xth, xrt, xam, kk, r, c, xr_off, omr, omr8, xa, dre, dim);
        } else {
#pragma unroll 1
          for (int kk = 0; kk < kn8; kk += 8)
            xt_step<NB>(xth, xrt, xam, kk, r, c, xr_off, omr, omr8, xa, dre, dim);
        }
        __syncwarp();
      }
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      float4* p = l2 + b * THREADS + threadIdx.x;
      float4* q = p + NB * THREADS;
      const float4 x = *p, y = *q;
      *p = make_float4(x.x + dre[b][0], x.y + dre[b][1], x.z + dre[b][2], x.w + dre[b][3]);
      *q = make_float4(y.x + dim[b][0], y.y + dim[b][1], y.z + dim[b][2], y.w + dim[b][3]);
#pragma unroll
      for (int e = 0; e < 4; ++e) dre[b][e] = dim[b][e] = 0.0f;
    }
    if (t.last && live && slot) {
      // node sums, hi and lo parts together (lane c < 2 holds columns 2c, 2c + 1)
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const float4 re4 = l2[b * THREADS + threadIdx.x], im4 = l2[(NB + b) * THREADS + threadIdx.x];
        l2[b * THREADS + threadIdx.x] = l2[(NB + b) * THREADS + threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
        const float re[4] = {re4.x, re4.y, re4.z, re4.w}, im[4] = {im4.x, im4.y, im4.z, im4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float vr = re[e] + __shfl_xor_sync(0xffffffffu, re[e], 2);
          const float vi = im[e] + __shfl_xor_sync(0xffffffffu, im[e], 2);
          if (c < 2)
            *reinterpret_cast<float2*>(ns + (16 * b + r + 8 * (e >> 1)) * kComps + 2 * (2 * c + (e & 1))) =
                make_float2(vr, vi);
        }
      }
      __syncwarp();
#pragma unroll 1
      for (int j = lane; j < L.js; j += 32) {
        const float4* wt = reinterpret_cast<const float4*>(L.wts + (size_t)j * kLowWt);
        const float4 w0 = __ldg(wt), w1 = __ldg(wt + 1), w2 = __ldg(wt + 2);
        const float w[kLowTaps] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w, w2.x, w2.y};
        const float4* p = reinterpret_cast<const float4*>(ns) + 2 * __float_as_int(w2.z);
        float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u;
#pragma unroll
        for (int k = 0; k < kLowTaps; ++k) {
          const float4 x = p[2 * k], y = p[2 * k + 1];
          u.x = fmaf(w[k], x.x, u.x), u.y = fmaf(w[k], x.y, u.y), u.z = fmaf(w[k], x.z, u.z), u.w = fmaf(w[k], x.w, u.w);
          v.x = fmaf(w[k], y.x, v.x), v.y = fmaf(w[k], y.y, v.y), v.z = fmaf(w[k], y.z, v.z), v.w = fmaf(w[k], y.w, v.w);
        }
        const float oh = __ldg(J.om_tab + j), wh = __ldg(J.om_tab + J.n_omega + j),
                    wl = __ldg(J.om_tab + 2 * J.n_omega + j);
        const float2 ph = phase2(make_float2(oh, oh), make_float2(wh, wh), make_float2(wl, wl),
                                 make_float2(tch, tch), make_float2(tcl, tcl));
        const float cp = cos_approx(ph.x), sp = sin_approx(ph.x);
        const float sum[kComps] = {u.x * cp - u.y * sp, u.x * sp + u.y * cp, u.z * cp - u.w * sp, u.z * sp + u.w * cp,
                                   v.x * cp - v.y * sp, v.x * sp + v.y * cp, v.z * cp - v.w * sp, v.z * sp + v.w * cp};
#pragma unroll
        for (int k = 0; k < kComps; ++k) {
          float* o = part + k * cs + j;
          __stcg(o, first ? sum[k] : __ldcg(o) + sum[k]);
        }
      }
      first = false;
      __syncwarp();
    }
    if (__syncthreads_or(landed ? 0 : 1)) {
      // a copy did not land within the bound: record it, wait (bounded) for both
      // buffers' copies in flight, and leave
      if (threadIdx.x == 0) {
        atomicOr(J.status, ST_TIMEOUT);
        mbar_wait(&bars[buf], ((phases >> buf) & 1u) ^ 1u);
        if (next < k1) mbar_wait(&bars[buf ^ 1], (phases >> (buf ^ 1)) & 1u);
      }
      return false;
    }
    if (next >= k1) return true;
  }
}

// The block's shared state: the current item and its job (one round trip to
// global memory per job instead of one per use).
struct BlockState {
  JobStatic J;
  JobCall K;
  ItemShared it;
  long long item;          // -1: a pass's first item is still to come
  int job, cur_job;        // the item's job, and the one loaded (-1: none)
  int any_wide, any_low;   // some job of the launch is wide, takes the low band
  LowPlan plan;            // the job's low-band plan (set -1: none), and its alternative
  LowSet low;
  LowTile tiles[2];
};

template <int THREADS>
__device__ __forceinline__ void load_job(BlockState& b, const LaunchArgs& a, int j) {
  copy_words<THREADS>(&b.J, &a.js[j], sizeof(JobStatic));
  copy_words<THREADS>(&b.K, a.use_inline ? &a.inline_call : &a.jc[j], sizeof(JobCall));
}

// One thread, once the kernels before this one are complete: the job's low-band
// plan; a call that takes the band has its tiles over the other bins only,
// chunked for them.
__device__ __forceinline__ void settle_plan(BlockState& b) {
  b.plan.set = -1;
  if (!b.K.low_ok) return;
  b.plan = *b.J.plan;
  if (b.plan.set < 0) return;
  b.low = b.J.low[b.plan.set];
  const LowSet& L = b.low;
  const LowCall& C = b.K.low[b.plan.set];
  // (rows without the band's bins; a frequency keeps its index)
  b.J.partials -= L.js;
  b.J.part_row -= L.js;
  b.J.part_bins -= b.J.n_dir * L.js;
  b.J.n_tiles = L.n_tiles;
  b.J.n_seg = L.n_seg;
  for (int i = 0; i < kMaxSegs; ++i) b.J.seg[i] = L.seg[i];
  b.K.ck = C.ck_hi;
  b.K.n_chunks = C.n_hi;
  b.K.run = 1;
  for (int l = 0; l < kTailLevels; ++l) {
    b.K.tail_tiles[l] = C.tail_tiles[l];
    b.K.ck_f[l] = C.ck_f[l];
    b.K.n_chunks_f[l] = C.n_chunks_f[l];
  }
}

// Claims the pass's next item (thread 0's counter; a block's first item is its
// index) and finds its job, into b.item and b.job; by the first warp.
__device__ __forceinline__ void claim_item(const LaunchArgs& a, BlockState& b, int counter, long long n_items,
                                           bool low) {
  long long item = blockIdx.x;
  if (b.item >= 0) {
    unsigned long long v = 0;
    if (threadIdx.x == 0) v = atomicAdd(a.item_counter + counter, 1ULL);
    item = (long long)(gridDim.x + __shfl_sync(0xffffffffu, v, 0));
  }
  const int j = item < n_items ? find_job_warp(a, item, low) : 0;
  __syncwarp();
  if (threadIdx.x == 0) {
    b.item = item;
    b.job = j;
  }
}

// Loads the claimed item's job if it is another than the last.
template <int THREADS>
__device__ __forceinline__ void switch_job(const LaunchArgs& a, BlockState& b) {
  if (b.job == b.cur_job) return;
  __syncthreads();
  load_job<THREADS>(b, a, b.job);
  __syncthreads();
  if (threadIdx.x == 0) {
    b.cur_job = b.job;
    settle_plan(b);
  }
  __syncthreads();
}

// The work items of the jobs whose call is not wide (WIDE = false) or is (true),
// each from its own counter.  Two instantiations, so the common path keeps
// its register allocation free of the wide-call code.  False: a wait gave up.
template <int THREADS, int W, bool TC, bool LIT, int PASSES, bool WIDE, bool XT>
__device__ __forceinline__ bool run_items(const LaunchArgs& a, BlockState& b, unsigned char* smem,
                                          uint64_t* bar, uint32_t& phase) {
  for (;;) {
    __syncthreads();  // the last item's shared state is used up
    if (threadIdx.x < 32) claim_item(a, b, WIDE ? 1 : 0, a.n_items, false);
    __syncthreads();
    const long long item = b.item;
    if (item >= a.n_items) return true;
    switch_job<THREADS>(a, b);
    if (b.any_wide && (b.J.wide_flag != nullptr && *b.J.wide_flag != 0) != WIDE) continue;  // the other pass's
    // Tile-major order: one tile's chunks run close together in time.
    const long long local = item - b.K.item_begin;
    // (the range holds the most items over the call's alternatives)
    if (XT && b.K.low_ok) {
      const int t0 = b.K.tail_tiles[0], t1 = b.K.tail_tiles[1];
      const int per_tile = (b.K.n_chunks + b.K.run - 1) / b.K.run;
      if (local >= (long long)(b.J.n_tiles - t0 - t1) * per_tile + (long long)t0 * b.K.n_chunks_f[0] +
                       (long long)t1 * b.K.n_chunks_f[1])
        continue;
    }
    const ItemRef it = decode_item<TC>(b.J, b.K, local);
    if (threadIdx.x == 0) {
      b.it.it = it;
      b.it.k_begin = (long long)it.chunk * it.ck;
      b.it.n_item = (int)min((long long)it.run * it.ck, b.K.n - b.it.k_begin);
    }
    bool ok;
    if constexpr (TC)
      ok = process_item_tc<THREADS, PASSES, 2 * W, WIDE, XT>(b.J, b.K, it, b.it, smem, bar, phase);
    else
      ok = process_item_fma<THREADS, W, 8, LIT, WIDE>(b.J, b.K, it, b.it, smem, bar, phase);
    if (!ok) return false;
  }
}

// The low bands' work items.
template <int THREADS>
__device__ __forceinline__ bool run_low(const LaunchArgs& a, BlockState& b, unsigned char* smem, uint64_t* bars) {
  uint32_t phases = 0u;
  for (;;) {
    __syncthreads();  // the last item's shared state is used up
    if (threadIdx.x < 32) claim_item(a, b, kCounterLow, a.n_items_low, true);
    __syncthreads();
    const long long item = b.item;
    if (item >= a.n_items_low) return true;
    switch_job<THREADS>(a, b);
    if (b.plan.set < 0) continue;
    int tile, chunk;
    div_rem(item - b.K.low_begin, b.K.low[b.plan.set].n_lo, tile, chunk);
    if (tile * kLowDirs >= b.J.n_dir) continue;
    if (!process_item_low<THREADS>(b.J, b.K, b.plan, b.low, tile, chunk, b.tiles, smem, bars, phases)) return false;
  }
}

template <int THREADS, int W, int MINB, bool TC, bool LIT, int PASSES = 1, bool XT = false>
__global__ void __launch_bounds__(THREADS, MINB) accumulate_kernel(const __grid_constant__ LaunchArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ __align__(8) uint64_t bars_low[2];
  __shared__ __align__(8) BlockState b;
  // Profiling: the block's start, kept in shared memory rather than in
  // registers live across the whole loop.
  __shared__ long long s_clk0;
  __shared__ unsigned long long s_ns0;
  pdl_trigger();
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_init(&bars_low[0], 1);
    mbar_init(&bars_low[1], 1);
    mbar_fence_init();
  }
  // A single job's tables, before the wait where no kernel writes them.  (The
  // allocation-free entry's set-up kernel does: the pre-pass triggers before its own
  // wait, so this kernel can be running before those writes are visible to it.  That
  // entry runs an FP32 variant: the others need no test.)
  if (a.n_jobs == 1 && (TC || a.use_inline != kJsFromKernel)) load_job<THREADS>(b, a, 0);
  pdl_wait();
  if (!TC && a.use_inline == kJsFromKernel) load_job<THREADS>(b, a, 0);
  // Whether any job of the launch is wide is final by now; without, the first
  // pass takes every item without looking at the jobs' flags.
  if (a.n_jobs == 1) __syncthreads();
  if (threadIdx.x == 0) {
    b.any_wide = a.any_wide != nullptr && a.any_wide[0] != 0;
    b.any_low = a.n_items_low > 0 && a.any_wide[1] != 0;
    b.cur_job = a.n_jobs == 1 ? 0 : -1;
    b.item = -1;
    if (a.n_jobs == 1) settle_plan(b);
  }
  if (a.prof_clk && threadIdx.x == 0) {
    s_clk0 = clock64();
    s_ns0 = global_ns();
  }
  uint32_t phase = 0u;
  // The low bands first: the bin tiles' fine-chunked last items end the launch
  // (with the bands' items last the SMs were active for 96.1 % of it).
  bool ok = true;
  if constexpr (XT) {
    __syncthreads();
    if (b.any_low) {
      ok = run_low<THREADS>(a, b, smem, bars_low);
      __syncthreads();
      if (threadIdx.x == 0) b.item = -1;
    }
  }
  if (ok) ok = run_items<THREADS, W, TC, LIT, PASSES, false, XT>(a, b, smem, &bar, phase);
  if (ok && b.any_wide) {
    __syncthreads();
    if (threadIdx.x == 0) b.item = -1;
    run_items<THREADS, W, TC, LIT, PASSES, true, XT>(a, b, smem, &bar, phase);
  }
  if (threadIdx.x == 0) {
    if (a.prof_clk) {
      atomicAdd(&a.prof_clk[0], (unsigned long long)(clock64() - s_clk0));
      atomicAdd(&a.prof_clk[1], global_ns() - s_ns0);
    }
    // The last block to leave puts the counter block back to zero for the next
    // call (no block claims an item after it has counted itself out).
    unsigned* out = reinterpret_cast<unsigned*>(a.item_counter + kCounterExit);
    if (atomicAdd(out, 1u) == gridDim.x - 1) {
      a.item_counter[0] = a.item_counter[1] = a.item_counter[kCounterLow] = 0ULL;
      *out = 0u;
      if (a.any_wide) a.any_wide[0] = a.any_wide[1] = 0;
    }
  }
}

// ------------------------------------------------------------ tile reduction
// Adds the chunks' partial sums of every bin, multiplies by e^{i omega
// tau_ref(n)} (reduced in FP64) and adds the result into the resident state
// with compensated (Kahan) FP32 sums.  A kernel of its own after the accumulate
// kernel: summed by the block that finished a tile last, a tile of many chunks
// was read by one SM at the end of the launch (90 of 157 us for 79 chunks of 4
// tiles, 35 us of the 6.9 ms LWFA step), and every item paid a fence and a
// counter.  Bound by the partials' bytes (mostly in L2) and, for small
// grids, by latency: kRedBins bins per block, a thread takes a quad of bins and
// a component pair over a quarter of the chunks, several chunks' loads in
// flight.  The quarters are added in chunk order, so results are a function of the
// chunking alone.  With it and the chunks of small calls (auto_chunk_for):
// 20000 particles, 128 x 16 bins, FP32 variant, 467 -> 76 us a call; 1777
// particles, 96 x 25 bins 64 -> 32 us; the LWFA step 6.96 -> 6.82 ms.
constexpr int kRedBins = 128;
constexpr int kRedGroups = 4;  // chunk ranges
constexpr int kRedThreads = kRedBins / 4 * 4 * kRedGroups;

// Four bins' values at p (vec: 16-byte aligned and all inside the grid).
__device__ __forceinline__ float4 load_quad(const float* p, bool vec, int live) {
  if (vec) return __ldcg(reinterpret_cast<const float4*>(p));
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (live > 0) v.x = __ldcg(p);
  if (live > 1) v.y = __ldcg(p + 1);
  if (live > 2) v.z = __ldcg(p + 2);
  if (live > 3) v.w = __ldcg(p + 3);
  return v;
}

// LATE: the job table comes from a kernel (kJsFromKernel).
// PER_SM: blocks per SM by the registers.  One for a single job: launched while the
// accumulate kernel still runs (pdl_trigger), two would fit in next to its blocks, and
// the next step's accumulate blocks then found the SMs unevenly taken (2000
// particles, 125 x 60 bins: 53 us a step at 64 registers, 33 at 71 and more).  Two for
// a batch, whose next round begins with copies (64 jobs of 1e3-1e4 particles: 1.31e12
// updates/s, with one 1.26e12).
template <bool LATE, int PER_SM>
__global__ void __launch_bounds__(kRedThreads, PER_SM) reduce_kernel(const __grid_constant__ LaunchArgs a) {
  __shared__ __align__(8) BlockState b;
  __shared__ float4 part[kRedGroups - 1][2][kRedBins];
  __shared__ float2 rot[kRedBins];
  pdl_trigger();
  if (a.n_jobs == 1) {
    if (!LATE) load_job<kRedThreads>(b, a, 0);  // (as accumulate_kernel)
  } else {
    if (threadIdx.x < 32) {
      int n = 0;
      for (int i = threadIdx.x; i < a.n_jobs; i += 32) n += a.jc[i].red_begin <= blockIdx.x;
      n = __reduce_add_sync(0xffffffffu, n) - 1;
      if (threadIdx.x == 0) b.job = n;
    }
    __syncthreads();
    load_job<kRedThreads>(b, a, b.job);
  }
  pdl_wait();
  if (LATE) load_job<kRedThreads>(b, a, 0);
  __syncthreads();
  if (threadIdx.x == 0) settle_plan(b);
  __syncthreads();
  const JobStatic& J = b.J;
  const JobCall& K = b.K;
  const int per_tile = J.bpt / kRedBins;
  const long long local = (long long)blockIdx.x - K.red_begin;
  const long long hi_blocks = (long long)J.n_tiles * per_tile;
  const int nb = J.n_bins, n_om = J.n_omega;
  const bool om4 = (n_om & 3) == 0;
  const int q = threadIdx.x & 31, pair = (threadIdx.x >> 5) & 3, cg = threadIdx.x >> 7;
  ItemRef it;
  PartMap m;
  int d, o, rd, ro;  // direction and frequency of the thread's first bin, and of its rotation
  size_t off;        // the first bin's offset in the partials
  bool part4;        // four bins at 16-byte aligned addresses
  it.chunk = it.run = it.ck = 0;
  const int rt = threadIdx.x & (kRedBins - 1);
  if (local < hi_blocks) {
    int s;
    div_rem(local, per_tile, it.tile, s);
    const int first1 = J.n_tiles - K.tail_tiles[1], first0 = first1 - K.tail_tiles[0];
    it.fine = it.tile >= first1 ? it.tile - first1 : (it.tile >= first0 ? it.tile - first0 : -1);
    it.n_chunks = it.fine < 0 ? K.n_chunks : K.n_chunks_f[it.tile >= first1 ? 1 : 0];
    const TileGeom g = tile_geom(J, it.tile, 256);
    m = part_map(J, K, it, g);
    if (!bounds_ok(part_fits(J, it, m), J.status)) return;
    const int sh = __ffs(g.WT) - 1;  // tile widths are powers of two
    const int i = s * kRedBins + 4 * q, ti = s * kRedBins + rt;
    d = g.d0 + (i >> sh), o = g.o0 + (i & (g.WT - 1));
    rd = g.d0 + (ti >> sh), ro = g.o0 + (ti & (g.WT - 1));
    off = it.fine < 0 ? (size_t)d * J.part_row + o : (size_t)i;
    part4 = it.fine >= 0 || om4;  // (js is a multiple of 64)
  } else {
    // the low band's bins, direction by direction
    const long long f = (local - hi_blocks) * kRedBins;
    const int js = b.plan.set >= 0 ? b.low.js : 0;
    if (f >= (long long)J.n_dir * js) return;
    div_rem(f + 4 * q, js, d, o);
    div_rem(f + rt, js, rd, ro);
    it.n_chunks = K.low[b.plan.set].n_lo;
    it.fine = -1;
    m.base = J.partials_l;
    m.comp_stride = (size_t)J.n_dir * js;
    m.chunk_stride = kComps * m.comp_stride;
    off = (size_t)f + 4 * q;
    part4 = true;  // (js is a multiple of 64)
    if (!bounds_ok(it.n_chunks * (long long)m.chunk_stride <= J.low_cap, J.status)) return;
  }
  const int live = d < J.n_dir ? min(4, n_om - o) : 0;  // bins inside the grid (<= 0: none)
  const size_t bin = (size_t)d * n_om + o;
  const bool vec = live > 0 && part4;
  // rotations: the last chunk range's threads, one bin each
  if (cg == kRedGroups - 1) {
    const double* nd = J.dirs + 3 * (size_t)min(rd, J.n_dir - 1);
    const double tref = J.ref[3] - (nd[0] * J.ref[0] + nd[1] * J.ref[1] + nd[2] * J.ref[2]) * kInvC;
    double psi = J.om_turns[min(ro, n_om - 1)] * tref;  // turns
    psi -= rint(psi);
    float2 cs;
    sincospif(2.0f * (float)psi, &cs.y, &cs.x);
    rot[rt] = cs;
  }
  const int per = (it.n_chunks + kRedGroups - 1) / kRedGroups;
  const int c0 = min(cg * per, it.n_chunks), c1 = min(c0 + per, it.n_chunks);
  // set 0: U and V; set 1: the literal sum's two pairs
  for (int set = 0; set < (J.literal ? 2 : 1); ++set) {
    const bool mine = live > 0 && (set == 0 || pair < 2);
    const float* base = set ? J.partials_p + bin : m.base + off;
    const size_t cs = set ? (size_t)nb : m.comp_stride, chs = set ? (size_t)4 * nb : m.chunk_stride;
    float4 re = make_float4(0.f, 0.f, 0.f, 0.f), im = re;
    if (mine) {
      const float* p = base + (size_t)(2 * pair) * cs + (size_t)c0 * chs;
#pragma unroll 8
      for (int ch = c0; ch < c1; ++ch, p += chs) {
        const float4 x = load_quad(p, vec, live), y = load_quad(p + cs, vec, live);
        re.x += x.x; re.y += x.y; re.z += x.z; re.w += x.w;
        im.x += y.x; im.y += y.y; im.z += y.z; im.w += y.w;
      }
    }
    __syncthreads();  // (set 1: the first set's sums are used up)
    if (cg > 0) {
      part[cg - 1][0][threadIdx.x & 127] = re;
      part[cg - 1][1][threadIdx.x & 127] = im;
    }
    __syncthreads();
    if (cg > 0 || !mine) continue;
#pragma unroll
    for (int k = 0; k < kRedGroups - 1; ++k) {
      const float4 x = part[k][0][threadIdx.x], y = part[k][1][threadIdx.x];
      re.x += x.x; re.y += x.y; re.z += x.z; re.w += x.w;
      im.x += y.x; im.y += y.y; im.z += y.z; im.w += y.w;
    }
    float* st = (set ? J.state_p : J.state) + bin;
    const int nc = set ? 4 : kComps, c = 2 * pair;
    const bool st4 = om4 && (reinterpret_cast<uintptr_t>(set ? J.state_p : J.state) & 15) == 0;
    float* sp[4] = {st + (size_t)c * nb, st + (size_t)(c + 1) * nb, st + (size_t)(nc + c) * nb,
                    st + (size_t)(nc + c + 1) * nb};
    float v[4][4];  // sum re, sum im, compensation re, compensation im of the four bins
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 x = load_quad(sp[k], st4, live);
      v[k][0] = x.x, v[k][1] = x.y, v[k][2] = x.z, v[k][3] = x.w;
    }
    const float re4[4] = {re.x, re.y, re.z, re.w}, im4[4] = {im.x, im.y, im.z, im.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 t = rot[4 * q + k];
      kahan_add(&v[0][k], &v[2][k], re4[k] * t.x - im4[k] * t.y);
      kahan_add(&v[1][k], &v[3][k], re4[k] * t.y + im4[k] * t.x);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (st4) {
        *reinterpret_cast<float4*>(sp[k]) = make_float4(v[k][0], v[k][1], v[k][2], v[k][3]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (e < live) sp[k][e] = v[k][e];
      }
    }
  }
}

template <int T, int W, int MINB, bool TC, bool LIT, int P = 1, bool XT = false>
cudaError_t launch_acc(const LaunchArgs& a, int grid, cudaStream_t s) {
  const size_t smem = Smem<T, TC, LIT, TC ? P * W : P, XT>::bytes;
  // The shared-memory opt-in is per kernel and device, and idempotent.
  static std::atomic<bool> attr_set[kMaxDevices];
  const int dev = current_device();
  if (dev < 0 || dev >= kMaxDevices || !attr_set[dev].load(std::memory_order_acquire)) {
    const cudaError_t e = cudaFuncSetAttribute(accumulate_kernel<T, W, MINB, TC, LIT, P, XT>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < kMaxDevices) attr_set[dev].store(true, std::memory_order_release);
  }
  count_launches(1);
  return launch_pdl(accumulate_kernel<T, W, MINB, TC, LIT, P, XT>, grid, T, smem, s, a);
}

template <int T, int W, int MINB, bool TC, bool LIT, int P = 1, bool XT = false>
int blocks_per_sm() {
  int nb = 0;
  const size_t smem = Smem<T, TC, LIT, TC ? P * W : P, XT>::bytes;
  cudaFuncSetAttribute(accumulate_kernel<T, W, MINB, TC, LIT, P, XT>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &nb, accumulate_kernel<T, W, MINB, TC, LIT, P, XT>, T, smem) != cudaSuccess ||
      nb < 1)
    nb = 1;
  return nb;
}

}  // namespace

int reduce_blocks(const JobStatic& js, const LowSet* low_sets) {
  const int per_tile = js.bpt / kRedBins;
  long long n = (long long)js.n_tiles * per_tile;
  for (int s = 0; s < js.n_low; ++s) {
    const long long low = ((long long)js.n_dir * low_sets[s].js + kRedBins - 1) / kRedBins;
    n = std::max(n, (long long)low_sets[s].n_tiles * per_tile + low);
  }
  return (int)n;
}

cudaError_t launch_reduce(const LaunchArgs& a, long long blocks, cudaStream_t s) {
  count_launches(1);
  auto* const kernel = a.use_inline == kJsFromKernel ? reduce_kernel<true, 1>
                       : a.use_inline                ? reduce_kernel<false, 1>
                                                     : reduce_kernel<false, 2>;
  return launch_pdl(kernel, blocks, kRedThreads, 0, s, a);
}

// Variants (rad_impl.h: variant_info): 0 FP32 256x2, 1 FP32 256x4, 2 FP32 128x2,
// 3 tensor-core 256 (3 CTAs/SM), 4 tensor-core 256 (4 CTAs/SM), 5 FP32 256x2 (4 CTAs/SM),
// 6 FP32 256x2 with the literal sum (2 CTAs/SM), 7 tensor-core 256 sweeping each staged
// particle tile in two frequency passes, 8 tensor-core 256 with four 16-frequency blocks
// per warp (512 frequencies per tile, 2 CTAs/SM), 9 as 8 with the phases' cross
// terms on tensor cores.
size_t accumulate_smem_bytes(int variant) {
  switch (variant) {
    case 2: return Smem<128, false>::bytes;
    case 3:
    case 4: return Smem<256, true>::bytes;
    case 6: return Smem<256, false, true>::bytes;
    case 7:
    case 8: return Smem<256, true, false, 2>::bytes;
    case 9: return Smem<256, true, false, 2, true>::bytes;
    default: return Smem<256, false>::bytes;
  }
}

int accumulate_blocks_per_sm(int variant) {
  static std::atomic<int> cached[kMaxDevices][kNumVariants];  // per device; 0 = not yet
  if (variant < 0 || variant >= kNumVariants) variant = 0;
  const int dev = current_device();
  const bool cache = dev >= 0 && dev < kMaxDevices;
  if (cache) {
    const int c = cached[dev][variant].load(std::memory_order_relaxed);
    if (c > 0) return c;
  }
  int nb;
  switch (variant) {
    case 1: nb = blocks_per_sm<256, 4, 2, false, false>(); break;
    case 2: nb = blocks_per_sm<128, 2, 6, false, false>(); break;
    case 3: nb = blocks_per_sm<256, 1, 3, true, false>(); break;
    case 4: nb = blocks_per_sm<256, 1, 4, true, false>(); break;
    case 5: nb = blocks_per_sm<256, 2, 4, false, false>(); break;
    case 6: nb = blocks_per_sm<256, 2, 2, false, true>(); break;
    case 7: nb = blocks_per_sm<256, 1, 3, true, false, 2>(); break;
    case 8: nb = blocks_per_sm<256, 2, 2, true, false>(); break;
    case 9: nb = blocks_per_sm<256, 2, 2, true, false, 1, true>(); break;
    default: nb = blocks_per_sm<256, 2, 3, false, false>(); break;
  }
  if (cache) cached[dev][variant].store(nb, std::memory_order_relaxed);
  return nb;
}

cudaError_t launch_accumulate(int variant, const LaunchArgs& a, int grid, cudaStream_t s) {
  switch (variant) {
    case 1: return launch_acc<256, 4, 2, false, false>(a, grid, s);
    case 2: return launch_acc<128, 2, 6, false, false>(a, grid, s);
    case 3: return launch_acc<256, 1, 3, true, false>(a, grid, s);
    case 4: return launch_acc<256, 1, 4, true, false>(a, grid, s);
    case 5: return launch_acc<256, 2, 4, false, false>(a, grid, s);
    case 6: return launch_acc<256, 2, 2, false, true>(a, grid, s);
    case 7: return launch_acc<256, 1, 3, true, false, 2>(a, grid, s);
    case 8: return launch_acc<256, 2, 2, true, false>(a, grid, s);
    case 9: return launch_acc<256, 2, 2, true, false, 1, true>(a, grid, s);
    default: return launch_acc<256, 2, 3, false, false>(a, grid, s);
  }
}

}  // namespace radimpl
