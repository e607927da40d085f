// qs_batch.cu -- many shots in one persistent launch (qs_scatter_batch).
//
// B0 k_bsetup   one thread per shot: validate the device-side descriptors,
//               derive the shot's launch constants, point them at its slice
//               of the samples and of the accumulators.
// B1 k_btable   one thread per (shot, phase cell): the shot's envelope table.
// B2 k_bscan    one CTA: tile sizes, exclusive prefix sum of the tile counts.
// B3 k_batch    persistent grid; each CTA pulls tiles from a device counter,
//               stages the tile's shot constants and table in shared memory,
//               evaluates the samples exactly as k_scatter does, writes the
//               tile's moment partials to the tile's own slot and merges its
//               shared-memory spectrum into the shot's accumulators (the
//               shot's divergence map and a_eff histogram take global
//               integer atomics directly).  Launched once per kind of shot
//               over the same schedule: quantum, classical, model variants.
// B4 k_bfinal   one CTA per shot: the tiles' partials summed in a fixed
//               order, histograms converted, moments written.
// G3 k_bgrad    (qs_scatter_grad_batch) the adjoint over the same (shot,
//               tile) schedule: each tile's samples recomputed with tangents,
//               the tile's 8 gradient partials to its own slot.
// G4 k_bgfinal  one CTA per shot: gradient slots summed in a fixed order.
//
// Paper: Amaro & Vranic, "QScatter", arXiv 2308.09348 (Sec. 3.2: parallel
// plane-wave runs; Sec. 6: high-repetition-rate data).
#include "qscatter.h"
#include "qs_device.cuh"
#include "qs_derive.cuh"
#include "qs_grad.cuh"
#include "qs_layout.hpp"
#include "qs_tiles.hpp"
#include "qs_host.hpp"

#include <type_traits>

namespace qs {

struct BatchArgs {
  int32_t n_shots, max_phase, wbits;
  int32_t tile, tile_rule;      // samples per work item, or the rule for them
  const qs_laser* lasers;
  const qs_beam* beams;
  const int64_t* offsets;
  qs_samples samples;
  qs_bins bins;
  const double* ranges;
  Params* shot;                 // [n_shots]
  int64_t* tiles;               // [n_shots + 1] counts, then exclusive offsets
  void* tables;                 // [n_shots * max_phase] float4 (FP32) or double (FP64)
  unsigned long long* acc;      // [n_shots * (n_bins + 2)]
  unsigned long long* acc_smooth;  // [n_shots * n_bins] (smoothed spectrum) or null
  unsigned long long* acc_map;     // [n_shots * (n_tx n_ty + 1)] (divergence maps) or null
  unsigned long long* acc_aeff;    // [n_shots * (n_aeff + 1)] (a_eff histograms) or null
  double* partials;             // [tiles * kNumMom]
  unsigned long long* counter;  // [kind] work counters, [kKinds + kind]
                                // nonzero if any shot with work is of the kind
  double* seeds;                // [n_shots * kSeeds] (adjoint) or null
  const qs_moments* moms;       // forward moments and their upstream gradient
  const double* dLdm;           // (adjoint)
  int64_t max_tiles;            // tile slots in the workspace
  const double* cyc_gl;         // cycle-resolved chi tables of this context
  const float4* cyc_m;          // (null: shots with that variant are invalid)
  int32_t precision, grid;      // grid: the caller's, or 0
};

// One warp per CTA, one shot per thread.  What bounds it is latency (a chain
// of FP64 divisions) and the write of 1.1 KB per shot: the constants go
// through shared memory and out coalesced, with few threads per SM (128
// threads writing their structs field by field took 68 us).
constexpr int kSetupThreads = 32;
constexpr int kParamWords = (int)(sizeof(Params) / 4);
constexpr int kParamStride = (kParamWords | 1);       // odd: conflict-free
static_assert(sizeof(Params) % 8 == 0, "Params is copied in words");

__global__ void __launch_bounds__(kSetupThreads) k_bsetup(const BatchArgs a) {
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  extern __shared__ uint32_t sp[];                    // [kSetupThreads][kParamStride]
  const int s0 = blockIdx.x * kSetupThreads, s = s0 + threadIdx.x;
  if (s < a.n_shots) {
    Params p;
    const qs_laser L = a.lasers[s];
    const qs_beam B = a.beams[s];
    qs_bins b = a.bins;
    if (a.ranges) {
      b.lo = a.ranges[2 * s];
      b.hi = a.ranges[2 * s + 1];
    }
    // shared samples (parameter sweep) when no offsets are given
    const int64_t o0 = a.offsets ? a.offsets[s] : 0;
    const int64_t o1 = a.offsets ? a.offsets[s + 1] : a.samples.n;
    // a model variant runs in its own kernels; cycle-resolved chi needs this
    // context's tables
    const bool cells = L.model == QS_MODEL_QFP || (L.variant & QS_VARIANT_CELL_FOCUS);
    const bool ok = check_laser(L) == QS_OK &&
                    (!(L.variant & QS_VARIANT_CYCLE_CHI) || (a.cyc_m && a.cyc_gl)) &&
                    check_beam(B) == QS_OK && check_bins(b) == QS_OK && o0 >= 0 && o1 >= o0 &&
                    o1 <= a.samples.n && (!cells || L.n_phase <= a.max_phase);
    int64_t work = 0;              // samples and kind, for k_bscan
    if (!ok) {
      memset(&p, 0, sizeof(Params));
      p.n = -1;                  // invalid shot
    } else {
      derive_params(p, L, B, &b, a.wbits);
      const size_t esz = a.samples.dtype == QS_F32 ? 4 : 8;
      p.n = o1 - o0;
      for (int k = 0; k < 8; ++k)
        p.xi[k] = a.samples.xi[k]
                      ? static_cast<const unsigned char*>(a.samples.xi[k]) + o0 * esz
                      : nullptr;
      p.w = a.samples.w ? static_cast<const unsigned char*>(a.samples.w) + o0 * esz : nullptr;
      p.dtype = a.samples.dtype;
      p.weighted = a.samples.w != nullptr;
      p.acc_spec = a.bins.n_bins > 0 ? a.acc + (size_t)s * (a.bins.n_bins + 2) : nullptr;
      p.acc_smooth = a.acc_smooth ? a.acc_smooth + (size_t)s * a.bins.n_bins : nullptr;
      p.acc_map = a.acc_map ? a.acc_map + (size_t)s * ((size_t)a.bins.n_tx * a.bins.n_ty + 1)
                            : nullptr;
      p.acc_aeff = a.acc_aeff ? a.acc_aeff + (size_t)s * (a.bins.n_aeff + 1) : nullptr;
      p.cyc_gl = a.cyc_gl;
      p.cyc_m = a.cyc_m;
      const int kind = L.variant != 0 ? kKindVar : (L.model == QS_MODEL_QFP ? kKindQfp : kKindLL);
      work = (p.n << 2) | kind;
      if (p.n > 0) a.counter[kKinds + kind] = 1ull;
      if (a.seeds) write_seeds(a.moms + s, a.dLdm + (size_t)s * 13, a.seeds + (size_t)s * kSeeds);
    }
    a.tiles[s] = work;
    uint32_t w[kParamWords];
    memcpy(w, &p, sizeof(Params));
#pragma unroll 8
    for (int k = 0; k < kParamWords; ++k) sp[threadIdx.x * kParamStride + k] = w[k];
  }
  __syncwarp();
  const int ns = min(kSetupThreads, a.n_shots - s0);
  uint32_t* dst = reinterpret_cast<uint32_t*>(a.shot + s0);
  for (int t = 0; t < ns; ++t)
    for (int k = threadIdx.x; k < kParamWords; k += kSetupThreads)
      dst[t * kParamWords + k] = sp[t * kParamStride + k];
}

// The shot whose phase table shot s reads: shot 0's if their windows are the
// same (the usual data set has one pulse shape; its entries are then the
// same numbers), else its own.
__device__ __forceinline__ int table_shot(const Params& p, const Params& p0, int s) {
  const bool same = p0.n >= 0 && (p0.model == QS_MODEL_QFP || p0.focus) && p.n_phase == p0.n_phase &&
                    p.envelope == p0.envelope && p.focus == p0.focus && p.h == p0.h &&
                    p.win_lo == p0.win_lo && p.Phi == p0.Phi && p.PhiT == p0.PhiT &&
                    p.phic == p0.phic && p.inv2k == p0.inv2k;
  return same ? 0 : s;
}

__global__ void k_btable(const BatchArgs a) {
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int s = (int)(idx / a.max_phase), j = (int)(idx % a.max_phase);
  if (s >= a.n_shots) return;
  const Params& p = a.shot[s];
  if (p.n < 0 || !(p.model == QS_MODEL_QFP || p.focus) || j >= p.n_phase) return;
  if (table_shot(p, a.shot[0], s) != s) return;
  if (a.precision == QS_F32)
    table_entry(p, j, static_cast<float4*>(a.tables) + (size_t)s * a.max_phase);
  else
    table_entry(p, j, static_cast<double*>(a.tables) + (size_t)s * a.max_phase);
}

// The tile sizes of the kinds, the shots' tile counts and their exclusive
// prefix sum in tiles[0..n) in place of k_bsetup's numbers of samples, total
// in tiles[n].  The per-shot checks of k_bsetup see one shot's range only; here the offsets
// are checked as a whole: if they decrease anywhere (shot ranges could then
// overlap), or the tiles would exceed the workspace's slots, every shot is
// made invalid and the total set to 0, so no shot does any work.
__global__ void __launch_bounds__(1024) k_bscan(const BatchArgs a) {
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  __shared__ int64_t wsum[32], ksum[kKinds][32];
  __shared__ int s_bad, s_tile[kKinds];
  const int n = a.n_shots;
  const int per = (n + blockDim.x - 1) / blockDim.x;
  const int b0 = threadIdx.x * per, b1 = min(n, b0 + per);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t w0 = b0 < b1 ? a.tiles[b0] : 0;            // read once for up to 1024 shots
  if (a.tile_rule == kTileFixed) {
    if (threadIdx.x < kKinds) s_tile[threadIdx.x] = a.tile;     // samples
  } else {
    int64_t t[kKinds] = {0, 0, 0};
    for (int i = b0; i < b1; ++i) {
      const int64_t w = i == b0 ? w0 : a.tiles[i];
#pragma unroll
      for (int k = 0; k < kKinds; ++k) t[k] += (w & 3) == k ? w >> 2 : 0;
    }
#pragma unroll
    for (int k = 0; k < kKinds; ++k) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
      if (lane == 0) ksum[k][warp] = t[k];
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
      for (int k = 0; k < kKinds; ++k) {
        t[k] = ksum[k][lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
      }
      if (lane == 0) {
        int tile[kKinds];
        choose_tiles(a.tile_rule, a.grid, t, a.acc_smooth ? a.bins.n_bins : 0, a.max_tiles - n - 1,
                     tile);
        for (int k = 0; k < kKinds; ++k) s_tile[k] = tile[k];   // exponents
      }
    }
  }
  __syncthreads();
  int64_t s = 0;
  int bad = 0;
  for (int i = b0; i < b1; ++i) {
    const int64_t w = i == b0 ? w0 : a.tiles[i];
    const bool fixed = a.tile_rule == kTileFixed;
    const int e = s_tile[w & 3], t = fixed ? e : 1 << e;
    const int64_t up = (w >> 2) + t - 1, v = fixed ? up / t : up >> e;
    a.tiles[i] = v;
    a.shot[i].tile = t;
    s += v;
    if (a.offsets && a.offsets[i + 1] < a.offsets[i]) bad = 1;
  }
  // inclusive sums: within the warp, then of the warps' totals by warp 0
  int64_t incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) wsum[warp] = incl;
  bad = __syncthreads_or(bad);
  if (warp == 0) {
    int64_t w = wsum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t v = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += v;
    }
    wsum[lane] = w;
    if (lane == 31) {
      s_bad = bad || w > a.max_tiles;
      a.tiles[n] = s_bad ? 0 : w;
    }
  }
  __syncthreads();
  if (s_bad) {
    for (int i = b0; i < b1; ++i) {
      a.shot[i].n = -1;
      a.tiles[i] = 0;
    }
    return;
  }
  int64_t run = incl - s + (warp > 0 ? wsum[warp - 1] : 0);
  for (int i = b0; i < b1; ++i) {
    const int64_t v = a.tiles[i];
    a.tiles[i] = run;
    run += v;
  }
}

__device__ __forceinline__ int kind_of(const Params& p) {
  return (p.focus != 0 || p.cycle != 0) ? kKindVar : (p.model == QS_MODEL_QFP ? kKindQfp : kKindLL);
}

// Thread 0 of a CTA takes the next tile of the kinds in `mask` (bits) from
// their counter (the first kind's) and finds its shot: the last one whose
// first tile is <= t (shots with no tiles are skipped).  Tiles of other kinds
// are passed over.
__device__ __forceinline__ int64_t next_tile(const BatchArgs& a, int kind, int mask, int64_t total,
                                             int* shot) {
  int64_t t;
  int s;
  do {
    t = (int64_t)atomicAdd(a.counter + kind, 1ull);
    s = -1;
    if (t < total) {
      int lo = 0, hi = a.n_shots - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.tiles[mid] <= t) lo = mid;
        else hi = mid - 1;
      }
      s = lo;
    }
  } while (t < total && !((mask >> kind_of(a.shot[s])) & 1));
  *shot = s;
  return t;
}

// Samples [first, last) of a classical shot (FP32, FP32 streams, no smoothed
// spectrum, map or a_eff histogram) four at a time: a shot's slice starts at
// any sample, so the few before the first 16-byte boundary, the same in
// every stream, and those after the last are left to the caller ([first,
// *v0) and [*v1, last)).  False if the streams' alignments differ, or for
// fewer samples than one step of the CTA (nothing to gain, and a handful of
// samples is then summed pair by pair in float pairs).
template <typename H>
__device__ __forceinline__ bool ll_tile_vector(const Params& p, int64_t first, int64_t last,
                                               AccF& acc, H* hs, int ns, int64_t* v0,
                                               int64_t* v1) {
  if (last - first < 4 * (int64_t)blockDim.x) return false;
  const uintptr_t mis = ((uintptr_t)p.xi[0] >> 2) & 3;
  for (int c = 0; c < 6; ++c)
    if (!p.xi[c] || (((uintptr_t)p.xi[c] >> 2) & 3) != mis) return false;
  if (p.weighted && (((uintptr_t)p.w >> 2) & 3) != mis) return false;
  const int64_t head = (int64_t)((4 - mis) & 3);        // samples before the boundary
  // groups of four samples, counted from the boundary
  const int64_t g0 = (first - head + 3) >> 2, g1 = (last - head) >> 2;
  Params q = p;                                         // the streams from the boundary on
  for (int c = 0; c < 6; ++c) q.xi[c] = static_cast<const float*>(p.xi[c]) + head;
  if (p.weighted) q.w = static_cast<const float*>(p.w) + head;
  // bins equal to the one-sample path's, whatever a shot's alignment
  ll_vector_range<H, true, true>(q, g0 + threadIdx.x, g1, blockDim.x, acc, hs, nullptr, nullptr,
                                 ns, 0, 0);
  *v0 = head + 4 * g0;
  *v1 = head + 4 * g1;
  return true;
}

// Shared memory of k_batch.
template <typename T, typename H, int KIND>
__host__ __device__ __forceinline__ BatchLayout batch_smem(const BatchArgs& a, int block) {
  return batch_layout(
      sizeof(Params), KIND == kKindVar && sizeof(T) == 4 ? 2 * kCycN * sizeof(float4) : 0,
      KIND == kKindLL ? 0 : (size_t)a.max_phase * sizeof(typename Tab<T>::type), block >> 5,
      kNumMom * sizeof(double), (size_t)(a.bins.n_bins > 0 ? a.bins.n_bins + 2 : 0) * sizeof(H),
      a.acc_smooth ? (size_t)a.bins.n_bins * 8 : 0);
}

// Block limit and registers of k_batch (FP32): the quantum model 64 (four
// 256-thread CTAs per SM), the classical one 80 (three), as k_scatter's.
// SMOOTH: classical FP32 shots whose spectrum is smoothed take one sample per
// thread and step, and the deposits (a kernel sum per sample, warp by warp)
// wait for shared memory: 64 registers for more warps (1000 shots of 20000
// samples, 128 threads: 1898 us with 80, 1583 with 64; 64 shots of 160000:
// 1013 and 849).
template <typename T, typename H, int KIND, bool SMOOTH>
__global__ void __launch_bounds__(KIND == kKindQfp ? 512 : 256,
                                  sizeof(T) == 8 ? 1 : (KIND == kKindLL ? (SMOOTH ? 4 : 3) : 2))
    k_batch(const BatchArgs a) {
  constexpr bool VARK = KIND == kKindVar;
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  using TT = typename Tab<T>::type;
  extern __shared__ __align__(16) unsigned char smem[];
  const BatchLayout at = batch_smem<T, H, KIND>(a, blockDim.x);
  Params& p = *reinterpret_cast<Params*>(smem);
  TT* tab = reinterpret_cast<TT*>(smem + at.table);
  // FP32 cycle-resolved chi: the per-interval monomial tables of G and H
  float4* cA = VARK ? reinterpret_cast<float4*>(smem + at.cycle) : nullptr;
  double* red = reinterpret_cast<double*>(smem + at.red);
  H* hs = reinterpret_cast<H*>(smem + at.hist);
  // work-item broadcast slots live in the dynamic allocation, so the kernel
  // has no static shared memory
  int64_t& s_tile = *reinterpret_cast<int64_t*>(smem + at.item);
  int& s_shot = *reinterpret_cast<int*>(smem + at.item + 8);
  // the tile's smoothed-spectrum accumulators (when smoothing)
  const int64_t nsm = a.acc_smooth ? (int64_t)a.bins.n_bins : 0;
  unsigned long long* hsm = nsm ? reinterpret_cast<unsigned long long*>(smem + at.smooth) : nullptr;
  const int64_t total = a.tiles[a.n_shots];
  const int64_t nspec = a.bins.n_bins > 0 ? (int64_t)a.bins.n_bins + 2 : 0;
  // per-shot divergence map and a_eff histogram: global accumulators
  const int64_t nmap = a.acc_map ? (int64_t)a.bins.n_tx * a.bins.n_ty + 1 : 0;
  const int64_t naeff = a.acc_aeff ? (int64_t)a.bins.n_aeff + 1 : 0;
  const int lane = threadIdx.x & 31;
  int cur = -1;
  if (a.counter[kKinds + KIND] == 0ull) return;    // no shot of this kind

  for (;;) {
    if (threadIdx.x == 0) {
      int sh;
      s_tile = next_tile(a, KIND, 1 << KIND, total, &sh);
      s_shot = sh;
    }
    __syncthreads();
    const int64_t t = s_tile;
    const int s = s_shot;
    if (t >= total) break;
    if (s != cur) {
      // stage the shot's constants and envelope table
      const int nw = (int)(sizeof(Params) / 4);
      const uint32_t* src = reinterpret_cast<const uint32_t*>(&a.shot[s]);
      uint32_t* dst = reinterpret_cast<uint32_t*>(&p);
      for (int k = threadIdx.x; k < nw; k += blockDim.x) dst[k] = src[k];
      __syncthreads();
      if (KIND != kKindLL && (p.model == QS_MODEL_QFP || p.focus)) {
        const TT* tg = static_cast<const TT*>(a.tables) +
                       (size_t)table_shot(p, a.shot[0], s) * a.max_phase;
        for (int j = threadIdx.x; j < p.n_phase; j += blockDim.x) tab[j] = tg[j];
      }
      if (VARK && sizeof(T) == 4 && p.cycle) {
        // per-interval monomial coefficients of G and H (the forward lookup)
        for (int j = threadIdx.x; j < kCycN - 1; j += blockDim.x) {
          cA[j] = p.cyc_m[j];
          cA[kCycN + j] = p.cyc_m[kCycN + j];
        }
      }
      cur = s;
    }
    for (int64_t b = threadIdx.x; b < nspec; b += blockDim.x) hs[b] = 0;
    for (int64_t b = threadIdx.x; b < nsm; b += blockDim.x) hsm[b] = 0;
    __syncthreads();

    typename AccT<T>::type acc;
    acc_init(acc);
    const int64_t first = (t - a.tiles[s]) * p.tile;
    const int64_t last = min(p.n, first + p.tile);
    // loops advance warp by warp (bounds uniform across the lanes), so that
    // the smoothed deposits run warp-cooperatively after each step
    auto single = [&](int64_t lo, int64_t hi, auto tqfp, auto tvar) {
      // one sample per thread
      constexpr int VAR = decltype(tvar)::value;
      constexpr bool Q = decltype(tqfp)::value;
      for (int64_t ib = lo + threadIdx.x - lane; ib < hi; ib += blockDim.x) {
        const int64_t i = ib + lane;
        typename DepT<T>::type d;
        bool ok = false;
        if (i < hi) {
          const auto sm = eval_one<T, Q, VAR>(p, tab, i, cA);
          ok = accumulate<T, H, true>(p, sm, i, acc, hs, nullptr, nullptr, nspec, nmap, naeff);
          dep_set(d, sm);
        }
        if (hsm) deposit_warp(p, ok, d, i, hsm);
      }
    };
    auto run = [&](auto tvar) {
      constexpr int VAR = decltype(tvar)::value;
      using Tr = std::true_type;
      using Fa = std::false_type;
      if constexpr (KIND == kKindLL) {
        int64_t v0 = last, v1 = last;
        if constexpr (sizeof(T) == 4 && !SMOOTH) {
          if (p.dtype != QS_F32 || hsm || nmap || naeff ||
              !ll_tile_vector<H>(p, first, last, acc, hs, (int)nspec, &v0, &v1))
            v0 = v1 = last;
        }
        single(first, v0, Fa{}, tvar);
        single(v1, last, Fa{}, tvar);
        return;
      }
      if constexpr (KIND == kKindVar) {
        if (p.model != QS_MODEL_QFP) {
          single(first, last, Fa{}, std::integral_constant<int, VAR & kVarCell>{});
          return;
        }
      }
      if constexpr (KIND != kKindLL && sizeof(T) == 4) {
        // FP32 QFP: each thread carries samples 2k and 2k+1 (first is even)
        for (int64_t kb = first / 2 + threadIdx.x - lane; 2 * kb < last; kb += blockDim.x) {
          const int64_t k = kb + lane;
          const int64_t i0 = 2 * k, i1 = (2 * k + 1 < last) ? 2 * k + 1 : 2 * k;
          DepF d0, d1;
          bool ok0 = false, ok1 = false;
          if (i0 < last) {
            SampleF s0, s1;
            eval_pair_f32_qfp<VAR>(p, reinterpret_cast<const float4*>(tab), i0, i1, s0, s1, cA);
            ok0 = accumulate<T, H, true>(p, s0, i0, acc, hs, nullptr, nullptr, nspec, nmap, naeff);
            if (i1 != i0)
              ok1 = accumulate<T, H, true>(p, s1, i1, acc, hs, nullptr, nullptr, nspec, nmap, naeff);
            dep_set(d0, s0);
            dep_set(d1, s1);
          }
          if (hsm) {
            deposit_warp(p, ok0, d0, i0, hsm);
            deposit_warp(p, ok1, d1, i1, hsm);
          }
        }
      } else if constexpr (KIND != kKindLL) {
        single(first, last, Tr{}, tvar);
      }
    };
    if constexpr (!VARK) {
      run(std::integral_constant<int, 0>{});
    } else {
      switch ((p.focus ? kVarCell : 0) | (p.cycle ? kVarCycle : 0)) {
        case kVarCell: run(std::integral_constant<int, kVarCell>{}); break;
        case kVarCycle: run(std::integral_constant<int, kVarCycle>{}); break;
        default: run(std::integral_constant<int, kVarCell | kVarCycle>{}); break;
      }
    }
    block_reduce_write(acc, red, a.partials + (size_t)t * kNumMom);
    __syncthreads();
    for (int64_t b = threadIdx.x; b < nspec; b += blockDim.x)
      if (hs[b]) atomicAdd(&p.acc_spec[b], (unsigned long long)hs[b]);
    for (int64_t b = threadIdx.x; b < nsm; b += blockDim.x)
      if (hsm[b]) atomicAdd(&p.acc_smooth[b], hsm[b]);
    __syncthreads();
  }
}

// One CTA per shot: its tiles' partials reduced (reduce_slots), its histograms
// converted.  (One warp per shot with a lane walking the tiles one by one, a
// division each, took 74 us for 400 shots and 104 us for 256 shots of 49
// tiles.)
__global__ void __launch_bounds__(kRedThreads)
    k_bfinal(const BatchArgs a, double* spectra, double* smooth, double* divmaps,
             double* aeff_hists, qs_moments* moments) {
  __shared__ double tot[kNumMom];
  cudaGridDependencySynchronize();
  const int s = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
  const Params& p = a.shot[s];
  const int nb = a.bins.n_bins;
  const bool sm = a.acc_smooth != nullptr;
  const int64_t nm = a.acc_map ? (int64_t)a.bins.n_tx * a.bins.n_ty : 0;
  const int na = a.acc_aeff ? a.bins.n_aeff : 0;
  if (p.n < 0) {
    for (int b = tid; b < nb; b += nt) spectra[(size_t)s * nb + b] = 0.0;
    if (sm)
      for (int b = tid; b < nb; b += nt) smooth[(size_t)s * nb + b] = 0.0;
    for (int64_t b = tid; b < nm; b += nt) divmaps[(size_t)s * nm + b] = 0.0;
    for (int b = tid; b < na; b += nt) aeff_hists[(size_t)s * na + b] = 0.0;
    if (tid == 0) {
      qs_moments m;
      memset(&m, 0, sizeof(m));
      m.nonfinite = -1.0;
      moments[s] = m;
    }
    return;
  }
  const double scale = p.weighted ? p.inv_wscale : 1.0;
  const int64_t t0 = a.tiles[s], t1 = a.tiles[s + 1];
  reduce_slots<true>(a.partials + (size_t)t0 * kNumMom, t1 - t0, tot);
  const unsigned long long* acc = p.acc_spec;
  if (tid < 32)
    write_moments(tot, nb > 0 ? (double)acc[nb] * scale : 0.0,
                  nb > 0 ? (double)acc[nb + 1] * scale : 0.0,
                  nm ? (double)p.acc_map[nm] * scale : 0.0, moments + s);
  for (int b = tid; b < nb; b += nt) spectra[(size_t)s * nb + b] = (double)acc[b] * scale;
  if (sm)
    for (int b = tid; b < nb; b += nt)
      smooth[(size_t)s * nb + b] = (double)p.acc_smooth[b] * p.inv_wscale;
  for (int64_t b = tid; b < nm; b += nt) divmaps[(size_t)s * nm + b] = (double)p.acc_map[b] * scale;
  for (int b = tid; b < na; b += nt) aeff_hists[(size_t)s * na + b] = (double)p.acc_aeff[b] * scale;
}

// Largest smoothed spectrum whose upstream gradient the FP32 batched adjoint
// stages in shared memory (larger ones are read from global memory).
constexpr int kBGradStageBins = 8192;

// G3: the adjoint of every shot over the (shot, tile) schedule of k_batch.
// Per tile: the shot's launch constants, envelope table and (FP32, when it
// fits) its upstream smoothed-spectrum gradient staged in shared memory, the
// upstream coefficients of its moments (formed once per shot by k_bsetup: a
// dozen FP64 divisions, 12 us when every thread of a CTA repeats them) in
// registers; the tile's samples recomputed with tangents exactly as k_grad
// does; the tile's 8 partials reduced in a fixed order into its own slot.
//   dLdS: n_shots x n_bins or null.
template <typename T, bool VARK>
__global__ void __maxnreg__((grad_regs(sizeof(T) == 8, VARK ? kVarCell : 0)))
    k_bgrad(const BatchArgs a, const double* __restrict__ dLdS) {
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  constexpr int KIND = VARK ? kKindVar : kKindQfp;      // kKindQfp: with the classical shots
  constexpr int MASK = VARK ? 1 << kKindVar : (1 << kKindQfp) | (1 << kKindLL);
  using TT = typename Tab<T>::type;
  extern __shared__ __align__(16) unsigned char smem[];
  Params& p = *reinterpret_cast<Params*>(smem);
  const size_t par_bytes = (sizeof(Params) + 15) & ~(size_t)15;
  TT* tab = reinterpret_cast<TT*>(smem + par_bytes);
  const size_t tab_bytes = ((size_t)a.max_phase * sizeof(TT) + 15) & ~(size_t)15;
  double* red = reinterpret_cast<double*>(smem + par_bytes + tab_bytes);
  unsigned char* after_red = smem + par_bytes + tab_bytes +
                             (((size_t)(blockDim.x >> 5) * kNumGrad * sizeof(double) + 15) &
                              ~(size_t)15);
  int64_t& s_tile = *reinterpret_cast<int64_t*>(after_red);
  int& s_shot = *reinterpret_cast<int*>(after_red + 8);
  const int nb = a.bins.n_bins;
  const bool smooth = dLdS != nullptr && a.bins.smooth_sigma_bins > 0.0;
  const bool stage = smooth && sizeof(T) == 4 && nb <= kBGradStageBins;
  T* sdS = reinterpret_cast<T*>(after_red + 16);
  // FP32 cycle-resolved chi: the monomial tables after the stage
  float4* cA = reinterpret_cast<float4*>(
      after_red + 16 + (((stage ? (size_t)nb * sizeof(T) : 0) + 15) & ~(size_t)15));
  const int64_t total = a.tiles[a.n_shots];
  int cur = -1;
  Seeds<T> sd{};
  T w0 = (T)1;
  if (VARK && a.counter[kKinds + kKindVar] == 0ull) return;      // no shot of this kind

  for (;;) {
    if (threadIdx.x == 0) {
      int sh;
      s_tile = next_tile(a, KIND, MASK, total, &sh);
      s_shot = sh;
    }
    __syncthreads();
    const int64_t t = s_tile;
    const int s = s_shot;
    if (t >= total) break;
    if (s != cur) {
      const int nw = (int)(sizeof(Params) / 4);
      const uint32_t* src = reinterpret_cast<const uint32_t*>(&a.shot[s]);
      uint32_t* dst = reinterpret_cast<uint32_t*>(&p);
      for (int k = threadIdx.x; k < nw; k += blockDim.x) dst[k] = src[k];
      __syncthreads();
      if (p.model == QS_MODEL_QFP || p.focus) {
        const TT* tg = static_cast<const TT*>(a.tables) +
                       (size_t)table_shot(p, a.shot[0], s) * a.max_phase;
        for (int j = threadIdx.x; j < p.n_phase; j += blockDim.x) tab[j] = tg[j];
      }
      if (VARK && sizeof(T) == 4 && p.cycle) {
        for (int j = threadIdx.x; j < 2 * kCycN; j += blockDim.x) cA[j] = p.cyc_m[j];
      }
      if (stage)
        for (int k = threadIdx.x; k < nb; k += blockDim.x) sdS[k] = (T)dLdS[(size_t)s * nb + k];
      sd = load_seeds<T>(a.seeds + (size_t)s * kSeeds);
      w0 = (T)sqrt(1.0 / p.inv_w0sq);
      cur = s;
      __syncthreads();
    }
    GAcc<T> acc;
    acc.init();
    const int64_t first = (t - a.tiles[s]) * p.tile;
    const int64_t last = min(p.n, first + p.tile);
    const int64_t tid = threadIdx.x, nthr = blockDim.x;
    const double* gS = smooth ? dLdS + (size_t)s * nb : nullptr;
    auto run = [&](auto tqfp, auto tvar) {
      constexpr bool Q = decltype(tqfp)::value;
      constexpr int VAR = decltype(tvar)::value;
      if (!smooth)
        grad_range<T, Q, T, VAR>(p, tab, sd, static_cast<const T*>(nullptr), w0, acc, first, last,
                                 tid, nthr, cA);
      else if (stage)
        grad_range<T, Q, T, VAR>(p, tab, sd, sdS, w0, acc, first, last, tid, nthr, cA);
      else
        grad_range<T, Q, double, VAR>(p, tab, sd, gS, w0, acc, first, last, tid, nthr, cA);
    };
    using std::integral_constant;
    using Tr = std::true_type;
    using Fa = std::false_type;
    if constexpr (!VARK) {
      if (p.model == QS_MODEL_QFP) run(Tr{}, integral_constant<int, 0>{});
      else run(Fa{}, integral_constant<int, 0>{});
    } else {
      const int var = (p.focus ? kVarCell : 0) | (p.cycle ? kVarCycle : 0);
      if (p.model != QS_MODEL_QFP) run(Fa{}, integral_constant<int, kVarCell>{});
      else if (var == kVarCell) run(Tr{}, integral_constant<int, kVarCell>{});
      else if (var == kVarCycle) run(Tr{}, integral_constant<int, kVarCycle>{});
      else run(Tr{}, integral_constant<int, kVarCell | kVarCycle>{});
    }
    grad_block_reduce(acc, red, a.partials + (size_t)t * kNumMom);
    __syncthreads();
  }
}

// G4: one CTA per shot, one warp per gradient component (a fixed order over
// the shot's tiles); invalid shots get zeros.
__global__ void __launch_bounds__(32 * kNumGrad) k_bgfinal(const BatchArgs a, double* grad) {
  cudaGridDependencySynchronize();
  const int s = blockIdx.x, k = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int64_t t0 = a.tiles[s], n = a.shot[s].n >= 0 ? a.tiles[s + 1] - t0 : 0;
  const double* q = a.partials + (size_t)t0 * kNumMom;
  double* g = grad + (size_t)s * kNumGrad;
  if (n <= kFewSlots) {
    if (k > 0) return;
    const double sum = warp_fields_sum((int)n, [&](int b, int f) { return q[b * kNumMom + f]; });
    if (lane < kNumGrad) g[lane] = sum;
    return;
  }
  const double sum = warp_slot_sum<true>(n, [&](int64_t b) { return q[b * kNumMom + k]; });
  if (lane == 0) g[k] = sum;
}

}  // namespace qs

using namespace qs;
using namespace qs::detail;

namespace {

struct BatchPlan {
  size_t off_counter = 0, off_params = 0, off_tiles = 0, off_seeds = 0, off_tables = 0,
         off_acc = 0, off_smooth = 0, off_map = 0, off_aeff = 0, off_part = 0, bytes = 0;
  int64_t max_tiles = 0;
};

bool batch_plan(BatchPlan& bp, int32_t n_shots, int64_t n_total, const qs_bins* bins,
                int32_t max_phase, int precision, int tile, bool shared) {
  if (n_shots < 1 || n_total < 0 || max_phase < 1 || max_phase > kMaxPhase) return false;
  // tile slots, of a given size: disjoint shots need at most n_total/tile + n_shots; a sweep
  // (every shot covers all samples) needs n_shots * ceil(n_total/tile)
  if (tile == 0)
    bp.max_tiles = open_tiles(n_shots, total_samples(n_shots, n_total, shared));
  else
    bp.max_tiles = shared ? (int64_t)n_shots * ((n_total + tile - 1) / tile) + 1
                          : n_total / tile + n_shots + 1;
  size_t off = 0;
  bp.off_counter = off; off = align_up(off + 2 * kKinds * 8, 256);
  bp.off_params = off; off = align_up(off + (size_t)n_shots * sizeof(Params), 256);
  bp.off_tiles = off; off = align_up(off + (size_t)(n_shots + 1) * 8, 256);
  bp.off_seeds = off; off = align_up(off + (size_t)n_shots * kSeeds * 8, 256);
  bp.off_tables = off;
  off = align_up(off + (size_t)n_shots * max_phase * (precision == QS_F64 ? 8 : 16), 256);
  bp.off_acc = off;
  off = align_up(off + (size_t)n_shots * (bins->n_bins > 0 ? bins->n_bins + 2 : 0) * 8, 256);
  bp.off_smooth = off;
  off = align_up(off + (size_t)n_shots * (bins->smooth_sigma_bins > 0 ? bins->n_bins : 0) * 8, 256);
  bp.off_map = off;
  off = align_up(off + (size_t)n_shots *
                           (bins->n_tx > 0 ? (size_t)bins->n_tx * bins->n_ty + 1 : 0) * 8, 256);
  bp.off_aeff = off;
  off = align_up(off + (size_t)n_shots * (bins->n_aeff > 0 ? bins->n_aeff + 1 : 0) * 8, 256);
  bp.off_part = off; off = align_up(off + (size_t)bp.max_tiles * kNumMom * 8, 256);
  bp.bytes = off;
  return true;
}

int32_t batch_checks(int32_t n_shots, const qs_samples* samples, const qs_bins* bins,
                     int32_t max_phase, const qs_exec* exec, int* prec, int* wbits, int* block,
                     int* grid, int* tile) {
  // *tile: the caller's, or 0 for one chosen by the launch
  int32_t st;
  if (n_shots < 1 || max_phase < 1 || max_phase > kMaxPhase) return QS_ERR_INVALID_ARG;
  if ((st = validate_samples(samples)) || (st = validate_bins(bins))) return st;
  if ((st = exec_opts(exec, prec, wbits, block, grid))) return st;
  if ((st = exec_tile(exec, tile))) return st;
  return QS_OK;
}

// small: CTAs of 128 threads instead of `block`, so that the CTAs of an SM are at
// different points of their tiles (loads, evaluation, merging), unless fewer
// threads of them fit on an SM (long spectra).
template <typename T, typename H, int KIND, bool SMOOTH = false>
int32_t launch_batch_kind(const BatchArgs& a, int block, bool small, int grid_req, int sms,
                          cudaStream_t st) {
  const size_t full = batch_smem<T, H, KIND>(a, block).bytes;
  if (full > (size_t)kSmemLimit) return QS_ERR_UNSUPPORTED;
  auto kern = k_batch<T, H, KIND, SMOOTH>;
  static CtxMark smem_mark;
  if (int32_t e = allow_smem(kern, smem_mark, kSmemLimit)) return e;
  int occ = 0;
  auto resident = [&](int b, size_t bytes) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, b, bytes) == cudaSuccess;
  };
  // (the registers allow 768 threads on an SM, 1024 with smoothed spectra)
  constexpr int most = SMOOTH ? 1024 : 768;
  size_t smem = full;
  int threads = 0;
  if (small && block > 128) {
    smem = batch_smem<T, H, KIND>(a, 128).bytes;
    if (!resident(128, smem)) return cuda_fail();
    threads = 128 * occ;
  }
  if (threads < most) {
    if (!resident(block, full)) return cuda_fail();
    if (threads < block * occ) {
      threads = 0;
      smem = full;
    }
  }
  if (threads > 0) {
    occ = threads / 128;
    block = 128;
  }
  // As many CTAs as fit at once.  Not more than there can be tiles (the
  // classical kernel apart, which is as fast without), nor an overlapping
  // launch of a caller's grid: CTAs placed while the kernel before holds the
  // SMs may share an SM where others stay idle (16 shots of 1000 samples with a
  // variant 75 us, 69; 152 CTAs on 256 shots of 20000 samples, cycle-resolved,
  // 2713 us, 1679).
  int grid = grid_req > 0 ? grid_req : sms * (occ > 0 ? occ : 1);
  if (KIND != kKindLL && grid_req == 0 && a.max_tiles < grid) grid = (int)a.max_tiles;
  return launch(kern, grid, block, smem, st, grid_req == 0, a);
}

// One kernel per kind of shot (it returns at once when no shot is of its
// kind).  small_ll: small CTAs for the classical shots.
template <typename T, typename H>
int32_t launch_batch(const BatchArgs& a, int block, bool small_ll, int grid_req, int sms,
                     cudaStream_t st) {
  if (int32_t e = launch_batch_kind<T, H, kKindQfp>(a, block, false, grid_req, sms, st)) return e;
  const int32_t e =
      sizeof(T) == 4 && a.acc_smooth
          ? launch_batch_kind<T, H, kKindLL, sizeof(T) == 4>(a, block, small_ll, grid_req, sms, st)
          : launch_batch_kind<T, H, kKindLL>(a, block, small_ll, grid_req, sms, st);
  if (e) return e;
  return launch_batch_kind<T, H, kKindVar>(a, block, false, grid_req, sms, st);
}

}  // namespace

extern "C" size_t qs_batch_workspace_bytes(int32_t n_shots, int64_t n_total, const qs_bins* bins,
                                           int32_t max_phase, const qs_exec* exec,
                                           int32_t shared_samples) {
  int prec, wbits, block, grid, tile;
  if (!bins || validate_bins(bins) != QS_OK) return 0;
  if (exec_opts(exec, &prec, &wbits, &block, &grid) || exec_tile(exec, &tile)) return 0;
  BatchPlan bp;
  if (!batch_plan(bp, n_shots, n_total, bins, max_phase, prec, tile, shared_samples != 0))
    return 0;
  return bp.bytes;
}

namespace {

// Device descriptors, workspace layout and the set-up kernels shared by the
// batched forward and adjoint: validates on the host, fills `a`, zeroes the
// work counters (and, for the forward, the accumulators) and launches
// k_bsetup, k_btable and k_bscan on `cs`.
int32_t batch_prepare(BatchArgs& a, int32_t n_shots, const qs_laser* d_lasers,
                      const qs_beam* d_beams, const int64_t* d_offsets,
                      const qs_samples* samples, const qs_bins* bins, const double* d_ranges,
                      int32_t max_phase, int prec, int wbits, int tile, int rule,
                      int grid, const qs_moments* moms, const double* dLdm,
                      void* d_workspace, size_t ws_bytes, bool zero_acc, int sms,
                      cudaStream_t cs) {
  if (!d_lasers || !d_beams) return QS_ERR_INVALID_ARG;
  BatchPlan bp;
  if (!batch_plan(bp, n_shots, samples->n, bins, max_phase, prec, tile, d_offsets == nullptr))
    return QS_ERR_INVALID_ARG;
  if (!d_workspace || ((uintptr_t)d_workspace % 256)) return QS_ERR_WORKSPACE;
  if (ws_bytes < bp.bytes) {
    // open tiles grow to what a smaller workspace (made for larger ones) holds
    const size_t slots = ws_bytes > bp.off_part ? (ws_bytes - bp.off_part) / (kNumMom * 8) : 0;
    if (tile != 0 || slots < (size_t)least_tiles(n_shots, samples->n, d_offsets == nullptr))
      return QS_ERR_WORKSPACE;
    bp.max_tiles = (int64_t)slots;
  }
  unsigned char* ws = static_cast<unsigned char*>(d_workspace);
  memset(&a, 0, sizeof(a));
  a.n_shots = n_shots;
  a.max_phase = max_phase;
  a.tile = tile;
  a.tile_rule = tile ? kTileFixed : rule;
  a.grid = grid;
  a.moms = moms;
  a.dLdm = dLdm;
  a.seeds = moms ? reinterpret_cast<double*>(ws + bp.off_seeds) : nullptr;
  a.wbits = wbits;
  a.lasers = d_lasers;
  a.beams = d_beams;
  a.offsets = d_offsets;
  a.samples = *samples;
  a.bins = *bins;
  a.ranges = d_ranges;
  a.shot = reinterpret_cast<Params*>(ws + bp.off_params);
  a.tiles = reinterpret_cast<int64_t*>(ws + bp.off_tiles);
  a.tables = ws + bp.off_tables;
  a.acc = reinterpret_cast<unsigned long long*>(ws + bp.off_acc);
  a.acc_smooth = bins->smooth_sigma_bins > 0
                     ? reinterpret_cast<unsigned long long*>(ws + bp.off_smooth)
                     : nullptr;
  a.acc_map = bins->n_tx > 0 ? reinterpret_cast<unsigned long long*>(ws + bp.off_map) : nullptr;
  a.acc_aeff = bins->n_aeff > 0 ? reinterpret_cast<unsigned long long*>(ws + bp.off_aeff) : nullptr;
  a.partials = reinterpret_cast<double*>(ws + bp.off_part);
  a.counter = reinterpret_cast<unsigned long long*>(ws + bp.off_counter);
  a.max_tiles = bp.max_tiles;
  a.precision = prec;
  // this context's cycle-resolved chi tables, built here on first use unless
  // the stream is being captured (then shots with that variant are invalid)
  {
    Params tp;
    const int32_t e = cycle_tables(tp, cs);
    if (e == QS_OK) {
      a.cyc_gl = tp.cyc_gl;
      a.cyc_m = tp.cyc_m;
    } else if (e != QS_ERR_UNSUPPORTED) {
      return e;
    }
  }
  // the counters lie before the accumulators' region: two clearings at most
  if (zero_acc && bp.off_part > bp.off_acc)
    if (int32_t e = clear(ws + bp.off_acc, bp.off_part - bp.off_acc, sms, cs)) return e;
  if (int32_t e = clear(ws + bp.off_counter, 256, sms, cs)) return e;
  constexpr size_t setup_smem = (size_t)kSetupThreads * kParamStride * 4;
  static_assert(setup_smem <= 48 * 1024, "fits the default shared memory");
  if (int32_t e = launch(k_bsetup, (n_shots + kSetupThreads - 1) / kSetupThreads, kSetupThreads,
                         setup_smem, cs, true, a))
    return e;
  const int64_t cells = (int64_t)n_shots * max_phase;
  if (int32_t e = launch(k_btable, (int)((cells + 255) / 256), 256, 0, cs, true, a)) return e;
  return launch(k_bscan, 1, 1024, 0, cs, true, a);
}

template <typename T>
int32_t launch_bgrad_kind(const BatchArgs& a, int block, int grid_req, int sms,
                          const double* dLdS, cudaStream_t st, bool vark) {
  using TT = typename Tab<T>::type;
  const bool stage = dLdS && a.bins.smooth_sigma_bins > 0 && sizeof(T) == 4 &&
                     a.bins.n_bins <= kBGradStageBins;
  const int most = grad_block(sizeof(T) == 8, vark ? kVarCell : 0);
  if (block > most && (vark || block > 512)) block = most;
  const size_t smem = align_up(sizeof(Params), 16) + align_up((size_t)a.max_phase * sizeof(TT), 16) +
                      align_up((size_t)(block / 32) * kNumGrad * sizeof(double), 16) + 16 +
                      align_up(stage ? (size_t)a.bins.n_bins * sizeof(T) : 0, 16) +
                      (vark && sizeof(T) == 4 ? (size_t)2 * kCycN * sizeof(float4) : 0);
  if (smem > (size_t)kSmemLimit) return QS_ERR_UNSUPPORTED;
  auto kern = vark ? k_bgrad<T, true> : k_bgrad<T, false>;
  static CtxMark smem_mark[2];
  if (int32_t e = allow_smem(kern, smem_mark[vark ? 1 : 0], kSmemLimit)) return e;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, block, smem) != cudaSuccess)
    return cuda_fail();
  const int grid = grid_req > 0 ? grid_req : sms * (occ > 0 ? occ : 1);
  // (a caller's grid: not overlapping, as in launch_batch_kind)
  return launch(kern, grid, block, smem, st, grid_req == 0, a, dLdS);
}

template <typename T>
int32_t launch_bgrad(const BatchArgs& a, int block, int grid_req, int sms, const double* dLdS,
                     cudaStream_t st) {
  if (int32_t e = launch_bgrad_kind<T>(a, block, grid_req, sms, dLdS, st, false)) return e;
  return launch_bgrad_kind<T>(a, block, grid_req, sms, dLdS, st, true);
}

}  // namespace

extern "C" int32_t qs_scatter_batch(int32_t n_shots, const qs_laser* d_lasers,
                                    const qs_beam* d_beams, const int64_t* d_offsets,
                                    const qs_samples* samples, const qs_bins* bins,
                                    const double* d_ranges, int32_t max_phase,
                                    const qs_exec* exec, double* d_spectra,
                                    double* d_spec_smooth, double* d_divmaps,
                                    double* d_aeff_hists, qs_moments* d_moments,
                                    void* d_workspace, size_t ws_bytes, void* stream) {
  int prec, wbits, block, grid, tile, sms;
  int32_t st = batch_checks(n_shots, samples, bins, max_phase, exec, &prec, &wbits, &block, &grid,
                            &tile);
  if (st) return st;
  if (!d_moments) return QS_ERR_INVALID_ARG;
  if (bins->n_bins > 0 && !d_spectra) return QS_ERR_INVALID_ARG;
  if (bins->smooth_sigma_bins > 0 && !d_spec_smooth) return QS_ERR_INVALID_ARG;
  if ((bins->n_tx > 0 && !d_divmaps) || (bins->n_aeff > 0 && !d_aeff_hists))
    return QS_ERR_INVALID_ARG;
  if (block > 256) block = 256;
  // classical shots, FP32, block and grid left open: 128 threads (the 256-shot
  // sweep 159 us with 256 threads, 149 with 128)
  const bool small_ll = prec == QS_F32 && !(exec && exec->block) && grid == 0;
  if ((st = device_sms(&sms))) return st;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  const bool check = exec_check_finite(exec);
  if (check && (st = sync_allowed(cs))) return st;
  BatchArgs a;
  if ((st = batch_prepare(a, n_shots, d_lasers, d_beams, d_offsets, samples, bins, d_ranges,
                          max_phase, prec, wbits, tile, kTileForward, grid, nullptr, nullptr,
                          d_workspace, ws_bytes, true, sms, cs)))
    return st;
  if (prec == QS_F64)
    st = samples->w ? launch_batch<double, unsigned long long>(a, block, false, grid, sms, cs)
                    : launch_batch<double, unsigned int>(a, block, false, grid, sms, cs);
  else
    st = samples->w ? launch_batch<float, unsigned long long>(a, block, small_ll, grid, sms, cs)
                    : launch_batch<float, unsigned int>(a, block, small_ll, grid, sms, cs);
  if (st) return st;
  if ((st = launch(k_bfinal, n_shots, kRedThreads, 0, cs, true, a, d_spectra, d_spec_smooth,
                   d_divmaps, d_aeff_hists, d_moments)))
    return st;
  return check ? nonfinite_status(&d_moments[0].nonfinite, n_shots, sizeof(qs_moments), cs)
               : QS_OK;
}

extern "C" int32_t qs_scatter_grad_batch(int32_t n_shots, const qs_laser* d_lasers,
                                         const qs_beam* d_beams, const int64_t* d_offsets,
                                         const qs_samples* samples, const qs_bins* bins,
                                         const double* d_ranges, int32_t max_phase,
                                         const qs_exec* exec, const qs_moments* d_moments,
                                         const double* d_dL_dmoments,
                                         const double* d_dL_dsmooth, double* d_grad,
                                         void* d_workspace, size_t ws_bytes, void* stream) {
  int prec, wbits, block, grid, tile, sms;
  int32_t st = batch_checks(n_shots, samples, bins, max_phase, exec, &prec, &wbits, &block, &grid,
                            &tile);
  if (st) return st;
  if (!d_moments || !d_dL_dmoments || !d_grad) return QS_ERR_INVALID_ARG;
  if (d_dL_dsmooth && !(bins->smooth_sigma_bins > 0)) return QS_ERR_INVALID_ARG;
  if ((st = device_sms(&sms))) return st;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  // block left open: one CTA per SM that fills the register file, as for the
  // single-shot adjoint (launch_bgrad_kind lowers it for the variants)
  const int kblock = (exec && exec->block) ? block : grad_block(prec == QS_F64, 0);
  BatchArgs a;
  if ((st = batch_prepare(a, n_shots, d_lasers, d_beams, d_offsets, samples, bins, d_ranges,
                          max_phase, prec, wbits, tile, kTileAdjoint, grid, d_moments,
                          d_dL_dmoments, d_workspace, ws_bytes, false, sms, cs)))
    return st;
  st = prec == QS_F64
           ? launch_bgrad<double>(a, kblock, grid, sms, d_dL_dsmooth, cs)
           : launch_bgrad<float>(a, kblock, grid, sms, d_dL_dsmooth, cs);
  if (st) return st;
  return launch(k_bgfinal, n_shots, 32 * kNumGrad, 0, cs, true, a, d_grad);
}
