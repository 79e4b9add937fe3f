// fused.cu -- a whole mixed-degree batch in persistent kernels over job lists.
//
// The fused batch plan serves the jobs of every degree of a ts_batch with one
// persistent kernel per tier of degrees that the batch holds: blocks pull work
// items from the tier's counter, stage the job's tables into shared memory
// with cp.async.bulk on an mbarrier (bounded wait) when they move to another
// triangulation, draw the job's splitmix64 sign vectors on the device (or
// read the caller's, ts_batch_set_signs), classify them with Algorithm 1
// (Sec. 2) and add the codes to the job's device histogram.  The degree of a
// job selects the code path inside the kernel (a switch over degree-templated
// bodies):
//
//   bit-sliced           (TS_KERNEL_TABLE)  the block classifies 128 sign
//        vectors at a time (tc_sliced.cuh), everything in shared memory;
//   warp per instance    (TS_KERNEL_WARP)   the 32 lanes of a warp classify
//        one sign vector together (lock-free union-find in shared memory,
//        tc_warp_sweep.cuh), 32 sign vectors per warp between histogram
//        inserts.
//
// Tiers: a block's shared memory grows with the degree (14 KB at d = 5, 54 KB
// at d = 10, 195 KB at d = 16), and one launch has one size, so the degrees of
// a launch share the occupancy of its largest.  The tiers run on forked
// streams, the largest degrees first: the blocks of one fill the SMs that the
// last blocks of another leave.  3.7e8 sign vectors of d = 5..10: 388 ms (one
// thread per sign vector, one launch) -> 122 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include "engine.h"
#include "tc_layout.h"
#include "tc_sliced.cuh"
#include "tc_stage.cuh"
#include "tc_table_sweep.cuh"
#include "tc_warp_sweep.cuh"

namespace tcurve {
namespace {

constexpr u32 kFT = kFusedThreads;  // threads per block: 4 warps

// Largest degree of the bit-sliced tiers.
constexpr int kTierD[kFusedTiers] = {6, 8, 10, 16};

// Resident blocks per SM a kernel of degrees up to DHI is compiled for: what
// its shared memory lets in (warp tiles: 80 registers).
constexpr int min_blocks(int dhi, bool warp) { return warp ? 6 : dhi <= 6 ? 9 : dhi <= 8 ? 7 : dhi <= 10 ? 4 : 2; }

// Sign vector idx of job J: the caller's (J.signs, W words each) or word w
// of the splitmix64 stream, splitmix64((base + idx) * W + w); bits >= |A|
// cleared.
template <u32 W, u32 NPOINTS>
__device__ __forceinline__ TcSig<W> job_sig(const FusedJob &__restrict__ J, u64 idx) {
  TcSig<W> sg;
  if (J.signs) {
#pragma unroll
    for (u32 w = 0; w < W; ++w) sg.w[w] = J.signs[idx * W + w];
  } else {
#pragma unroll
    for (u32 w = 0; w < W; ++w) sg.w[w] = tc_splitmix64((J.base + idx) * W + w);
  }
  sg.w[W - 1] &= tc_top_mask(NPOINTS, W);
  return sg;
}

// Bit-sliced: the J.chunk sign vectors of job J from index `first`, a block
// of 128 at a time.
template <int D>
__device__ __forceinline__ void sliced_item(const FusedJob &__restrict__ J, u64 first, const u32 *tab, u32 *area,
                                            u32 *err_word, u32 &err, unsigned long long &failed) {
  typedef TcSlK<D, (int)kFT / 32> K;
  const TcSlMem M = tc_sl_carve<K>(tab, area, J.sl.chunks);
  const u32 t = threadIdx.x, lane = t & 31u, mine = tc_sl_instance<K>(t);
  for (u32 k = 0; k < J.chunk && first + k < J.n; k += kFT) {
    TcSig<K::W> sg{};
    if (first + k + t < J.n) sg = job_sig<K::W, K::NPOINTS>(J, first + k + t);
    u32 e = 0;
    u64 code[K::CW];
    tc_sl_classify<K>(M, sg, t, e, code);
    const u64 idx = first + k + mine;
    u64 any = 0;
    const bool live = idx < J.n;
#pragma unroll
    for (u32 w = 0; w < K::CW; ++w) {
      code[w] = live ? code[w] : 0ull;
      any |= code[w];
      if (live && J.codes) J.codes[idx * K::CW + w] = code[w];
    }
    err |= live ? e : 0u;
    failed += live && any == 0;
    if constexpr (K::CW == 1) {
      const unsigned peers = __match_any_sync(0xffffffffu, code[0]);
      if (code[0] != 0 && lane == (u32)(__ffs(peers) - 1))
        tc_global_add(J.hkeys, J.hcnt, J.hslots, err_word, code[0], (unsigned long long)__popc(peers));
    } else {
      tc_hist_add_wide<K::CW>(code, J.hkeys, J.hcnt, J.hslots, err_word);
    }
    __syncthreads();
  }
}

// Warp per instance: warp w of the block takes sign vectors first + g + r,
// g = 32 w, 32 w + 128, ..., r < 32, one at a time; lane r keeps the code of
// the r-th and the warp inserts its 32 codes together.
template <int D>
__device__ __forceinline__ void warp_item(const FusedJob &__restrict__ J, u64 first, const u32 *tab, u32 *ws,
                                          u32 *err_word, u32 &err, unsigned long long &failed) {
  typedef TcWarpK<D> K;
  const u32 warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
  for (u32 g = warp * 32u; g < J.chunk; g += kFT) {
    u64 mine[K::CW];
#pragma unroll
    for (u32 w = 0; w < K::CW; ++w) mine[w] = 0;
    for (u32 r = 0; r < 32u; ++r) {
      const u64 idx = first + g + r;
      if (idx >= J.n) break;  // warp-uniform
      const TcSig<K::W> sg = job_sig<K::W, K::NPOINTS>(J, idx);
      u64 code[K::CW];
#pragma unroll
      for (u32 w = 0; w < K::CW; ++w) code[w] = 0;
      err |= tc_warp_classify<D>(sg, tab + J.wl.off_v, tab + J.wl.off_e, J.wl.E,
                                 tab + J.wl.off_anti, J.wl.nanti, tab + J.wl.off_bedge,
                                 J.wl.nbedge, ws, code);
#pragma unroll
      for (u32 w = 0; w < K::CW; ++w) {
        const u64 c = __shfl_sync(0xffffffffu, code[w], 0);  // lane 0 holds the code
        if (lane == 0 && J.codes) J.codes[idx * K::CW + w] = c;
        mine[w] = lane == r ? c : mine[w];
      }
    }
    u64 any = 0;
#pragma unroll
    for (u32 w = 0; w < K::CW; ++w) any |= mine[w];
    failed += first + g + lane < J.n && any == 0;
    if constexpr (K::CW == 1) {
      const unsigned peers = __match_any_sync(0xffffffffu, mine[0]);
      if (mine[0] != 0 && lane == (u32)(__ffs(peers) - 1))
        tc_global_add(J.hkeys, J.hcnt, J.hslots, err_word, mine[0],
                      (unsigned long long)__popc(peers));
    } else {
      tc_hist_add_wide<K::CW>(mine, J.hkeys, J.hcnt, J.hslots, err_word);
    }
  }
}

// Body of a degree-D job in the kernel of degrees DLO..DHI.
template <int D, int DLO, int DHI, bool WARP>
__device__ __forceinline__ void run_item(const FusedJob &__restrict__ J, u64 first, const u32 *tab, u32 *area,
                                         u32 ws_stride, u32 *err_word, u32 &err, unsigned long long &failed) {
  if constexpr (D >= DLO && D <= DHI) {
    if constexpr (WARP)
      warp_item<D>(J, first, tab, area + (threadIdx.x >> 5) * ws_stride, err_word, err, failed);
    else
      sliced_item<D>(J, first, tab, area, err_word, err, failed);
  }
}

// smem: tables (toff bytes) | mbarrier, work slot (128 bytes) | the block's
// areas (bit-sliced) or 4 x ws_stride words (warp states).
template <int DLO, int DHI, bool WARP>
__global__ void __launch_bounds__(kFT, min_blocks(DHI, WARP))
    fused_jobs_kernel(const FusedJob *__restrict__ jobs, u32 njobs, u64 total_items,
                      unsigned long long *work, u32 *err_word, unsigned long long *failed_word, u32 toff,
                      u32 ws_stride) {
  extern __shared__ __align__(128) uint8_t smem[];
  u32 *tab = reinterpret_cast<u32 *>(smem);
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem + toff);
  unsigned long long *slot = reinterpret_cast<unsigned long long *>(smem + toff + 64);
  u32 *area = reinterpret_cast<u32 *>(smem + toff + 128);
  if (threadIdx.x == 0) mbar_init(bar, 1);
  __syncthreads();
  const u32 *cur = nullptr;
  u32 phase = 0, err = 0;
  unsigned long long failed = 0;
  for (;;) {
    if (threadIdx.x == 0) *slot = atomicAdd(work, 1ull);
    __syncthreads();
    const u64 c = *slot;
    __syncthreads();  // also: every thread is done with the previous tables
    if (c >= total_items) break;
    u32 lo = 0, hi = njobs;  // the job holding item c: last j with item0 <= c
    while (hi - lo > 1) {
      const u32 mid = (lo + hi) / 2;
      if (jobs[mid].item0 <= c) lo = mid; else hi = mid;
    }
    const FusedJob &J = jobs[lo];  // fields read where used (L1): no copy to keep live
    if (J.tab != cur) {  // stage the job's tables (cp.async.bulk, bounded wait)
      if (threadIdx.x == 0) {
        mbar_expect_tx(bar, J.tab_words * 4u);
        bulk_g2s(tab, J.tab, J.tab_words * 4u, bar);
      }
      bool ok = false;
      for (long it = 0; it < kWaitIters && !ok; ++it) ok = mbar_try_wait(bar, phase);
      if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) atomicOr(err_word, kErrTimeout);
        // let a late copy land before the block's shared memory is released
        for (long it = 0; it < kWaitIters && !ok; ++it) ok = mbar_try_wait(bar, phase);
        return;
      }
      phase ^= 1u;
      cur = J.tab;
    }
    const u64 first = (c - J.item0) * (u64)J.chunk;
    switch (J.d) {
#define TC_FUSED_CASE(d) \
  case d: run_item<d, DLO, DHI, WARP>(J, first, tab, area, ws_stride, err_word, err, failed); break;
      TC_FUSED_CASE(1) TC_FUSED_CASE(2) TC_FUSED_CASE(3) TC_FUSED_CASE(4) TC_FUSED_CASE(5)
      TC_FUSED_CASE(6) TC_FUSED_CASE(7) TC_FUSED_CASE(8) TC_FUSED_CASE(9) TC_FUSED_CASE(10)
      TC_FUSED_CASE(11) TC_FUSED_CASE(12) TC_FUSED_CASE(13) TC_FUSED_CASE(14)
      TC_FUSED_CASE(15) TC_FUSED_CASE(16)
#undef TC_FUSED_CASE
      default: err |= kErrInternal; break;
    }
  }
  if (err) atomicOr(err_word, err);
  if (failed) atomicAdd(failed_word, failed);
}

typedef void (*FusedFn)(const FusedJob *, u32, u64, unsigned long long *, u32 *, unsigned long long *, u32, u32);

FusedFn tier_fn(int tier) {
  switch (tier) {
    case 0: return fused_jobs_kernel<1, kTierD[0], false>;
    case 1: return fused_jobs_kernel<kTierD[0] + 1, kTierD[1], false>;
    case 2: return fused_jobs_kernel<kTierD[1] + 1, kTierD[2], false>;
    case 3: return fused_jobs_kernel<kTierD[2] + 1, kTierD[3], false>;
    case kFusedWarpTier: return fused_jobs_kernel<kFusedWarpFrom, kTierD[3], true>;
    default: return nullptr;
  }
}

template <int D>
u32 warp_words_d() {
  return TcWarpK<D>::WORDS;
}

}  // namespace

int fused_tier(int d) {
  for (int t = 0; t < kFusedTiers; ++t)
    if (d <= kTierD[t]) return t;
  return -1;
}

size_t fused_area_bytes(int d, const SlicedLayout &l) {
  switch (d) {
#define TC_AREA(x) \
  case x: return (size_t)tc_sl_words<TcSlK<x, (int)kFT / 32>>(l.chunks) * 4;
    TC_AREA(1) TC_AREA(2) TC_AREA(3) TC_AREA(4) TC_AREA(5) TC_AREA(6) TC_AREA(7) TC_AREA(8) TC_AREA(9)
    TC_AREA(10) TC_AREA(11) TC_AREA(12) TC_AREA(13) TC_AREA(14) TC_AREA(15) TC_AREA(16)
#undef TC_AREA
    default: return 0;
  }
}

uint32_t fused_warp_words(int d) {
  switch (d) {
#define TC_WW(x) \
  case x: return warp_words_d<x>();
    TC_WW(1) TC_WW(2) TC_WW(3) TC_WW(4) TC_WW(5) TC_WW(6) TC_WW(7) TC_WW(8) TC_WW(9) TC_WW(10)
    TC_WW(11) TC_WW(12) TC_WW(13) TC_WW(14) TC_WW(15) TC_WW(16)
#undef TC_WW
    default: return 0;
  }
}

// The kernel may use any dynamic shared memory a block can have, whichever
// batch was planned last: the size of a launch is its own.
cudaError_t fused_occupancy(int tier, size_t smem, int *blocks_per_sm) {
  const FusedFn fn = tier_fn(tier);
  if (!fn) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kMaxBlockSmem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, (const void *)fn, (int)kFT, smem);
}

cudaError_t fused_attrs(int tier, int *regs, int *local_bytes) {
  const FusedFn fn = tier_fn(tier);
  if (!fn) return cudaErrorInvalidValue;
  cudaFuncAttributes fa{};
  cudaError_t e = cudaFuncGetAttributes(&fa, (const void *)fn);
  if (e != cudaSuccess) return e;
  *regs = fa.numRegs;
  *local_bytes = (int)fa.localSizeBytes;
  return cudaSuccess;
}

cudaError_t fused_launch(int tier, unsigned grid, size_t smem, uint32_t toff, uint32_t ws_stride,
                         const FusedJob *jobs, uint32_t njobs, uint64_t items, unsigned long long *work,
                         uint32_t *err, unsigned long long *failed, cudaStream_t st) {
  const FusedFn fn = tier_fn(tier);
  if (!fn) return cudaErrorInvalidValue;
  fn<<<grid, kFT, smem, st>>>(jobs, njobs, items, work, err, failed, toff, ws_stride);
  return cudaGetLastError();
}

}  // namespace tcurve
