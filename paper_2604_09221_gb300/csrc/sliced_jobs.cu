// sliced_jobs.cu -- the bit-sliced kernel of a degree group of a batch
// (ts_batch, one persistent kernel per degree; batch.cu plans and launches
// it).
#include <cuda_runtime.h>
#include <stdint.h>

#include "engine.h"
#include "tc_sliced.cuh"
#include "tc_stage.cuh"

namespace tcurve {
namespace {

// Work items of chunk sign vectors, K::T of them at a time (tc_sliced.cuh),
// everything in shared memory.  smem: tables (toff bytes) | mbarrier, work slot
// (128 bytes) | the block's areas.
//
// Blocks of 128, but at d = 13 and 14 of 64 or 192 (tc_sl_wide): 128 are one
// block per multiprocessor there, and four jobs of 2^20 took 15.1 and 21.1 ms
// against 14.0 and 18.9 with one thread per sign vector; now 10.4 and 15.1.
// Their work items are two blocks long, so that short jobs wait for no more
// phases.
// (d = 15 and 16 have two blocks of 64 or one of 128: 20.2 and 27.6 ms with
// 128, 19.7 and 27.6 with 64, whose short jobs take up to twice as long.)
template <class K>
__global__ void __launch_bounds__(K::T)
    sliced_jobs_kernel(const DevJob *__restrict__ jobs, u32 njobs, u64 total_items, u32 chunk, u32 toff,
                       unsigned long long *work, u32 *err_word, unsigned long long *failed_word) {
  extern __shared__ __align__(128) uint8_t smem[];
  u32 *tab = reinterpret_cast<u32 *>(smem);
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem + toff);
  unsigned long long *slot = reinterpret_cast<unsigned long long *>(smem + toff + 64);
  if (threadIdx.x == 0) mbar_init(bar, 1);
  __syncthreads();
  const u32 t = threadIdx.x, lane = t & 31u, mine = tc_sl_instance<K>(t);
  u32 cur = 0xFFFFFFFFu, phase = 0, err = 0;
  unsigned long long failed = 0;
  for (;;) {
    if (t == 0) *slot = atomicAdd(work, 1ull);
    __syncthreads();
    const u64 c = *slot;
    __syncthreads();  // also: every thread is done with the previous job's tables
    if (c >= total_items) break;
    u32 lo = 0, hi = njobs;  // the job holding item c: last j with chunk0 <= c
    while (hi - lo > 1) {
      const u32 mid = (lo + hi) / 2;
      if (jobs[mid].chunk0 <= c) lo = mid; else hi = mid;
    }
    const DevJob &J = jobs[lo];
    if (lo != cur) {  // stage the job's tables (cp.async.bulk, bounded wait)
      if (t == 0) {
        mbar_expect_tx(bar, J.swords * 4u);
        bulk_g2s(tab, J.stab, J.swords * 4u, bar);
      }
      bool ok = false;
      for (long it = 0; it < kWaitIters && !ok; ++it) ok = mbar_try_wait(bar, phase);
      if (__syncthreads_or(!ok)) {
        if (t == 0) atomicOr(err_word, kErrTimeout);
        for (long it = 0; it < kWaitIters && !ok; ++it) ok = mbar_try_wait(bar, phase);
        return;
      }
      phase ^= 1u;
      cur = lo;
    }
    const TcSlMem M = tc_sl_carve<K>(tab, reinterpret_cast<u32 *>(smem + toff + 128), J.schunks);
    const u64 first = (c - J.chunk0) * (u64)chunk, end = first + chunk < J.n ? first + chunk : J.n;
    for (u32 k = 0; first + k < end; k += K::T) {
      // the sign vector of counter base + idx, as ts_splitmix_masks writes it
      TcSig<K::W> sg;
#pragma unroll
      for (u32 w = 0; w < K::W; ++w) sg.w[w] = tc_splitmix64((J.base + first + k + t) * K::W + w);
      sg.w[K::W - 1] &= tc_top_mask(K::NPOINTS, K::W);
      u32 e = 0;
      u64 code[K::CW];
      tc_sl_classify<K>(M, sg, t, e, code);
      const u64 idx = first + k + mine;
      u64 any = 0;
      const bool live = idx < end;
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
  if (err) atomicOr(err_word, err);
  if (failed) atomicAdd(failed_word, failed);
}

typedef void (*SlicedJobsFn)(const DevJob *, u32, u64, u32, u32, unsigned long long *, u32 *,
                             unsigned long long *);

template <class K>
SlicedJobs plan_k(const SlicedLayout &l) {
  return SlicedJobs{(const void *)sliced_jobs_kernel<K>, K::T, K::T == 128 ? 1024 : 2 * K::T,
                    (l.words * 4 + 127) / 128 * 128, tc_sl_bytes<K>(l.words, l.chunks)};
}
template <int D>
SlicedJobs plan_d(const SlicedLayout &l, u64 n) {
  if constexpr (D == 13 || D == 14)
    return tc_sl_wide<D>(l.words, l.chunks, n) ? plan_k<TcSlWide<D>>(l) : plan_k<TcSlNarrow<D>>(l);
  else
    return plan_k<TcSlK<D, 4>>(l);
}

}  // namespace

SlicedJobs sliced_jobs(int d, const SlicedLayout &largest, uint64_t n) {
  switch (d) {
#define TC_CASE(x) \
  case x: return plan_d<x>(largest, n);
    TC_CASE(1) TC_CASE(2) TC_CASE(3) TC_CASE(4) TC_CASE(5) TC_CASE(6) TC_CASE(7) TC_CASE(8) TC_CASE(9)
    TC_CASE(10) TC_CASE(11) TC_CASE(12) TC_CASE(13) TC_CASE(14) TC_CASE(15) TC_CASE(16)
#undef TC_CASE
    default: return SlicedJobs{};
  }
}

cudaError_t sliced_jobs_launch(const SlicedJobs &p, unsigned grid, const DevJob *jobs, uint32_t njobs,
                               uint64_t items, uint32_t chunk, unsigned long long *work, uint32_t *err,
                               unsigned long long *failed, cudaStream_t st) {
  if (!p.fn) return cudaErrorInvalidValue;
  reinterpret_cast<SlicedJobsFn>(const_cast<void *>(p.fn))<<<grid, p.threads, p.smem, st>>>(
      jobs, njobs, items, chunk, p.toff, work, err, failed);
  return cudaGetLastError();
}

}  // namespace tcurve
