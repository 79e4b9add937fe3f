// block_sweep.cu -- exhaustive sweeps in whole blocks of middle-row patterns
// (tc_block_sweep.cuh): the kernel, and the split of a range into whole
// blocks, for 4 <= d <= 9.
//
// A persistent block takes 128 high parts at a time, or for short ranges one
// of 2^lparts equal parts of their patterns.  What bounds it is integer issue:
// at d = 7 the halves and their records take about as long as two words (64
// patterns) of the middle phase (ALU pipe 68 % busy, three blocks of 168
// registers per multiprocessor).  2^30 masks at d = 7: 162 ms (specialised block
// sweep) -> 10.5 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "engine.h"
#include "tc_block_sweep.cuh"
#include "tc_stage.cuh"

namespace tcurve {
namespace {

// Masks (h << oshift) | (t << ishift) for h = hi0 .. hi0 + n_hi - 1 (with
// TS_ENUM_ORBITS in flags, h = the block's high part, tc_orbit_high) and
// t < 2^ib, in work items of 128 high parts and 2^(ib - lparts) patterns.
// smem: tables (toff bytes) | mbarrier, work slot (128 bytes) |
// the areas | hash table.
template <int D>
__global__ void __launch_bounds__(128, D <= 7 ? 3 : 2)
    block_sweep_kernel(SlicedLayout L, const uint32_t *__restrict__ gtab, uint64_t hi0, uint64_t n_hi,
                       uint32_t oshift, uint32_t ishift, uint32_t ib, uint32_t lparts, uint32_t flags,
                       ts_hist h) {
  typedef TcSbK<D> K;
  typedef typename K::Base B;
  extern __shared__ __align__(128) uint8_t smem[];
  const uint32_t toff = (L.words * 4 + 127) / 128 * 128;
  u32 *const tab = reinterpret_cast<u32 *>(smem);
  u32 *const area = reinterpret_cast<u32 *>(smem + toff + 128);
  unsigned long long *const slot = reinterpret_cast<unsigned long long *>(smem + toff + 64);
  const TcSbMem M = tc_sb_carve<K>(tab, area, L.chunks);
  u64 *const hkeys = reinterpret_cast<u64 *>(area + tc_sb_words<K>(L.chunks));
  u32 *const hcnt = reinterpret_cast<u32 *>(hkeys + K::HASH);
  const TcSbOut out{hkeys, hcnt, reinterpret_cast<u64 *>(h.d_keys), h.d_counts, h.slots, h.d_err};
  const u32 t = threadIdx.x, mine = tc_sl_instance<B>(t), lw = ib - 5u - lparts;
  for (u32 s = t; s < K::HASH; s += K::T) {
    hkeys[s] = 0;
    hcnt[s] = 0;
  }
  for (u32 s = t; s < K::STARS; s += K::T) M.stars[s] = 0;
  if (t == 0) *M.queued = 0;
  if (t == 0) *slot = atomicAdd(h.d_work, 1ull);
  if (!stage_tables(tab, gtab, L.words * 4, reinterpret_cast<uint64_t *>(smem + toff), h.d_err)) return;
  uint32_t err = 0, items = 0;
  unsigned long long failed = 0;
  auto flush = [&] {  // the block's counts to the device table, by the thread that owns the slot
    for (u32 s = t; s < K::HASH; s += K::T)
      if (hcnt[s]) {
        tc_global_add(out.gkeys, h.d_counts, h.slots, h.d_err, hkeys[s], hcnt[s]);
        hcnt[s] = 0;
      }
    for (u32 R = t; R < K::STARS; R += K::T)
      if (M.stars[R]) {
        tc_global_add(out.gkeys, h.d_counts, h.slots, h.d_err, tc_sb_star_code(R), M.stars[R]);
        M.stars[R] = 0;
      }
    __syncthreads();
  };
  auto mask_of = [&](uint64_t i) -> u64 {  // of block i of the range, middle row zero
    const u64 u = hi0 + i;
    return ((flags & TS_ENUM_ORBITS) ? tc_orbit_high(u, flags) : u) << oshift;
  };
  for (;;) {
    const uint64_t item = *slot, base = (item >> lparts) * K::T;
    const u32 part = (u32)item & ((1u << lparts) - 1u);
    if (base >= n_hi) break;
    __syncthreads();
    // the next work item is fetched while this one runs
    if (t == 0) *slot = atomicAdd(h.d_work, 1ull);
    tc_sl_clear<B>(M.s, t);
    tc_sl_planes<B>(M.s, TcSig<1>{{base + t < n_hi ? mask_of(base + t) : 0ull}}, t);
    __syncthreads();
    tc_sl_logic<B>(M.s, t);
    __syncthreads();
    tc_sl_tiles<B>(M.s, t);
    tc_sl_events<B>(M.s, t);
    __syncthreads();
    const bool live = base + mine < n_hi;
    const u64 sig = live ? mask_of(base + mine) : 0ull;
    tc_sb_record<K>(M, t, sig);
    if (!live) M.rec[K::R_HDR * K::T + t] = 1u << 31;  // behind the range
    __syncthreads();
    for (u32 task = t; task < K::T << lw; task += K::T) {
      const u32 hl = task >> lw, w = part << lw | (task & ((1u << lw) - 1u)), hdr = M.rec[K::R_HDR * K::T + hl];
      const bool valid = (hdr >> 25) & 1u;
      // the larger size when a lane of the warp needs it
      if (__any_sync(0xffffffffu, valid && ((hdr >> 8) & 255u) > K::NA)) {
        if (valid) tc_sb_middle<K, K::NB>(M, t, hl, w, ishift, out, err, failed);
      } else if (valid) {
        tc_sb_middle<K, K::NA>(M, t, hl, w, ishift, out, err, failed);
      }
      tc_sb_flush_queue<K>(M, t, task + K::T >= K::T << lw, out, err, failed);
    }
    for (u32 hl = 0; hl < K::T; ++hl) {  // high parts the middle phase does not take
      const u32 hdr = M.rec[K::R_HDR * K::T + hl];
      if ((hdr >> 25) & 1u || hdr >> 31) continue;
      const u64 hm = mask_of(base + tc_sl_instance<B>(hl));
      const u32 pend = (part + 1u) << (lw + 5u);
      for (u32 p = part << (lw + 5u); p < pend; p += K::T) {
        u32 e = 0;
        u64 code = 0;
        tc_sl_classify<B>(M.s, TcSig<1>{{hm | ((u64)(p + t < pend ? p + t : p) << ishift)}}, t, e, &code);
        const bool in = p + mine < pend;
        code = in ? code : 0ull;
        err |= in ? e : 0u;
        failed += in && code == 0;
        if (code) tc_sb_insert<K::HASH>(code, 1, hkeys, hcnt, out.gkeys, h.d_counts, h.slots, h.d_err);
        __syncthreads();
      }
    }
    __syncthreads();
    // at most 2^10 patterns per high part: counts stay below 2^32 for fewer than
    // 2^15 items
    if ((++items & 63u) == 0) flush();
  }
  __syncthreads();
  flush();
  if (err) atomicOr(h.d_err, err);
  if (failed) atomicAdd(h.d_failed, failed);
}

struct Split {
  uint32_t ib, ishift, oshift;
};

template <int D>
cudaError_t launch_d(const ts_tri *t, uint64_t h0, uint64_t n, const Split &s, uint32_t flags, ts_hist *h,
                     cudaStream_t st) {
  typedef TcSbK<D> K;
  const size_t smem = (t->slay.words * 4 + 127) / 128 * 128 + 128 +
                      (size_t)tc_sb_words<K>(t->slay.chunks) * 4 + (size_t)K::HASH * 16;
  cudaError_t e = cudaFuncSetAttribute(block_sweep_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kMaxBlockSmem);
  int per_sm = 0, sms = 0, dev = 0;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, block_sweep_kernel<D>, 128, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  e = cudaMemsetAsync(h->d_work, 0, sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  // Parts: those for which the items' time on the blocks the device holds plus
  // one item's (the last to start; high parts differ, so no wave is full) is
  // least, in words of the middle phase, the halves counted as two (0.28, 0.45,
  // 0.57 of 6.6, 4.4, 2.5 ms at d = 9, 8, 7).  One part -> these: 2^19 masks
  // 736, 306, 114 -> 100, 80, 64 us; d = 9, three ranges each, 2^24 masks 1.38,
  // 0.95, 2.1 -> 0.80, 0.72, 0.90 ms, 2^26 modulo the flip 3.9, 2.1, 4.6 -> 3.3,
  // 2.2, 3.6 ms.  Counting full waves instead: 1.01, 0.74, 1.37 and 3.6, 2.2, 3.5.
  const uint64_t groups = (n + 127) / 128, held = (uint64_t)per_sm * sms;
  uint32_t lparts = 0;
  uint64_t best = ~0ull;
  for (uint32_t l = 0; l <= s.ib - 5; ++l) {
    const uint64_t time = ((groups << l) + held) * (2 + (1ull << (s.ib - 5 - l)));
    if (time < best) {
      best = time;
      lparts = l;
    }
  }
  const unsigned grid = (unsigned)std::min<uint64_t>(groups << lparts, held);
  block_sweep_kernel<D><<<grid, 128, smem, st>>>(t->slay, t->d_stables, h0, n, s.oshift, s.ishift, s.ib, lparts,
                                                 flags, *h);
  return cudaGetLastError();
}

cudaError_t launch(const ts_tri *t, uint64_t h0, uint64_t n, const Split &s, uint32_t flags, ts_hist *h,
                   cudaStream_t st) {
  switch (t->d) {
    case 4: return launch_d<4>(t, h0, n, s, flags, h, st);
    case 5: return launch_d<5>(t, h0, n, s, flags, h, st);
    case 6: return launch_d<6>(t, h0, n, s, flags, h, st);
    case 7: return launch_d<7>(t, h0, n, s, flags, h, st);
    case 8: return launch_d<8>(t, h0, n, s, flags, h, st);
    case 9: return launch_d<9>(t, h0, n, s, flags, h, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

// In terms of the sweep index k, the mask m(k) is (h << oshift) |
// (t << ishift) with t = k mod 2^ib the middle-row pattern (ib free
// middle-row bits) and h = k >> ib (with TS_ENUM_ORBITS its high part with
// the pivots zero, tc_orbit_high).
bool block_range(const ts_tri *t, uint64_t lo, uint64_t hi, uint32_t flags, uint64_t *a, uint64_t *b) {
  if (t->d < 4 || t->d > 9 || (flags & TS_ENUM_SPLITMIX)) return false;
  // More open components than the middle phase holds: the sliced kernel's own
  // sweep, with more blocks per multiprocessor and no halves in vain (2^22 masks
  // of three triangulations each, in this kernel -> there: d = 6 4.0 -> 0.73 ms,
  // d = 8 6.2 -> 1.5, d = 9 6.7 -> 2.0; specialised 1.3, 1.8 and 1.7).
  if (t->open > tc_block_nodes(t->d)) return false;
  const uint32_t ib = t->d + 1 - ((flags & TS_ENUM_FLIP) ? 1 : 0) - ((flags & TS_ENUM_REDUCED) ? 2 : 0);
  if (ib < 5) return false;  // fewer patterns than a word has bits
  const uint64_t first = (lo >> ib) + ((lo & ((1ull << ib) - 1)) != 0), last = hi >> ib;
  if (first >= last || last - first < (kBlockSweepMin >> ib)) return false;
  *a = first << ib;
  *b = last << ib;
  return true;
}

cudaError_t launch_block_sweep(const ts_tri *t, uint64_t lo, uint64_t hi, uint32_t flags, ts_hist *h,
                               cudaStream_t st) {
  const int d = t->d;
  Split s{(uint32_t)d + 1, 0, (uint32_t)d + 1};
  if (flags & TS_ENUM_FLIP) s = Split{(uint32_t)d, 1, (uint32_t)d + 1};
  if (flags & TS_ENUM_REDUCED) s = Split{(uint32_t)d - 1, 2, (uint32_t)d + 2};
  if (flags & TS_ENUM_ORBITS) s.oshift = d + 2;
  uint64_t h0 = lo >> s.ib, h1 = hi >> s.ib;  // whole blocks [h0, h1)
  cudaError_t e = cudaSuccess;
  if (flags & TS_ENUM_FLIP) {
    // Global sign flip: block h (masks with bit 0 clear) and block M - h (all
    // high bits complemented) hold one representative of each class {sigma,
    // ~sigma} whose high part is h or M - h; flipping the second block's masks
    // gives block h with bit 0 set.  So a pair of blocks in the range is swept
    // as the one unreduced block h with all 2^(d+1) patterns: the same schemes
    // (the flip keeps the curve), and the halves once for both.  Paired: h in
    // [p, q] (symmetric about M / 2, both ends in the range); the rest as is.
    const uint64_t M = (1ull << (t->np - 1 - s.ib)) - 1;
    const uint64_t p = std::max<uint64_t>(h0, h1 > M ? 0 : M + 1 - h1);
    const uint64_t q1 = std::min<uint64_t>(h1, h0 > M ? 0 : M - h0 + 1);  // q + 1
    if (p < q1) {
      const uint64_t half = (q1 - p) / 2;  // q1 - p is even: p + q = M, M odd
      if (h0 < p && (e = launch(t, h0, p - h0, s, 0, h, st)) != cudaSuccess) return e;
      if ((e = launch(t, p, half, Split{(uint32_t)d + 1, 0, (uint32_t)d + 1}, 0, h, st)) != cudaSuccess)
        return e;
      h0 = q1;
    }
  }
  return h0 < h1 ? launch(t, h0, h1 - h0, s, flags & (TS_ENUM_ORBITS | 0xFFFF00u), h, st) : e;
}

}  // namespace tcurve
