// batch.cu -- many triangulations of mixed degree in one graph launch.
//
// A batch is a list of jobs (triangulation, number of sign vectors, splitmix64
// stream of the sign vectors, optional code output).  For each degree present
// the batch runs ONE persistent kernel over all jobs of that degree: blocks
// pull (job, chunk) work items from a counter, re-stage a job's tables into
// shared memory with cp.async.bulk when the job changes, generate the sign
// vectors on the device, classify them with Algorithm 1 (bit-sliced,
// sliced_jobs.cu; other tiles than the default with one thread per sign
// vector) and add the codes to the job's own device hash histogram
// (warp-aggregated atomics).  The per-degree kernels run on forked streams
// inside one CUDA graph that is captured on the first run and replayed after;
// each degree has its own tile shape (threads per block, instances per work
// item, scratch in shared or global memory), which ts_batch_set_tile
// changes (the autotuner's knob).
//
// A degree group with many sign vectors (or whose triangulations ask for
// TS_KERNEL_SPECIALIZED) runs specialised code instead: its persistent
// kernel tcj_jobs (jit.cpp) calls, per job, the straight-line sweep generated
// for that job's triangulation; all of the batch's objects are compiled in
// parallel at creation and linked per degree.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "engine.h"
#include "tc_layout.h"
#include "tc_stage.cuh"
#include "tc_table_sweep.cuh"

namespace tcurve {
namespace {

// Largest table of degree d: 2V + |E(T^diamond)| words, V = 2d^2 + 2d + 1 and
// |E(T^diamond)| = 6d^2 + 2d, padded to 16 bytes.
constexpr size_t max_table_bytes(int d) {
  return (size_t)(((10 * d * d + 6 * d + 2) + 3) & ~3) * 4;
}

// Degree-D_ kernel with T_ threads per block; per-thread scratch in shared
// memory, or (G_) in global memory, L1/L2-resident.
template <int D_, int T_, bool G_>
struct JobK : TcTableK<D_, T_, true> {
  static constexpr bool fits = JobK::L.ok && (max_table_bytes(D_) + 127) / 128 * 128 + 128 +
                                                     (G_ ? 0 : (size_t)JobK::WORDS * 4 * T_) <=
                                                 227 * 1024;
};


// Degree groups of at least this many sign vectors run specialised code
// (TS_KERNEL_AUTO, d <= kMaxBatchSpecialized), compiled at creation (about a
// second per triangulation, in parallel).  The rule is from before the
// bit-sliced kernels, which are faster now: four jobs of 2^20 at d = 3, 4, 5, 6
// 0.43, 0.96, 1.30, 2.68 ms specialised, 0.25, 0.46, 0.48, 0.80 bit-sliced
// (TS_KERNEL_TABLE or ts_batch_set_fused takes them).
constexpr uint64_t kJitGroupMin = 1ull << 22;

template <int D, int T, bool G>
__global__ void __launch_bounds__(T)
    jobs_kernel(const DevJob *__restrict__ jobs, u32 njobs, u64 total_items, u32 chunk,
                u32 table_words, u32 off_fan, u32 off_vext, unsigned long long *work, u32 *err_word,
                unsigned long long *failed_word, u32 *gscratch) {
  typedef JobK<D, T, G> K;
  extern __shared__ __align__(128) uint8_t smem[];
  u32 *tab = reinterpret_cast<u32 *>(smem);
  const size_t toff = ((size_t)table_words * 4 + 127) / 128 * 128;
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem + toff);
  unsigned long long *slot = reinterpret_cast<unsigned long long *>(smem + toff + 64);
  const TcScratch<K> S{(G ? gscratch + (size_t)blockIdx.x * K::WORDS * T
                         : reinterpret_cast<u32 *>(smem + toff + 128)) +
                        threadIdx.x};
  // global scratch: the label slots of the sweep in shared memory
  u32 *const ls = G ? reinterpret_cast<u32 *>(smem + toff + 128) + threadIdx.x : nullptr;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(1u));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const u32 lane = threadIdx.x & 31u;
  u32 cur = 0xFFFFFFFFu, phase = 0, err = 0;
  unsigned long long failed = 0;
  for (;;) {
    if (threadIdx.x == 0) *slot = atomicAdd(work, 1ull);
    __syncthreads();
    const u64 c = *slot;
    __syncthreads();  // also: every thread is done with the previous job's tables
    if (c >= total_items) break;
    u32 lo = 0, hi = njobs;  // the job holding item c: last j with chunk0 <= c
    while (hi - lo > 1) {
      const u32 mid = (lo + hi) / 2;
      if (jobs[mid].chunk0 <= c) lo = mid; else hi = mid;
    }
    const u32 j = lo;
    if (j != cur) {  // stage the job's tables (cp.async.bulk, bounded wait)
      if (threadIdx.x == 0) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                     "r"(table_words * 4u) : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
                "r"(smem_u32(tab)), "l"(jobs[j].tab), "r"(table_words * 4u), "r"(smem_u32(bar))
            : "memory");
      }
      bool ok = false;
      for (long it = 0; it < kWaitIters && !ok; ++it) {
        uint32_t r;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}"
            : "=r"(r) : "r"(smem_u32(bar)), "r"(phase) : "memory");
        ok = r != 0;
      }
      if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) atomicOr(err_word, kErrTimeout);
        for (long it = 0; it < kWaitIters && !ok; ++it) {
          uint32_t r;
          asm volatile(
              "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
              " selp.u32 %0, 1, 0, p;\n}"
              : "=r"(r) : "r"(smem_u32(bar)), "r"(phase) : "memory");
          ok = r != 0;
        }
        return;
      }
      phase ^= 1u;
      cur = j;
      if (G) {  // label slots in shared memory, found by the fan entries' offsets
        tc_fan_to_offsets(tab + off_fan, off_vext - off_fan, TcScratch<K>::EPW, K::LBYTES, T,
                          threadIdx.x, T);
        __syncthreads();
      }
    }
    const DevJob J = jobs[j];
    const u64 first = (c - J.chunk0) * (u64)chunk;
    for (u32 k = 0; k < chunk; k += T) {
      const u64 idx = first + k + threadIdx.x;
      TcCodeOut<K> key{};
      if (idx < J.n) {
        // the sign vector of counter base + idx, as ts_splitmix_masks writes it
        TcSig<K::W> sg;
#pragma unroll
        for (u32 w = 0; w < K::W; ++w) sg.w[w] = tc_splitmix64((J.base + idx) * K::W + w);
        sg.w[K::W - 1] &= tc_top_mask(K::NPOINTS, K::W);
        key = tc_table_classify<K, G>(sg, tab, off_fan, off_vext, S, err, ls);
        u64 any = 0;
#pragma unroll
        for (u32 w = 0; w < K::CW; ++w) {
          any |= key.w[w];
          if (J.codes) J.codes[idx * K::CW + w] = key.w[w];
        }
        failed += any == 0;
      }
      if constexpr (K::CW == 1) {
        const unsigned peers = __match_any_sync(0xffffffffu, key.w[0]);
        if (key.w[0] != 0 && lane == (u32)(__ffs(peers) - 1))
          tc_global_add(J.hkeys, J.hcnt, J.hslots, err_word, key.w[0],
                        (unsigned long long)__popc(peers));
      } else {
        tc_hist_add_wide<K::CW>(key.w, J.hkeys, J.hcnt, J.hslots, err_word);
      }
    }
  }
  if (err) atomicOr(err_word, err);
  if (failed) atomicAdd(failed_word, failed);
}

// (degree, threads, scratch) -> kernel; only instantiations whose block fits.
typedef void (*JobsFn)(const DevJob *, u32, u64, u32, u32, u32, u32, unsigned long long *, u32 *,
                       unsigned long long *, u32 *);

template <int D, int T, bool G>
JobsFn jobs_fn() {
  if constexpr (JobK<D, T, G>::fits) return jobs_kernel<D, T, G>;
  else return nullptr;
}

template <int D, bool G>
JobsFn jobs_fn_tg(int t) {
  switch (t) {
    case 32: return jobs_fn<D, 32, G>();
    case 64: return jobs_fn<D, 64, G>();
    case 96: return jobs_fn<D, 96, G>();
    case 128:  // bit-sliced unless the scratch is global (table_tile)
      if constexpr (G) return jobs_fn<D, 128, G>();
      else return nullptr;
    case 192: return jobs_fn<D, 192, G>();
    case 256: return jobs_fn<D, 256, G>();
    default: return nullptr;
  }
}

template <int D>
JobsFn jobs_fn_t(int t, bool g) {
  return g ? jobs_fn_tg<D, true>(t) : jobs_fn_tg<D, false>(t);
}

JobsFn jobs_fn_dt(int d, int t, bool g) {
  switch (d) {
    case 1: return jobs_fn_t<1>(t, g);
    case 2: return jobs_fn_t<2>(t, g);
    case 3: return jobs_fn_t<3>(t, g);
    case 4: return jobs_fn_t<4>(t, g);
    case 5: return jobs_fn_t<5>(t, g);
    case 6: return jobs_fn_t<6>(t, g);
    case 7: return jobs_fn_t<7>(t, g);
    case 8: return jobs_fn_t<8>(t, g);
    case 9: return jobs_fn_t<9>(t, g);
    case 10: return jobs_fn_t<10>(t, g);
    case 11: return jobs_fn_t<11>(t, g);
    case 12: return jobs_fn_t<12>(t, g);
    case 13: return jobs_fn_t<13>(t, g);
    case 14: return jobs_fn_t<14>(t, g);
    case 15: return jobs_fn_t<15>(t, g);
    case 16: return jobs_fn_t<16>(t, g);
    default: return nullptr;
  }
}

// ls_words: label-slot words per thread (global scratch: kept in shared memory)
size_t jobs_smem(int d, int t, uint32_t table_words, uint32_t ls_words, bool g) {
  const TcLayout L = tc_layout(d, true, t);
  return ((size_t)table_words * 4 + 127) / 128 * 128 + 128 +
         (g ? (size_t)ls_words * 4 * t : (size_t)L.words * 4 * t);
}

size_t scratch_words(int d, int t) { return (size_t)tc_layout(d, true, t).words * t; }

ts_status cuda_st(cudaError_t e) {
  if (e == cudaSuccess) return TS_OK;
  return e == cudaErrorMemoryAllocation ? TS_ENOMEM : TS_ECUDA;
}

// Makes a device current for a scope (its calls are ordered by that device's
// legacy stream), then the caller's again.
struct DeviceScope {
  cudaError_t status = cudaSuccess;
  int device = -1;  // the caller's, if it is another
  explicit DeviceScope(int wanted) {
    int now = wanted;
    status = cudaGetDevice(&now);
    if (status != cudaSuccess || now == wanted) return;
    status = cudaSetDevice(wanted);
    if (status == cudaSuccess) device = now;
  }
  ~DeviceScope() {
    if (device >= 0) cudaSetDevice(device);
  }
};

// Packed histogram of one job: entries found, failed instances, error word, 0;
// then per entry its code words and its count.
constexpr uint64_t kPackHeader = 4;
constexpr uint64_t kPackMax = 1 << 14;   // entries there is room for
constexpr uint64_t kPackFirst = 1 << 10;  // entries read along with the header

// The occupied slots (a nonzero key word) of a job's table, in any order, at
// most cap of them stored: one atomic per warp, lanes ranked by a ballot.
// Bound by the table's bytes (512 KB of 2^15 slots: 3 us).
__global__ void batch_pack_kernel(const uint64_t *__restrict__ keys, const unsigned long long *__restrict__ counts,
                                  uint64_t slots, int cw, uint64_t cap, const uint32_t *err,
                                  const unsigned long long *failed, unsigned long long *out) {
  const uint32_t lane = threadIdx.x & 31u;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    out[1] = *failed;
    out[2] = *err;
  }
  for (uint64_t base = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31ull; base < slots;
       base += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t s = base + lane;
    bool nz = false;
    if (s < slots)
      for (int w = 0; w < cw; ++w) nz |= keys[s * cw + w] != 0;
    const unsigned ball = __ballot_sync(0xffffffffu, nz);
    unsigned long long first = 0;
    if (lane == 0 && ball) first = atomicAdd(out, (unsigned long long)__popc(ball));
    first = __shfl_sync(0xffffffffu, first, 0);
    const uint64_t o = first + __popc(ball & ((1u << lane) - 1u));
    if (nz && o < cap) {
      unsigned long long *e = out + kPackHeader + o * (cw + 1);
      for (int w = 0; w < cw; ++w) e[w] = keys[s * cw + w];
      e[cw] = counts[s] & kCountMask;
    }
  }
}

}  // namespace
}  // namespace tcurve

using namespace tcurve;

struct ts_batch {
  struct Group {  // all jobs of one degree
    int d = 0, threads = 64, chunk = 1024;
    bool global = false;        // per-thread scratch in global memory
    bool sliced = false;        // the bit-sliced kernel (shared memory)
    SlicedLayout slargest{};    // its largest tables and most event chunks
    uint64_t n = 0;             // sign vectors of its jobs
    SlicedJobs splan;
    std::shared_ptr<JitJobsModule> jit;  // specialised kernel (null: table-driven)
    std::string jit_log;        // why the specialised kernel could not be built
    JobsFn fn = nullptr;        // the kernel of this tile, its launch shape
    size_t smem = 0;
    unsigned grid = 1;
    u32 *scratch = nullptr;     // global scratch (grid x threads x words)
    size_t scratch_bytes = 0;
    uint32_t table_words = 0, off_fan = 0, off_vext = 0;
    uint32_t ls_words = 0;      // label-slot words per thread (largest of the group's tables)
    std::vector<int> jobs;      // indices into the batch's job list
    DevJob *d_jobs = nullptr;   // device job table (sorted as `jobs`)
    uint64_t items = 0;
    unsigned long long *d_work = nullptr;
    cudaStream_t stream = nullptr;
    cudaEvent_t done = nullptr;
    int fwarp = 0;              // fused launch: warp (1) or thread (0) per instance
    int fchunk = kFusedThreads * 8;  // fused launch: sign vectors per work item
  };
  std::vector<DevJob> jobs;  // host copies (chunk0 per group)
  std::vector<int> degree, cws;       // degree and code words of every job
  std::vector<size_t> kofs;           // first key word of every job's histogram
  std::vector<size_t> cofs;           // first count of every job's histogram
  std::vector<uint64_t> jslots;       // slots of every job's histogram
  size_t key_words = 0, count_words = 0;
  std::vector<Group> groups;
  uint64_t *d_keys = nullptr;  // per job: slots x code_words
  unsigned long long *d_counts = nullptr;
  uint32_t *d_err = nullptr;
  unsigned long long *d_failed = nullptr;
  std::mutex read_mu;               // of the packed entries (ts_batch_read)
  unsigned long long *d_pack = nullptr;  // kPackHeader words, then pack_cap entries
  uint64_t pack_cap = 0;
  cudaEvent_t fork = nullptr;
  cudaGraphExec_t exec = nullptr;
  int device = 0;
  std::vector<ts_tri *> tris;  // triangulation of every job
  std::vector<const uint64_t *> signs;  // caller sign vectors of every job (null: splitmix64)
  bool serial = false;         // degree groups one after the other (else concurrent streams)
  // fused plan (ts_batch_set_fused): one persistent kernel per tier of degrees
  struct Tier {
    int tier = -1;
    uint32_t job0 = 0, njobs = 0, toff = 0, ws = 0;
    uint64_t items = 0;
    unsigned grid = 1;
    size_t smem = 0;
  };
  bool fused = false;
  std::vector<Tier> tiers;     // largest degrees first
  FusedJob *d_fjobs = nullptr;  // jobs tier by tier
  unsigned long long *d_fwork = nullptr;  // one counter per tier
  cudaStream_t fstream[kFusedTiers + 1] = {};  // of the tiers after the first
  cudaEvent_t fdone[kFusedTiers + 1] = {};
};

namespace {

cudaError_t upload_group(ts_batch *b, ts_batch::Group &g) {
  std::vector<DevJob> dj;
  uint64_t items = 0;
  for (int j : g.jobs) {
    DevJob x = b->jobs[j];
    x.chunk0 = items;
    items += (x.n + g.chunk - 1) / g.chunk;
    dj.push_back(x);
  }
  g.items = items;
  if (!g.d_jobs) {
    cudaError_t e = cudaMalloc(&g.d_jobs, sizeof(DevJob) * dj.size());
    if (e != cudaSuccess) return e;
  }
  return cudaMemcpy(g.d_jobs, dj.data(), sizeof(DevJob) * dj.size(), cudaMemcpyHostToDevice);
}

// Kernel, shared memory, persistent grid and global scratch of the group's
// tile (host work only: done at creation and on a tile change, never while a
// stream is being captured).
cudaError_t prepare_group(ts_batch::Group &g) {
  int per_sm = 0, sms = 0, dev = 0;
  cudaError_t e = cudaSuccess;
  if (!g.jit && g.sliced) {
    g.splan = sliced_jobs(g.d, g.slargest, g.n);
    if (!g.splan.fn) return cudaErrorInvalidConfiguration;
    g.fn = nullptr;
    g.smem = g.splan.smem;
    e = cudaFuncSetAttribute(g.splan.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxBlockSmem);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, g.splan.fn, g.splan.threads, g.smem);
    if (e != cudaSuccess) return e;
  } else if (g.jit) {  // specialised: 128-thread blocks, global scratch, grid from its occupancy
    g.fn = nullptr;
    g.smem = 0;
    per_sm = jit_jobs_blocks_per_sm(*g.jit);
  } else {
    g.fn = jobs_fn_dt(g.d, g.threads, g.global);
    if (!g.fn) return cudaErrorInvalidConfiguration;
    g.smem = jobs_smem(g.d, g.threads, g.table_words, g.ls_words, g.global);
    // whichever batch was planned last, every launch may have its own size
    e = cudaFuncSetAttribute((const void *)g.fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kMaxBlockSmem);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void *)g.fn, g.threads, g.smem);
    if (e != cudaSuccess) return e;
  }
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const uint64_t cap = (uint64_t)per_sm * sms;
  g.grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(cap, g.items));
  if (g.global) {
    const size_t need = g.jit ? (size_t)g.grid * jit_jobs_slab_bytes(*g.jit)
                              : (size_t)g.grid * scratch_words(g.d, g.threads) * 4;
    if (need > g.scratch_bytes) {
      if (g.scratch) cudaFree(g.scratch);
      g.scratch = nullptr;
      g.scratch_bytes = 0;
      e = cudaMalloc(&g.scratch, need);
      if (e != cudaSuccess) return e;
      g.scratch_bytes = need;
    }
  }
  return cudaSuccess;
}

cudaError_t launch_group(ts_batch *b, ts_batch::Group &g, cudaStream_t st) {
  if (!g.fn && !g.jit && !g.sliced) return cudaErrorInvalidConfiguration;
  cudaError_t e = cudaMemsetAsync(g.d_work, 0, sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  if (!g.jit && g.sliced)
    return sliced_jobs_launch(g.splan, g.grid, g.d_jobs, (uint32_t)g.jobs.size(), g.items,
                              (uint32_t)g.chunk, g.d_work, b->d_err, b->d_failed, st);
  if (g.jit)
    return jit_jobs_launch(*g.jit, g.grid, g.d_jobs, (uint32_t)g.jobs.size(), g.items,
                           (uint32_t)g.chunk, g.d_work, b->d_err, b->d_failed, g.scratch, st);
  g.fn<<<g.grid, g.threads, g.smem, st>>>(g.d_jobs, (u32)g.jobs.size(), g.items, (u32)g.chunk,
                                          g.table_words, g.off_fan, g.off_vext, g.d_work, b->d_err,
                                          b->d_failed, g.scratch);
  return cudaGetLastError();
}

// Job table and launches of the fused plan (host work only, never while a
// stream is captured): the jobs tier by tier, each with its degree's tile,
// and per tier the shared memory of its largest job and a persistent grid.
cudaError_t prepare_fused(ts_batch *b) {
  std::vector<FusedJob> fj;
  std::vector<ts_batch::Tier> tiers;
  int sms = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  for (int tier = kFusedTiers; tier >= 0; --tier) {
    ts_batch::Tier T;
    T.tier = tier;
    T.job0 = (uint32_t)fj.size();
    uint32_t maxtab = 0;
    size_t area = 0;
    for (const auto &g : b->groups) {
      if ((g.fwarp ? kFusedWarpTier : fused_tier(g.d)) != tier) continue;
      for (int j : g.jobs) {
        const DevJob &dj = b->jobs[j];
        const ts_tri *t = b->tris[j];
        FusedJob x{};
        x.n = dj.n;
        x.base = dj.base;
        x.codes = dj.codes;
        x.hkeys = dj.hkeys;
        x.hcnt = dj.hcnt;
        x.hslots = dj.hslots;
        x.item0 = T.items;
        x.signs = reinterpret_cast<const unsigned long long *>(b->signs[j]);
        x.d = (uint32_t)g.d;
        x.chunk = (uint32_t)g.fchunk;
        x.sl = t->slay;
        x.wl = t->wlay;
        if (g.fwarp) {
          x.tab = t->d_wtables;
          x.tab_words = t->wlay.words;
          T.ws = std::max(T.ws, fused_warp_words(g.d));
          area = std::max(area, (size_t)4 * T.ws * 4);
        } else {
          x.tab = t->d_stables;
          x.tab_words = t->slay.words;
          area = std::max(area, fused_area_bytes(g.d, t->slay));
        }
        maxtab = std::max(maxtab, x.tab_words);
        T.items += (x.n + x.chunk - 1) / x.chunk;
        fj.push_back(x);
      }
    }
    T.njobs = (uint32_t)fj.size() - T.job0;
    if (!T.njobs) continue;
    T.toff = (maxtab * 4 + 127) / 128 * 128;
    T.smem = (size_t)T.toff + 128 + area;
    if (T.smem > (size_t)kMaxBlockSmem) return cudaErrorInvalidConfiguration;
    int per_sm = 0;
    cudaError_t e = fused_occupancy(tier, T.smem, &per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    T.grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)per_sm * sms, T.items));
    tiers.push_back(T);
  }
  if (fj.empty()) return cudaErrorInvalidConfiguration;
  cudaError_t e = cudaSuccess;
  for (size_t k = 1; k < tiers.size() && e == cudaSuccess; ++k) {
    if (!b->fstream[k]) e = cudaStreamCreateWithFlags(&b->fstream[k], cudaStreamNonBlocking);
    if (e == cudaSuccess && !b->fdone[k]) e = cudaEventCreateWithFlags(&b->fdone[k], cudaEventDisableTiming);
  }
  if (e == cudaSuccess && !b->d_fjobs) e = cudaMalloc(&b->d_fjobs, sizeof(FusedJob) * fj.size());
  if (e == cudaSuccess && !b->d_fwork) e = cudaMalloc(&b->d_fwork, sizeof(unsigned long long) * (kFusedTiers + 1));
  if (e == cudaSuccess)
    e = cudaMemcpy(b->d_fjobs, fj.data(), sizeof(FusedJob) * fj.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return e;
  b->tiers = tiers;
  return cudaSuccess;
}

// The whole batch as stream work on `st`: clear, then either the fused
// launch or fork, one kernel per degree, join.
cudaError_t enqueue(ts_batch *b, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(b->d_keys, 0, b->key_words * 8, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(b->d_counts, 0, b->count_words * 8, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(b->d_err, 0, 4, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(b->d_failed, 0, 8, st);
  if (b->fused) {  // one persistent kernel per tier, the later ones on forked streams
    if (e == cudaSuccess)
      e = cudaMemsetAsync(b->d_fwork, 0, sizeof(unsigned long long) * (kFusedTiers + 1), st);
    if (e == cudaSuccess && b->tiers.size() > 1) e = cudaEventRecord(b->fork, st);
    for (size_t k = 0; k < b->tiers.size(); ++k) {
      const auto &T = b->tiers[k];
      cudaStream_t s = k ? b->fstream[k] : st;
      if (e == cudaSuccess && k) e = cudaStreamWaitEvent(s, b->fork, 0);
      if (e == cudaSuccess)
        e = fused_launch(T.tier, T.grid, T.smem, T.toff, T.ws, b->d_fjobs + T.job0, T.njobs, T.items,
                         b->d_fwork + k, b->d_err, b->d_failed, s);
      if (e == cudaSuccess && k) e = cudaEventRecord(b->fdone[k], s);
      if (e == cudaSuccess && k) e = cudaStreamWaitEvent(st, b->fdone[k], 0);
    }
    return e;
  }
  if (b->serial) {  // one degree after the other, each persistent kernel on the whole GPU
    for (auto &g : b->groups)
      if (e == cudaSuccess) e = launch_group(b, g, st);
    return e;
  }
  if (e == cudaSuccess) e = cudaEventRecord(b->fork, st);
  for (auto &g : b->groups) {
    if (e == cudaSuccess) e = cudaStreamWaitEvent(g.stream, b->fork, 0);
    if (e == cudaSuccess) e = launch_group(b, g, g.stream);
    if (e == cudaSuccess) e = cudaEventRecord(g.done, g.stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, g.done, 0);
  }
  return e;
}

// Tile of a table-driven group: the bit-sliced kernel for blocks of 128
// threads unless global scratch is asked for, else the sweep with one thread
// per sign vector, its scratch placed as asked (TS_SCRATCH_AUTO: global from
// d = 7).
void table_tile(ts_batch::Group &g, int threads, int chunk, int scratch) {
  g.sliced = threads == kSlicedThreads && scratch != TS_SCRATCH_GLOBAL;
  g.global = !g.sliced && (scratch == TS_SCRATCH_GLOBAL ||
                           (scratch == TS_SCRATCH_AUTO && g.d >= kGlobalScratchFrom));
  g.threads = threads;
  g.chunk = chunk;
}
void table_defaults(ts_batch::Group &g) {
  g.jit.reset();
  table_tile(g, kSlicedThreads, (int)sliced_jobs(g.d, g.slargest, g.n).chunk, TS_SCRATCH_AUTO);
}

// TS_KERNEL_AUTO at creation: specialised code for groups of at least
// kJitGroupMin sign vectors up to degree kMaxBatchSpecialized, or when a
// triangulation of the group asks for it; never when one asks for tables.
bool wants_specialised(const ts_batch *b, const ts_batch::Group &g) {
  bool table = false, forced = false;
  uint64_t total = 0;
  for (int j : g.jobs) {
    table |= b->tris[j]->kernel == TS_KERNEL_TABLE;
    forced |= b->tris[j]->kernel == TS_KERNEL_SPECIALIZED;
    total += b->jobs[j].n;
  }
  return !table && (forced || (total >= kJitGroupMin && g.d <= kMaxBatchSpecialized));
}

// Build the specialised modules of the groups `gids` at once (one parallel
// compile): every job gets the index of its triangulation's function (one
// per distinct ts_tri of the group).  A group whose module cannot be built
// gets the table-driven tile and the log.  Returns false if any failed.
bool make_specialised(ts_batch *b, const std::vector<int> &gids) {
  if (gids.empty()) return true;
  std::vector<std::vector<const Diamond *>> want;
  std::vector<int> min_blocks;
  for (int gi : gids) {
    auto &g = b->groups[gi];
    std::map<const ts_tri *, uint32_t> fn;
    std::vector<const Diamond *> dias;
    int occ = 0;  // a register budget asked for with ts_set_occupancy
    for (int j : g.jobs) {
      occ = std::max(occ, b->tris[j]->occupancy);
      auto it = fn.find(b->tris[j]);
      if (it == fn.end()) {
        it = fn.emplace(b->tris[j], (uint32_t)dias.size()).first;
        dias.push_back(&b->tris[j]->dia);
      }
      b->jobs[j].fn = it->second;
    }
    want.push_back(dias);
    min_blocks.push_back(occ);
  }
  std::vector<std::shared_ptr<JitJobsModule>> mods;
  std::vector<std::string> logs;
  jit_jobs_build(want, min_blocks, &mods, &logs);
  bool all = true;
  for (size_t k = 0; k < gids.size(); ++k) {
    auto &g = b->groups[gids[k]];
    if (k < mods.size() && mods[k]) {
      g.jit = mods[k];
      g.jit_log.clear();
      g.global = true;
      g.sliced = false;
      g.threads = jit_jobs_threads();
      g.chunk = g.threads * 16;
    } else {
      table_defaults(g);
      g.jit_log = k < logs.size() && !logs[k].empty() ? logs[k] : "specialised batch kernel unavailable";
      all = false;
    }
  }
  return all;
}

}  // namespace

extern "C" {

ts_status ts_batch_create(int njobs, ts_tri *const *tris, const uint64_t *counts,
                          const uint64_t *bases, uint64_t *const *code_outputs,
                          uint64_t hist_capacity, ts_batch **out) {
  if (!out || njobs < 1 || !tris || !counts || !bases || hist_capacity == 0 ||
      hist_capacity > (1u << 20))
    return TS_EINVAL;
  *out = nullptr;
  ts_batch *b = new (std::nothrow) ts_batch();
  if (!b) return TS_ENOMEM;
  cudaError_t e = cudaGetDevice(&b->device);
  for (int j = 0; j < njobs; ++j) {
    if (!tris[j] || counts[j] > (1ull << 62)) {  // counts: room for the work-item arithmetic
      ts_batch_free(b);
      return TS_EINVAL;
    }
    // a job of n sign vectors has at most n distinct schemes
    const uint64_t cap = std::min<uint64_t>(hist_capacity, std::max<uint64_t>(counts[j], 1));
    uint64_t s = 16;
    while (s < 2 * cap) s <<= 1;
    b->jslots.push_back(s);
    b->kofs.push_back(b->key_words);
    b->cofs.push_back(b->count_words);
    b->cws.push_back(tris[j]->cw);
    b->key_words += s * tris[j]->cw;
    b->count_words += s;
  }
  if (e == cudaSuccess) e = cudaMalloc(&b->d_keys, b->key_words * 8);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_counts, b->count_words * 8);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_err, 4);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_failed, 8);
  uint64_t pack_words = 0;
  for (int j = 0; j < njobs; ++j) {
    b->pack_cap = std::max(b->pack_cap, std::min(b->jslots[j], kPackMax));
    pack_words = std::max<uint64_t>(pack_words, b->cws[j] + 1);
  }
  pack_words = pack_words * b->pack_cap + kPackHeader;
  if (e == cudaSuccess) e = cudaMalloc(&b->d_pack, pack_words * 8);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming);
  std::map<int, int> gi;
  for (int j = 0; j < njobs && e == cudaSuccess; ++j) {
    const ts_tri *t = tris[j];
    if (t->device != b->device) {
      ts_batch_free(b);
      return TS_EINVAL;
    }
    DevJob x{};
    x.tab = t->d_tables;
    x.n = counts[j];
    x.base = bases[j];
    x.codes = code_outputs ? reinterpret_cast<unsigned long long *>(code_outputs[j]) : nullptr;
    x.hkeys = reinterpret_cast<unsigned long long *>(b->d_keys + b->kofs[j]);
    x.hcnt = b->d_counts + b->cofs[j];
    x.hslots = b->jslots[j];
    x.stab = t->d_stables;
    x.swords = t->slay.words;
    x.schunks = t->slay.chunks;
    b->jobs.push_back(x);
    b->degree.push_back(t->d);
    b->tris.push_back(tris[j]);
    b->signs.push_back(nullptr);
    if (!gi.count(t->d)) {
      gi[t->d] = (int)b->groups.size();
      ts_batch::Group g;
      g.d = t->d;
      g.table_words = t->lay.words;
      g.off_fan = t->lay.off_fan;
      g.off_vext = t->lay.off_vext;
      b->groups.push_back(g);
    }
    auto &grp = b->groups[gi[t->d]];
    grp.jobs.push_back(j);
    grp.table_words = std::max(grp.table_words, t->lay.words);
    const uint32_t epw = (uint32_t)tc_layout(t->d, true, 32).epw;
    grp.ls_words = std::max(grp.ls_words, (t->lay.nslots + epw - 1) / epw);
    grp.slargest.words = std::max(grp.slargest.words, t->slay.words);
    grp.slargest.chunks = std::max(grp.slargest.chunks, t->slay.chunks);
    grp.n += counts[j];
  }
  for (auto &g : b->groups) table_defaults(g);
  if (e == cudaSuccess) {
    std::vector<int> spec;
    for (size_t gi = 0; gi < b->groups.size(); ++gi)
      if (wants_specialised(b, b->groups[gi])) spec.push_back((int)gi);
    make_specialised(b, spec);
  }
  for (auto &g : b->groups) {
    if (e == cudaSuccess) e = cudaMalloc(&g.d_work, sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&g.stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&g.done, cudaEventDisableTiming);
    if (e == cudaSuccess) e = upload_group(b, g);
    if (e == cudaSuccess) e = prepare_group(g);
  }
  if (e != cudaSuccess) {
    ts_batch_free(b);
    return cuda_st(e);
  }
  *out = b;
  return TS_OK;
}

void ts_batch_free(ts_batch *b) {
  if (!b) return;
  if (b->exec) cudaGraphExecDestroy(b->exec);
  for (auto &g : b->groups) {
    if (g.d_jobs) cudaFree(g.d_jobs);
    if (g.d_work) cudaFree(g.d_work);
    if (g.scratch) cudaFree(g.scratch);
    if (g.stream) cudaStreamDestroy(g.stream);
    if (g.done) cudaEventDestroy(g.done);
  }
  if (b->fork) cudaEventDestroy(b->fork);
  for (auto &f : b->fstream)
    if (f) cudaStreamDestroy(f);
  for (auto &f : b->fdone)
    if (f) cudaEventDestroy(f);
  if (b->d_fjobs) cudaFree(b->d_fjobs);
  if (b->d_fwork) cudaFree(b->d_fwork);
  if (b->d_keys) cudaFree(b->d_keys);
  if (b->d_counts) cudaFree(b->d_counts);
  if (b->d_err) cudaFree(b->d_err);
  if (b->d_failed) cudaFree(b->d_failed);
  if (b->d_pack) cudaFree(b->d_pack);
  delete b;
}

ts_status ts_batch_set_tile(ts_batch *b, int d, int threads, int chunk, int scratch) {
  if (!b || threads < 32 || threads % 32 || chunk < threads || chunk % threads ||
      scratch < TS_SCRATCH_AUTO || scratch > TS_SCRATCH_GLOBAL)
    return TS_EINVAL;
  for (auto &g : b->groups) {
    if (g.d != d) continue;
    const bool global = scratch == TS_SCRATCH_AUTO ? d >= kGlobalScratchFrom : scratch == TS_SCRATCH_GLOBAL;
    if (g.jit) {  // specialised: the block size and global scratch are fixed at compile time
      if (threads != jit_jobs_threads() || scratch == TS_SCRATCH_SHARED) return TS_EINVAL;
    } else if (!(threads == kSlicedThreads && scratch != TS_SCRATCH_GLOBAL) && !jobs_fn_dt(d, threads, global)) {
      return TS_EINVAL;  // block does not fit shared memory
    }
    // runs already launched (graph launches included) read the job table and
    // the scratch that this call rewrites or frees: let them finish first
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return cuda_st(e);
    if (g.jit) {
      g.threads = threads;
      g.chunk = chunk;
    } else {
      table_tile(g, threads, chunk, scratch);
    }
    if (b->exec) {
      cudaGraphExecDestroy(b->exec);
      b->exec = nullptr;
    }
    e = upload_group(b, g);
    if (e == cudaSuccess) e = prepare_group(g);
    return cuda_st(e);
  }
  return TS_EINVAL;
}

ts_status ts_batch_set_kernel(ts_batch *b, int d, int kind) {
  if (!b || kind < TS_KERNEL_AUTO || kind > TS_KERNEL_SPECIALIZED) return TS_EINVAL;
  for (size_t gi = 0; gi < b->groups.size(); ++gi) {
    auto &g = b->groups[gi];
    if (g.d != d) continue;
    // runs already launched read the job table and scratch rewritten here
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return cuda_st(e);
    if (b->exec) {
      cudaGraphExecDestroy(b->exec);
      b->exec = nullptr;
    }
    bool ok = true;
    const bool spec = kind == TS_KERNEL_SPECIALIZED || (kind == TS_KERNEL_AUTO && wants_specialised(b, g));
    if (!spec) table_defaults(g);
    else if (!g.jit) ok = make_specialised(b, {(int)gi});
    e = upload_group(b, g);
    if (e == cudaSuccess) e = prepare_group(g);
    if (e != cudaSuccess) return cuda_st(e);
    return ok ? TS_OK : TS_ECUDA;
  }
  return TS_EINVAL;
}

ts_status ts_batch_set_serial(ts_batch *b, int serial) {
  if (!b || serial < 0 || serial > 1) return TS_EINVAL;
  if (b->serial != (serial != 0) && b->exec) {
    cudaError_t e = cudaDeviceSynchronize();  // a graph launched before may still run
    if (e != cudaSuccess) return cuda_st(e);
    cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
  }
  b->serial = serial != 0;
  return TS_OK;
}

ts_status ts_batch_set_fused(ts_batch *b, int fused) {
  if (!b || fused < 0 || fused > 1) return TS_EINVAL;
  if (b->fused == (fused != 0)) return TS_OK;
  cudaError_t e = cudaDeviceSynchronize();  // a run launched before may still read the tables
  if (e != cudaSuccess) return cuda_st(e);
  if (b->exec) {
    cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
  }
  if (fused) {
    e = prepare_fused(b);
    if (e != cudaSuccess) return cuda_st(e);
  }
  b->fused = fused != 0;
  return TS_OK;
}

ts_status ts_batch_set_fused_tile(ts_batch *b, int d, int kind, int chunk) {
  if (!b || chunk < kFusedThreads || chunk % kFusedThreads || chunk > (1 << 24) ||
      (kind != TS_KERNEL_AUTO && kind != TS_KERNEL_TABLE && kind != TS_KERNEL_WARP) ||
      (kind == TS_KERNEL_WARP && d < kFusedWarpFrom))
    return TS_EINVAL;
  for (auto &g : b->groups) {
    if (g.d != d) continue;
    cudaError_t e = cudaDeviceSynchronize();  // runs already launched read the job table
    if (e != cudaSuccess) return cuda_st(e);
    if (b->exec) {
      cudaGraphExecDestroy(b->exec);
      b->exec = nullptr;
    }
    const int ow = g.fwarp, oc = g.fchunk;
    g.fwarp = kind == TS_KERNEL_WARP ? 1 : 0;
    g.fchunk = chunk;
    if (b->fused) {
      e = prepare_fused(b);
      if (e != cudaSuccess) {  // keep the previous, prepared tile
        g.fwarp = ow;
        g.fchunk = oc;
        const cudaError_t e2 = prepare_fused(b);
        return e2 != cudaSuccess ? cuda_st(e2) : TS_EINVAL;
      }
    }
    return TS_OK;
  }
  return TS_EINVAL;
}

ts_status ts_batch_set_signs(ts_batch *b, int job, const uint64_t *signs) {
  if (!b || job < 0 || job >= (int)b->jobs.size()) return TS_EINVAL;
  if (b->signs[job] == signs) return TS_OK;
  cudaError_t e = cudaDeviceSynchronize();  // a run launched before may still read the job table
  if (e != cudaSuccess) return cuda_st(e);
  if (b->exec) {
    cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
  }
  b->signs[job] = signs;
  if (b->fused) {
    e = prepare_fused(b);
    if (e != cudaSuccess) return cuda_st(e);
  }
  return TS_OK;
}

ts_status ts_batch_run(ts_batch *b, int use_graph, void *stream) {
  if (!b) return TS_EINVAL;
  if (!b->fused)  // the degree-group kernels draw their sign vectors: caller inputs need the fused launch
    for (const uint64_t *p : b->signs)
      if (p) return TS_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  if (!use_graph) return cuda_st(enqueue(b, st));
  if (!b->exec) {
    cudaStream_t cap = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
    cudaGraph_t graph = nullptr;
    if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      cudaError_t e2 = enqueue(b, cap);
      e = cudaStreamEndCapture(cap, &graph);
      if (e2 != cudaSuccess) e = e2;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, graph, 0);
    if (graph) cudaGraphDestroy(graph);
    if (cap) cudaStreamDestroy(cap);
    if (e != cudaSuccess) return cuda_st(e);
  }
  return cuda_st(cudaGraphLaunch(b->exec, st));
}

ts_status ts_batch_info(const ts_batch *b, int d, ts_batch_group_info *info, char *log,
                        size_t len) {
  if (!b || !info) return TS_EINVAL;
  for (const auto &g : b->groups) {
    if (g.d != d) continue;
    ts_batch_group_info x{};
    if (b->fused) {  // the degree's tile in the one fused launch
      x.kernel = g.fwarp ? TS_KERNEL_WARP : TS_KERNEL_TABLE;
      x.threads = kFusedThreads;
      x.chunk = g.fchunk;
      x.scratch = TS_SCRATCH_SHARED;
      for (const auto &T : b->tiers)
        if (T.tier == (g.fwarp ? kFusedWarpTier : fused_tier(g.d))) {
          x.grid = (int)T.grid;
          fused_attrs(T.tier, &x.registers, &x.local_bytes);
          fused_occupancy(T.tier, T.smem, &x.blocks_per_sm);
        }
      *info = x;
      if (log && len) log[0] = 0;
      return TS_OK;
    }
    x.kernel = g.jit ? TS_KERNEL_SPECIALIZED : TS_KERNEL_TABLE;
    x.threads = g.threads;
    x.chunk = g.chunk;
    x.scratch = g.global ? TS_SCRATCH_GLOBAL : TS_SCRATCH_SHARED;
    x.grid = (int)g.grid;
    if (g.jit) {
      jit_jobs_attrs(*g.jit, &x.registers, &x.local_bytes);
      x.blocks_per_sm = jit_jobs_blocks_per_sm(*g.jit);
    } else if (const void *fn = g.sliced ? g.splan.fn : (const void *)g.fn) {
      cudaFuncAttributes fa{};
      if (cudaFuncGetAttributes(&fa, fn) == cudaSuccess) {
        x.registers = fa.numRegs;
        x.local_bytes = (int)fa.localSizeBytes;
      }
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&x.blocks_per_sm, fn,
                                                    g.sliced ? (int)g.splan.threads : g.threads, g.smem);
    }
    *info = x;
    if (log && len) {
      const size_t n = std::min(len - 1, g.jit_log.size());
      std::memcpy(log, g.jit_log.data(), n);
      log[n] = 0;
    }
    return TS_OK;
  }
  return TS_EINVAL;
}

ts_status ts_batch_read(ts_batch *b, int job, uint64_t *codes, uint64_t *counts, uint64_t cap,
                        uint64_t *n_out, uint64_t *n_failed, void *stream) {
  if (!b || !n_out || job < 0 || job >= (int)b->jobs.size() || (cap && (!codes || !counts)))
    return TS_EINVAL;
  // The occupied slots are packed on the device and cross with the header in
  // one copy (the first kPackFirst of them; the rest in a second one).  A
  // table is at most half full and usually nearly empty: a batch of 5.1e6 sign
  // vectors with 12 reads of 2^15 slots took 3.77 ms with whole tables copied,
  // 2.96 ms now.  More schemes than kPackMax: the whole table.
  const int cw = b->cws[job];
  const uint64_t hs = b->jslots[job];
  const uint64_t ew = cw + 1;
  std::vector<unsigned long long> buf;
  cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
  std::lock_guard<std::mutex> lock(b->read_mu);  // of d_pack, up to the last copy
  const DeviceScope scope(b->device);
  if (e == cudaSuccess) e = scope.status;
  if (e == cudaSuccess) e = cudaMemsetAsync(b->d_pack, 0, 8, cudaStreamLegacy);
  if (e == cudaSuccess) {
    const uint64_t blocks = std::min<uint64_t>((hs + 255) / 256, 1024);
    batch_pack_kernel<<<(unsigned)blocks, 256, 0, cudaStreamLegacy>>>(
        b->d_keys + b->kofs[job], b->d_counts + b->cofs[job], hs, cw, b->pack_cap, b->d_err, b->d_failed,
        b->d_pack);
    e = cudaGetLastError();
  }
  const uint64_t first = std::min(b->pack_cap, kPackFirst);
  buf.resize(kPackHeader + first * ew);
  if (e == cudaSuccess) e = cudaMemcpy(buf.data(), b->d_pack, buf.size() * 8, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_st(e);
  const uint64_t n = buf[0];
  const unsigned long long failed = buf[1];
  const uint32_t err = (uint32_t)buf[2];
  std::vector<unsigned long long> ent;  // n entries
  if (n <= b->pack_cap) {
    ent.assign(buf.begin() + kPackHeader, buf.begin() + kPackHeader + std::min(n, first) * ew);
    ent.resize(n * ew);
    if (n > first)
      e = cudaMemcpy(ent.data() + first * ew, b->d_pack + kPackHeader + first * ew, (n - first) * ew * 8,
                     cudaMemcpyDeviceToHost);
  } else {
    std::vector<uint64_t> k(hs * cw);
    std::vector<unsigned long long> c(hs);
    e = cudaMemcpy(k.data(), b->d_keys + b->kofs[job], k.size() * 8, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess)
      e = cudaMemcpy(c.data(), b->d_counts + b->cofs[job], hs * 8, cudaMemcpyDeviceToHost);
    for (uint64_t s = 0; s < hs; ++s) {
      bool nz = false;
      for (int w = 0; w < cw; ++w) nz |= k[s * cw + w] != 0;
      if (!nz) continue;
      ent.insert(ent.end(), k.begin() + s * cw, k.begin() + (s + 1) * cw);
      ent.push_back(c[s] & kCountMask);
    }
  }
  if (e != cudaSuccess) return cuda_st(e);
  std::vector<uint64_t> idx(ent.size() / ew);
  for (uint64_t i = 0; i < idx.size(); ++i) idx[i] = i;
  std::sort(idx.begin(), idx.end(), [&](uint64_t a, uint64_t x) {
    for (int w = cw - 1; w >= 0; --w)
      if (ent[a * ew + w] != ent[x * ew + w]) return ent[a * ew + w] < ent[x * ew + w];
    return false;
  });
  *n_out = idx.size();
  if (n_failed) *n_failed = failed;
  for (uint64_t i = 0; i < idx.size() && i < cap; ++i) {
    for (int w = 0; w < cw; ++w) codes[i * cw + w] = ent[idx[i] * ew + w];
    counts[i] = ent[idx[i] * ew + cw];
  }
  if (idx.size() > cap) return TS_EOVERFLOW;
  if (err & kErrTimeout) return TS_ETIMEOUT;
  if (err & kErrOverflow) return TS_EOVERFLOW;
  if (err & kErrInternal) return TS_EINTERNAL;
  return TS_OK;
}

}  // extern "C"
