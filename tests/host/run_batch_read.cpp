// Test infrastructure: ts_batch_read against a fake of the CUDA runtime with two
// devices (this program's definitions come before the shared library's).
// Exit 0 when the copies of a read are ordered behind the kernel that packs
// its entries, i.e. made with the batch's device current, whatever the
// caller's is, when a reader whose stream is busy holds up no other, and when a
// triangulation is loaded by one allocation and one copy.
#include <cuda_runtime_api.h>

#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <thread>
#include <vector>

#include "tcurve.h"

namespace {
struct Call {
  char what;  // 'k' kernel launch, 'r' copy to the host
  int device;
};
thread_local int device = 0;
thread_local std::vector<Call> calls;
std::atomic<unsigned long long> packed{0};  // entries the pack kernel "finds"
const cudaStream_t kBusy = (cudaStream_t)0xA0, kIdle = (cudaStream_t)0xB0;
std::mutex mu;
std::condition_variable cv;
bool waiting = false, released = false;
int allocations = 0, uploads = 0;
}  // namespace

extern "C" {
void **__cudaRegisterFatBinary(void *) {
  static void *h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **args, size_t, cudaStream_t) {
  calls.push_back({'k', device});
  **(unsigned long long **)args[7] = packed;  // the out of batch_pack_kernel
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  device = d;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) {
  ++allocations;
  *p = calloc(n, 1);
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind k) {
  if (k == cudaMemcpyDeviceToHost) calls.push_back({'r', device});
  else ++uploads;
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) {
  ++uploads;
  memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  if (s == kBusy) {
    std::unique_lock<std::mutex> l(mu);
    waiting = true;
    cv.notify_all();
    cv.wait(l, [] { return released; });
  }
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = (cudaStream_t)0xC0;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
  *e = (cudaEvent_t)0xD0;
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
}

int main() {
  const int32_t edges[] = {0, 0, 1, 0, 0, 0, 0, 1, 1, 0, 0, 1, 1, 0, 2, 0, 1, 0, 1, 1,
                           0, 1, 1, 1, 0, 1, 0, 2, 2, 0, 1, 1, 1, 1, 0, 2};
  device = 1;
  ts_tri *tri = nullptr;
  ts_batch *batch = nullptr;
  const uint64_t count = 1 << 20, base = 0;
  if (ts_load_triangulation(2, edges, 9, &tri) != TS_OK) return 2;
  int bad = 0;
  if (allocations != 1 || uploads != 1) {
    printf("a load makes %d allocations, %d copies\n", allocations, uploads);
    ++bad;
  }
  if (ts_batch_create(1, &tri, &count, &base, nullptr, 1 << 15, &batch) != TS_OK) return 3;
  std::vector<uint64_t> codes(1 << 16), counts(1 << 16);
  auto read = [&](cudaStream_t st) {
    uint64_t n = 0, failed = 0;
    return ts_batch_read(batch, 0, codes.data(), counts.data(), codes.size(), &n, &failed, st);
  };
  for (int current : {0, 1})
    for (unsigned long long n : {3ull, 2000ull, 20000ull}) {  // one copy, two, the whole table
      packed = n;
      device = current;
      calls.clear();
      if (read(nullptr) != TS_OK) return 4;
      size_t copies = 0;
      bool ok = !calls.empty() && calls[0].what == 'k' && device == current;
      for (const Call &c : calls) {
        ok &= c.device == 1;
        copies += c.what == 'r';
      }
      if (!ok || copies != (n == 3 ? 1u : n == 2000 ? 2u : 3u)) {
        printf("current device %d, %llu entries: %zu copies, in order %d\n", current, n, copies, (int)ok);
        ++bad;
      }
    }
  packed = 3;
  std::atomic<bool> done{false};
  std::thread a([&] { read(kBusy); });
  {
    std::unique_lock<std::mutex> l(mu);
    cv.wait(l, [] { return waiting; });
  }
  std::thread b([&] {
    read(kIdle);
    done = true;
  });
  for (int i = 0; i < 200 && !done; ++i) std::this_thread::sleep_for(std::chrono::milliseconds(20));
  if (!done) {
    puts("a reader waits for another reader's stream");
    ++bad;
  }
  {
    std::lock_guard<std::mutex> l(mu);
    released = true;
  }
  cv.notify_all();
  a.join();
  b.join();
  ts_batch_free(batch);
  ts_free_triangulation(tri);
  return bad != 0;
}
