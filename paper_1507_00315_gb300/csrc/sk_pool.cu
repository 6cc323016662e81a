// sk_pool.cu -- the pool behind CallScope (sk_pool.h).
#include <mutex>
#include <vector>

#include "sk_exact_launch.cuh"
#include "sk_host_common.h"
#include "sk_pool.h"

namespace sk {
namespace {

struct Pool {
  std::mutex mu;
  std::vector<CallSet> free_sets[kMaxDevices];
};

// Never destroyed: a call may still run in another thread while the process
// exits, and the driver releases what is left.
Pool& pool() {
  static Pool* p = new Pool;
  return *p;
}

void destroy(CallSet& s) {
  if (s.e0) cudaEventDestroy(s.e0);
  if (s.e1) cudaEventDestroy(s.e1);
  if (s.stream) cudaStreamDestroy(s.stream);
  if (s.dmem) cudaFree(s.dmem);
  if (s.hmem) cudaFreeHost(s.hmem);
  s = CallSet{};
}

size_t rounded(size_t bytes) { return (bytes + 4095) / 4096 * 4096; }

cudaError_t host_malloc(void** p, size_t bytes) {
  cudaError_t e = cudaHostAlloc(p, bytes, cudaHostAllocDefault);
  if (e != cudaErrorMemoryAllocation) return e;
  cudaGetLastError();
  e = pool_release();
  return e == cudaSuccess ? cudaHostAlloc(p, bytes, cudaHostAllocDefault) : e;
}

}  // namespace

cudaError_t pool_release() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::vector<CallSet> idle;
  if (dev >= 0 && dev < kMaxDevices) {
    Pool& p = pool();
    std::lock_guard<std::mutex> lock(p.mu);
    idle.swap(p.free_sets[dev]);
  }
  for (CallSet& s : idle) destroy(s);
  return cudaSuccess;
}

cudaError_t device_malloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaErrorMemoryAllocation) return e;
  cudaGetLastError();
  e = pool_release();
  return e == cudaSuccess ? cudaMalloc(p, bytes) : e;
}

CallScope::CallScope(size_t dbytes, size_t hbytes, void* user_stream)
    : user_((cudaStream_t)user_stream) {
  int dev = 0;
  err_ = cudaGetDevice(&dev);
  if (err_ != cudaSuccess) return;
  if (dev >= 0 && dev < kMaxDevices) {
    Pool& p = pool();
    std::lock_guard<std::mutex> lock(p.mu);
    if (!p.free_sets[dev].empty()) {
      set_ = p.free_sets[dev].back();
      p.free_sets[dev].pop_back();
    }
  }
  // a set from before a device reset is of no use (and nothing of it is left
  // to free)
  if (set_.stream && cudaStreamQuery(set_.stream) != cudaSuccess) {
    cudaGetLastError();
    set_ = CallSet{};
  }
  set_.dev = dev;
  if (!set_.stream) err_ = cudaStreamCreateWithFlags(&set_.stream, cudaStreamNonBlocking);
  if (err_ == cudaSuccess && !set_.e0) err_ = cudaEventCreate(&set_.e0);
  if (err_ == cudaSuccess && !set_.e1) err_ = cudaEventCreate(&set_.e1);
  if (err_ == cudaSuccess && set_.dcap < dbytes) {
    if (set_.dmem) cudaFree(set_.dmem);
    set_.dmem = nullptr;
    set_.dcap = 0;
    err_ = device_malloc((void**)&set_.dmem, rounded(dbytes));
    if (err_ == cudaSuccess) set_.dcap = rounded(dbytes);
  }
  if (err_ == cudaSuccess && set_.hcap < hbytes) {
    if (set_.hmem) cudaFreeHost(set_.hmem);
    set_.hmem = nullptr;
    set_.hcap = 0;
    err_ = host_malloc((void**)&set_.hmem, rounded(hbytes));
    if (err_ == cudaSuccess) set_.hcap = rounded(hbytes);
  }
}

cudaError_t CallScope::drain() {
  const cudaError_t e = cudaStreamSynchronize(stream());
  if (e == cudaSuccess) drained_ = true;
  else err_ = e;
  return e;
}

CallScope::~CallScope() {
  if (set_.dev < 0) return;
  if (!drained_) drain();
  if (err_ == cudaSuccess && set_.dev < kMaxDevices) {
    if (set_.dcap > kPoolBytes) {
      cudaFree(set_.dmem);
      set_.dmem = nullptr;
      set_.dcap = 0;
    }
    if (set_.hcap > kPoolBytes) {
      cudaFreeHost(set_.hmem);
      set_.hmem = nullptr;
      set_.hcap = 0;
    }
    Pool& p = pool();
    std::lock_guard<std::mutex> lock(p.mu);
    if ((int)p.free_sets[set_.dev].size() < kPoolSlots) {
      p.free_sets[set_.dev].push_back(set_);
      return;
    }
  }
  destroy(set_);                               // surplus, or after an error
}

}  // namespace sk

extern "C" int sk_release_memory(void) { return sk::cuda_status(sk::pool_release()); }
