// sk_pool.h -- what a synchronous call needs for its duration: a stream, two
// timing events, device memory and pinned host memory, taken from a pool.
//
// Creating and destroying them (cudaMalloc, cudaFree's device-wide wait, stream
// and event creation) took most of a small count: S(8) 168 us with them, 36 us
// from the pool.  A call takes a set of its own and gives it back when it returns,
// after its stream has drained, so calls of several threads and streams never
// share one.  At most kPoolSlots sets a device are kept, each with at most
// kPoolBytes of device and of host memory; the rest is freed at once.  Idle sets
// never stand in the way of an allocation of the library (device_malloc), and
// a caller can have them freed (sk_release_memory).
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

namespace sk {

constexpr int kPoolSlots = 8;
constexpr size_t kPoolBytes = 32u << 20;

struct CallSet {
  int dev = -1;
  cudaStream_t stream = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  char* dmem = nullptr;
  char* hmem = nullptr;
  size_t dcap = 0, hcap = 0;
};

// Holds a set for one call.  user_stream: run there instead of the set's own
// stream.  The destructor waits for the stream if it was handed out after the
// last drain() (work may have been enqueued, on an error path too) and gives
// the set back.
class CallScope {
 public:
  CallScope(size_t dbytes, size_t hbytes, void* user_stream);
  ~CallScope();
  CallScope(const CallScope&) = delete;
  CallScope& operator=(const CallScope&) = delete;
  cudaError_t error() const { return err_; }
  // The stream to enqueue on; take it again after a drain() before new work.
  cudaStream_t stream() {
    drained_ = false;
    return user_ ? user_ : set_.stream;
  }
  cudaEvent_t e0() const { return set_.e0; }
  cudaEvent_t e1() const { return set_.e1; }
  char* dmem() const { return set_.dmem; }
  char* hmem() const { return set_.hmem; }
  // Waits for the stream; after success nothing of the call is in flight.
  cudaError_t drain();

 private:
  CallSet set_;
  cudaStream_t user_ = nullptr;
  cudaError_t err_ = cudaSuccess;
  bool drained_ = true;            // nothing enqueued since
};

// Frees the idle sets of the current device.
cudaError_t pool_release();

// cudaMalloc; where the device is full, once more without the idle sets.
cudaError_t device_malloc(void** p, size_t bytes);

}  // namespace sk
