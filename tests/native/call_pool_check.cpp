// Host check of the call pool (csrc/sk_pool.cu) against a fake of the CUDA
// runtime calls it makes, defined here (linked ahead of the runtime): no GPU
// work is done.  A fake stream knows whether work is enqueued on it; memory may
// go back to the pool (or to the runtime) only when the stream it was used on
// has none left.  Prints one line per scenario; exit status 1 if any fails.
#include <cstdio>
#include <cstdlib>
#include <map>

#include "sk_pool.h"

namespace {
struct FakeStream {
  bool pending = false;
};
std::map<void*, size_t> g_mem;                   // live allocations
size_t g_limit = ~(size_t)0;                     // bytes the fake device (and host) can hold
bool g_early = false;                            // something freed with work in flight
FakeStream* g_user = nullptr;
FakeStream* g_last = nullptr;
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  g_last = new FakeStream;
  *s = (cudaStream_t)g_last;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t s) {
  return ((FakeStream*)s)->pending ? cudaErrorNotReady : cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  ((FakeStream*)s)->pending = false;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
  size_t used = 0;
  for (const auto& m : g_mem) used += m.second;
  if (n > g_limit - used) return cudaErrorMemoryAllocation;
  *p = std::malloc(1);
  g_mem[*p] = n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (p && g_user && g_user->pending) g_early = true;
  if (p) { g_mem.erase(p); std::free(p); }
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
}

extern "C" int sk_release_memory(void);
using sk::CallScope;

// A call of `chunks` launches whose last one fails after it enqueued work and
// before its wait.
static int failing_call(FakeStream* user, int chunks) {
  FakeStream* used = nullptr;
  char* mem = nullptr;
  {
    CallScope cs(256, 256, user);
    if (cs.error() != cudaSuccess) return 1;
    mem = cs.dmem();
    for (int c = 0; c < chunks; ++c) {
      used = (FakeStream*)cs.stream();
      used->pending = true;
      if (c + 1 < chunks && cs.drain() != cudaSuccess) return 1;
    }
  }
  if (used->pending) return 1;                   // handed back with work in flight
  CallScope next(256, 256, nullptr);             // and it serves the next call
  return next.error() != cudaSuccess || next.dmem() != mem;
}

// Eight idle sets of the largest size kept.
static void fill_pool() {
  CallScope* s[8];
  for (auto& p : s) p = new CallScope(sk::kPoolBytes, sk::kPoolBytes, nullptr);
  for (auto& p : s) delete p;
}

// Idle sets give way to an allocation that would fail beside them, of a call
// and of the rest of the library; what cannot be had at all still fails.
static int full_device() {
  int bad = 0;
  for (int device = 0; device < 2; ++device) {
    fill_pool();
    if (g_mem.size() != 16) ++bad;
    g_limit = 17 * sk::kPoolBytes;
    if (device) {
      void* p = nullptr;
      if (sk::device_malloc(&p, 17 * sk::kPoolBytes) != cudaSuccess) ++bad;
      cudaFree(p);
      if (sk::device_malloc(&p, 18 * sk::kPoolBytes) != cudaErrorMemoryAllocation) ++bad;
    } else {
      CallScope cs(8 * sk::kPoolBytes, 8 * sk::kPoolBytes, nullptr);
      if (cs.error() != cudaSuccess) ++bad;
      CallScope more(4 * sk::kPoolBytes, 256, nullptr);
      if (more.error() != cudaErrorMemoryAllocation) ++bad;
    }
    g_limit = ~(size_t)0;
  }
  return bad;
}

static int released() {
  fill_pool();
  CallScope running(4096, 4096, nullptr);
  const int st = sk_release_memory();
  return st != 0 || g_mem.size() != 2;           // the running call's own stay
}

int main() {
  int bad = 0;
  auto report = [&](const char* what, int b) {
    std::printf("%s bad=%d\n", what, b);
    bad += b;
  };
  FakeStream user;
  report("first launch fails, own stream", failing_call(nullptr, 1));
  report("third launch fails, own stream", failing_call(nullptr, 3));
  g_user = &user;
  report("first launch fails, caller's stream", failing_call(&user, 1));
  report("third launch fails, caller's stream", failing_call(&user, 3));
  {
    // a call that waited leaves the caller's stream alone afterwards
    CallScope cs(256, 256, &user);
    FakeStream* s = (FakeStream*)cs.stream();
    s->pending = true;
    cs.drain();
    s->pending = true;                           // the caller's own work
  }
  report("no second wait after a drain", user.pending ? 0 : 1);
  report("nothing freed early", g_early ? 1 : 0);
  g_user = nullptr;
  report("idle sets give way on a full device", full_device());
  report("release frees the idle sets", released());
  std::printf("total bad=%d\n", bad);
  return bad ? 1 : 0;
}
