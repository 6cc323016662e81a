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
  std::printf("total bad=%d\n", bad);
  return bad ? 1 : 0;
}
