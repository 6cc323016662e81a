// sk_batch.cuh -- work function of the persistent batched sweep.
//
// The batch kernel (sk_batch.cu) serves many exact-count jobs of different
// (variant, n) in one launch.  Jobs are laid end to end in a space of chunks
// (32 work items of the dense walk below n = kSparseMinN, one unit of tiles of
// the zero-skipping walk from there on), largest job first; every warp takes
// the next chunk from a device counter, finds its job, and calls the compiled
// walk of that job's (delta, n) -- one non-inlined device function per
// instance, defined in the per-n translation units and linked at device-link
// time.
#pragma once
#include "sk_exact_launch.cuh"
#include "sk_sparse.cuh"

namespace sk {

// One job of a batch as the device sees it.
struct BatchJobDev {
  unsigned long long pres;       // position mask
  unsigned long long items;      // work items of the job
  unsigned long long chunk_lo;   // first global chunk of the job
  SpJob sp;                      // n >= kSparseMinN: its tiles
  int m;                         // walk bits per item
  int code;                      // delta * 32 + n
};

// Tiles whose survivors a warp evaluates together, and its shared memory (two
// CTAs of 8 warps an SM, beside the dense walk's columns).
constexpr int kBatchGroup = 2;
constexpr int kBatchWarp = sp_warp_bytes(8, kBatchGroup);

// Shared memory of a CTA as the work functions see it.
struct BatchSmem {
  signed char* ws_col;           // this thread's column of the dense walk's copy of w
  unsigned tab, wsm;             // the zero-skipping walk's tables and this warp's area
};

// Residues of this lane's part of chunk c of a job.
template <int DELTA, int N>
__device__ __forceinline__ Res4 batch_chunk_impl(const BatchJobDev* job, const Primes* P,
                                                 int nprimes, unsigned long long c,
                                                 const BatchSmem& sm) {
  if constexpr (N >= kSparseMinN) {
    const unsigned long long off = c * (unsigned long long)job->sp.tpu;
    return sparse_unit<DELTA, N, 0, kBatchGroup>(&job->sp, off, job->sp.tpu, P, nprimes, sm.tab, sm.wsm);
  } else {
    const unsigned long long item = c * 32ULL + (threadIdx.x & 31);
    if (item < job->items)
      return limb_item<DELTA, N>(job->pres, job->m, item, P, nprimes, sm.ws_col);
    Res4 out = {{0, 0, 0, 0}};
    return out;
  }
}

}  // namespace sk

#define SK_BATCH_FN(D, N) sk_batch_chunk_d##D##_n##N
#define SK_DECLARE_BATCH(N)                                                                  \
  extern __device__ sk::Res4 SK_BATCH_FN(0, N)(const sk::BatchJobDev*, const sk::Primes*, int, \
                                               unsigned long long, const sk::BatchSmem&);     \
  extern __device__ sk::Res4 SK_BATCH_FN(1, N)(const sk::BatchJobDev*, const sk::Primes*, int, \
                                               unsigned long long, const sk::BatchSmem&);
#define SK_DEFINE_BATCH(N)                                                                   \
  __device__ __noinline__ sk::Res4 SK_BATCH_FN(0, N)(const sk::BatchJobDev* j,               \
                                                     const sk::Primes* P, int np,            \
                                                     unsigned long long c,                   \
                                                     const sk::BatchSmem& sm) {              \
    return sk::batch_chunk_impl<0, N>(j, P, np, c, sm);                                      \
  }                                                                                          \
  __device__ __noinline__ sk::Res4 SK_BATCH_FN(1, N)(const sk::BatchJobDev* j,               \
                                                     const sk::Primes* P, int np,            \
                                                     unsigned long long c,                   \
                                                     const sk::BatchSmem& sm) {              \
    return sk::batch_chunk_impl<1, N>(j, P, np, c, sm);                                      \
  }
