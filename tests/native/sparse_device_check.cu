// GPU check of the zero-skipping walk at the orders that no whole count
// reaches: a part of a job (2^17 tiles from a random aligned one, or mirrored
// items around a change of weight or side) through the library's own
// launcher, and the batch's unit function (its group of tiles) at the widest
// rows, against the definition summed on the host: every assignment's sign
// times the product of its n correlations, modulo three primes.  2^17 tiles
// make units of several groups, so accumulators are split and lists reused.
// Arguments: delta, n.  Prints one line per case; exit status 1 if any fails.
#include <cstdio>
#include <cstdlib>
#include <random>
#include <thread>
#include <vector>

#include "sk_batch.cuh"
#include "sk_host_common.h"

using namespace sk;
typedef unsigned long long u64;

constexpr int kLgTiles = 17;

static u64 mask_of(int variant, int n) {
  return variant == 2 ? ((1ULL << (2 * n + 1)) - 1) & ~(1ULL << (2 * n - 1)) : (1ULL << (2 * n)) - 1;
}

// The term of one assignment modulo the primes, added weight times.
struct Sum {
  u64 r[3] = {0, 0, 0};
  void add(u64 x, u64 pres, int delta, int n, const u64* p, int weight) {
    int c[kMaxN];
    for (int pass = 0; pass < 2; ++pass)         // even distances first: most terms end there
      for (int d = 1 + delta; d <= n + delta; ++d) {
        if ((d & 1) != pass) continue;
        const u64 m = pres & (pres >> d);
        const int v = __builtin_popcountll(m) - 2 * __builtin_popcountll((x ^ (x >> d)) & m);
        if (v == 0) return;
        c[d - 1 - delta] = v;
      }
    long long part[4] = {weight, 1, 1, 1};       // |c| < 64: ten of them fit
    for (int k = 0; k < n; ++k) part[k / 10] *= c[k];
    if (__builtin_popcountll(x) & 1) part[0] = -part[0];
    for (int i = 0; i < 3; ++i) {
      u64 v = 1;
      for (long long g : part) {
        const long long y = g % (long long)p[i];
        v = mulmod(v, (u64)(y < 0 ? y + (long long)p[i] : y), p[i]);
      }
      r[i] = (r[i] + v) % p[i];
    }
  }
};

// Sum over the tiles of every range of J.
static void host_sum(const SpJob& J, int delta, int n, const u64* p, u64* out) {
  const int nt = (int)std::max(1u, std::thread::hardware_concurrency());
  std::vector<Sum> part(nt);
  std::vector<std::thread> th;
  const MirrorShape sh = J.h ? mirror_shape(n, J.h) : MirrorShape{};
  for (int t = 0; t < nt; ++t)
    th.emplace_back([&, t] {
      Sum s;
      for (int g = 0; g < J.nrange; ++g)
        for (u64 k = t; k < J.range[g].tiles; k += nt) {
          const u64 T = J.range[g].tile_lo + k;
          u64 x0;
          int weight = 1;
          if (J.h) {
            const int wb = 2 * (J.h - 5);
            x0 = mirror_item_bits(sh, T >> wb, &weight) |
                 sp_mirror_walk(J, n, T & ((1ULL << wb) - 1));
          } else {
            x0 = sp_tile_bits(J, T);
          }
          for (u64 i = 0; i < 1024; ++i)
            s.add(x0 | ((i & 31) << (J.h ? 1 : 0)) | ((i >> 5) << J.hb), J.pres, delta, n, p, weight);
        }
      part[t] = s;
    });
  for (auto& t : th) t.join();
  for (int i = 0; i < 3; ++i) {
    out[i] = 0;
    for (const Sum& s : part) out[i] = (out[i] + s.r[i]) % p[i];
  }
}

// One unit a warp of a batch's job.
template <int D, int N>
__global__ void __launch_bounds__(256, SK_EXACT_MIN_BLOCKS)
    batch_units(const BatchJobDev* job, u64 first, u64 units, const Primes* P, ExactScratch* scr) {
  extern __shared__ __align__(16) unsigned char smem[];
  BatchSmem sm;
  sm.tab = (unsigned)__cvta_generic_to_shared(smem);
  sm.wsm = sm.tab + sp_table_bytes(0) + (threadIdx.x >> 5) * kBatchWarp;
  sm.ws_col = nullptr;
  sp_build_tables<0>(smem);
  __syncthreads();
  u64 tot[kMaxPrimes] = {0, 0, 0, 0};
  const u64 warp = blockIdx.x * 8ULL + (threadIdx.x >> 5);
  for (u64 u = warp; u < units; u += gridDim.x * 8ULL) {
    const Res4 r = batch_chunk_impl<D, N>(job, P, 3, first + u, sm);
    for (int i = 0; i < 3; ++i) tot[i] = addmod(tot[i], r.r[i], (u64)P->pr[i].p);
  }
  warp_flush(tot, 3, *P, scr);
}

template <int D, int N>
static cudaError_t run_batch(const SpJob& part, const Primes& P, ExactScratch* dscr) {
  char* d = nullptr;
  BatchJobDev j{};
  j.pres = part.pres;
  j.sp = part;
  j.sp.tpu = 16;
  j.code = D * 32 + N;
  cudaError_t e = cudaMalloc(&d, 4096);
  if (e != cudaSuccess) return e;
  static_assert(sizeof(BatchJobDev) <= 2048 && sizeof(Primes) <= 2048, "layout");
  cudaMemcpy(d, &j, sizeof(j), cudaMemcpyHostToDevice);
  cudaMemcpy(d + 2048, &P, sizeof(P), cudaMemcpyHostToDevice);
  const int smem = sp_table_bytes(0) + 8 * kBatchWarp;
  e = cudaFuncSetAttribute(batch_units<D, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) {
    const SpRange& R = part.range[0];
    batch_units<D, N><<<304, 256, smem>>>((const BatchJobDev*)d, R.tile_lo / 16, R.tiles / 16,
                                          (const Primes*)(d + 2048), dscr);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  cudaFree(d);
  return e;
}

int main(int argc, char** argv) {
  if (argc != 3) return 2;
  const int delta = std::atoi(argv[1]), n = std::atoi(argv[2]);
  u64 p[4];
  int np = 3, bad = 0;
  Primes P;
  sk_count_opts o{};
  o.nprimes = 3;
  if (prepare_primes(&o, &np, (uint64_t*)p, &P)) return 2;
  ExactScratch* dscr = nullptr;
  if (cudaMalloc(&dscr, sizeof(ExactScratch)) != cudaSuccess) return 2;
  std::mt19937_64 rng(100 * n + delta);
  auto compare = [&](const char* what, cudaError_t e, const u64* want) {
    ExactScratch h{};
    if (e == cudaSuccess) e = cudaMemcpy(&h, dscr, sizeof(h), cudaMemcpyDeviceToHost);
    int b = e != cudaSuccess;
    for (int i = 0; i < 3; ++i) b |= scratch_residue(h, i, p[i]) != want[i];
    std::printf("delta=%d n=%d %s bad=%d\n", delta, n, what, b);
    bad += b;
  };
  auto launch = [&](const SpJob& J, bool mirrored) {
    SpLaunch L{};
    L.job = J;
    L.P = P;
    L.nprimes = 3;
    L.scratch = dscr;
    cudaError_t e = cudaMemset(dscr, 0, sizeof(ExactScratch));
    if (e == cudaSuccess) e = sparse_launcher(delta, n, mirrored)(L);
    return e == cudaSuccess ? cudaDeviceSynchronize() : e;
  };
  u64 want[3];
  for (int variant = delta; variant <= 2; variant += 2) {    // Skolem and hooked, or Langford
    const int m = 9;
    SpJob J;
    if (!sp_plain_job(mask_of(variant, n), delta, n, m, 0, 0, 1ULL << (2 * n - 1 - m), &J)) return 2;
    SpRange& R = J.range[0];
    R.tile_lo = (rng() % (R.tiles >> kLgTiles)) << kLgTiles;
    R.tiles = 1ULL << kLgTiles;
    host_sum(J, delta, n, p, want);
    compare(variant == 2 ? "hooked" : "plain", launch(J, false), want);
    if (variant != 2 && (n == 29 || n == 31)) {
      cudaError_t e = cudaMemset(dscr, 0, sizeof(ExactScratch));
      if (e == cudaSuccess)
        e = delta ? (n == 29 ? run_batch<1, 29>(J, P, dscr) : run_batch<1, 31>(J, P, dscr))
                  : (n == 29 ? run_batch<0, 29>(J, P, dscr) : run_batch<0, 31>(J, P, dscr));
      compare("batch unit", e, want);
    }
  }
  for (int h = 5; h <= 8; h += 3) {
    const MirrorShape sh = mirror_shape(n, h);
    const u64 half = (1ULL << (kLgTiles - 1)) >> (2 * (h - 5));
    const u64 mid[2] = {sh.block_lo[sh.depth], sh.per_side};
    SpJob J;
    if (!sp_mirror_job(mask_of(delta, n), delta, n, 2 * h, mid[h == 5] - half, mid[h == 5] + half, &J))
      return 2;
    host_sum(J, delta, n, p, want);
    compare(h == 5 ? "mirrored, both sides" : "mirrored, both weights", launch(J, true), want);
  }
  std::printf("total bad=%d\n", bad);
  return bad ? 1 : 0;
}
