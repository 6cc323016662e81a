// Host check of the zero-skipping walk's tables, tile set-up and products for
// every (delta, n, walk) the library compiles, against the definition:
//   * every table address a lane forms lies inside the tables and is aligned;
//   * the rows' bytes give c_d (odd d) and c_d / 2 (even d) of the term, the
//     zero masks exactly the terms with c_d = 0 at an even d;
//   * T sum_i r_i 2^{31 i} = prod_k of those factors, modulo two primes, for
//     the sampled terms and for factors at their bounds; |T| < 2^tail_bits;
//   * the fast index bits of a tile leave the low block's addresses alone;
//   * the tiles of a job cover each assignment once (n = 13, whole and part
//     jobs, plain, with a held bit, hooked, mirrored: weights included).
// Prints one line per check; exit status 1 if any fails.
#include <algorithm>
#include <cstdio>
#include <random>
#include <utility>
#include <vector>

#include "sk_sparse.cuh"

using namespace sk;

typedef unsigned long long u64;
static const u64 kP[2] = {(1ULL << 61) - 1, 1000000007ULL};

static u64 mod_p(long long x, u64 p) {
  const long long y = x % (long long)p;
  return (u64)(y < 0 ? y + (long long)p : y);
}

static u64 mask_of(int variant, int n) {
  return variant == 2 ? ((1ULL << (2 * n + 1)) - 1) & ~(1ULL << (2 * n - 1)) : (1ULL << (2 * n)) - 1;
}

template <int D, int N>
static int product_bad(const int (&c)[N]) {
  constexpr DigitPlan dp = make_sparse_plan(D, N);
  int r[dp.kd], T, bad = 0;
  sparse_product<D, N>(c, r, T);
  if (T >= (1 << dp.tail_bits) || -T >= (1 << dp.tail_bits)) ++bad;
  for (u64 p : kP) {
    u64 want = 1, h = 0;
    for (int k = 0; k < N; ++k) want = (u64)((unsigned __int128)want * mod_p(c[k], p) % p);
    for (int i = dp.kd - 1; i >= 0; --i)
      h = (u64)((((unsigned __int128)h << 31) + mod_p(r[i], p)) % p);
    if ((u64)((unsigned __int128)h * mod_p(T, p) % p) != want) ++bad;
  }
  return bad;
}

// The rows, masks and products of sampled tiles of one job.
template <int D, int N, int LB>
static int check_tiles(const SpJob& J, std::mt19937_64& rng, int samples) {
  constexpr int NQ = sp_quads(D, N), NT = sp_tested(D, N), D0 = 1 + D;
  static std::vector<unsigned> tab(sp_table_bytes(1) / 4);
  for (int o = 0; o < sp_table_bytes(LB); o += 4) tab[o / 4] = sp_table_word(LB, o);
  int bad = 0;
  const int hb = J.hb;
  auto at = [&](unsigned a) -> unsigned {
    if (a % 4 || a >= (unsigned)sp_table_bytes(LB)) { ++bad; return 0; }
    return tab[a / 4];
  };
  const u64 pres = J.pres;
  const MirrorShape sh = LB ? mirror_shape(N, J.h) : MirrorShape{};
  for (int it = 0; it < samples; ++it) {
    const SpRange& R = J.range[rng() % (unsigned)J.nrange];
    const u64 T = R.tile_lo + rng() % R.tiles;
    u64 x;
    if (LB == 0) {
      x = sp_tile_bits(J, T);
    } else {
      const int wb = 2 * (J.h - 5);
      int w = 0;
      x = mirror_item_bits(sh, T >> wb, &w) | sp_mirror_walk(J, N, T & ((1ULL << wb) - 1));
      if (w != R.weight) ++bad;
    }
    // the fast index bits leave the low block's partners alone
    u64 x_first;
    {
      const u64 T0 = T & ~((1ULL << J.fast) - 1);
      const int wb = LB ? 2 * (J.h - 5) : 0;
      x_first = LB ? (x & ~sp_mirror_walk(J, N, T & ((1ULL << wb) - 1))) |
                         sp_mirror_walk(J, N, T0 & ((1ULL << wb) - 1))
                   : sp_tile_bits(J, T0);
    }
    const u64 blocks = (31ULL << LB) | (31ULL << hb);
    if (x & blocks) ++bad;
    const u64 y = x >> (LB + 5), yr = sp_brevll(x) >> (64 - hb);
    unsigned u[NQ] = {}, addr[32];
    for (int t = 0; t < 32; ++t) {
      if (t < 4 * NQ) {
        unsigned b = kSparseBias;
        if (t < N) {
          const u64 M = pres & ~blocks, pm = M & (M >> (D0 + t));
          b += sp_popcll(pres & (pres >> (D0 + t))) / 2 - sp_popcll((x ^ (x >> (D0 + t))) & pm);
        }
        u[t / 4] |= b << (8 * (t & 3));
      }
      const SpTask k = sp_task(D, NQ, NT, LB, t);
      addr[t] = k.base + ((unsigned)((t >= 8 && t < 16 ? yr : y) >> k.sh) & k.msk) * k.mul +
                (LB && (x & 1) ? k.x0add : 0u);
      unsigned used = k.msk;                       // bits behind the bytes in use
      if (t < NQ && N - 4 * t < 4) used &= (1u << (N - 4 * t + (t ? 4 : D))) - 1;
      if ((t < 8 || t >= 16) && ((((x ^ x_first) >> (LB + 5)) >> k.sh) & used)) ++bad;
    }
    const u64 x_fixed = LB ? 0 : x & ~((1ULL << hb) - 1);
    const int odd_first = (sp_popcll(pres & (pres >> 1)) & 1) ? -255 : -256;
    for (unsigned i = 0; i < 32; ++i) {
      unsigned a[NQ];
      const u64 X = x_fixed | ((u64)i << hb), hm = 31ULL << hb;
      for (int q = 0; q < NQ; ++q) {
        a[q] = u[q] - at(addr[8 + q] + 4 * sp_rev5(i));
        for (int e = 0; e < 4 && 4 * q + e < N; ++e) {
          const int d = D0 + 4 * q + e;
          a[q] -= sp_popcll((X ^ (X >> d)) & hm & (pres >> d) & ~(hm >> d)) << (8 * e);
        }
      }
      unsigned zero = 0;
      for (int j = 0; j < NT; ++j) {
        const int k = 2 + 2 * j - D0;
        zero |= at(addr[16 + j] + 4 * ((a[k / 4] >> (8 * (k & 3))) & 255u));
      }
      for (unsigned s = 0; s < 32; ++s) {
        unsigned w[NQ];
        for (int q = 0; q < NQ; ++q) w[q] = a[q] - at(addr[q] + 4 * s);
        if (LB)
          for (int j = 0; j < 5; ++j) {
            const int k = 1 + j - D0;
            if (k >= 0) w[k / 4] -= (unsigned)((x & 1) ^ ((s >> j) & 1)) << (8 * (k & 3));
          }
        int c[N];
        sp_factors<D, N>(w, odd_first, -255, make_uint2(0, 0), c);
        const u64 full = x | ((u64)s << LB) | ((u64)i << hb);
        bool none = true;
        for (int k = 0; k < N; ++k) {
          const int d = D0 + k;
          const int L = (int)sp_popcll(pres & (pres >> d));
          const int cd = L - 2 * (int)sp_popcll((full ^ (full >> d)) & pres & (pres >> d));
          if ((d % 2 ? c[k] : 2 * c[k]) != cd) ++bad;
          if (d % 2 == 0 && cd == 0) none = false;
        }
        if (none != !((zero >> s) & 1u)) ++bad;
        if (it < 4 && (s & 7) == 0) bad += product_bad<D, N>(c);
      }
    }
  }
  return bad;
}

template <int D, int N>
static int check_order(std::mt19937_64& rng) {
  int bad = 0;
  SpJob J;
  for (int variant = D; variant <= 2; variant += 2) {       // Skolem and hooked, or Langford
    const u64 pres = mask_of(variant, N);
    const int F = 2 * N - 1, m = 9;
    if (!sp_plain_job(pres, D, N, m, 0, 0, 1ULL << (F - m), &J)) ++bad;
    else bad += check_tiles<D, N, 0>(J, rng, 24);
    const int held = variant == 2 ? 2 * N - 3 : 2 * N - 2;   // Lemma 2.4's bit
    if (!sp_plain_job(pres, D, N, m, held, 0, 1ULL << (F - 1 - m), &J)) ++bad;
    else bad += check_tiles<D, N, 0>(J, rng, 24);
    if (N >= 16) {                                           // an aligned part of the items
      if (!sp_plain_job(pres, D, N, m, 0, 3ULL << (F - m - 2), 4ULL << (F - m - 2), &J)) ++bad;
      else bad += check_tiles<D, N, 0>(J, rng, 24);
    }
    if (sp_plain_job(pres, D, N, m, 0, 1, 3, &J) || sp_plain_job(pres, D, N, m, 0, 0, 3, &J)) ++bad;
  }
  for (int h = 5; h <= (N < 14 ? 8 : 10); ++h) {
    const u64 side = mirror_shape(N, h).per_side;
    if (!sp_mirror_job(mask_of(D, N), D, N, 2 * h, 0, 2 * side, &J)) ++bad;
    else bad += check_tiles<D, N, 1>(J, rng, 24);
    if (!sp_mirror_job(mask_of(D, N), D, N, 2 * h, side / 3, side + 2, &J)) ++bad;
    else bad += check_tiles<D, N, 1>(J, rng, 8);
  }
  for (int t = 0; t < 2000; ++t) {
    int c[N];
    for (int k = 0; k < N; ++k) {
      const long long L = sp_bound(D, N, k);
      long long v = (t & 1) ? L : (long long)(rng() % (u64)(2 * L + 1)) - L;
      c[k] = (int)((rng() & 1) ? -v : v);
    }
    bad += product_bad<D, N>(c);
  }
  constexpr DigitPlan dp = make_sparse_plan(D, N);
  std::printf("delta=%d n=%2d groups=%d tail=%d tail_bits=%2d digits=%d bad=%d\n", D, N, dp.ng,
              dp.ntail, dp.tail_bits, dp.kd, bad);
  return bad;
}

template <int D, int... Ns>
static int check_all(std::mt19937_64& rng, std::integer_sequence<int, Ns...>) {
  return (check_order<D, Ns + kSparseMinN>(rng) + ...);
}

// Every assignment once: the patterns of all tiles, times the low and lane
// bits, against the items' own patterns.
static int check_cover(int variant, int held) {
  constexpr int n = kSparseMinN;
  const int m = 9, F = 2 * n - 1;
  const u64 pres = mask_of(variant, n);
  const u64 items = 1ULL << (F - (held ? 1 : 0) - m);
  SpJob J;
  if (!sp_plain_job(pres, variant == 1, n, m, held, 0, items, &J)) return 1;
  std::vector<unsigned char> seen(1ULL << F, 0);
  for (u64 T = 0; T < J.range[0].tiles; ++T)
    for (u64 i = 0; i < 32; ++i)
      for (u64 s = 0; s < 32; ++s) {
        const u64 x = sp_tile_bits(J, T) | s | (i << J.hb);
        if (x >> F) return 1;
        ++seen[x];
      }
  int bad = 0;
  for (u64 x = 0; x < (1ULL << F); ++x) bad += seen[x] != (held && ((x >> held) & 1) ? 0 : 1);
  return bad;
}

static int check_cover_mirror(int delta, int h) {
  constexpr int n = kSparseMinN;
  const u64 side = mirror_shape(n, h).per_side;
  const MirrorShape sh = mirror_shape(n, h);
  SpJob J;
  if (!sp_mirror_job(mask_of(delta, n), delta, n, 2 * h, 0, 2 * side, &J)) return 1;
  std::vector<unsigned char> seen(1ULL << (2 * n - 1), 0);
  const int wb = 2 * (h - 5);
  for (int g = 0; g < J.nrange; ++g)
    for (u64 T = J.range[g].tile_lo; T < J.range[g].tile_lo + J.range[g].tiles; ++T) {
      int w = 0;
      const u64 x0 = mirror_item_bits(sh, T >> wb, &w) | sp_mirror_walk(J, n, T & ((1ULL << wb) - 1));
      if (w != J.range[g].weight) return 1;
      for (u64 i = 0; i < 32; ++i)
        for (u64 s = 0; s < 32; ++s) {
          const u64 x = x0 | (s << 1) | (i << J.hb);
          if (x >> (2 * n - 1)) return 1;
          seen[x] += (unsigned char)w;
        }
    }
  // each assignment and its image under the reversal symmetry together twice
  int bad = 0;
  for (u64 x = 0; x < (1ULL << (2 * n - 1)); ++x) {
    u64 r = sp_brevll(x) >> (64 - 2 * n);
    if (x & 1) r ^= (1ULL << (2 * n)) - 1;
    bad += (int)seen[x] + (int)seen[r] != 2;
  }
  return bad;
}

int main() {
  std::mt19937_64 rng(1);
  constexpr int count = kMaxN + 1 - kSparseMinN;
  int bad = check_all<0>(rng, std::make_integer_sequence<int, count>{});
  bad += check_all<1>(rng, std::make_integer_sequence<int, count>{});
  const int cover[5][2] = {{0, 0}, {1, 0}, {2, 0}, {0, 2 * kSparseMinN - 2}, {2, 2 * kSparseMinN - 3}};
  for (const auto& v : cover) {
    const int b = check_cover(v[0], v[1]);
    std::printf("cover variant=%d held=%d bad=%d\n", v[0], v[1], b);
    bad += b;
  }
  for (int h = 5; h <= 6; ++h) {
    const int b = check_cover_mirror(h & 1, h);
    std::printf("cover mirrored h=%d bad=%d\n", h, b);
    bad += b;
  }
  std::printf("total bad=%d\n", bad);
  return bad ? 1 : 0;
}
