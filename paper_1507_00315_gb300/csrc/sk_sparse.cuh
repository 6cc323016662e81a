// sk_sparse.cuh -- the exact signed sum with the zero terms skipped: the walk
// of whole counts, aligned chunks of work items and mirrored items, n >= 13.
//
// A term prod_k c_k(x) vanishes when any factor does.  c_d has the parity of
// its number of pairs L_d = 2n - d, so the factors of even distance d can be
// 0, each with probability about sqrt(2 / (pi L_d)): 80 % of the terms of
// S(20) are zero (76 % at n = 16, 82 % at n = 24).  The dense walk
// (sk_exact.cuh) forms every product; this one finds the nonzero terms with a
// few table lookups per 32 of them and multiplies only those.
//
// Tile.  A warp takes 2^10 terms at a time: 5 "low" bits LB..LB+4 (state s)
// and 5 "lane" bits hb..hb+4 (lane i holds state i), every other bit fixed by
// the tile index.  hb - (LB+4) > N + DELTA, so no pair (a, a+d) joins a low
// bit and a lane bit and the number of disagreeing pairs at distance d is a
// sum of three parts:
//   D_d = U_d (neither end a low or lane bit) + H_d(i) + R_d(s).
// Rows.  Four consecutive distances share a word, one byte each (bias 128):
//   a_i = 128 + floor(L_d / 2) - U_d - H_d(i),   byte = a_i - R_d(s),
// so that c_d = 2 byte - 256 (+ 1 for odd L_d).  For even d the common factor
// 2 is left out of every product and restored once per unit.  R_d(s) of a quad
// depends on the 5 low bits and the 8 bits its partners span: a 32 KB table
// of words [window][s] in shared memory, read without bank conflicts (lane =
// s); the same table serves H with both bit orders reversed.  U_d: lane t
// counts distance D0 + t over the 64-bit pattern.
// Zero test.  Term (i, s) has c_d = 0 iff R_d(s) = v_i, v_i = L_d/2 - U_d -
// H_d(i): a table word [pattern of the partners][v] holds one bit per s.
// Lane i ORs the words of every even d: the zeros of its 32 terms.
// Survivors are appended to the warp's list (lane-major, entry = tile, lane, s)
// and evaluated 32 at a time: a_i comes from shared memory, R(s) by a shuffle
// per word, the bytes are multiplied in int32 groups and the groups in signed radix-2^31 digits
// as in sk_exact.cuh, and tail * digit enters 64-bit accumulators (split into
// 32-bit halves before they can overflow).
//
// Group.  The survivors of up to 4 tiles that differ in the fast bits (next to
// the lane bits, out of the low block's reach: R and the mask rows stay) share
// one list, so that few evaluations run part empty; the tiles' a rows wait in
// shared memory, where the 32 entries of an evaluation read few of them.
//
// Bound by instruction issue (82 % of the issue slots, ALU 70 %, multiply pipe
// 58 %, shared-memory pipe 70 % busy, S(18) under ncu): 857 warp instructions a
// tile (928 at n = 17), about 600 of them the survivors' evaluation (73 for 32).
// Whole counts, dense walk (56 instructions a term) and this one: S(20) 1086
// and 426 ms, hooked n = 18 65.0 and 28.1 ms, mirrored L(19) (Lemmas 2.3 + 2.4)
// 71.5 and 25.8 ms; on the way, one list a tile: 482, 31.4, 35.1 ms.  (24 warps
// an SM with 80 registers in place of 20 with 96: 447, 28.2, 28.9 ms.)  Below
// n = 13 no lane block is clear of the low block's partners.
#pragma once
#include <cuda_runtime.h>

#include "sk_exact_launch.cuh"
#include "sk_mirror.cuh"

namespace sk {

constexpr int kSparseMinN = 13;   // smallest order of this walk: hb >= LB + 5 + N + DELTA
constexpr int kSparseBias = 128;

__host__ __device__ constexpr int sp_quads(int DELTA, int N) { return (N + 3) / 4; }
// even distances 2, 4, .. <= N + DELTA (both DELTA start at or below 2)
__host__ __device__ constexpr int sp_tested(int DELTA, int N) { return (N + DELTA) / 2; }

// ------------------------------------------------------------ table layout

// Shared-memory tables of a CTA (bytes): quad words [256 windows][32 states],
// first-quad words [DELTA][32 windows][32 states], zero masks [rows][64 v].
constexpr int kSpQuad = 0;
constexpr int kSpFirst = 256 * 128;
constexpr int kSpMask = kSpFirst + 2 * 32 * 128;
__host__ __device__ constexpr int sp_mask_rows(int LB) { return LB ? 72 : 52; }
__host__ __device__ constexpr int sp_table_bytes(int LB) { return kSpMask + sp_mask_rows(LB) * 256; }
// Per warp, for groups of TG tiles (bytes): the survivors' list (two-byte
// entries; at least one tile's 1024, for TG = 4 half as many again as usually
// survive), the tiles' masks [TG][32], their rows a
// [TG][32][first 4 words] and [TG][32][other words], 32 table addresses and 32
// bytes of U.
__host__ __device__ constexpr int sp_list_cap(int TG) { return TG >= 4 ? 1536 : 1024; }
__host__ __device__ constexpr int sp_row2(int NQ) { return NQ <= 4 ? 0 : NQ == 5 ? 4 : NQ == 6 ? 8 : 16; }
__host__ __device__ constexpr int sp_warp_bytes(int NQ, int TG) {
  return 2 * sp_list_cap(TG) + TG * 32 * (4 + 16 + sp_row2(NQ)) + 128 + 32;
}

__host__ __device__ inline unsigned sp_popc(unsigned x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__popc(x);
#else
  return (unsigned)__builtin_popcount(x);
#endif
}
__host__ __device__ inline unsigned sp_popcll(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__popcll((long long)x);
#else
  return (unsigned)__builtin_popcountll(x);
#endif
}
__host__ __device__ inline unsigned long long sp_brevll(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __brevll(x);
#else
  unsigned long long r = 0;
  for (int i = 0; i < 64; ++i) r |= ((x >> i) & 1ULL) << (63 - i);
  return r;
#endif
}
__host__ __device__ inline unsigned sp_rev5(unsigned s) {
  return ((s & 1) << 4) | ((s & 2) << 2) | (s & 4) | ((s & 8) >> 2) | ((s & 16) >> 4);
}

// Disagreements of state s with its partners at distances d0 .. d0+3, one byte
// each; the bits after the block are w_0, w_1, ... (bit j pairs with s_{j+d}
// inside the block, w_{j+d-5} beyond it).  d0 >= 5: only the window counts
// (w = the 8 bits from w_{d0-5} on).
__host__ __device__ inline unsigned sp_quad_word(unsigned w, unsigned s) {
  return sp_popc(s ^ (w & 31)) | (sp_popc(s ^ ((w >> 1) & 31)) << 8) |
         (sp_popc(s ^ ((w >> 2) & 31)) << 16) | (sp_popc(s ^ ((w >> 3) & 31)) << 24);
}
__host__ __device__ inline unsigned sp_near(unsigned w, unsigned s, int d) {
  const unsigned line = s | (w << 5);              // the block, then the bits after it
  return sp_popc((s ^ (line >> d)) & 31);
}
__host__ __device__ inline unsigned sp_first_word(int delta, unsigned w, unsigned s) {
  unsigned v = 0;
  for (int e = 0; e < 4; ++e) v |= sp_near(w, s, 1 + delta + e) << (8 * e);
  return v;
}
// Zero-mask word: bit s iff R_d(s) == v, v = column - 32.  Rows 0..31: d >= 6,
// the 5 partner bits; then d = 2 (partners w_0, w_1) and d = 4 (w_0..w_3),
// LB = 1: once for each value of bit 0, which pairs with low bit d - 1.
__host__ __device__ inline unsigned sp_mask_word(int LB, int row, int col) {
  int d = 0;
  unsigned w = 0, x0 = 0;
  const int rows2 = LB ? 8 : 4;
  if (row < 32) {
    d = 6;
    w = (unsigned)row;
  } else if (row < 32 + rows2) {
    d = 2;
    w = (unsigned)(row - 32) & 3u;
    x0 = (unsigned)(row - 32) >> 2;
  } else {
    d = 4;
    w = (unsigned)(row - 32 - rows2) & 15u;
    x0 = (unsigned)(row - 32 - rows2) >> 4;
  }
  unsigned m = 0;
  for (unsigned s = 0; s < 32; ++s) {
    int r = d == 6 ? (int)sp_popc(s ^ w) : (int)sp_near(w, s, d);
    if (LB && d < 6) r += (int)(x0 ^ ((s >> (d - 1)) & 1u));
    if (r == col - 32) m |= 1u << s;
  }
  return m;
}

// One 4-byte word of the tables, by its byte offset.
__host__ __device__ inline unsigned sp_table_word(int LB, int off) {
  if (off < kSpFirst) return sp_quad_word((unsigned)off >> 7, (unsigned)(off >> 2) & 31u);
  if (off < kSpMask) {
    const int o = off - kSpFirst;
    return sp_first_word(o >> 12, (unsigned)(o >> 7) & 31u, (unsigned)(o >> 2) & 31u);
  }
  const int o = off - kSpMask;
  return sp_mask_word(LB, o >> 8, (o >> 2) & 63);
}

// ------------------------------------------------------------ tile set-up

// Lane t prepares one table address per tile: t = q: the low block's quad q,
// t = 8 + q: the lane block's, t = 16 + i: the zero masks of d = 2 + 2 i.
// address = base + ((stream >> sh) & msk) * mul (+ x0add when bit 0 is set).
struct SpTask {
  int sh;
  unsigned msk, mul, base, x0add;
};
__host__ __device__ inline SpTask sp_task(int DELTA, int NQ, int NT, int LB, int t) {
  SpTask k = {0, 0u, 0u, (unsigned)kSpQuad, 0u};
  if (t < 16) {
    const int q = t & 7;
    if (q >= NQ) return k;
    k.mul = 128;
    if (q == 0) {
      k.msk = (16u << DELTA) - 1u;
      k.base = (unsigned)(kSpFirst + DELTA * 4096);
    } else {
      k.sh = 4 * q - 4 + DELTA;
      k.msk = 255u;
    }
    return k;
  }
  const int i = t - 16, d = 2 + 2 * i;
  if (i >= NT) return k;
  k.mul = 256;
  // the column of byte b = 128 + v is v + 32 = b - 96
  if (d == 2) {
    k.msk = 3u;
    k.base = (unsigned)(kSpMask + 32 * 256);
    k.x0add = LB ? 4u * 256u : 0u;
  } else if (d == 4) {
    k.msk = 15u;
    k.base = (unsigned)(kSpMask + (LB ? 40 : 36) * 256);
    k.x0add = LB ? 16u * 256u : 0u;
  } else {
    k.sh = d - 5;
    k.msk = 31u;
    k.base = (unsigned)kSpMask;
  }
  k.base -= 96u * 4u;
  return k;
}

// A range of tiles with one weight (mirrored items: 2 for each of a pair).
struct SpRange {
  unsigned long long tile_lo, tiles, unit_lo;
  int weight, pad;
};

// One job as the kernel sees it.
struct SpJob {
  unsigned long long pres;        // position mask
  unsigned long long fixed;       // bits above the lane bits held at -1 (LB = 0)
  unsigned long long units;       // work units of all ranges
  SpRange range[4];
  int nrange;
  int tpu;                        // tiles per unit
  int hb;                         // first lane bit
  int fast;                       // fastest index bits: just below the lane bits, out of
                                  // reach of the low block, whose rows they leave alone
  int mid_bits;                   // LB = 0: free bits between the low and the lane bits
  int upper_shift;                // LB = 0: the tile index beyond them starts at this bit
  int h;                          // LB = 1: walk bits at each end
};

// Pattern of a tile: the fixed and middle bits (1 = x of -1); the low and
// lane bits are 0.
__host__ __device__ inline unsigned long long sp_tile_bits(const SpJob& J, unsigned long long T) {
  const unsigned long long in = T & ((1ULL << J.fast) - 1ULL), out = T >> J.fast;
  const int slow = J.mid_bits - J.fast;
  return (in << (J.hb - J.fast)) | ((out & ((1ULL << slow) - 1ULL)) << 5) | J.fixed |
         ((out >> slow) << J.upper_shift);
}
// The walk bits of a mirrored item's tile t: the fast ones, the others of the
// h - 5 below the lane block, the h - 5 beyond the low block.
__host__ __device__ inline unsigned long long sp_mirror_walk(const SpJob& J, int n,
                                                            unsigned long long t) {
  const int w = J.h - 5, rest = w - J.fast;
  const unsigned long long out = t >> J.fast;
  return ((t & ((1ULL << J.fast) - 1ULL)) << (J.hb - J.fast)) |
         ((out & ((1ULL << rest) - 1ULL)) << (2 * n - 1 - J.h)) | ((out >> rest) << 6);
}

// ------------------------------------------------------------ product plan

__host__ __device__ constexpr long long sp_bound(int DELTA, int N, int k) {   // k = 0-based factor
  const int d = 1 + DELTA + k;
  long long L = 2LL * N - d;
  if (d % 2 == 0) L /= 2;
  return L < 1 ? 1 : L;
}

// Factors in int32 groups (bounds below 2^31), the last ones in a tail below
// 2^tail_bits: of the tails up to 2^26 (accumulators hold 2^6 terms and more
// between flushes), the one of least multiply-pipe cost.
constexpr int kSpTailBits = 26;
__host__ __device__ constexpr DigitPlan make_sparse_plan(int DELTA, int N) {
  DigitPlan best{};
  best.cost = 1 << 30;
  for (int tb = 4; tb <= kSpTailBits; ++tb) {
    long long L[kMaxN] = {};
    for (int i = 0; i < N; ++i) L[i] = sp_bound(DELTA, N, i);
    DigitPlan dp{};
    // the tail takes the smallest factors that fit
    bool used[kMaxN] = {};
    int tail[kMaxN] = {}, nt = 0;
    long long tp = 1;
    while (nt < N) {
      int m = -1;
      for (int i = 0; i < N; ++i)
        if (!used[i] && (m < 0 || L[i] < L[m])) m = i;
      if (tp * L[m] >= (1LL << tb)) break;
      tp *= L[m];
      used[m] = true;
      tail[nt++] = m;
    }
    if (nt == 0 || nt == N) continue;
    // the rest: largest first, each into the fullest group that still fits
    int ng = 0, cnt[kMaxGroups] = {}, member[kMaxGroups][kMaxN] = {};
    long long prod[kMaxGroups] = {};
    bool ok = true;
    for (int n = N - nt; n > 0; --n) {
      int m = -1;
      for (int i = 0; i < N; ++i)
        if (!used[i] && (m < 0 || L[i] > L[m])) m = i;
      used[m] = true;
      int g = -1;
      for (int j = 0; j < ng; ++j)
        if (prod[j] * L[m] < 2147483648LL && (g < 0 || prod[j] > prod[g])) g = j;
      if (g < 0) {
        if (ng >= kMaxGroups) { ok = false; break; }
        g = ng++;
        prod[g] = 1;
      }
      prod[g] *= L[m];
      member[g][cnt[g]++] = m;
    }
    if (!ok) continue;
    int pos = 0;
    for (int g = 0; g < ng; ++g) {
      dp.start[g] = pos;
      for (int i = 0; i < cnt[g]; ++i) dp.fac[pos++] = member[g][i];
    }
    dp.ng = ng;
    dp.start[ng] = pos;
    for (int i = 0; i < nt; ++i) dp.fac[pos + i] = tail[i];
    dp.ntail = nt;
    dp.tail_form = 1;
    dp.tail_bits = tb;
    dp.max_m = 32 - tb;              // terms between flushes: 2^max_m
    // digits of the product of the groups so far
    unsigned w[8] = {1, 0, 0, 0, 0, 0, 0, 0};
    int wide = 0;
    for (int g = 0; g < ng; ++g) {
      for (int i = 0; i < cnt[g]; ++i) {
        unsigned long long carry = 0;
        for (int j = 0; j < 8; ++j) {
          const unsigned long long x = (unsigned long long)w[j] * (unsigned long long)L[member[g][i]] + carry;
          w[j] = (unsigned)x;
          carry = x >> 32;
        }
      }
      int top = 7;
      while (top > 0 && w[top] == 0) --top;
      int bits = 0;
      while (bits < 32 && (w[top] >> bits)) ++bits;
      bits += top * 32;
      if (g > 0) wide += dp.digits[g - 1];
      dp.digits[g] = (bits + 30) / 31 < 1 ? 1 : (bits + 30) / 31;
      dp.kd = dp.digits[g];
    }
    wide += dp.kd;
    dp.cost = 2 * (N - ng - 1) + 4 * wide;
    if (dp.cost < best.cost) best = dp;
  }
  return best;
}

// prod_k c_k = T * sum_i r_i 2^{31 i}
template <int DELTA, int N>
__host__ __device__ __forceinline__ void sparse_product(const int (&c)[N],
                                                       int (&r)[make_sparse_plan(DELTA, N).kd],
                                                       int& T) {
  constexpr DigitPlan dp = make_sparse_plan(DELTA, N);
  constexpr int K = dp.kd;
  T = group_product(c, dp.fac + dp.start[dp.ng], dp.ntail, true);
  int G[dp.ng];
#pragma unroll
  for (int g = 0; g < dp.ng; ++g)
    G[g] = group_product(c, dp.fac + dp.start[g], dp.start[g + 1] - dp.start[g], true);
  r[0] = G[0];
#pragma unroll
  for (int g = 1; g < dp.ng; ++g) {
    const int kc = dp.digits[g - 1], kn = dp.digits[g];
    long long carry = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      if (i < kn) {
        const long long v = (i < kc) ? (i == 0 ? wide_mul_s32(r[i], G[g])
                                               : wide_mad_s32(r[i], G[g], carry))
                                     : carry;
        if (i < kn - 1) {
          r[i] = (int)((unsigned)v & 0x7FFFFFFFu);
          carry = v >> 31;
        } else {
          r[i] = (int)v;
        }
      }
    }
  }
}

// Factor k (distance 1 + DELTA + k) from the row words (bias 128): half of c_d
// for even d (a sign-extended byte), c_d for odd d (twice the byte plus odd0,
// -255, or -256 where L_d is even after all: hooked Skolem's d = 1).
template <int DELTA, int K>
__host__ __device__ __forceinline__ int sp_factor(unsigned w, int odd0, uint2 unit) {
  constexpr int e = K & 3;
  constexpr int d = 1 + DELTA + K;
#ifdef __CUDA_ARCH__
  // even d on the ALU, odd d on the multiply pipe: both are near 60 % busy
  if constexpr (d % 2 == 0) {
    unsigned v;
    asm("prmt.b32 %0, %1, %1, %2;" : "=r"(v) : "r"(w ^ 0x80808080u), "n"(0x8880 + 0x1111 * e));
    return (int)v;
  } else {
    return (int)__dp4a(w, e < 2 ? unit.x : unit.y, (unsigned)odd0);
  }
#else
  const int b = (int)((w >> (8 * e)) & 255u);
  return d % 2 == 0 ? b - 128 : 2 * b + odd0;
#endif
}

template <int DELTA, int N, int K = 0>
__host__ __device__ __forceinline__ void sp_factors(const unsigned (&w)[sp_quads(DELTA, N)],
                                                   int odd_first, int odd, uint2 unit,
                                                   int (&c)[N]) {
  if constexpr (K < N) {
    c[K] = sp_factor<DELTA, K>(w[K / 4], K == 0 ? odd_first : odd, unit);
    sp_factors<DELTA, N, K + 1>(w, odd_first, odd, unit, c);
  }
}

// (hi 2^32 + lo) mod p for signed words.
__host__ __device__ __forceinline__ unsigned long long sp_mod_pair(long long hi, long long lo,
                                                                  unsigned long long p) {
  unsigned long long u = horner31_mod(signed_mod(hi, p), 0ULL, p);
  u = u + u >= p ? u + u - p : u + u;
  const unsigned long long v = signed_mod(lo, p);
  return u + v >= p ? u + v - p : u + v;
}

// Residues of 2^twos * sum_i (hi_i 2^32 + lo_i) 2^{31 i}; out of line for the
// reason given at reduce_digits.
static __device__ __noinline__ void sp_reduce(const long long (&hi)[kMaxDigits],
                                              const long long (&lo)[kMaxDigits], int K, int twos,
                                              int nprimes, const Primes* P,
                                              unsigned long long (&res)[kMaxPrimes]) {
#pragma unroll 1
  for (int j = 0; j < kMaxPrimes; ++j) {
    res[j] = 0;
    if (j >= nprimes) continue;
    const unsigned long long p = (unsigned long long)P->pr[j].p;
    unsigned long long u = 0;
#pragma unroll 1
    for (int i = K - 1; i >= 0; --i) u = horner31_mod(u, sp_mod_pair(hi[i], lo[i], p), p);
#pragma unroll 1
    for (int i = 0; i < twos; ++i) u = u + u >= p ? u + u - p : u + u;
    res[j] = u;
  }
}

// ------------------------------------------------------------ device walk

__device__ __forceinline__ unsigned lds32(unsigned a) {
  unsigned v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint4 lds128(unsigned a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(a)
               : "memory");
  return v;
}
__device__ __forceinline__ unsigned lds_u16(unsigned a) {
  unsigned short v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts_u16(unsigned a, unsigned v) {
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((unsigned short)v) : "memory");
}
__device__ __forceinline__ void sts_u8(unsigned a, unsigned v) {
  asm volatile("st.shared.u8 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts32(unsigned a, unsigned v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void lds64(unsigned a, unsigned& x, unsigned& y) {
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(x), "=r"(y) : "r"(a) : "memory");
}
__device__ __forceinline__ void sts64(unsigned a, unsigned x, unsigned y) {
  asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void sts128(unsigned a, unsigned x, unsigned y, unsigned z, unsigned w) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w)
               : "memory");
}
// Takes the highest set bit b of `left` and stores tag | b; nothing where
// left = 0.
__device__ __forceinline__ void sp_pop(unsigned& left, unsigned to, unsigned tag) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b32 b, v;\n\t.reg .b16 h;\n\t"
      "setp.ne.u32 p, %0, 0;\n\tbfind.u32 b, %0;\n\tor.b32 v, b, %2;\n\tcvt.u16.u32 h, v;\n\t"
      "@p st.shared.u16 [%1], h;\n\tshl.b32 v, 1, b;\n\txor.b32 %0, %0, v;\n\t}"
      : "+r"(left)
      : "r"(to), "r"(tag)
      : "memory");
}
// NW (<= 16) words from a 16-byte aligned shared address
template <int NW>
__device__ __forceinline__ void lds_words(unsigned a, unsigned (&w)[NW]) {
#pragma unroll
  for (int i = 0; i < NW; i += 4) {
    const uint4 v = lds128(a + 4 * i);
    w[i] = v.x;
    if (i + 1 < NW) w[i + 1] = v.y;
    if (i + 2 < NW) w[i + 2] = v.z;
    if (i + 3 < NW) w[i + 3] = v.w;
  }
}

template <int LB>
__device__ __forceinline__ void sp_build_tables(unsigned char* smem) {
  for (int o = threadIdx.x * 4; o < sp_table_bytes(LB); o += blockDim.x * 4)
    *(unsigned*)(smem + o) = sp_table_word(LB, o);
}

// (x ^ (x >> d)) & m counted, 1 <= d <= 32.
template <bool WIDE>
__device__ __forceinline__ unsigned sp_disagree(unsigned xl, unsigned xh, int d, unsigned ml,
                                                unsigned mh) {
  if constexpr (WIDE) {
    const unsigned long long x = ((unsigned long long)xh << 32) | xl;
    return sp_popcll((x ^ (x >> d)) & (((unsigned long long)mh << 32) | ml));
  } else {
    return __popc((xl ^ __funnelshift_r(xl, xh, d)) & ml) + __popc((xh ^ (xh >> d)) & mh);
  }
}

// Residues of one work unit (tiles tile_lo .. tile_lo + ntiles - 1), this
// lane's part.  tab, wsm: shared addresses of the CTA's tables and this
// warp's area.
template <int DELTA, int N, int LB, int TG>
__device__ __forceinline__ Res4 sparse_unit(const SpJob* Jp, unsigned long long tile_lo, int ntiles,
                                            const Primes* P, int nprimes, unsigned tab,
                                            unsigned wsm) {
  constexpr int NQ = sp_quads(DELTA, N), NT = sp_tested(DELTA, N), D0 = 1 + DELTA;
  constexpr DigitPlan dp = make_sparse_plan(DELTA, N);
  constexpr int K = dp.kd;
  constexpr bool kWide = N + DELTA >= 32;
  static_assert(NQ >= 4 && NQ <= 8 && NT <= 16 && K <= kMaxDigits, "one lane per task");
  constexpr int kCap = sp_list_cap(TG);
  // evaluations between flushes: 2^max_m; a batch adds at most kCap / 32
  constexpr int kFlush = (1 << dp.max_m) - kCap / 32;
  static_assert(kFlush >= 0, "accumulators hold one batch");
  const SpJob& J = *Jp;
  const int lane = threadIdx.x & 31;
  const unsigned long long pres = J.pres;
  const int hb = J.hb;
  // this lane's distance and address task
  const int du = D0 + lane;
  unsigned pml = 0, pmh = 0;
  unsigned ubase = kSparseBias;
  if (lane < N) {
    const unsigned long long M = pres & ~((31ULL << LB) | (31ULL << hb));
    const unsigned long long pm = M & (M >> du);
    pml = (unsigned)pm;
    pmh = (unsigned)(pm >> 32);
    ubase += sp_popcll(pres & (pres >> du)) / 2;
  }
  SpTask task = sp_task(DELTA, NQ, NT, LB, lane);
  task.base += tab;
  // the task's window starts at bit `from` of x, or of x reversed for the lane
  // block's quads
  const bool hi_stream = lane >= 8 && lane < 16;
  const int from = task.sh + (hi_stream ? 64 - hb : LB + 5);
  const bool upper = from >= 32;
  const int odd_first = (sp_popcll(pres & (pres >> 1)) & 1) ? -255 : -256;   // hooked: L_1 even
  // constants of the odd factors in registers, not rebuilt for every use
  int odd;
  uint2 unit;                                    // twice the byte of an odd distance
  asm volatile("mov.u32 %0, -255;" : "=r"(odd));
  asm volatile("mov.u32 %0, %1;" : "=r"(unit.x) : "n"(DELTA ? 0x200 : 0x2));
  asm volatile("mov.u32 %0, %1;" : "=r"(unit.y) : "n"(DELTA ? 0x2000000 : 0x20000));
  // fixed bits above the lane bits: their pairs with the lane bits
  unsigned long long x_fixed = 0;
  if constexpr (LB == 0) x_fixed = sp_tile_bits(J, tile_lo) & ~((1ULL << hb) - 1ULL);
  unsigned st[NQ];
  {
    const unsigned long long hm = 31ULL << hb;
    const unsigned long long X = x_fixed | ((unsigned long long)lane << hb);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      st[q] = 0;
#pragma unroll 1
      for (int e = 0; e < 4; ++e) {
        const int d = D0 + 4 * q + e;
        if (4 * q + e < N)
          st[q] |= sp_popcll((X ^ (X >> d)) & hm & (pres >> d) & ~(hm >> d)) << (8 * e);
      }
    }
  }
  const unsigned lane4 = (unsigned)lane * 4u, rlane4 = sp_rev5((unsigned)lane) * 4u;
  const unsigned a_row = wsm, a_row2 = a_row + TG * 32 * 16, a_mask = a_row2 + TG * 32 * sp_row2(NQ),
                 a_list = a_mask + TG * 32 * 4, a_addr = a_list + 2 * kCap, a_u = a_addr + 128;
  long long acc[K], alo[K], ahi[K];
#pragma unroll
  for (int i = 0; i < K; ++i) acc[i] = alo[i] = ahi[i] = 0;
  int evals = 0;
  unsigned long long q_cur = ~0ULL, q_bits = 0;   // LB = 1: the item whose bits are decoded
  MirrorShape sh;
  if constexpr (LB == 1) sh = mirror_shape(N, J.h);
  unsigned r[NQ];
  const unsigned fast_mask = (1u << J.fast) - 1u;
  const unsigned long long fast_step = 1ULL << (hb - J.fast);
  const int group = J.fast >= 2 ? TG : (TG < (1 << J.fast) ? TG : (1 << J.fast));
  // 32 list entries from e on: T r_i of each into the accumulators
  auto evaluate = [&](unsigned e, int sgn) {
    unsigned w[NQ];
    const unsigned slot = e >> 6;
    {
      const uint4 v = lds128(a_row + slot * 16u);
      w[0] = v.x;
      w[1] = v.y;
      w[2] = v.z;
      w[3] = v.w;
    }
    if constexpr (NQ == 5) {
      w[4] = lds32(a_row2 + slot * 4u);
    } else if constexpr (NQ == 6) {
      lds64(a_row2 + slot * 8u, w[4], w[5]);
    } else if constexpr (NQ >= 7) {
      const uint4 v = lds128(a_row2 + slot * 16u);
      w[4] = v.x;
      w[5] = v.y;
      w[6] = v.z;
      if constexpr (NQ == 8) w[7] = v.w;
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) w[q] -= __shfl_sync(0xffffffffu, r[q], (int)e);
    int c[N], rd[K], Tl;
    sp_factors<DELTA, N>(w, odd_first, odd, unit, c);
    sparse_product<DELTA, N>(c, rd, Tl);
    Tl *= sgn;
#pragma unroll
    for (int i = 0; i < K; ++i) acc[i] = wide_mad_s32(rd[i], Tl, acc[i]);
  };
  for (int tt = 0; tt < ntiles; tt += group) {
    const int here = ntiles - tt < group ? ntiles - tt : group;
    unsigned tags = 0;                              // sign bit of each tile of the group
    int cnt = 0;
    // the group's first pattern; its tiles count up the fast bits
    const unsigned long long T0 = tile_lo + (unsigned)tt;
    unsigned long long x;
    if constexpr (LB == 0) {
      x = sp_tile_bits(J, T0);
    } else {
      const int wb = 2 * (J.h - 5);
      const unsigned long long q = T0 >> wb;
      if (q != q_cur) {
        int weight;
        q_cur = q;
        q_bits = mirror_item_bits(sh, q, &weight);
      }
      x = q_bits | sp_mirror_walk(J, N, T0 & ((1ULL << wb) - 1ULL));
    }
    bool fresh = tt == 0 || ((unsigned)T0 & fast_mask) == 0;        // new rows r
#pragma unroll 1
    for (int g = 0; g < here; ++g, x += fast_step, fresh = false) {
      const unsigned xl = (unsigned)x, xh = (unsigned)(x >> 32);
      // one distance and one table address per lane
      {
        const unsigned zl = hi_stream ? __brev(xh) : xl, zh = hi_stream ? __brev(xl) : xh;
        const unsigned win =
            __funnelshift_r(upper ? zh : zl, upper ? 0u : zh, (unsigned)from) & task.msk;
        unsigned addr = task.base + win * task.mul;
        if constexpr (LB == 1) addr += (xl & 1u) ? task.x0add : 0u;
        sts32(a_addr + lane4, addr);
      }
      sts_u8(a_u + lane, ubase - sp_disagree<kWide>(xl, xh, du, pml, pmh));
      tags |= (((unsigned)__popc(xl ^ xh ^ (unsigned)g)) & 1u) << g;
      __syncwarp();
      if (fresh) {
        unsigned al[NQ];
        lds_words<NQ>(a_addr, al);
#pragma unroll
        for (int q = 0; q < NQ; ++q) r[q] = lds32(al[q] + lane4);
        if constexpr (LB == 1) {
          // bit 0 pairs with low bit j at distance 1 + j
#pragma unroll
          for (int j = 0; j < 5; ++j) {
            const int k = 1 + j - D0;
            if (k >= 0 && k < N) r[k / 4] += (((unsigned)(lane >> j) ^ xl) & 1u) << (8 * (k & 3));
          }
        }
      }
      unsigned a[NQ];
      {
        unsigned ah[NQ], u[NQ];
        lds_words<NQ>(a_addr + 32, ah);
        lds_words<NQ>(a_u, u);
#pragma unroll
        for (int q = 0; q < NQ; ++q) a[q] = u[q] - lds32(ah[q] + rlane4) - st[q];
      }
      const unsigned slot = (unsigned)(g * 32 + lane);
      sts128(a_row + slot * 16u, a[0], a[1], a[2], a[3]);
      if constexpr (NQ == 5) sts32(a_row2 + slot * 4u, a[4]);
      if constexpr (NQ == 6) sts64(a_row2 + slot * 8u, a[4], a[5]);
      if constexpr (NQ >= 7) sts128(a_row2 + slot * 16u, a[4], a[5], a[6], NQ == 8 ? a[NQ - 1] : 0u);
      // zeros of this lane's 32 terms
      unsigned zero = 0;
      {
        unsigned am[NT];
        lds_words<NT>(a_addr + 64, am);
#pragma unroll
        for (int i = 0; i < NT; ++i) {
          const int k = 2 + 2 * i - D0;             // d = 2 + 2 i
          zero |= lds32(__dp4a(a[k / 4], 4u << (8 * (k & 3)), am[i]));
        }
      }
      sts32(a_mask + (unsigned)g * 128u + lane4, ~zero);
      cnt += __popc(~zero);
      __syncwarp();                                 // before the next tile's addresses
    }
    // the group's survivors in one batch, or, if the list could not hold
    // them, tile by tile
    // (sums by warp reduction: uniform, so the loops below are too)
    int total = (int)__reduce_add_sync(0xffffffffu, (unsigned)cnt);
    const bool whole = total <= kCap;
    for (int g0 = 0; g0 < here;) {
      const int g1 = whole ? here : g0 + 1;
      if (!whole) {
        cnt = __popc(lds32(a_mask + (unsigned)g0 * 128u + lane4));
        total = (int)__reduce_add_sync(0xffffffffu, (unsigned)cnt);
      }
      int incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      // lane-major; entry = tile, lane, sign of tile, s
      unsigned at = a_list + 2u * (unsigned)(incl - cnt);
      for (int g = g0; g < g1; ++g) {
        unsigned left = lds32(a_mask + (unsigned)g * 128u + lane4);
        const unsigned tag = ((unsigned)(g * 32 + lane) << 6) | (((tags >> g) & 1u) << 5);
        const int mine = __popc(left), most = __reduce_max_sync(0xffffffffu, mine);
        unsigned to = at;
        for (int j = 0; j < most; j += 2) {
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            sp_pop(left, to + 2 * i, tag);
          }
          to += 4;
        }
        at += 2u * (unsigned)mine;
      }
      __syncwarp();
      // (the next entry is fetched ahead; past the end it reads the addresses
      // that follow the list, unused)
      int i0 = 0;
      unsigned e = lds_u16(a_list + 2u * (unsigned)lane);
      for (; i0 + 32 <= total; i0 += 32) {
        const unsigned en = lds_u16(a_list + 2u * (unsigned)(i0 + 32 + lane));
        evaluate(e, 1 - 2 * (int)(__popc(e) & 1u));
        e = en;
      }
      if (i0 < total) {
        const bool in = i0 + lane < total;
        evaluate(in ? e : 0u, in ? 1 - 2 * (int)(__popc(e) & 1u) : 0);
      }
      evals += (total + 31) >> 5;
      if (evals > kFlush) {
        evals = 0;
#pragma unroll
        for (int i = 0; i < K; ++i) {
          alo[i] += (long long)(unsigned)acc[i];
          ahi[i] += acc[i] >> 32;
          acc[i] = 0;
        }
      }
      __syncwarp();
      g0 = g1;
    }
  }
  long long h6[kMaxDigits] = {}, l6[kMaxDigits] = {};
#pragma unroll
  for (int i = 0; i < K; ++i) {
    l6[i] = alo[i] + (long long)(unsigned)acc[i];
    h6[i] = ahi[i] + (acc[i] >> 32);
  }
  Res4 out;
  sp_reduce(h6, l6, K, NT, nprimes, P, out.r);
  return out;
}

// ------------------------------------------------------------ kernel

// One CTA an SM: 20 warps (96 registers a thread; 24 warps of 80 registers, kernel
// time: S(20) 447.1 for 425.4 ms, S(17) 7.87 for 7.79, S(18) 28.2 for 28.0, L(19)
// with Lemmas 2.3 + 2.4 28.9 for 25.7, but L(20) 444.4 for 445.4), 16 where the
// rows of the largest orders would not fit beside the tables.
constexpr int kSpGroup = 4;
__host__ __device__ constexpr int sp_max_warps(int DELTA, int N) {
  return sp_quads(DELTA, N) <= 6 ? 20 : 16;
}

template <int DELTA, int N, int LB>
__global__ void __launch_bounds__(32 * sp_max_warps(DELTA, N), 1)
    sparse_kernel(SpJob J, Primes P, int nprimes, ExactScratch* scr) {
  extern __shared__ __align__(16) unsigned char sp_smem[];
  __shared__ SpJob sJ;
  __shared__ Primes sP;
  if (threadIdx.x == 0) {
    sJ = J;
    sP = P;
  }
  sp_build_tables<LB>(sp_smem);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const unsigned tab = (unsigned)__cvta_generic_to_shared(sp_smem);
  const unsigned wsm =
      tab + sp_table_bytes(LB) + (threadIdx.x >> 5) * sp_warp_bytes(sp_quads(DELTA, N), kSpGroup);
  unsigned long long tot[kMaxPrimes] = {0, 0, 0, 0};
  for (;;) {
    unsigned long long u = 0;
    if (lane == 0) u = atomicAdd(&scr->counter, 1ULL);
    // lane 0's unit, by warp reduction: uniform registers hold it from here on
    u = ((unsigned long long)__reduce_max_sync(0xffffffffu, (unsigned)(u >> 32)) << 32) |
        __reduce_max_sync(0xffffffffu, lane == 0 ? (unsigned)u : 0u);
    if (u >= sJ.units) break;
    int g = 0;
    while (g + 1 < sJ.nrange && u >= sJ.range[g + 1].unit_lo) ++g;
    const SpRange& R = sJ.range[g];
    const unsigned long long off = (u - R.unit_lo) * (unsigned long long)sJ.tpu;
    const unsigned long long rest = R.tiles - off;
    const int nt = rest < (unsigned long long)sJ.tpu ? (int)rest : sJ.tpu;
    const Res4 r =
        sparse_unit<DELTA, N, LB, kSpGroup>(&sJ, R.tile_lo + off, nt, &sP, nprimes, tab, wsm);
#pragma unroll
    for (int i = 0; i < kMaxPrimes; ++i) {
      if (i >= nprimes) break;
      const unsigned long long p = (unsigned long long)sP.pr[i].p;
      tot[i] = addmod(tot[i], r.r[i], p);
      if (R.weight == 2) tot[i] = addmod(tot[i], r.r[i], p);
    }
  }
  warp_flush(tot, nprimes, sP, scr);
}

// ------------------------------------------------------------ host side

// Tiles per unit: enough units for every resident warp to take several,
// between 1 and 128 tiles (a unit's reduction costs about as much as one
// tile).
inline int sp_tiles_per_unit(unsigned long long tiles, unsigned long long warps) {
  int t = 1;
  while (t < 128 && tiles / (2ULL * t) >= 6ULL * warps) t *= 2;
  return t;
}

// The job of work items [lo, hi) of the plain walk (fixed: Lemma 2.4's held
// bit, 0 if none), or false where the tiles do not apply: the items must be
// one aligned power-of-two block, and the lane bits clear of the low bits'
// partners.
inline bool sp_plain_job(unsigned long long pres, int delta, int n, int m, int fixed_bit,
                         unsigned long long lo, unsigned long long hi, SpJob* J) {
  if (n < kSparseMinN || hi <= lo) return false;
  const unsigned long long size = hi - lo;
  if ((size & (size - 1)) || (lo & (size - 1))) return false;
  int lg = 0;
  while ((1ULL << lg) < size) ++lg;
  // c_d must have the parity of d (all but hooked Skolem's d = 1, where L_1
  // is even: odd0 of sp_factor): an extended sequence's hole can break it
  for (int d = 1 + delta; d <= n + delta; ++d)
    if (d > 1 && ((sp_popcll(pres & (pres >> d)) ^ (unsigned)d) & 1u)) return false;
  *J = SpJob{};
  J->pres = pres;
  int free_lo = m + lg;                       // the block's free bits are 0 .. free_lo-1 ...
  int upper = 0;
  if (fixed_bit && m + lg > fixed_bit) {      // ... those at and above the held bit move up
    upper = m + lg - fixed_bit;
    free_lo = fixed_bit;
    J->upper_shift = fixed_bit + 1;
  }
  J->hb = free_lo - 5;
  if (J->hb < 5 + n + delta) return false;
  J->mid_bits = J->hb - 5;
  J->fast = J->hb - (5 + n + delta);
  if (((pres >> J->hb) & 31ULL) != 31ULL || (pres & 31ULL) != 31ULL) return false;
  // every position the low block can pair with must be present
  if ((~pres >> 5) & ((1ULL << (n + delta)) - 1ULL)) return false;
  // and every position below the lane block it can pair with
  if ((~pres >> (J->hb - n - delta)) & ((1ULL << (n + delta)) - 1ULL)) return false;
  if (!upper) {
    unsigned long long q = lo;                // the block's index bits, all zero below lg
    J->fixed = (fixed_bit && m <= fixed_bit ? insert_zero_bit(q, fixed_bit - m) : q) << m;
    J->upper_shift = 63;                      // no upper index bits
  } else {
    J->fixed = (insert_zero_bit(lo, fixed_bit - m)) << m;
  }
  J->range[0].tiles = 1ULL << (J->mid_bits + upper);
  J->range[0].weight = 1;
  J->nrange = 1;
  return true;
}

// Mirrored items [lo, hi) of walk width m = 2h (sk_mirror.cuh): up to two
// weights on each side.
inline bool sp_mirror_job(unsigned long long pres, int delta, int n, int m, unsigned long long lo,
                          unsigned long long hi, SpJob* J) {
  const int h = m / 2;
  if (n < kSparseMinN || h < 5 || hi <= lo) return false;
  *J = SpJob{};
  J->pres = pres;
  J->h = h;
  J->hb = 2 * n - 6;
  if (J->hb < 6 + n + delta) return false;
  J->fast = h - 5 < J->hb - (6 + n + delta) ? h - 5 : J->hb - (6 + n + delta);
  const MirrorShape sh = mirror_shape(n, h);
  const int wb = 2 * (h - 5);
  for (int side = 0; side < 2; ++side)
    for (int part = 0; part < 2; ++part) {
      unsigned long long a = side * sh.per_side + (part ? sh.block_lo[sh.depth] : 0ULL);
      unsigned long long b = side * sh.per_side + (part ? sh.per_side : sh.block_lo[sh.depth]);
      if (a < lo) a = lo;
      if (b > hi) b = hi;
      if (a >= b) continue;
      SpRange& R = J->range[J->nrange++];
      R.tile_lo = a << wb;
      R.tiles = (b - a) << wb;
      R.weight = part ? 1 : 2;
    }
  return J->nrange > 0;
}

// Splits the ranges into units of at most tpu tiles; a plain unit (h = 0)
// stays inside one pattern of the bits above the lane bits.
inline void sp_split(SpJob* J, int tpu) {
  while (!J->h && J->mid_bits < 7 && tpu > (1 << J->mid_bits)) tpu /= 2;
  J->tpu = tpu;
  J->units = 0;
  for (int g = 0; g < J->nrange; ++g) {
    J->range[g].unit_lo = J->units;
    J->units += (J->range[g].tiles + (unsigned)tpu - 1) / (unsigned)tpu;
  }
}

struct SpLaunch {
  SpJob job;
  Primes P;
  int nprimes;
  ExactScratch* scratch;
  int grid;                       // 0: SMs x resident blocks
  cudaStream_t stream;
};

// The CTA size is the walk's own: its warps share 54 KB of tables, so the
// caller's block size (the dense walk's) would leave SMs short of warps: S(17)
// at 32 threads 24.9 ms, dense walk 17.1; at 640 threads 7.8 ms.
template <int DELTA, int N, int LB>
cudaError_t launch_sparse(const SpLaunch& L) {
  static OccupancyCache occ;
  if (L.nprimes < 1 || L.nprimes > kMaxPrimes) return cudaErrorInvalidValue;
  constexpr int warps = sp_max_warps(DELTA, N);
  constexpr int kArea = sp_warp_bytes(sp_quads(DELTA, N), kSpGroup);
  constexpr int smem = sp_table_bytes(LB) + warps * kArea;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool keyed = dev >= 0 && dev < kMaxDevices;
  int nb = keyed ? occ.per_sm[dev][0].load(std::memory_order_relaxed) : 0;
  if (nb <= 0) {                  // first launch on the device
    e = cudaFuncSetAttribute(sparse_kernel<DELTA, N, LB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, sparse_kernel<DELTA, N, LB>,
                                                        32 * warps, smem);
    if (e != cudaSuccess) return e;
    if (nb <= 0) nb = 1;
    if (keyed) occ.per_sm[dev][0].store(nb, std::memory_order_relaxed);
  }
  const unsigned long long wave = (unsigned long long)device_sm_count(dev) * nb;
  SpJob J = L.job;
  unsigned long long tiles = 0;
  for (int g = 0; g < J.nrange; ++g) tiles += J.range[g].tiles;
  sp_split(&J, sp_tiles_per_unit(tiles, wave * warps));
  unsigned long long grid = L.grid > 0 ? (unsigned long long)L.grid : wave;
  if (L.grid <= 0) {
    const unsigned long long need = (J.units + warps - 1) / warps;
    if (grid > need) grid = need;
  }
  sparse_kernel<DELTA, N, LB>
      <<<(unsigned)grid, 32 * warps, smem, L.stream>>>(J, L.P, L.nprimes, L.scratch);
  return cudaGetLastError();
}

typedef cudaError_t (*SparseLaunchFn)(const SpLaunch&);
// Launchers for delta in {0, 1}, n in [kSparseMinN, kMaxN]; mirrored: LB = 1.
SparseLaunchFn sparse_launcher(int delta, int n, bool mirrored);

}  // namespace sk

#define SK_INSTANTIATE_SPARSE(N)                                                  \
  template cudaError_t sk::launch_sparse<0, N, 0>(const sk::SpLaunch&);           \
  template cudaError_t sk::launch_sparse<1, N, 0>(const sk::SpLaunch&);           \
  template cudaError_t sk::launch_sparse<0, N, 1>(const sk::SpLaunch&);           \
  template cudaError_t sk::launch_sparse<1, N, 1>(const sk::SpLaunch&);
