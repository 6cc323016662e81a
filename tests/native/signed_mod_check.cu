// Host check of the signed reduction of an item's 64-bit sums: a mod p in
// [0, p) for moduli at both ends of the library's window and any 64-bit a
// (multiples of p and the range's ends +-3, uniform values).  Exit status 1
// if any differs.
#include <cstdio>
#include <random>

#include "sk_exact.cuh"

int main() {
  const unsigned long long ps[4] = {(1ULL << 62) - 1, (1ULL << 62) - 57,
                                    (1ULL << 62) - (1ULL << 30) + 3, (1ULL << 62) - (1ULL << 31) + 1};
  std::mt19937_64 rng(1);
  long bad = 0;
  for (unsigned long long p : ps) {
    auto check = [&](__int128 a) {
      if (a < -((__int128)1 << 63) || a >= ((__int128)1 << 63)) return;
      __int128 want = a % (__int128)p;
      if (want < 0) want += p;
      if ((unsigned long long)want != sk::signed_mod((long long)a, p)) ++bad;
    };
    for (int d = -3; d <= 3; ++d) {
      for (int k = -3; k <= 3; ++k) check((__int128)k * p + d);
      check(((__int128)1 << 63) + d);
      check(-((__int128)1 << 63) + d);
    }
    for (int i = 0; i < 1000000; ++i) check((long long)rng());
  }
  std::printf("bad=%ld\n", bad);
  return bad ? 1 : 0;
}
