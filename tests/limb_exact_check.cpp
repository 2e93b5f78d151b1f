// Host check of the adjoint terms' limb sums (csrc/fixedpoint.cuh): fx::ImSum is exact, against plain
// 128-bit sums, fx::WeightedImSum against the weighted sum of the terms rounded to 2^32.  Exit 0 = all good.
#include <cstdint>
#include <cstdio>
#include <random>

#include "fixedpoint.cuh"

using namespace qaoa::fx;

static std::mt19937_64 rng(40711);
static int fails = 0;

// |x| < 2^bits, at times with a low word at its extremes
static long long below(int bits) {
  const unsigned long long lim = (1ull << bits) - 1;
  long long x = (long long)(rng() % (2 * lim + 1)) - (long long)lim;
  if (bits > 33 && rng() % 5 == 0) x = (x & ~0xffffffffll) | (rng() & 1 ? 0x80000000ll : 0x7fffffffll);
  return x;
}

int main() {
  for (int it = 0; it < 500000; ++it) {
    // eight terms with weights 0..3 (popcounts), 2-norms of v and w up to 1.1 x 2^60: 16 components of
    // 2^58 each, or of independent magnitudes down to single bits
    const int kind = it % 4, gm = 1 + (int)(rng() % 7);
    const int bv = kind == 0 ? 58 : 1 + (int)(rng() % 58), bw = kind == 0 ? 58 : 1 + (int)(rng() % 58);
    ImSum S, T;
    i128 ws = 0, wt = 0;
    for (int r = 7; r >= 0; --r) {
      const long long vx = below(bv), vy = below(bv), wx = below(bw), wy = below(bw);
      S.add(split(vx), split(vy), split(wx), split(wy));
      const int pr = __builtin_popcount(r & gm);
      if (r > 0) T.add_times(S, pr - __builtin_popcount((r - 1) & gm));
      const i128 t = (i128)wx * vy - (i128)wy * vx;
      ws += t;
      wt += t * pr;
    }
    if (S.value() != ws || T.value() != wt)
      if (fails++ < 10) printf("ImSum not exact at %d\n", it);
  }
  for (int it = 0; it < 500000; ++it) {
    WeightedImSum s;
    i128 want = 0;
    const int bits = 1 + (int)(rng() % 59), cb = 1 + (int)(rng() % 28);
    for (int r = 0; r < 8; ++r) {
      const long long vx = below(bits), vy = below(bits), wx = below(bits), wy = below(bits);
      const int c = it % 5 ? (int)below(cb) : ((rng() & 1) ? 1 : -1) * (1 << 28);
      s.add(vx, vy, wx, wy, c);
      want += (((i128)wx * vy - (i128)wy * vx + ((i128)1 << 31)) >> 32) * c;
    }
    if (s.value() != want)
      if (fails++ < 10) printf("WeightedImSum not exact at %d\n", it);
  }
  printf(fails ? "FAIL %d\n" : "OK\n", fails);
  return fails ? 1 : 0;
}
