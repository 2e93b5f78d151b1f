// Host check of fx::turn_phase and fx::mul_unit (csrc/fixedpoint.cuh) against long double.  Exit 0 = good.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <random>

#include "fixedpoint.cuh"

using namespace qaoa::fx;

int main() {
  const long double tau = 2 * 3.14159265358979323846264338327950288L;
  static C64 tt[512];
  for (int j = 0; j < 512; ++j) {
    const long double th = tau * (j % 256) * ldexpl(1.0L, j < 256 ? -8 : -16);
    tt[j].x = llrintl(ldexpl(cosl(th), 62));
    tt[j].y = llrintl(ldexpl(-sinl(th), 62));
  }
  std::mt19937_64 rng(7);
  int fails = 0;
  long double worst = 0;
  for (int it = 0; it < 2000000; ++it) {
    unsigned long long t = rng();
    const int kind = it % 8;
    if (kind == 1) t >>= rng() % 64;                                            // small turns
    if (kind == 2) t = (t << 48) + (1ull << 47) - (rng() & 1);                  // ends of the residual's range
    if (kind == 3) t = (t << (rng() % 64));                                     // table points
    if (kind == 4) t = 0ull - (t >> (rng() % 64));
    const C64 e = turn_phase(t, tt);
    const long double th = tau * ldexpl((long double)t, -64);
    const long double dx = fabsl(ldexpl((long double)e.x, -62) - cosl(th)), dy = fabsl(ldexpl((long double)e.y, -62) + sinl(th));
    worst = fmaxl(worst, fmaxl(dx, dy));
    // rho^4/24 < 2^-57.8, the tables and their product 6 x 2^-62, the truncated terms 2^-57.5;
    // the reference's own argument rounds at 2^-61
    if (dx > ldexpl(1.0L, -56) || dy > ldexpl(1.0L, -56)) {
      if (fails++ < 10) printf("turn_phase(%llu) off by %Lg %Lg\n", t, dx, dy);
    }
    const long long x = (long long)(rng() >> (5 + rng() % 58)) * ((rng() & 1) ? 1 : -1);
    const long long c = it % 31 ? (long long)(rng() >> 2) * ((rng() & 1) ? 1 : -1) : (1ll << 62);
    const __int128 d = ((__int128)mul_unit(x, split(c)) << 62) - (__int128)x * c;
    if (d > ((__int128)1 << 62) || d < -((__int128)1 << 62)) {
      if (fails++ < 10) printf("mul_unit(%lld, %lld)\n", x, c);
    }
  }
  printf("worst %Lg = 2^%.2Lf\n", worst, log2l(worst));
  printf(fails ? "FAIL %d\n" : "OK\n", fails);
  return fails ? 1 : 0;
}
