// Host check of fx::two_turns_f32 (csrc/fixedpoint.cuh) against long double.  Exit 0 = good.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <random>

#include "fixedpoint.cuh"

using namespace qaoa::fx;

static int fails = 0;

static void check(double d) {
  const long double want = 2.0L * ((long double)d - rintl((long double)d));  // exact
  const float got = two_turns_f32(d);
  // half a unit of float32 in the last place (three quarters below 2^-21 of a turn, unless that is the
  // number itself), 2^-55 of a turn at which the lower part of the fraction ends, zero below 2^-126
  const int e = want == 0 ? -149 : ilogbl(want) - 24;
  const bool whole = fabs(d) < 0.5 || fabsl(want) >= ldexpl(1.0L, -20);
  const long double tol = ldexpl(1.0L, e) * (whole ? 1.0L + ldexpl(1.0L, -4) : 1.5L) +
                          (fabs(d) >= ldexp(1.0, -12) && fabs(d) < 0.5 ? ldexpl(1.0L, -54) : 0.0L) + ldexpl(1.0L, -125);
  // 2 is a whole turn: at +-1/2 of one the sign may differ
  if (!(fabsl(remainderl((long double)got - want, 2.0L)) <= tol) && fails++ < 10) printf("two_turns_f32(%a) = %a, want %La\n", d, got, want);
}

int main() {
  const double edges[] = {0.0, -0.0, 0.25, -0.25, 0.5, -0.5, 0.75, 1.0, 1.5, 2.5, 0x1.0p-12, -0x1.0p-12, 0x1.fffffffffffffp-13,
                          0x1.0p-20, 0x1.fffffffffffffp-21, 0x1.0p-126, 0x1.8p-127, 0x1.0p-511, 0x1.8p-600,
                          0x1.0p-24, 0x1.fffffffffffffp-25,
                          0x1.0p-1022, 0x1.0p-1074, 0x1.0p-60, 0x1.0p52 + 0.5, 0x1.0p53, 0x1.fffffffffffffp-2, 0x1.0000000000001p-1,
                          1 + 0x1.0p-52, 1 - 0x1.0p-53, 1e6 + 0x1.0p-33, -1e6 - 0x1.0p-33, 1e300, -1e300};
  for (double d : edges) check(d), check(-d);
  std::mt19937_64 rng(11);
  std::uniform_real_distribution<double> u(-1.0, 1.0);
  for (int it = 0; it < 3000000; ++it) {
    double d = u(rng) * std::ldexp(1.0, (int)(rng() % 170) - 130);       // every magnitude, 2^-130 .. 2^39
    if (it % 4 == 1) d = std::rint(d) + u(rng) * std::ldexp(1.0, -(int)(rng() % 53));  // near whole turns
    if (it % 4 == 2) {                                                    // near ties of the rounding
      const float f = (float)(u(rng) * 0.5);
      d = ((double)f + (double)std::nextafterf(f, 1.0f)) / 2 + u(rng) * std::ldexp(1.0, -50);
      if (it & 4) d += std::ldexp(1.0, (int)(rng() % 12));
    }
    check(d);
  }
  printf(fails ? "FAIL %d\n" : "OK\n", fails);
  return fails ? 1 : 0;
}
