// Host check of fx::from_double (csrc/fixedpoint.cuh) at the end of its range.  Exit 0 = good.
#include <cmath>
#include <cstdio>

#include "fixedpoint.cuh"

using namespace qaoa::fx;

int main() {
  int fails = 0;
  for (int k = -40; k <= 1000; ++k) {
    const double d = std::ldexp(1.0, k), below = std::nextafter(d, 0.0);
    for (int top = 58; top <= 62; ++top) {  // |d| 2^s = 2^top, and the double below it
      const long long want = 1ll << top, less = want - (top >= 53 ? 1ll << (top - 53) : 0);
      if (from_double(d, top - k) != want || from_double(-d, top - k) != -want || from_double(below, top - k) != less ||
          from_double(-below, top - k) != -less)
        if (fails++ < 10) printf("2^%d at 2^%d: %lld\n", k, top, from_double(d, top - k));
    }
  }
  printf(fails ? "FAIL %d\n" : "OK\n", fails);
  return fails ? 1 : 0;
}
