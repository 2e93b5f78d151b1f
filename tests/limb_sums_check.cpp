// Host check of the limb sums and limb-shared multiplies of csrc/fixedpoint.cuh against plain
// 128-bit arithmetic.  Exit 0 = all good.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <random>

#include "fixedpoint.cuh"

using namespace qaoa::fx;

static std::mt19937_64 rng(2407);
static int fails = 0;

static long long below(int bits) {  // |x| < 2^bits
  const unsigned long long lim = (1ull << bits) - 1;
  return (long long)(rng() % (2 * lim + 1)) - (long long)lim;
}
static bool far(i128 a, i128 b, i128 tol) { return a - b > tol || b - a > tol; }
static void bad(const char* what, int it) {
  if (fails++ < 10) printf("%s mismatch at %d\n", what, it);
}

int main() {
  std::uniform_real_distribution<double> ang(0.0, 6.283185307179586);
  for (int it = 0; it < 1000000; ++it) {  // unit-factor and mixer-diagonal multiplies
    const double th = ang(rng);
    long long ur = llrint(ldexp(std::cos(th), 62)), ui = llrint(ldexp(std::sin(th), 62));
    if (it % 97 == 0) ur = 0, ui = -(1ll << 62);
    if (it % 89 == 0) ur = 1ll << 62, ui = 0;
    const Factor f = factor(ur, ui);
    const int b1 = 1 + (int)(rng() % 60);
    const long long x = below(b1), y = it % 53 ? below(b1) : 1ll << 60;
    const C64 a = cmul_unit<false>(x, y, f), c = cmul_unit<true>(x, y, f);
    const C64 wa = cmul_q62_exact(x, y, ur, ui, 0), wc = cmul_q62_exact(x, y, ur, -ui, 0);
    if (far(a.x, wa.x, 1) || far(a.y, wa.y, 1) || far(c.x, wc.x, 1) || far(c.y, wc.y, 1)) bad("cmul_unit", it);
    const int e = 3 + (int)(rng() % 11);
    const long long p = below(61), q = below(61);
    const C64 d = cmul_big(split(p), split(q), f, e), wd = cmul_q62_exact(p, q, ur, ui, e);
    if (far(d.x, wd.x, 1) || far(d.y, wd.y, 1)) bad("cmul_big", it);
  }
  for (int it = 0; it < 300000; ++it) {
    // eight terms with weights 0..3 (as popcounts of 0..7), both vectors of 2-norm up to 1.1 x 2^60:
    // spread evenly, all in one component, or of random magnitudes
    double v[16], w[16], nv = 0, nw = 0;
    const int kind = it % 4;
    for (int k = 0; k < 16; ++k) {
      v[k] = ldexp((double)below(53), -53);
      w[k] = ldexp((double)below(53), -53);
      if (kind == 1) v[k] = v[k] < 0 ? -1 : 1, w[k] = w[k] < 0 ? -1 : 1;
      if (kind == 2) v[k] = ldexp(v[k], -(int)(rng() % 60)), w[k] = ldexp(w[k], -(int)(rng() % 60));
      if (kind == 3) v[k] *= k == 14, w[k] *= k == 15;
      nv += v[k] * v[k];
      nw += w[k] * w[k];
    }
    const double sv = nv > 0 ? ldexp(1.1, 60) / std::sqrt(nv) : 0, sw = nw > 0 ? ldexp(1.1, 60) / std::sqrt(nw) : 0;
    const double cv = ldexp(0.9, 61), cs = it % 8 < 4 ? 1.0 : ldexp(1.0, -(int)(rng() % 40));
    long long V[16], W[16];
    for (int k = 0; k < 16; ++k) {
      V[k] = (long long)std::fmax(-cv, std::fmin(cv, v[k] * sv * cs));
      W[k] = (long long)std::fmax(-cv, std::fmin(cv, w[k] * sw * cs));
    }
    if (kind == 1)  // low words at their extremes
      for (int k = 0; k < 16; ++k) V[k] = (V[k] & ~0xffffffffll) | 0x80000000ll, W[k] = (W[k] & ~0xffffffffll) | 0x80000000ll;
    const int gm = 1 + (int)(rng() % 7);
    ImSum S, T;
    i128 ws = 0, wt = 0;
    for (int r = 7; r >= 0; --r) {
      S.add(split(V[2 * r]), split(V[2 * r + 1]), split(W[2 * r]), split(W[2 * r + 1]));
      const int pr = __builtin_popcount(r & gm);
      if (r > 0) T.add_times(S, pr - __builtin_popcount((r - 1) & gm));
      const i128 t = (i128)W[2 * r] * V[2 * r + 1] - (i128)W[2 * r + 1] * V[2 * r];
      ws += t;
      wt += t * pr;
    }
    // left out: up to 15 units of two low words per term, each times a low word
    if (far(S.value(), ws, (i128)8 * 30 << 31) || far(T.value(), wt, (i128)12 * 30 << 31)) bad("ImSum", it);
  }
  for (int it = 0; it < 300000; ++it) {
    WeightedImSum s;
    i128 want = 0, room = 0;
    const int bits = 1 + (int)(rng() % 56), cb = 1 + (int)(rng() % 28);
    for (int r = 0; r < 8; ++r) {
      long long v[4];
      for (long long& x : v) x = it % 7 ? below(bits) : ((rng() & 1) ? 1 : -1) * ((1ll << 56) - 1) ^ 0x80000000ll;
      for (long long& x : v) x = x >= (1ll << 56) ? (1ll << 56) - 1 : x <= -(1ll << 56) ? -(1ll << 56) + 1 : x;
      const int c = it % 5 ? (int)below(cb) : ((rng() & 1) ? 1 : -1) * (1 << 28);
      s.add(v[0], v[1], v[2], v[3], c);
      want += ((i128)v[2] * v[1] - (i128)v[3] * v[0]) * c;
      room += c < 0 ? -c : c;
    }
    // per term and unit of c: half a unit of 2^32 from the rounding, 30 x 2^31 left out
    if (far(s.value() << 32, want, room * (((i128)1 << 31) + ((i128)30 << 31)))) bad("WeightedImSum", it);
  }
  printf(fails ? "FAIL %d\n" : "OK\n", fails);
  return fails ? 1 : 0;
}
