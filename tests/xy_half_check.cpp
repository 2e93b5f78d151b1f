// Host check of the half states of csrc/xy_window.cuh: for balanced n = 14..20 (two and three windows),
// every window of the half state visits every amplitude of the first D / 2 ranks that its classes
// cover exactly once, and the half plan's layer (windows, closing pair) on a symmetric vector gives
// what the ring mixer's gates give on all D amplitudes.  Both sides are about n rounded float64
// rotations of a unit vector: 1e-13.
// Exit 0 = all good.
#include <cmath>
#include <complex>
#include <cstdio>
#include <random>
#include <vector>

#include "xy_window.cuh"

using namespace qaoa::xyw;
using Cx = std::complex<double>;

static u64 B[kBN][kBN];
static int fails = 0;
#define CHECK(ok, ...) do { if (!(ok) && fails++ < 10) { printf(__VA_ARGS__); printf("\n"); } } while (0)

static void rotate(Cx& x, Cx& y, double cb, double sb) {
  const Cx u = cb * x - Cx(0, sb) * y, v = cb * y - Cx(0, sb) * x;
  x = u;
  y = v;
}

int main() {
  for (int c = 0; c < kBN; ++c) binom_row(B, c);
  std::mt19937_64 rng(3);
  std::normal_distribution<double> nd;
  const double cb = std::cos(0.6), sb = std::sin(0.6);
  for (int n = 14; n <= 20; n += 2) {
    const int k = n / 2;
    const u64 D = B[n][k], half = D / 2;
    std::vector<u64> states;
    for (u64 z = 0; z < (1ull << n); ++z)
      if (__builtin_popcountll(z) == k) states.push_back(z);
    std::vector<int64_t> rank_of(1ull << n, -1);
    for (u64 r = 0; r < D; ++r) {
      rank_of[states[r]] = (int64_t)r;
      CHECK(states[D - 1 - r] == (~states[r] & ((1ull << n) - 1)), "n %d: complement of rank %llu", n, r);
      CHECK((states[r] >> (n - 1)) == (r >= half), "n %d: top bit of rank %llu", n, r);
    }
    std::vector<Cx> full(D), h(half);
    double nn = 0;
    for (u64 r = 0; r < half; ++r) {
      full[r] = full[D - 1 - r] = Cx(nd(rng), nd(rng));
      nn += 2 * std::norm(full[r]);
    }
    for (Cx& x : full) x /= std::sqrt(nn);
    for (u64 r = 0; r < half; ++r) h[r] = full[r];
    auto gate = [&](int a, int b) {
      for (u64 r = 0; r < D; ++r) {
        const u64 z = states[r];
        if ((z >> a & 1) && !(z >> b & 1)) rotate(full[r], full[(u64)rank_of[z ^ (1ull << a) ^ (1ull << b)]], cb, sb);
      }
    };
    for (int par = 0; par < 2; ++par)
      for (int a = par; a + 1 < n; a += 2) gate(a, a + 1);
    gate(0, n - 1);
    int lo[kMaxWindows + 1], w[kMaxWindows + 1];
    const int nwin = plan_ring_windows(n, lo, w);
    CHECK(nwin >= 2, "n %d: one window", n);
    for (int i = 0; i < nwin; ++i) {
      static Window W;
      plan_window(W, n, k, lo[i], w[i], 512, B, i == 0, true);
      const u64 last = W.nh == 0 ? W.f.last : ~0ull;
      std::vector<char> seen(half, 0);
      u64 visited = 0, tiles = 0;
      for (int ci = 0; ci < W.ncls; ++ci) {
        const Class& C = W.cls[ci];
        CHECK(C.half_first == tiles, "n %d window %d: class %d starts at tile %llu", n, i, ci, C.half_first);
        for (u64 t = 0; t < (C.half_cols + C.m - 1) / C.m; ++t)
          CHECK(find_class(W, tiles + t, true) == ci, "n %d window %d: class of tile %llu", n, i, tiles + t);
        tiles += (C.half_cols + (u64)C.m - 1) / (u64)C.m;
        std::vector<unsigned> pat(C.rows);
        for (int r = 0; r < C.rows; ++r) pat[r] = (unsigned)unrank_bits((u64)r, W.w, C.kw, B);
        for (u64 col = 0; col < C.half_cols; ++col) {
          auto at = [&](int r) { return fold_rank(last, rank_part(pat[r], W.lo, C.kL, B) + col_base(W, C, col, B)); };
          for (int r = 0; r < C.rows; ++r) {
            const u64 x = at(r);
            CHECK(x < half && !seen[x], "n %d window %d: rank %llu", n, i, x);
            if (x < half) seen[x] = 1;
            ++visited;
          }
          if (fails) return 1;
          for (int g = 0; g < W.ngates; ++g)
            for (int r = 0; r < C.rows; ++r)
              if (((pat[r] >> W.ga[g]) & 3u) == 1u) rotate(h[at(r)], h[at(partner_row(r, pat[r], W.ga[g], B))], cb, sb);
        }
      }
      CHECK(visited == W.half_elems && tiles == W.half_tiles && (i > 0 || visited == half), "n %d window %d: %llu of %llu", n, i,
            visited, W.half_elems);
    }
    const Closing K = plan_closing(n, k, B, true);
    u64 pairs = 0;
    std::vector<char> seen(half, 0);
    for (int ci = 0; ci < K.ncls; ++ci) {
      const Closing::Cls& C = K.cls[ci];
      for (u64 col = 0; col < C.half_cols; ++col)
        for (u64 x = 0; x < (1ull << K.lb); ++x) {
          if (__builtin_popcountll(x) != C.kl) continue;
          const u64 y = (unrank_bits(col, K.nh, k - 1 - C.kl, B) << K.lb | x) << 1;
          const u64 rz = (u64)rank_of[y | 1], rp = fold_rank(K.f.last, (u64)rank_of[y | 1ull << (n - 1)]);
          CHECK(rz < half && rp < half && rz != rp && !seen[rz] && !seen[rp], "n %d closing: %llu %llu", n, rz, rp);
          if (fails) return 1;
          seen[rz] = seen[rp] = 1;
          rotate(h[rz], h[rp], cb, sb);
          ++pairs;
        }
    }
    CHECK(pairs == K.half_pairs && pairs == B[n - 2][k - 1] / 2, "n %d closing: %llu pairs", n, pairs);
    double e = 0;
    for (u64 r = 0; r < half; ++r) e += 2 * std::norm(h[r] - full[r]);
    CHECK(std::sqrt(e) < 1e-13, "n %d: state error %g", n, std::sqrt(e));
  }
  puts(fails ? "FAILED" : "OK");
  return fails != 0;
}
