// Windowed passes of the ring XY mixer on the Hamming-weight subspace F_k (states in rank
// order, as in xy.cu).  Everything here compiles for the device and for the host, so the
// tile addressing can be checked exhaustively on the CPU (tests/xy_window_check.cpp).
//
// A window is a run of w consecutive qubits [lo, lo + w).  A state z of F_k splits into the
// bits below the window (L, popcount kL), in it (P, popcount kw) and above it (H, popcount
// h).  The rank of z is the sum over its set bits c_1 < ... < c_k of binom(c_i, i), so
//   rank(z) = rank(L) + sum_j binom(lo + p_j, kL + j) + sum_j binom(lo + w + q_j, kL + kw + j)
// with p_j, q_j the positions (inside P and H) of their j-th set bit, j = 1, 2, ..., and
// rank(L) running over 0 .. binom(lo, kL) - 1 in the order of L.  A pair gate on two qubits
// of the window keeps L, H and popcount(P).  So for a class (h, kw) every column (H, L)
// holds the binom(w, kw) patterns P of popcount kw ("rows"), every gate of the window acts
// inside columns, and element (row r, column c) sits at rank rowoff[r] + colbase[c]:
//   rowoff[r]  = sum_j binom(lo + p_j, kL + j), P the r-th pattern of popcount kw,
//   colbase[c] = rank(L) + sum_j binom(lo + w + q_j, kL + kw + j).
// Columns are ordered H-major (H by its rank among the patterns of nh = n - lo - w bits with
// popcount h) and rank(L)-minor, so a row of a tile reads runs of consecutive ranks.  A tile
// is up to m consecutive columns of one class.  Classes with kw = 0 or kw = w have a single
// row that no gate of the window changes; only a pass that also applies the cost unitary
// (to every amplitude) visits them.
//
// The ring mixer applies the pairs (a, a + 1) with a even, then those with a odd, then the
// closing pair (0, n - 1).  The windows [0, e_0), [e_0 - 1, e_1), [e_1 - 1, e_2), ... (every
// e_i even except the last, e_last = n) share one qubit with their neighbour, so every pair
// (a, a + 1) lies in exactly one window.  A window applies its even pairs, then its odd
// pairs; pairs of different windows either commute or come in the order of the sets (an odd
// pair that crosses e_i - 1 needs the even pair (e_i, e_i + 1), which its own window applies
// first).  The closing pair is a pass of its own.
//
// Half states.  With k = n / 2 the complement ~z of a state is in F_k too, at rank D - 1 - rank(z)
// (D = binom(n, k): complementing reverses the order), and it commutes with every pair gate.  So if
// C(z) = C(~z) (every cut), psi(z) = psi(~z) from the Dicke state on, and the first D / 2 ranks, the
// states with qubit n - 1 clear, carry the whole state.  A window below qubit n - 1 runs on the
// columns whose H has a clear top bit: a prefix of each class's.  The last window and the closing
// pair move qubit n - 1: they visit one of every two complementary columns (pairs), those whose top
// bit below the window (of the middle bits) is clear, again a prefix of each class's, and an
// element of rank r lives at min(r, D - 1 - r).
#pragma once

#include <stdint.h>

#include <algorithm>

#ifdef __CUDACC__
#define XYW_HD __host__ __device__ __forceinline__
#else
#define XYW_HD inline
#endif

namespace qaoa {
namespace xyw {

constexpr int kMaxN = 40;                                // qubits (QAOA_XY_MAX_N)
constexpr int kBN = kMaxN + 1;                           // binomial table side
constexpr int kMaxW = 9;                                 // qubits per window
constexpr int kMaxRows = 126;                            // binom(9, 4)
constexpr int kMaxPairs = 35;                            // binom(7, 3): rows one gate moves
constexpr int kMaxCols = 512;                            // columns per tile
constexpr int kMaxGates = kMaxW - 1;                     // pairs inside one window
constexpr int kMaxClasses = (kMaxN - 1) * (kMaxW + 1);  // h = 0..nh <= n - 2, kw = 0..w
constexpr int kMaxWindows = (kMaxN + 6) / 8 + 1;         // [0, 8), then 8 new qubits per window

typedef unsigned long long u64;

// Half states: a launch with a flag (device) runs on half the state if *flag == 0; D - 1.
struct Fold {
  u64 last;
  const unsigned* flag;
};
XYW_HD u64 fold_rank(u64 last, u64 r) { return r < last - r ? r : last - r; }

struct Class {
  u64 first_tile;  // tiles of the classes before this one
  u64 ncols;       // binom(nh, h) * len
  u64 half_first, half_cols;  // the same on a half state
  u64 len;         // binom(lo, kL): ranks per row run of one H
  unsigned char h, kw, kL;  // popcounts above, inside and below the window
  unsigned char mb;         // columns per tile, a power of two: m = 2^mb
  unsigned short rows, m;   // binom(w, kw)
};

struct Window {
  int n, k, lo, w, nh;
  int ngates;
  int ga[kMaxGates];  // window-relative low qubit of each pair (lo + ga, lo + ga + 1), in order
  int ncls;
  int tile_elems;     // largest rows * m over the classes
  u64 tiles;
  u64 elems;          // amplitudes visited by one pass
  u64 half_tiles, half_elems;
  Fold f;
  Class cls[kMaxClasses];
};

XYW_HD int ctz64(u64 x) {
#ifdef __CUDA_ARCH__
  return __ffsll((long long)x) - 1;
#else
  return __builtin_ctzll(x);
#endif
}
XYW_HD int popc32(unsigned x) {
#ifdef __CUDA_ARCH__
  return __popc(x);
#else
  return __builtin_popcount(x);
#endif
}

// the pattern of nb bits with popcount kk whose rank among those patterns (increasing order)
// is r, r < binom(nb, kk): the i-th set bit is the largest c with binom(c, i) <= r
XYW_HD u64 unrank_bits(u64 r, int nb, int kk, const u64 (*B)[kBN]) {
  u64 z = 0;
  int c = nb - 1;
  for (int i = kk; i >= 1; --i) {
    while (B[c][i] > r) --c;
    z |= 1ull << c;
    r -= B[c][i];
    --c;
  }
  return z;
}

// sum over the set bits of x (j = 1, 2, ... in increasing order) of binom(base + pos, first + j)
XYW_HD u64 rank_part(u64 x, int base, int first, const u64 (*B)[kBN]) {
  u64 s = 0;
  for (int j = first + 1; x != 0; ++j) {
    s += B[base + ctz64(x)][j];
    x &= x - 1;
  }
  return s;
}

// rank of the first element of column `col` of class C, without the row's part
XYW_HD u64 col_base(const Window& W, const Class& C, u64 col, const u64 (*B)[kBN]) {
  const u64 hi = col / C.len, l = col - hi * C.len;
  const u64 H = unrank_bits(hi, W.nh, C.h, B);
  return l + rank_part(H, W.lo + W.w, C.kL + C.kw, B);
}

// the row of pattern P moved by the pair at window bits (ga, ga + 1): P has bit ga set and
// bit ga + 1 clear, and moving its (j + 1)-th set bit up by one adds binom(ga, j) to its rank
XYW_HD int partner_row(int r, unsigned P, int ga, const u64 (*B)[kBN]) {
  return r + (int)B[ga][popc32(P & ((1u << ga) - 1u))];
}

// x / d for x, d < 2^16 as a multiply-high by m = floor(2^32 / d) + 1 (d >= 2): exact,
// because x (m d - 2^32) <= x d < 2^32; m = 0 stands for d = 1
XYW_HD unsigned div_magic(unsigned d) { return d < 2 ? 0u : (unsigned)((1ull << 32) / d + 1); }
XYW_HD unsigned div_small(unsigned x, unsigned m) {
  if (m == 0) return x;
#ifdef __CUDA_ARCH__
  return __umulhi(x, m);
#else
  return (unsigned)(((u64)x * m) >> 32);
#endif
}

XYW_HD int find_class(const Window& W, u64 tile, bool half = false) {
  int a = 0, b = W.ncls - 1;
  while (a < b) {
    const int mid = (a + b + 1) / 2;
    if ((half ? W.cls[mid].half_first : W.cls[mid].first_tile) <= tile) a = mid;
    else b = mid - 1;
  }
  return a;
}

// Pascal's triangle up to kMaxN
XYW_HD void binom_row(u64 (*B)[kBN], int c) {
  u64 v = 1;
  for (int i = 0; i < kBN; ++i) {
    B[c][i] = i <= c ? v : 0;
    v = i < c ? v * (u64)(c - i) / (u64)(i + 1) : 0;  // binom(c, i + 1), exact
  }
}

// ---------------------------------------------------------------- host planning

// The windows of the ring mixer on n qubits (n >= 2): their [lo, lo + w) ranges.
inline int plan_ring_windows(int n, int* lo, int* w) {
  if (n < 2) return 0;
  int nw = 0;
  int e = n <= kMaxW ? n : kMaxW - 1;  // the first window ends at an even bit unless it is the last
  lo[nw] = 0;
  w[nw++] = e;
  while (e < n) {
    const int s = e - 1;
    e = s + kMaxW < n ? s + kMaxW : n;  // s is odd, so s + kMaxW is even
    lo[nw] = s;
    w[nw++] = e - s;
  }
  return nw;
}

// Window [lo, lo + w) of the ring mixer on n qubits: its pairs and its tile classes.
// `target` = amplitudes per tile (per buffer); `every_state` also visits the single-row
// classes (kw = 0, kw = w), for a pass that applies the cost unitary to every amplitude.
// `half` (k = n / 2; not for a window of all qubits) also plans the pass over a half state.
inline void plan_window(Window& W, int n, int k, int lo, int w, int target, const u64 (*B)[kBN],
                        bool every_state = false, bool half = false) {
  W.n = n;
  W.k = k;
  W.lo = lo;
  W.w = w;
  W.nh = n - lo - w;
  W.ngates = 0;
  for (int par = 0; par < 2; ++par)  // even pairs, then odd pairs
    for (int a = lo; a + 1 < lo + w; ++a)
      if ((a & 1) == par) W.ga[W.ngates++] = a - lo;
  W.ncls = 0;
  W.tiles = 0;
  W.elems = 0;
  W.half_tiles = W.half_elems = 0;
  W.f.last = half ? B[n][k] - 1 : 0;
  W.f.flag = nullptr;
  W.tile_elems = 0;
  for (int h = 0; h <= W.nh; ++h) {
    for (int kw = every_state ? 0 : 1; kw <= (every_state ? w : w - 1); ++kw) {
      const int kL = k - h - kw;
      if (kL < 0 || kL > lo) continue;
      Class& C = W.cls[W.ncls++];
      C.h = (unsigned char)h;
      C.kw = (unsigned char)kw;
      C.kL = (unsigned char)kL;
      C.rows = (unsigned short)B[w][kw];
      C.len = B[lo][kL];
      C.ncols = B[W.nh][h] * C.len;
      C.half_cols = !half ? 0 : W.nh == 0 ? B[lo - 1][kL] : B[W.nh - 1][h] * C.len;
      u64 m = 1;  // the most columns of a power of two in the target, no more than the class needs
      C.mb = 0;
      while (2 * m * (u64)C.rows <= (u64)target && 2 * m <= (u64)kMaxCols && m < C.ncols) {
        m *= 2;
        ++C.mb;
      }
      C.m = (unsigned short)m;
      C.first_tile = W.tiles;
      W.tiles += (C.ncols + m - 1) / m;
      W.elems += C.ncols * (u64)C.rows;
      C.half_first = W.half_tiles;
      W.half_tiles += (C.half_cols + m - 1) / m;
      W.half_elems += C.half_cols * (u64)C.rows;
      if (C.rows * C.m > W.tile_elems) W.tile_elems = C.rows * C.m;
    }
  }
}

// ---------------------------------------------------------------- the closing pair

constexpr int kCloseBits = 10;   // most low bits: both parts are below binom(11, 5) + ... < 2^16
constexpr int kCloseCols = 256;  // columns per tile
constexpr int kClosePairs = 2048;
struct Closing {
  int n, k, lb, nh, ncls;
  u64 tiles, half_tiles;
  u64 pairs, half_pairs;  // visited by one pass
  Fold f;
  struct Cls {
    u64 first_tile, ncols, half_first, half_cols;
    int kl, rows, start, m;
  } cls[kCloseBits + 1];
};

// the closing pair's classes and tiles (n >= 3, 0 < k < n).  Half states (n >= lb + 3): one of every
// two complementary pairs, the one whose middle bits have a clear top bit.
inline Closing plan_closing(int n, int k, const u64 (*B)[kBN], bool half = false) {
  Closing W = {};
  W.n = n;
  W.k = k;
  W.lb = std::max(0, std::min(kCloseBits, n - 2));
  W.nh = std::max(0, n - 2 - W.lb);
  W.f.last = half ? B[n][k] - 1 : 0;
  int start = 0;
  for (int kl = 0; kl <= W.lb; ++kl) {
    const int rows = (int)B[W.lb][kl], kh = k - 1 - kl;
    if (kh >= 0 && kh <= W.nh) {
      Closing::Cls& C = W.cls[W.ncls++];
      C.kl = kl;
      C.rows = rows;
      C.start = start;
      C.ncols = B[W.nh][kh];
      C.half_cols = half ? B[W.nh - 1][kh] : 0;
      C.m = std::max(1, std::min(kCloseCols, kClosePairs / rows));
      C.first_tile = W.tiles;
      C.half_first = W.half_tiles;
      W.tiles += (C.ncols + C.m - 1) / C.m;
      W.half_tiles += (C.half_cols + C.m - 1) / C.m;
      W.pairs += C.ncols * (u64)rows;
      W.half_pairs += C.half_cols * (u64)rows;
    }
    start += rows;
  }
  return W;
}

}  // namespace xyw
}  // namespace qaoa
