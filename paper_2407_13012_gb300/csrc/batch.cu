// Batched adjoint gradients: thousands of small graphs (n ~ 8..20).
//
// The per-graph computation is the plain method (cost vector, Eq. 1's p layers, <C>, and
// the adjoint gradient of Sec. IV-D); only the scheduling differs from the one-graph path.
// One prep launch builds every graph's cost vector and tables.  Then the graphs run in one
// of two ways, by size (the host decides, capi.cu):
//  * grouped sweeps (the larger graphs, whose one-graph plan is all lean sweeps): the graphs
//    of one size run the one-graph gradient plan together, each sweep one launch of the
//    one-graph lean kernel over all of them, each block on its own graph's tiles, tables and
//    angles (GroupSlot), then one reduction per size;
//  * the persistent kernel below (the rest): one CTA owns one graph at a time and runs the
//    graph's whole sweep plan over the graph's own buffers, tile after tile, with CTA
//    barriers between sweeps, writing the graph's outputs from its block accumulators.
//    complex128 sweeps on full 2^12 tiles use the lean tile code, the rest the generic
//    program (for complex64 the lean form spilled and measured slower).  Graphs come off a
//    work counter largest first (longest-processing-time order).  Small graphs (n <= 10)
//    run on 2^10-amplitude tiles, larger ones on 2^12; the host may pick per qubit count
//    from measured times.
#include "batch_kernel.cuh"

namespace qaoa {
namespace {

constexpr int kPrepThreads = 256;
constexpr int kMaxBatchEdges = 512;
static_assert(QAOA_BATCH_MAX_EDGES <= kMaxBatchEdges, "edge staging holds every edge of a graph");
static_assert(QAOA_BATCH_MAX_N < 32, "cost-vector indices in 32 bits");

// The costs of one block's 2^12 entries z = (h, y, x), y and x six bits each, h fixed:
//   C(z) = Q0[x] + T1[y] + sum_{u < 6} x_u a_u[y],
// Q0 the edges inside x, T1 those inside y, between y and h and inside h, and
// a_u[y] = sum_{v >= 6} w_uv (1 - 2 z_v), which together with the cut edges' constant w z_v (part of
// T1) gives the edges leaving x.  The tables take a few operations per thread; an entry is then
// three additions (summing every edge per entry took 9.8 of the 191 ms of the 4096-graph batch).
// S: unsigned for integer weights (sums modulo 2^32 give the exact int32 cost), long long for
// fixed-point ones.  4096-graph batch, complex128: 174.4 -> 167.0 ms.
constexpr int kHalf = 6;
template <class S, class OUT>
__device__ __forceinline__ void batch_costs(int n, const int2* e_s, const S* w_s, int m, uint32_t z0, S* W, S* tab,
                                            OUT&& put) {
  constexpr int N = QAOA_BATCH_MAX_N, H = 1 << kHalf;
  S* Q0 = tab;              // [64]
  S* T1 = tab + H;          // [64]
  S* A = tab + 2 * H;       // [6][64]
  S* lin = tab + 8 * H;     // [12]: bits 0..5: sum over h of w (1 - 2 h_v); bits 6..11: the same
  S* kh = lin + 2 * kHalf;  // edges inside h, and the constants h_v w of edges into h
  const int tid = threadIdx.x;
  for (int i = tid; i < N * N; i += kPrepThreads) W[i] = 0;
  __syncthreads();
  for (int k = tid; k < m; k += kPrepThreads) {
    W[e_s[k].x * N + e_s[k].y] = w_s[k];
    W[e_s[k].y * N + e_s[k].x] = w_s[k];
  }
  __syncthreads();
  if (tid < 2 * kHalf) {
    S s = 0;
    for (int v = 2 * kHalf; v < n; ++v) s += (z0 >> v) & 1u ? -W[tid * N + v] : W[tid * N + v];
    lin[tid] = s;
  } else if (tid == 32) {
    S s = 0;
    for (int v = 2 * kHalf; v < n; ++v) {
      if (!((z0 >> v) & 1u)) continue;
      for (int u = 0; u < n; ++u)  // inside h: pairs with a clear bit; below h: the constant
        if (u < 2 * kHalf || !((z0 >> u) & 1u)) s += W[v * N + u];
    }
    *kh = s;
  }
  __syncthreads();
  for (int i = tid; i < 8 * H; i += kPrepThreads) {
    const int y = i % H, row = i / H;
    S s = 0;
    if (row == 0) {
      for (int u = 0; u < kHalf; ++u)
        for (int v = u + 1; v < kHalf; ++v)
          if (((y >> u) ^ (y >> v)) & 1) s += W[u * N + v];
    } else if (row == 1) {
      s = *kh;
      for (int u = 0; u < kHalf; ++u) {
        if (!((y >> u) & 1)) continue;
        s += lin[kHalf + u];
        for (int v = 0; v < kHalf; ++v)  // inside y: pairs with a clear bit; below y: the constant
          s += W[(kHalf + u) * N + v] + ((y >> v) & 1 ? 0 : W[(kHalf + u) * N + kHalf + v]);
      }
    } else {
      const int u = row - 2;
      s = lin[u];
      for (int v = 0; v < kHalf; ++v) s += (y >> v) & 1 ? -W[u * N + kHalf + v] : W[u * N + kHalf + v];
    }
    tab[i] = s;
  }
  __syncthreads();
  // thread: one y, 16 consecutive x
  const int y = tid >> 2, x0 = (tid & 3) * 16;
  S base = T1[y];
  if (x0 & 16) base += A[4 * H + y];
  if (x0 & 32) base += A[5 * H + y];
  const uint32_t z = z0 + (uint32_t)(y << kHalf) + (uint32_t)x0;
  if (z >= (1u << n)) return;
  S s[16];
  s[0] = base;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const S au = A[u * H + y];
#pragma unroll
    for (int i = 0; i < (1 << u); ++i) s[i + (1 << u)] = s[i] + au;
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) s[i] += Q0[x0 + i];
  put(z, s);
}

// One launch prepares every graph: blocks [0, cost_blocks) build the cost vectors (2^12
// entries per block, C(z) = sum over edges of w [z_u != z_v], Sec. III-B's MaxCut cost, int32
// for integer weights; float weights are quantised once to a common fixed point,
// 2^-(62 - e) with sum |w| < 2^e, summed exactly in int64 and rounded once to float64, as the
// one-graph cost kernel does); the next ngraphs blocks build each graph's per-layer terms and
// tables; the last block (fixed point) builds the shared turn tables.
__global__ void __launch_bounds__(kPrepThreads) batch_prep_kernel(const __grid_constant__ BatchArgs b,
                                                                   int64_t cost_blocks) {
  __shared__ int2 e_s[kMaxBatchEdges];
  __shared__ long long w_s[kMaxBatchEdges];  // integer weights (int) or float weights in fixed point
  __shared__ long long W_s[QAOA_BATCH_MAX_N * QAOA_BATCH_MAX_N];
  __shared__ long long tab_s[8 * (1 << kHalf) + 2 * kHalf + 1];
  __shared__ int shift_s;
  const int64_t blk = blockIdx.x;
  const int tid = threadIdx.x;
  const int p = b.p;
  const bool fx = b.dtype == QAOA_C128;
  if (blk < cost_blocks) {
    int lo = 0, hi = b.ngraphs - 1;  // last graph with blk_off <= blk
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (b.blk_off[mid] <= blk) lo = mid;
      else hi = mid - 1;
    }
    const BatchGraph G = b.graphs[lo];
    if (tid == 0) {
      int sh = 0;
      if (b.cost_f64) {  // sum |w| in edge order, as the host does for the one-graph kernel
        double sa = 0.0;
        for (int k = 0; k < G.m; ++k) sa += fabs(b.ew[G.edge + k]);
        int e2 = 0;
        frexp(sa > 0.0 ? sa : 1.0, &e2);
        sh = 62 - e2;
      }
      shift_s = sh;
    }
    __syncthreads();
    for (int k = tid; k < G.m; k += kPrepThreads) {
      e_s[k] = make_int2(b.edges[2 * (G.edge + k)], b.edges[2 * (G.edge + k) + 1]);
      const double w = b.ew[G.edge + k];
      if (b.cost_f64) w_s[k] = llrint(ldexp(w, shift_s));
      else ((int*)w_s)[k] = (int)w;
    }
    // n <= QAOA_BATCH_MAX_N < 32: 32-bit indices
    const uint32_t z0 = (uint32_t)(blk - b.blk_off[lo]) << kBatchCostBits;
    const int live = min(16, 1 << G.n);  // entries of a thread's 16 inside the vector
    if (b.cost_f64) {
      double* out = (double*)b.C + G.cost;
      batch_costs<long long>(G.n, e_s, w_s, G.m, z0, W_s, tab_s, [&](uint32_t z, const long long(&s)[16]) {
#pragma unroll
        for (int i = 0; i < 16; ++i)  // (to_double forms normal numbers: every entry's are down to 2^-1022)
          if (i < live) out[z + i] = shift_s <= 1022 ? fx::to_double(s[i], shift_s) : ldexp((double)s[i], -shift_s);
      });
    } else {
      int* out = (int*)b.C + G.cost;
      batch_costs<unsigned>(G.n, e_s, (const unsigned*)w_s, G.m, z0, (unsigned*)W_s, (unsigned*)tab_s,
                            [&](uint32_t z, const unsigned(&s)[16]) {
        if (live == 16) {  // graphs start 64-element aligned
#pragma unroll
          for (int i = 0; i < 16; i += 4) *(int4*)(out + z + i) =
            make_int4((int)s[i], (int)s[i + 1], (int)s[i + 2], (int)s[i + 3]);
        } else {
          for (int i = 0; i < live; ++i) out[z + i] = (int)s[i];
        }
      });
    }
    return;
  }
  const int64_t gi = blk - cost_blocks;
  if (gi < b.ngraphs) {
    const BatchGraph G = b.graphs[gi];
    const double* ang = b.angles + gi * 2 * p;
    double* trig = b.trig + gi * 3 * p;
    for (int l = tid; l < p; l += kPrepThreads) {
      trig[l] = ang[l] / (2.0 * 3.141592653589793238);
      double sn, cs;
      sincos(ang[p + l], &sn, &cs);
      trig[p + l] = cs;
      trig[2 * p + l] = sn;
    }
    const int64_t nph = (int64_t)p * G.span;
    for (int64_t i = tid; i < nph; i += kPrepThreads) {
      const int l = (int)(i / G.span);
      const double th = ang[l] * (double)(G.cmin + (i - (int64_t)l * G.span));
      if (fx) ((longlong2*)b.phase)[G.table + i] = unit_q62(th);
      else ((float2*)b.phase)[G.table + i] = unit_f32(th);
    }
    if (fx)
      for (int i = tid; i < p * 196; i += kPrepThreads)
        ((longlong2*)b.dtab)[gi * p * 196 + i] = d_entry(ang[p + i / 196], i % 196);
    return;
  }
  if (fx)
    for (int j = tid; j < kTurnEntries; j += kPrepThreads) ((longlong2*)b.turn)[j] = turn_entry(j);
}

// The persistent kernel: graphs [first, first + count) of the processing order, taken from
// *queue one at a time by each CTA.
}  // namespace

int batch_tile_bits(int tile) { return tile == 0 ? CfgXS::B : CfgXB::B; }
int batch_register_bits(int dtype, int tile) {
  if (tile == 0) return dtype == QAOA_C128 ? CfgXS::RB : CfgFS::RB;
  return dtype == QAOA_C128 ? CfgXB::RB : CfgFB::RB;
}

cudaError_t launch_batch_prep(const BatchArgs& b, int64_t cost_blocks, cudaStream_t s) {
  const int64_t blocks = cost_blocks + b.ngraphs + 1;
  note_launch(1, s, true);
  batch_prep_kernel<<<(unsigned)blocks, kPrepThreads, 0, s>>>(b, cost_blocks);
  note_launch(1, s, false);
  return cudaGetLastError();
}

cudaError_t launch_batch(const BatchArgs& b, int tile, int first, int count, int* queue, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  note_launch(0, s, true);
  cudaError_t e;
  if (b.dtype == QAOA_C128)
    e = tile == 0 ? launch_batch_cfg<CfgXS, true, false>(b, first, count, queue, s)
                  : launch_batch_c128_large(b, first, count, queue, s);
  else
    e = tile == 0 ? launch_batch_cfg<CfgFS, false, false>(b, first, count, queue, s)
                  : launch_batch_cfg<CfgFB, false, false>(b, first, count, queue, s);
  note_launch(0, s, false);
  return e;
}

}  // namespace qaoa
