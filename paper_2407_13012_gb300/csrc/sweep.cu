// Layer sweeps: phase separator, mixer, lambda = C psi and the fused reductions of <C>,
// the norm and the adjoint-gradient terms (Eq. 1; Sec. II-B, IV-B, IV-C, IV-D); the tile
// machinery and the arithmetic are described in sweeper.cuh.
#include "lean_kernel.cuh"

namespace qaoa {
namespace {


template <class CF, bool FX, bool TWO>
__global__ void __launch_bounds__(CF::NT, CF::MINB) sweep_kernel(const __grid_constant__ SweepArgs a) {
  using S = Sweeper<CF, FX, TWO>;
  using V = typename S::V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* X = (V*)smem_raw;  // exchange area: 2^B slots, twice that for two-buffer sweeps
  void* Cs = smem_raw + ((sizeof(V) << CF::B) << (TWO ? 1 : 0));
  V* Tsm = (V*)((unsigned char*)Cs + (a.needs_cost ? ((a.cost_dtype == QAOA_COST_F64 ? 8 : 4) << CF::B) : 0));
  __shared__ double blk[kMaxAcc];
  __shared__ double red[2 * (CF::NT / 32)];
  __shared__ fx::Factor dsm[16];
  for (int r = threadIdx.x; r < kMaxAcc; r += CF::NT) blk[r] = 0.0;

  S s(a, X, Cs, blk, red);
  s.Ds = dsm;
  if (a.smem_table_layer >= 0) {  // one layer's phase table in shared memory
    stage_table<FX>(s, a, Tsm, CF::NT);
    __syncthreads();
  }
  const SweepGeom& g = a.g;
  s.evalid = 1u << (g.t + g.c);
  if constexpr (FX) {
    if (a.scan != nullptr) s.set_scan(read_scan(a.scan, a.nscan));
    s.in_shift = input_shift(a.norm2_dev);
  }
  for (int64_t tile = blockIdx.x; tile < g.tiles; tile += gridDim.x) sweep_tile<CF, FX, TWO, false>(s, a, tile, Cs);

  __syncthreads();
  for (int r = threadIdx.x; r < a.nred; r += CF::NT)
    a.partials[(int64_t)a.red_slot[r] * a.grid + blockIdx.x] = blk[r];
}

// ------------------------------------------------------------------ small kernels

__global__ void reduce_kernel(const __grid_constant__ ReducePlan r, const double* __restrict__ partials,
                              double* __restrict__ out, const unsigned long long* scan, int nscan) {
  const bool twice = scan != nullptr && read_scan(scan, nscan).symmetric;
  const int o = blockIdx.x;
  __shared__ double sh[256];
  double v = 0.0;
  const int64_t n = (int64_t)r.ncontrib[o] * r.grid;
  const double* base = partials + (int64_t)o * kMaxContrib * r.grid;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) v += base[i];
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[o] = sh[0] * r.scale[o] * (twice ? 2.0 : 1.0);
}

// grouped sweeps: one warp per (graph, output), summing the graph's contributions and blocks
// in a fixed order
__global__ void group_reduce_kernel(const __grid_constant__ ReducePlan r, int ngraphs, int bpg,
                                    const int* __restrict__ out_row, const double* __restrict__ partials,
                                    double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t item = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (item >= (int64_t)ngraphs * r.nout) return;
  const int g = (int)(item / r.nout), o = (int)(item % r.nout);
  double v = 0.0;
  for (int i = lane; i < r.ncontrib[o] * bpg; i += 32) {
    const int k = i / bpg, j = i - k * bpg;
    v += partials[((int64_t)o * kMaxContrib + k) * r.grid + (int64_t)g * bpg + j];
  }
  for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
  if (lane == 0) out[(int64_t)out_row[g] * r.nout + o] = v * r.scale[o];
}

// integer-cost phase tables exp(-i gamma_l c), c = cmin + k; then (fixed point) the
// mixer diagonals exp(-i beta_l (t - 2k)) for t = 1..13, k = 0..t, and the turn tables
__host__ __device__ inline int64_t table_entries(const TableArgs& t) {
  return (int64_t)t.p * t.span + (t.fx ? (int64_t)t.p * 196 + kTurnEntries : 0) + (t.trig != nullptr ? t.p : 0);
}
// entries first, first + step, ... of the call's tables
__device__ void make_tables(const TableArgs& ta, int64_t first, int64_t step) {
  const int64_t nphase = (int64_t)ta.p * ta.span;
  const int64_t nd = ta.fx ? (int64_t)ta.p * 14 * 14 : 0;
  const int64_t nt = ta.fx ? kTurnEntries : 0;
  const int64_t total = table_entries(ta);
  for (int64_t i = first; i < total; i += step) {
    if (i >= nphase + nd + nt) {  // [g2pi p | cos(beta) p | sin(beta) p] from device angles [gamma p | beta p]
      const int l = (int)(i - nphase - nd - nt);
      ta.trig[l] = ta.dev_angles[l] / (2.0 * 3.141592653589793238);
      double sn, cs;
      sincos(ta.dev_angles[ta.p + l], &sn, &cs);
      ta.trig[ta.p + l] = cs;
      ta.trig[2 * ta.p + l] = sn;
    } else if (i < nphase) {
      const int l = (int)(i / ta.span);
      const int64_t c = ta.cmin + (i - (int64_t)l * ta.span);
      const double th = (ta.dev_angles ? ta.dev_angles[l] : ta.gamma[l]) * (double)c;
      if (ta.fx) ((longlong2*)ta.phase)[i] = unit_q62(th);
      else ((float2*)ta.phase)[i] = unit_f32(th);
    } else if (i < nphase + nd) {
      const int64_t j = i - nphase;
      const int l = (int)(j / 196);
      ((longlong2*)ta.dtab)[j] = d_entry(ta.dev_angles ? ta.dev_angles[ta.p + l] : ta.beta[l], (int)(j % 196));
    } else {
      ((longlong2*)ta.turn)[i - nphase - nd] = turn_entry((int)(i - nphase - nd));
    }
  }
}
__global__ void tables_kernel(const __grid_constant__ TableArgs ta) {
  make_tables(ta, blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x);
}

// One Adam ascent step on the angles from the gradient output g = [E, norm, dE/dgamma,
// dE/dbeta]; state = [m (2p) | v (2p)]; *step counts completed steps.  The record of this
// step (the 2p + 2 gradient outputs followed by the 2p angles it was evaluated at) goes to
// history[step * (4p + 2)] when history is non-null.
__global__ void adam_kernel(double* __restrict__ ang, const double* __restrict__ g, double* __restrict__ state,
                            long long* __restrict__ step, int p, double lr, double b1, double b2, double eps,
                            double* __restrict__ history, long long row0, long long max_rows) {
  const int i = threadIdx.x;
  const long long t = *step;  // completed steps before this one
  const int np2 = 2 * p;
  if (history != nullptr && t >= row0 && t - row0 < max_rows) {
    double* h = history + (t - row0) * (2 * np2 + 2);
    for (int k = i; k < np2 + 2; k += blockDim.x) h[k] = g[k];
    for (int k = i; k < np2; k += blockDim.x) h[np2 + 2 + k] = ang[k];
  }
  __syncthreads();
  const double c1 = 1.0 - pow(b1, (double)(t + 1)), c2 = 1.0 - pow(b2, (double)(t + 1));
  for (int k = i; k < np2; k += blockDim.x) {
    const double gk = g[2 + k];  // ascent on <C>
    double m = state[k], v = state[np2 + k];
    m = b1 * m + (1.0 - b1) * gk;
    v = b2 * v + (1.0 - b2) * gk * gk;
    state[k] = m;
    state[np2 + k] = v;
    ang[k] += lr * (m / c1) / (sqrt(v / c2) + eps);
  }
  __syncthreads();
  if (i == 0) *step = t + 1;
}

// |C| as an unsigned integer that orders like it
__device__ __forceinline__ unsigned cost_abs(unsigned c) { return (int)c < 0 ? 0u - c : c; }
__device__ __forceinline__ unsigned long long cost_abs(unsigned long long c) { return c & ~(1ull << 63); }

// One read of C (float64 bits or int32): per block, the bits of max |C| as a double, with the sign
// bit set if C[i] != C[count - 1 - i] for some i.  16 bytes at a time (both ends of C 16-byte
// aligned) or one by one.  The call's tables (ta.p = 0: none) ride along, a warp's worth of entries to
// each block before a second to any.  Without `bound` max |C| is not wanted, and a thread that has met
// an asymmetric pair stops: a cost that has them everywhere is told after 128 KB per block (p = 1 complex64
// layers with such a cost: n = 24 191.8 -> 182.2 us, n = 26 1298 -> 1253, n = 28 2863 -> 2691).
template <class T>
__global__ void __launch_bounds__(1024) cost_scan_kernel(const T* __restrict__ C, int64_t count, int vec, int bound,
                                                         unsigned long long* __restrict__ scan,
                                                         const __grid_constant__ TableArgs ta) {
  if (ta.p > 0)
    make_tables(ta, ((int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31),
                (int64_t)gridDim.x * blockDim.x);
  const int64_t half = count >> 1, stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  constexpr int E = 16 / sizeof(T);
  T mx = 0;
  bool asym = false;
  auto pair = [&](T x, T y) {
    mx = max(mx, max(cost_abs(x), cost_abs(y)));
    asym |= x != y;
  };
  union Q {
    uint4 v;
    T e[E];
  };
  if (vec) {
    const int64_t n16 = (half + E - 1) / E;
    for (int64_t i0 = first; i0 < n16 && (bound || !asym); i0 += 4 * stride) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int64_t i = i0 + u * stride;
        if (i >= n16) break;
        Q x, y;
        x.v = __ldg((const uint4*)C + i);
        y.v = __ldg((const uint4*)(C + count) - 1 - i);
#pragma unroll
        for (int e = 0; e < E; ++e) pair(x.e[e], y.e[E - 1 - e]);
      }
    }
  } else {
    for (int64_t i = first; i < half && (bound || !asym); i += stride) pair(__ldg(C + i), __ldg(C + count - 1 - i));
  }
  __shared__ T wmax[32];
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_down_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = mx;
  const bool any = __syncthreads_or(asym);
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) mx = max(mx, wmax[w]);
    const unsigned long long b = sizeof(T) == 4 ? (unsigned long long)__double_as_longlong((double)mx) : (unsigned long long)mx;
    scan[blockIdx.x] = b | (any ? 1ull << 63 : 0);
  }
}

__global__ void scan_flag_kernel(const unsigned long long* __restrict__ scan, int nscan, unsigned* flag) {
  const bool symmetric = read_scan(scan, nscan).symmetric;
  if (threadIdx.x == 0) *flag = symmetric ? 0u : 1u;
}

// state norm^2 of a user (float64 / float32) state, for the fixed-point input scale
__global__ void norm_kernel(const void* __restrict__ psi, int dtype, int64_t count, double* __restrict__ partials) {
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    if (dtype == QAOA_C128) {
      const double2 d = __ldg((const double2*)psi + i);
      s += d.x * d.x + d.y * d.y;
    } else {
      const float2 f = __ldg((const float2*)psi + i);
      s += (double)f.x * f.x + (double)f.y * f.y;
    }
  }
  __shared__ double sh[256];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int st = blockDim.x / 2; st > 0; st >>= 1) {
    if ((int)threadIdx.x < st) sh[threadIdx.x] += sh[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) partials[blockIdx.x] = sh[0];
}

// ------------------------------------------------------------------ launch plumbing

int num_sms() {
  static int cached = 0;
  if (!cached) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&cached, cudaDevAttrMultiProcessorCount, dev);
    if (cached <= 0) cached = 1;
  }
  return cached;
}

// blocks per SM for a configuration with a cost tile of cost_bytes per amplitude (0, 4, 8)
template <class CF, bool FX, bool TWO>
int blocks_per_sm(int cost_bytes) {
  static int cached[3] = {0, 0, 0};
  static std::mutex mu;
  static uint64_t done = 0;
  const int slot = cost_bytes == 0 ? 0 : (cost_bytes == 4 ? 1 : 2);
  once_per_device(mu, done, [] {
    cudaFuncSetAttribute(sweep_kernel<CF, FX, TWO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem_bytes<CF, FX, TWO>(8, kSmemTable));
  });
  if (!cached[slot]) {
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, sweep_kernel<CF, FX, TWO>, CF::NT,
                                                  smem_bytes<CF, FX, TWO>(cost_bytes, kSmemTable));
    cached[slot] = nb > 0 ? nb : 1;
  }
  return cached[slot];
}

// the lean kernels of this configuration (translation units lean_*.cu)
template <class CF, bool FX, bool TWO>
void lean_launch_cfg(const SweepArgs& a, size_t sm, cudaStream_t s) {
  if constexpr (CF::B == CfgXT::B) TWO ? lean_xt2(a, sm, s) : lean_xt1(a, sm, s);
  else if constexpr (CF::B == CfgXM::B) TWO ? lean_xm2(a, sm, s) : lean_xm1(a, sm, s);
  else if constexpr (FX && !TWO) lean_x1(a, sm, s);
  else if constexpr (FX) a.kind == SWEEP_LEAN_OPS ? lean_x2_ops(a, sm, s) : lean_x2_mix(a, sm, s);
  else if constexpr (!TWO) lean_f1(a, sm, s);
  else lean_f2(a, sm, s);
}

template <class CF, bool FX, bool TWO>
void launch_t(const SweepArgs& a, cudaStream_t s) {
  blocks_per_sm<CF, FX, TWO>(8);
  const int cb = a.needs_cost ? (a.cost_dtype == QAOA_COST_F64 ? 8 : 4) : 0;
  const int te = a.smem_table_layer >= 0 ? (int)a.span : 0;
  size_t sm = smem_bytes<CF, FX, TWO>(cb, te);
  if (a.kind == SWEEP_LEAN_MIX || a.kind == SWEEP_LEAN_OPS) {
    // complex128 two-buffer sweeps that load psi stage the next tile's psi when shared
    // memory allows (complex64: measured no gain)
    SweepArgs b = a;
    b.stage = 0;
    if (a.needs_cost) {
      sm = smem_bytes<CF, FX, TWO>(lean_cost_bytes<FX>(a.cost_dtype), te);
      b.smem_turns = FX && a.kind == SWEEP_LEAN_OPS && a.cost_dtype == QAOA_COST_F64;
      if (b.smem_turns) sm += sizeof(longlong2) * kTurnEntries;
    }
    if (TWO && FX && !(a.kind == SWEEP_LEAN_OPS && a.load_fmt == 2)) {
      const size_t st = ((sm + 15) & ~(size_t)15) + ((FX ? sizeof(longlong2) : sizeof(float2)) << CF::B);
      if (st <= lean_smem_cap<CF, FX, TWO>()) {
        b.stage = 1;
        lean_launch_cfg<CF, FX, TWO>(b, st, s);
        return;
      }
    }
    lean_launch_cfg<CF, FX, TWO>(b, sm, s);
    return;
  }
  sweep_kernel<CF, FX, TWO><<<a.grid, CF::NT, sm, s>>>(a);
}

// <C> and the norm of a user-format state, one pass (stand-alone expectation)
template <bool C128>
__global__ void expect_kernel(const void* __restrict__ psi, const void* __restrict__ C, int cost_f64, int64_t count,
                              double* __restrict__ partials, int grid) {
  double e0 = 0.0, e1 = 0.0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i0 < count; i0 += 32 * stride) {
    float f0 = 0.f, f1 = 0.f;
    for (int k = 0; k < 32; ++k) {
      const int64_t i = i0 + k * stride;
      if (i >= count) break;
      const double c = cost_f64 ? __ldg((const double*)C + i) : (double)__ldg((const int*)C + i);
      if (C128) {
        const double2 d = __ldg((const double2*)psi + i);
        const double pr = d.x * d.x + d.y * d.y;
        e0 += c * pr;
        e1 += pr;
      } else {
        const float2 f = __ldg((const float2*)psi + i);
        const float pr = f.x * f.x + f.y * f.y;
        f0 += (float)c * pr;
        f1 += pr;
      }
    }
    if (!C128) {
      e0 += f0;
      e1 += f1;
    }
  }
  __shared__ double sh[2][256];
  sh[0][threadIdx.x] = e0;
  sh[1][threadIdx.x] = e1;
  __syncthreads();
  for (int st = blockDim.x / 2; st > 0; st >>= 1) {
    if ((int)threadIdx.x < st) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + st];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + st];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = sh[0][0];
    partials[(int64_t)kMaxContrib * grid + blockIdx.x] = sh[1][0];
  }
}

}  // namespace

// complex128 sweeps of up to kSmallTileN qubits run on 512-amplitude tiles (from n = 13 on in two groups
// like 4096-amplitude tiles, so in as many sweeps): they fill the chip better while the large tiles of
// such a state are fewer than its SMs.  At n = 10..12, where one 4096-amplitude tile takes the whole
// circuit in one launch, two groups of small tiles are still faster: p = 6 layers 84 -> 62 us (n = 10) and
// 92 -> 56 (n = 12), p = 1 33 -> 24 and 27 -> 24, p = 6 gradient 270 -> 173 and 284 -> 156.  Measured,
// 4096- -> 512-amplitude tiles: n = 14, p = 4,
// 50 Adam steps 12.4 -> 5.5 ms; n = 16 and 18, p = 6 gradients 353 -> 175 and 366 -> 266 us; n = 17,
// p = 6 layers 151 -> 88 us.  n = 19 (4096- -> 1024-amplitude tiles, half states): p = 6 layers 151 -> 118 us,
// gradient 383 -> 314 us, 50 Adam steps 12.3 -> 10.2 ms.  At n = 20 those lose: layers 151 -> 153, gradient
// 389 -> 430 us, and a cost that is not symmetric 189 -> 230 us.
constexpr int kSmallTileN = 18, kMidTileN = 19;

int sweep_tile_bits(int dtype, int n) {
  return dtype == QAOA_C128 ? (n <= kSmallTileN ? CfgXT::B : n <= kMidTileN ? CfgXM::B : CfgX1::B) : CfgF1::B;
}

// values stay below 2^61 through a group's Walsh-Hadamard transform (growth 2^(t/2)) for
// states of norm < 2, as the limb multiply requires
int fx_shift_for(int tmax) { return 62 - (tmax + 1) / 2 - 2; }

int sweep_grid(int dtype, bool two, int tile_bits, int cost_bytes, int64_t tiles) {
  int per_sm;
  if (dtype == QAOA_C128 && tile_bits == CfgXT::B) {
    per_sm = two ? blocks_per_sm<CfgXT, true, true>(cost_bytes) : blocks_per_sm<CfgXT, true, false>(cost_bytes);
  } else if (dtype == QAOA_C128 && tile_bits == CfgXM::B) {
    per_sm = two ? blocks_per_sm<CfgXM, true, true>(cost_bytes) : blocks_per_sm<CfgXM, true, false>(cost_bytes);
  } else if (dtype == QAOA_C128) {
    per_sm = two ? blocks_per_sm<CfgX2, true, true>(cost_bytes) : blocks_per_sm<CfgX1, true, false>(cost_bytes);
  } else if (two) {
    per_sm = blocks_per_sm<CfgF3, false, true>(cost_bytes);
  } else {
    per_sm = blocks_per_sm<CfgF1, false, false>(cost_bytes);
  }
  const int64_t cap = (int64_t)num_sms() * per_sm;
  return (int)(tiles < cap ? tiles : cap);
}

cudaError_t launch_sweep(int dtype, bool two, const SweepArgs& a, cudaStream_t s) {
  note_launch(0, s, true);
  if (dtype == QAOA_C128 && a.tile_bits == CfgXT::B) {
    if (two) launch_t<CfgXT, true, true>(a, s);
    else launch_t<CfgXT, true, false>(a, s);
  } else if (dtype == QAOA_C128 && a.tile_bits == CfgXM::B) {
    if (two) launch_t<CfgXM, true, true>(a, s);
    else launch_t<CfgXM, true, false>(a, s);
  } else if (dtype == QAOA_C128) {
    if (two) launch_t<CfgX2, true, true>(a, s);
    else launch_t<CfgX1, true, false>(a, s);
  } else {
    if (two) launch_t<CfgF3, false, true>(a, s);
    else launch_t<CfgF1, false, false>(a, s);
  }
  note_launch(0, s, false, a.algo_bytes, a.half_bytes, a.timing_slot);
  return cudaGetLastError();
}

cudaError_t launch_expect(int dtype, const void* psi, const void* C, int cost_dtype, int n, double* partials,
                          int grid, cudaStream_t s) {
  const int64_t count = 1ll << n;
  const double bytes = (double)count * ((dtype == QAOA_C128 ? 16.0 : 8.0) + (cost_dtype == QAOA_COST_F64 ? 8.0 : 4.0));
  note_launch(0, s, true);
  if (dtype == QAOA_C128)
    expect_kernel<true><<<grid, 256, 0, s>>>(psi, C, cost_dtype == QAOA_COST_F64, count, partials, grid);
  else
    expect_kernel<false><<<grid, 256, 0, s>>>(psi, C, cost_dtype == QAOA_COST_F64, count, partials, grid);
  note_launch(0, s, false, bytes);
  return cudaGetLastError();
}

cudaError_t launch_reduce(const ReducePlan& r, const double* partials, double* out, cudaStream_t s,
                          const unsigned long long* scan, int nscan) {
  note_launch(3, s, true);
  reduce_kernel<<<r.nout, 256, 0, s>>>(r, partials, out, scan, nscan);
  note_launch(3, s, false);
  return cudaGetLastError();
}

cudaError_t launch_group_reduce(const ReducePlan& r, int ngraphs, int bpg, const int* out_row,
                                const double* partials, double* out, cudaStream_t s) {
  const int64_t items = (int64_t)ngraphs * r.nout;
  if (items == 0) return cudaSuccess;
  note_launch(3, s, true);
  group_reduce_kernel<<<(unsigned)((items + 7) / 8), 256, 0, s>>>(r, ngraphs, bpg, out_row, partials, out);
  note_launch(3, s, false);
  return cudaGetLastError();
}

cudaError_t launch_tables(const TableArgs& t, cudaStream_t s) {
  const int64_t total = table_entries(t);
  if (total <= 0) return cudaSuccess;
  // an entry is a float64 sincos, ~100 operations of which an SM quarter retires one per 64 cycles
  // and warp: one warp per block spreads them over the chip (with the angle terms in the same launch
  // and max |C| read once per run, 50 Adam steps at n = 14, p = 4 went from 5.5 to 5.05 ms)
  const int64_t blocks = std::min<int64_t>((total + 31) / 32, 4096);
  note_launch(3, s, true);
  tables_kernel<<<(int)blocks, 32, 0, s>>>(t);
  note_launch(3, s, false);
  return cudaGetLastError();
}

cudaError_t launch_scan_flag(const unsigned long long* scan, int nscan, unsigned* flag, cudaStream_t s) {
  note_launch(3, s, true);
  scan_flag_kernel<<<1, 32, 0, s>>>(scan, nscan, flag);
  note_launch(3, s, false);
  return cudaGetLastError();
}

int cost_scan_blocks(int n) {
  const int64_t blocks = ((1ll << n) + 16383) / 16384;
  return (int)std::min<int64_t>({blocks, (int64_t)num_sms(), (int64_t)kMaxScan});
}

cudaError_t launch_cost_scan(const void* C, int f64, int n, int bound, unsigned long long* scan, const TableArgs& t,
                             cudaStream_t s) {
  const int64_t count = 1ll << n;
  const int vec = ((uintptr_t)C & 15) == 0 && n >= 2;
  note_launch(3, s, true);
  if (f64) cost_scan_kernel<<<cost_scan_blocks(n), 1024, 0, s>>>((const unsigned long long*)C, count, vec, bound, scan, t);
  else cost_scan_kernel<<<cost_scan_blocks(n), 1024, 0, s>>>((const unsigned*)C, count, vec, bound, scan, t);
  note_launch(3, s, false, (double)count * (f64 ? 8.0 : 4.0));
  return cudaGetLastError();
}

cudaError_t launch_adam(double* ang, const double* g, double* state, long long* step, int p, double lr, double b1,
                        double b2, double eps, double* history, long long row0, long long max_rows, cudaStream_t s) {
  note_launch(3, s, true);
  adam_kernel<<<1, 128, 0, s>>>(ang, g, state, step, p, lr, b1, b2, eps, history, row0, max_rows);
  note_launch(3, s, false);
  return cudaGetLastError();
}

cudaError_t launch_norm(const void* psi, int dtype, int n, double* partials, int* nblocks, cudaStream_t s) {
  const int64_t count = 1ll << n;
  int64_t blocks = (count + 255) / 256;
  if (blocks > 1024) blocks = 1024;
  *nblocks = (int)blocks;
  note_launch(3, s, true);
  norm_kernel<<<(int)blocks, 256, 0, s>>>(psi, dtype, count, partials);
  note_launch(3, s, false, (double)count * (dtype == QAOA_C128 ? 16.0 : 8.0));
  return cudaGetLastError();
}

}  // namespace qaoa
