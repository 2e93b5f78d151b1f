// The lean sweep kernels, one per tile configuration and shape (complex64: also per number of
// carried bits; complex128: per last layout with group qubits, since code that is fixed for
// every number of carried bits measured slower there: n = 28 gradient 172.4 instead of 166.0 ms,
// n = 20 layers 261 instead of 241 us, with fewer instructions but more instruction-cache misses
// in the one-buffer kernels and less overlap in the two-buffer ones); the translation units lean_*.cu instantiate them (in parallel: they are most of the build).
#pragma once

#include "sweeper.cuh"

namespace qaoa {
namespace {

// One layer's phase table (the sweeper's graph's) in shared memory: float32 factors as they
// are, fixed-point factors prepared for the limb multiply (fx::Factor, 24 bytes per entry).
// Callers synchronise.
template <bool FX, class S>
__device__ __forceinline__ void stage_table(S& s, const SweepArgs& a, void* dst, int nt) {
  using V = typename S::V;
  const V* src = (const V*)s.ptab + (long long)a.smem_table_layer * s.pspan;
  if constexpr (FX) {
    fx::Factor* tf = (fx::Factor*)dst;
    for (int k = threadIdx.x; k < s.pspan; k += nt) {
      const longlong2 e = __ldg((const longlong2*)src + k);
      tf[k] = fx::factor(e.x, e.y);
    }
    s.Tf = tf;
  } else {
    V* ts = (V*)dst;
    for (int k = threadIdx.x; k < s.pspan; k += nt) ts[k] = __ldg(src + k);
    s.Ts = ts;
  }
  s.ts_layer = a.smem_table_layer;
}

// last layout with group bits [c, B)
template <class CF>
constexpr int lean_last(int c) {
  int last = 0;
  for (int k = 0; k < CF::NR; ++k)
    if (CF::newhi(k) > c) last = k;
  return last;
}

// bytes per amplitude of a lean sweep's cost tile (complex64 reads float64 costs from memory:
// their 64 KB tile left one block per SM; with the integer turn fractions of the computed phases,
// n = 29, p = 5 layers went from 57.7 to 36.7 ms)
template <bool FX>
__host__ __device__ constexpr int lean_cost_bytes(int cost_dtype) {
  return cost_dtype == QAOA_COST_F64 ? (FX ? 8 : 0) : 4;
}

// static shared memory of a lean kernel: per-warp accumulators and staged diagonals
template <class CF, bool FX>
constexpr size_t lean_static_smem() {
  const size_t slots = (size_t)kLeanAcc * (CF::NT / 32);
  return sizeof(double) * slots + (FX ? (sizeof(__int128) * slots + sizeof(fx::Factor) * kLeanMix * 16) : sizeof(float2) * slots) +
         sizeof(int) * kLeanAcc + sizeof(F32Mix) * kLeanMix + 256;
}

// dynamic shared memory a lean kernel may take on this device: the opt-in limit less its
// static shared memory (two-buffer kernels, which may add the psi staging area), else the
// largest exchange + cost + table layout
template <class CF, bool FX, bool TWO>
size_t lean_smem_cap() {
  static size_t cached[64] = {};
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(mu);
  size_t& c = cached[dev & 63];
  if (c == 0) {
    c = smem_bytes<CF, FX, TWO>(8, kSmemTable);
    if (TWO) {
      int optin = 0;
      const size_t fixed = lean_static_smem<CF, FX>() + 1024;
      if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
          (size_t)optin > fixed)
        c = std::max(c, (size_t)optin - fixed);
    }
  }
  return c;
}

// Lean sweeps: full tiles, affine layout-0 addresses, state loaded in the internal format
// or created as |+>, stored in the internal or the caller's format (complex64: the same).
template <class CF, bool FX, bool TWO, bool OPS, int C, int LAST>
__global__ void __launch_bounds__(CF::NT, CF::MINB) lean_kernel(const __grid_constant__ SweepArgs a) {
  using S = Lean<CF, FX, TWO, C>;
  using V = typename S::V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* X = (V*)smem_raw;  // exchange area: 2^B slots, twice that for two-buffer sweeps
  void* Cs = smem_raw + ((sizeof(V) << CF::B) << (TWO ? 1 : 0));
  const bool cost = OPS && a.needs_cost;
  V* Tsm = (V*)((unsigned char*)Cs + (cost ? lean_cost_bytes<FX>(a.cost_dtype) << CF::B : 0));
  constexpr int NW = CF::NT / 32;
  __shared__ double wacc[kLeanAcc * NW];
  __shared__ fx::Factor dpre[FX ? kLeanMix * 16 : 1];
  __shared__ __int128 iacc[FX ? kLeanAcc * NW : 1];
  __shared__ int ishift[kLeanAcc];
  __shared__ float2 facc[FX ? 1 : kLeanAcc * NW];
  __shared__ F32Mix fpre[kLeanMix];
  for (int r = threadIdx.x; r < kLeanAcc * NW; r += CF::NT) {
    wacc[r] = 0.0;
    if constexpr (FX) iacc[r] = 0;
    else facc[r] = make_float2(0.f, 0.f);
    if (r < kLeanAcc) ishift[r] = 0;
  }
  const CostScan scan = a.half == 2 ? read_scan(a.scan, a.nscan) : CostScan{a.half != 0, true, 0};
  const SweepGeom g = scan.symmetric ? half_geom(a.g) : a.g;
  S s(a, X, Cs, nullptr, nullptr);
  s.wacc = wacc;
  if constexpr (FX) {
    s.iacc = iacc;
    s.ishift = ishift;
  } else {
    s.facc = facc;
  }
  // grouped sweeps: this block's graph and its share of the graph's tiles
  int64_t t0 = blockIdx.x, tstep = gridDim.x;
  if (a.gslot != nullptr) {
    const GroupSlot& gsl = a.gslot[blockIdx.x / a.gbpg];
    s.zoff = gsl.zoff;
    s.ptab = gsl.phase_table;
    s.pcmin = gsl.cmin;
    s.pspan = gsl.span;
    s.trig = gsl.trig;
    s.dtab = gsl.d_table;
    t0 = blockIdx.x % a.gbpg;
    tstep = a.gbpg;
  }
  if constexpr (FX) {  // every mixer's diagonal exp(-i beta (t - 2k)), k = 0..t, as prepared factors
    const int t = s.gt();
    int m = 0;
    for (int k = 0; k < (OPS ? a.nops : 1) && m < kLeanMix; ++k) {
      const uint32_t op = a.ops[k];
      if ((op & 0xff) != OP_MIX) continue;
      if (threadIdx.x <= (uint32_t)t) {
        const longlong2 e = __ldg((const longlong2*)s.dtab + ((long long)((op >> 16) & 0xff) * 14 + t) * 14 + threadIdx.x);
        dpre[16 * m + threadIdx.x] = fx::factor(e.x, (op & F_SIGN) ? -e.y : e.y);
      }
      ++m;
    }
    s.dpre = dpre;
  }
  if constexpr (!FX) {
    int m = 0;
    for (int k = 0; k < (OPS ? a.nops : 1) && m < kLeanMix; ++k) {
      const uint32_t op = a.ops[k];
      if ((op & 0xff) != OP_MIX) continue;
      if (threadIdx.x == (uint32_t)m) fpre[m] = f32_mix(a, s.trig, (op >> 16) & 0xff, op & F_SIGN, s.gt());
      ++m;
    }
    s.fpre = fpre;
  }
  if (OPS && a.smem_table_layer >= 0) {
    stage_table<FX>(s, a, Tsm, CF::NT);
  }
  if (FX && OPS && a.smem_turns) {  // the turn tables of computed phases (no phase table then)
    longlong2* tt = (longlong2*)Tsm;
    for (int j = threadIdx.x; j < kTurnEntries; j += CF::NT) tt[j] = __ldg((const longlong2*)a.turn_table + j);
    s.turns = tt;
  }
  if (TWO && a.stage) {  // staging area after the phase table, 16-byte aligned
    const size_t tb = FX ? sizeof(fx::Factor) : sizeof(V);
    const size_t off = (size_t)((unsigned char*)Tsm - smem_raw) + (OPS && a.smem_table_layer >= 0 ? tb * a.span : 0) +
                       (OPS && a.smem_turns ? sizeof(longlong2) * kTurnEntries : 0);
    s.Ps = (V*)(smem_raw + ((off + 15) & ~(size_t)15));
  }
  s.evalid = 1u << CF::B;
  if constexpr (FX && !TWO) s.in_shift = input_shift(a.norm2_dev);
  if constexpr (FX && TWO) {
    if (a.gslot != nullptr) {
      s.lam_shift = a.gslot[blockIdx.x / a.gbpg].lam_shift;
      s.c_expo = a.gslot[blockIdx.x / a.gbpg].c_expo;
    } else if (a.scan != nullptr) {
      s.set_scan(a.half == 2 ? scan : read_scan(a.scan, a.nscan));
    }
  }
  __syncthreads();
  bool have = false;  // this tile's psi is in the staging area
  for (int64_t tile = t0; tile < g.tiles; tile += tstep) {
    const int64_t next = tile + tstep < g.tiles ? tile + tstep : -1;
    lean_tile<CF, FX, TWO, OPS, LAST, false, C>(s, a, g, tile, Cs, next, have);
    have = s.Ps != nullptr && next >= 0;
  }
  __syncthreads();
  for (int r = threadIdx.x; r < a.nred; r += CF::NT) {
    double v = 0.0;
    for (int w = 0; w < NW; ++w) v += wacc[r * NW + w];
    if constexpr (FX) {
      __int128 t = 0;
      for (int w = 0; w < NW; ++w) t += iacc[r * NW + w];
      v += i128_to_double(t, ishift[r]);
    } else {
      for (int w = 0; w < NW; ++w) v += (double)facc[r * NW + w].x + (double)facc[r * NW + w].y;
    }
    a.partials[(int64_t)a.red_slot[r] * a.grid + blockIdx.x] = v;
  }
}

template <class CF, bool FX, bool TWO, bool OPS, int C, int LAST>
void lean_launch_one(const SweepArgs& a, size_t sm, cudaStream_t s) {
  static std::mutex mu;
  static uint64_t done = 0;
  once_per_device(mu, done, [] {
    cudaFuncSetAttribute(lean_kernel<CF, FX, TWO, OPS, C, LAST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)lean_smem_cap<CF, FX, TWO>());
  });
  lean_kernel<CF, FX, TWO, OPS, C, LAST><<<a.grid, CF::NT, sm, s>>>(a);
}
// the kernel of a.g.c carried bits (0 <= c <= B - RB)
template <class CF, bool FX, bool TWO, bool OPS, int C = 0>
void lean_launch_c(const SweepArgs& a, size_t sm, cudaStream_t s) {
  if constexpr (C < CF::B - CF::RB) {
    if (a.g.c != C) {
      lean_launch_c<CF, FX, TWO, OPS, C + 1>(a, sm, s);
      return;
    }
  }
  lean_launch_one<CF, FX, TWO, OPS, C, lean_last<CF>(C)>(a, sm, s);
}
// the kernel of the sweep's last layout with group qubits, any number of carried bits
template <class CF, bool FX, bool TWO, bool OPS, int LAST = 0>
void lean_launch_last(const SweepArgs& a, size_t sm, cudaStream_t s) {
  if constexpr (LAST + 1 < CF::NR) {
    if (lean_last<CF>(a.g.c) != LAST) {
      lean_launch_last<CF, FX, TWO, OPS, LAST + 1>(a, sm, s);
      return;
    }
  }
  lean_launch_one<CF, FX, TWO, OPS, -1, LAST>(a, sm, s);
}

}  // namespace
}  // namespace qaoa
