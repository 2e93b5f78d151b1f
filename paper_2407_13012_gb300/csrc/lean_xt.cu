// Lean sweeps of small complex128 (fixed-point) states on 512-amplitude tiles.
#include "lean_kernel.cuh"

namespace qaoa {

void lean_xt1(const SweepArgs& a, size_t sm, cudaStream_t s) {
  if (a.kind == SWEEP_LEAN_OPS) lean_launch_last<CfgXT, true, false, true>(a, sm, s);
  else lean_launch_last<CfgXT, true, false, false>(a, sm, s);
}

void lean_xt2(const SweepArgs& a, size_t sm, cudaStream_t s) {
  if (a.kind == SWEEP_LEAN_OPS) lean_launch_last<CfgXT, true, true, true>(a, sm, s);
  else lean_launch_last<CfgXT, true, true, false>(a, sm, s);
}

}  // namespace qaoa
