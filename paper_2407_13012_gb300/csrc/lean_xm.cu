// Lean sweeps of complex128 (fixed-point) states of middling size on 1024-amplitude tiles.
#include "lean_kernel.cuh"

namespace qaoa {

void lean_xm1(const SweepArgs& a, size_t sm, cudaStream_t s) {
  if (a.kind == SWEEP_LEAN_OPS) lean_launch_last<CfgXM, true, false, true>(a, sm, s);
  else lean_launch_last<CfgXM, true, false, false>(a, sm, s);
}

void lean_xm2(const SweepArgs& a, size_t sm, cudaStream_t s) {
  if (a.kind == SWEEP_LEAN_OPS) lean_launch_last<CfgXM, true, true, true>(a, sm, s);
  else lean_launch_last<CfgXM, true, true, false>(a, sm, s);
}

}  // namespace qaoa
