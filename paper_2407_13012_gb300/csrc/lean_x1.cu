// Lean sweeps of one complex128 (fixed-point) state.
#include "lean_kernel.cuh"

namespace qaoa {

void lean_x1(const SweepArgs& a, size_t sm, cudaStream_t s) {
  if (a.kind == SWEEP_LEAN_OPS) lean_launch_last<CfgX1, true, false, true>(a, sm, s);
  else lean_launch_last<CfgX1, true, false, false>(a, sm, s);
}

}  // namespace qaoa
