// Lean sweeps of one complex64 state.
#include "lean_kernel.cuh"

namespace qaoa {

void lean_f1(const SweepArgs& a, size_t sm, cudaStream_t s) {
  if (a.kind == SWEEP_LEAN_OPS && a.needs_cost && a.cost_dtype == QAOA_COST_F64) lean_f1d(a, sm, s);
  else if (a.kind == SWEEP_LEAN_OPS) lean_launch_c<CfgF1, false, false, true>(a, sm, s);
  else lean_launch_c<CfgF1, false, false, false>(a, sm, s);
}

}  // namespace qaoa
