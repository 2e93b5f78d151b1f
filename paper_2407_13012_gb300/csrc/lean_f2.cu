// Lean sweeps of complex64 psi and lambda.
#include "lean_kernel.cuh"

namespace qaoa {

void lean_f2(const SweepArgs& a, size_t sm, cudaStream_t s) {
  if (a.kind == SWEEP_LEAN_OPS) lean_launch_c<CfgF3, false, true, true>(a, sm, s);
  else lean_launch_c<CfgF3, false, true, false>(a, sm, s);
}

}  // namespace qaoa
