// Lean sweeps of complex128 (fixed-point) psi and lambda: one mixer.
#include "lean_kernel.cuh"

namespace qaoa {

void lean_x2_mix(const SweepArgs& a, size_t sm, cudaStream_t s) {
  lean_launch_last<CfgX2, true, true, false>(a, sm, s);
}

}  // namespace qaoa
