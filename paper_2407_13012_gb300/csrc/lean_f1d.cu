// Lean op programs of one complex64 state with float64 costs.
#include "lean_kernel.cuh"

namespace qaoa {

void lean_f1d(const SweepArgs& a, size_t sm, cudaStream_t s) {
  lean_launch_c<CfgF1D, false, false, true>(a, sm, s);
}

}  // namespace qaoa
