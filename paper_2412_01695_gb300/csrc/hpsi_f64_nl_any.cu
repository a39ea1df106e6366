// Instantiation of the general H|psi> kernel (any sphere) with the projector terms inside
// (nl_fused.cuh): FP64.
#include "fused_kernel.cuh"

namespace pwk {
int launch_fused_f64_nl(int N, const FusedArgs& a, int nblocks, const LaunchShape& s, cudaStream_t st) {
  return launch_fused<double, double, false, true>(N, a, nblocks, s, st);
}
}  // namespace pwk
