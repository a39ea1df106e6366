// Instantiation of the general H|psi> kernel (any sphere) without the projector terms: FP64.
#include "fused_kernel.cuh"

namespace pwk {
int launch_fused_f64(int N, const FusedArgs& a, int nblocks, const LaunchShape& s, cudaStream_t st) {
  return launch_fused<double, double, false, false>(N, a, nblocks, s, st);
}
}  // namespace pwk
