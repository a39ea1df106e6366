// Instantiation of the window H|psi> kernel with the projector terms inside (nl_fused.cuh): FP64.
#include "fused_window.cuh"

namespace pwk {
int launch_window_f64_nl(int N, const FusedArgs& a, int nblocks, const LaunchShape& s, cudaStream_t st) {
  return launch_window<double, double, true>(N, a, nblocks, s, st);
}
}  // namespace pwk
