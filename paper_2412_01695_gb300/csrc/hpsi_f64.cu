// Instantiation of the window H|psi> kernel without the projector terms: FP64.
#include "fused_window.cuh"

namespace pwk {
int launch_window_f64(int N, const FusedArgs& a, int nblocks, const LaunchShape& s, cudaStream_t st) {
  return launch_window<double, double, false>(N, a, nblocks, s, st);
}
}  // namespace pwk
