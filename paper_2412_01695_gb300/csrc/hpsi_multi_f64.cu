// The FP64 instantiation of the window kernel over work lists that span several plans.
#include "fused_window.cuh"

namespace pwk {
int launch_window_multi_f64(int N, const FusedArgs& a, int nblocks, const LaunchShape& s, cudaStream_t st) {
  return launch_window_multi<double, double>(N, a, nblocks, s, st);
}
}  // namespace pwk
