// Largest error, in units of the last place, of fast_rcp and fast_rsqrt (csrc/recip.cuh) and of
// the division and 1.0 / sqrt(x), over the ranges the header states: prints the four.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../../paper_2412_01695_gb300/csrc/recip.cuh"

__global__ void eval_kernel(int n, const double* x, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i], a = fabs(v);
  const bool root = a >= 1e-280 && a <= 1e280;
  out[i] = pwk::fast_rcp(v);
  out[n + i] = 1.0 / v;
  out[2 * n + i] = root ? pwk::fast_rsqrt(a) : 0.0;
  out[3 * n + i] = root ? 1.0 / sqrt(a) : 0.0;
}

int main() {
  std::vector<double> x;
  unsigned long long s = 88172645463325252ull;
  for (int e = -963; e <= 963; ++e)
    for (int j = 0; j < 256; ++j) {
      s ^= s << 13, s ^= s >> 7, s ^= s << 17;   // xorshift64 (Marsaglia)
      unsigned long long m = s >> 12;
      if (j < 4) m = j < 2 ? j : (1ull << 52) - 3 + j;   // the ends of the binade
      const double v = std::ldexp(1.0 + (double)m / 4503599627370496.0, e);
      if (v < 1e-290 || v > 1e290) continue;
      x.push_back(j & 1 ? -v : v);
    }
  const int n = (int)x.size();
  double *dx = nullptr, *dy = nullptr;
  if (cudaMalloc(&dx, n * sizeof(double)) != cudaSuccess || cudaMalloc(&dy, 4 * (size_t)n * sizeof(double)) != cudaSuccess) return 1;
  cudaMemcpy(dx, x.data(), n * sizeof(double), cudaMemcpyHostToDevice);
  eval_kernel<<<(n + 255) / 256, 256>>>(n, dx, dy);
  std::vector<double> y(4 * (size_t)n);
  if (cudaMemcpy(y.data(), dy, y.size() * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  double worst[4] = {0, 0, 0, 0};
  for (int f = 0; f < 4; ++f)
    for (int i = 0; i < n; ++i) {
      const double a = std::fabs(x[i]);
      if (f >= 2 && !(a >= 1e-280 && a <= 1e280)) continue;
      const long double ref = f < 2 ? 1.0L / (long double)x[i] : 1.0L / std::sqrt((long double)a);
      const double r = std::fabs((double)ref), ulp = std::nextafter(r, INFINITY) - r;
      const double err = (double)(std::fabs((long double)y[(size_t)f * n + i] - ref) / (long double)ulp);
      if (!(err <= worst[f])) worst[f] = err;
    }
  std::printf("%.6f %.6f %.6f %.6f\n", worst[0], worst[1], worst[2], worst[3]);
  cudaFree(dx);
  cudaFree(dy);
  return 0;
}
