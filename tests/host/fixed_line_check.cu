// Host check of the fixed-point line transforms (csrc/fixed.cuh through csrc/fft_line.cuh):
// LineFFT<long long, N, DIR> against the direct DFT sum in long double, for inputs at the top of
// the range (sum of moduli just below 2^61) and for inputs with zeros outside |m| <= N/4.
// Prints per size:  N <n> <max error, inverse> <forward> <windowed inverse> <largest |output| / 2^61>
// with errors in units of the last place.
#include <cmath>
#include <cstdio>

#include "../../paper_2412_01695_gb300/csrc/fft_line.cuh"

using namespace pwk;

static unsigned long long state = 88172645463325252ull;
static double uniform() {   // (-1, 1)
  state ^= state << 13;
  state ^= state >> 7;
  state ^= state << 17;
  return (double)(long long)state / 9223372036854775808.0;
}

template <int N, int DIR>
static double check(bool window, bool peak, double& top) {
  const long double two_pi = 6.283185307179586476925286766559005768L;
  double worst = 0;
  for (int rep = 0; rep < 20; ++rep) {
    longlong2 x[N], in[N];
    double sum = 0, re[N], im[N];
    for (int i = 0; i < N; ++i) {
      const bool zero = (window && i > N / 4 && i < N - N / 4) || (peak && i != rep % N);
      re[i] = zero ? 0 : uniform();
      im[i] = zero ? 0 : uniform();
      sum += std::hypot(re[i], im[i]);
    }
    const double s = std::ldexp(0.999999, kFxBits) / sum;
    for (int i = 0; i < N; ++i) x[i] = in[i] = longlong2{(long long)(re[i] * s), (long long)(im[i] * s)};
    LineFFT<long long, N, DIR>::run(x);
    for (int k = 0; k < N; ++k) {
      long double a = 0, b = 0;
      for (int n = 0; n < N; ++n) {
        const long double w = DIR * two_pi * (long double)((n * k) % N) / N, c = cosl(w), d = sinl(w);
        a += in[n].x * c - in[n].y * d;
        b += in[n].x * d + in[n].y * c;
      }
      const longlong2 o = x[fft_out_slot(N, k)];
      worst = std::fmax(worst, std::fmax((double)fabsl(o.x - a), (double)fabsl(o.y - b)));
      top = std::fmax(top, std::hypot((double)o.x, (double)o.y) / std::ldexp(1.0, kFxBits));
    }
  }
  return worst;
}

template <int N>
static void line() {
  double top = 0;
  const double inv = std::fmax(check<N, 1>(false, false, top), check<N, 1>(false, true, top));
  const double fwd = std::fmax(check<N, -1>(false, false, top), check<N, -1>(false, true, top));
  std::printf("N %d %.3e %.3e %.3e %.6f\n", N, inv, fwd, check<N, 1>(true, false, top), top);
}

int main() {
  line<12>(); line<15>(); line<16>(); line<18>(); line<20>(); line<24>(); line<25>();
  line<27>(); line<30>(); line<32>(); line<36>(); line<40>(); line<45>(); line<48>();
  return 0;
}
