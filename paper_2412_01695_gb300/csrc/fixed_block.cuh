// Block-level parts of the fixed-point transforms (fixed.cuh): the scale of a vector, the
// shifts of a line, and the way back to double.
#pragma once
#include <type_traits>

#include "fft_line.cuh"
#include "fixed.cuh"

namespace pwk {

// arithmetic of the transforms of an H application in T
template <typename T>
using fft_arith_t = typename std::conditional<std::is_same<T, double>::value, long long, T>::type;

// right shift that brings a line whose high words have magnitude m below the cap of length N
template <int N>
__device__ __forceinline__ int fx_shift(unsigned m) {
  return max(0, 64 - __clz((int)m) - fx_cap(N));
}

// sc 2^e as the factor of an integer result; e far outside the normal range goes to fx_scaled
__device__ __forceinline__ bool fx_plain_scale(int e) { return e > -900 && e < 900; }
__device__ __forceinline__ double fx_factor(double sc, int e) {
  return fx_plain_scale(e) ? sc * __hiloint2double((1023 + e) << 20, 0) : sc;
}
__device__ __forceinline__ double fx_scaled(long long z, double f, int e) {
  const double d = __ll2double_rn(z) * f;
  return fx_plain_scale(e) ? d : ldexp(d, e);
}

// Block-wide scale of one vector, independent of the order and number of threads: the exponent
// S with sum_G |C(G)| 2^S <= 2^kFxBits.  pre: power of two the input is first multiplied by
// (exact; only vectors with no component above 2^-895 need it).  bad: a component is not
// finite.  Every thread of the block calls it; sh is shared scratch zeroed by the call.
struct FxScale {
  double pre, in;   // the integers hold (C pre) in
  int exp;          // = C 2^exp
  bool bad;
  int top;          // every |component of C| < 2^top (bad: kFxBadField)
};
__device__ __forceinline__ longlong2 fx_from(const FxScale& s, double2 v) {
  if (s.pre != 1.0) v = make_double2(v.x * s.pre, v.y * s.pre);   // uniform over the block
  return longlong2{__double2ll_rn(v.x * s.in), __double2ll_rn(v.y * s.in)};
}
struct FxScratch {
  unsigned hmax;
  unsigned lo, hi;
};
// the scratch in the 16 spare bytes at the end of a kernel's shared memory
__device__ __forceinline__ FxScratch* fx_scratch_at(unsigned char* end) {
  return reinterpret_cast<FxScratch*>((reinterpret_cast<size_t>(end) + 3) & ~(size_t)3);
}
__device__ __forceinline__ unsigned fx_abs_hi(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

__device__ __forceinline__ FxScale fx_block_scale(const double2* __restrict__ c, int n, FxScratch* sh) {
  const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31;
  double pre = 1.0;
  int pexp = 0;
  unsigned hm = 0;
  for (int pass = 0; pass < 2; ++pass) {
    if (tid == 0) sh->hmax = sh->lo = sh->hi = 0u;
    __syncthreads();
    hm = 0;
    for (int g = tid; g < n; g += nth) {
      double2 v = c[g];
      if (pass) v = make_double2(v.x * pre, v.y * pre);
      hm = max(hm, max(fx_abs_hi(v.x), fx_abs_hi(v.y)));
    }
    hm = __reduce_max_sync(0xffffffffu, hm);
    if (lane == 0) atomicMax(&sh->hmax, hm);
    __syncthreads();
    hm = sh->hmax;
    if ((hm >> 20) >= 128 || pass == 1) break;   // uniform
    pre = __hiloint2double((1023 + 600) << 20, 0);
    pexp = 600;
    __syncthreads();   // hmax is read before it is reset
  }
  const int em = (int)(hm >> 20);
  if (em == 0x7ff) return FxScale{1.0, 0.0, 0, true, kFxBadField};
  if (em < 128) return FxScale{1.0, 0.0, 0, false, 0};   // a zero vector (pre has lifted every other one)
  // sum of the component magnitudes in units of 2^(em - 1043), each rounded up
  unsigned s0 = 0, s1 = 0;
  for (int g = tid; g < n; g += nth) {
    double2 v = c[g];
    if (pexp) v = make_double2(v.x * pre, v.y * pre);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const unsigned h = fx_abs_hi(p ? v.y : v.x);
      const int d = min(em - (int)(h >> 20), 31);
      const unsigned q = ((((h & 0xfffffu) | 0x100000u) + 1u) >> d) + 1u;
      s0 += q & 0xffffu;
      s1 += q >> 16;
    }
  }
  s0 = __reduce_add_sync(0xffffffffu, s0);
  s1 = __reduce_add_sync(0xffffffffu, s1);
  if (lane == 0) {
    atomicAdd(&sh->lo, s0);
    atomicAdd(&sh->hi, s1);
  }
  __syncthreads();
  const unsigned long long q = ((unsigned long long)sh->hi << 16) + sh->lo;
  const int S = kFxBits - ((64 - __clzll((long long)q)) + em - 1043);
  return FxScale{pre, __hiloint2double((1023 + S) << 20, 0), S + pexp, false, em - 1022 - pexp};
}

// A line's values x (already loaded) shifted to one scale and below the cap of a forward
// transform of length N: element i carries the shift s[i * stride] of the pass before.  Returns
// the line's shift.
template <int N>
__device__ __forceinline__ int fx_align(longlong2 (&x)[N], const unsigned char* s, int stride) {
  int d[N];
  int top = 0;
  PWK_SFOR(N, i, {
    d[i] = s[i * stride];
    top = max(top, d[i]);
  });
  unsigned m = 0;
  PWK_SFOR(N, i, {
    const int hx = (int)(x[i].x >> 32) >> (top - d[i]), hy = (int)(x[i].y >> 32) >> (top - d[i]);
    m |= (unsigned)(hx ^ (hx >> 31)) | (unsigned)(hy ^ (hy >> 31));
  });
  top += fx_shift<N>(m);
  PWK_SFOR(N, i, {
    const int e = top - d[i];
    const long long half = (1LL << e) >> 1;
    x[i] = longlong2{(x[i].x + half) >> e, (x[i].y + half) >> e};
  });
  return top;
}

// y = u V of one x line: u the outputs of an inverse transform (in its output slots), V the
// limb pairs of the line; y brought below the cap of the forward transform.
// Returns the line's shift.
template <int N>
__device__ __forceinline__ int fx_v_product(const longlong2 (&u)[N], const int2* __restrict__ v, longlong2 (&y)[N]) {
  unsigned m = 0;
  auto put = [&](auto lc, int vh, int vl) {
    constexpr int l1 = decltype(lc)::value;
    const longlong2 t = u[OutSlot<N, l1>::value];
    y[l1] = longlong2{fx_mul(t.x, vh, vl), fx_mul(t.y, vh, vl)};
    m = fx_magnitude(fx_magnitude(m, y[l1].x), y[l1].y);
  };
  if constexpr (N % 2 == 0) {   // a line is N 8-byte pairs: 16-byte loads where N is even
    const int4* q = reinterpret_cast<const int4*>(v);
    static_for<N / 2>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      const int4 w = __ldg(q + j);
      put(std::integral_constant<int, 2 * j>{}, w.x, w.y);
      put(std::integral_constant<int, 2 * j + 1>{}, w.z, w.w);
    });
  } else {
    static_for<N>([&](auto jc) {
      const int2 w = __ldg(v + decltype(jc)::value);
      put(jc, w.x, w.y);
    });
  }
  const int sh = fx_shift<N>(m);
  const long long half = (1LL << sh) >> 1;
  PWK_SFOR(N, l1, y[l1] = longlong2{(y[l1].x + half) >> sh, (y[l1].y + half) >> sh});
  return sh;
}

// The same with a complex field: v holds (re, im) limb pairs, |re|, |im| <= 1/2.
template <int N>
__device__ __forceinline__ int fx_dv_product(const longlong2 (&u)[N], const int4* __restrict__ v, longlong2 (&y)[N]) {
  unsigned m = 0;
  PWK_SFOR(N, l1, {
    const longlong2 t = u[OutSlot<N, l1>::value];
    const int4 w = __ldg(v + l1);
    y[l1] = longlong2{fx_mul2(t.x, w.x, w.y, -t.y, w.z, w.w), fx_mul2(t.x, w.z, w.w, t.y, w.x, w.y)};
    m = fx_magnitude(fx_magnitude(m, y[l1].x), y[l1].y);
  });
  const int sh = fx_shift<N>(m);
  const long long half = (1LL << sh) >> 1;
  PWK_SFOR(N, l1, y[l1] = longlong2{(y[l1].x + half) >> sh, (y[l1].y + half) >> sh});
  return sh;
}

}  // namespace pwk
