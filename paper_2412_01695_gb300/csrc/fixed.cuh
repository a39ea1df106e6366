// 64-bit block fixed point: the arithmetic of the FP64 transforms.
//
// GB300 issues an FP64 instruction on 2 lanes per SM and clock, a 32 x 32 + 64 bit integer
// multiply-add (IMAD.WIDE) on about 30 and a 64-bit integer add on about 43 (measured with
// independent chains on every SM).  A line transform is adds and products with constants of
// modulus <= 1, so it runs on 64-bit integers with one common power-of-two scale per vector:
// values keep |x| <= 2^61 and about 56 significant bits below the vector's largest grid
// value, against 53 of FP64, at a tenth of the issue time.  Measured on 1280 band-k of the
// N = 24 cell with 9 projectors: H|psi> 1.94 ms with FP64 transforms, 0.48 ms with these (0.26 of
// 1.15 ms for H and S on 237 items at N = 27); against long-double sums the relative error
// went from 2.1e-16 to 1.8e-16 (both mostly that of the kinetic table).
//
//   * A constant c (|c| < 1, fx_cos2pi) is Q = c 2^63 = ch 2^32 + cl with ch, cl signed 32-bit.
//   * A value x is hp 2^32 + ls with hp, ls signed 32-bit (limbs()).
//   * x c = 2 hp ch + ((hp cl + ls ch + 2^30) >> 31): three IMAD.WIDE; the dropped ls cl and
//     the rounding are at most one unit in the last place together, without bias.
//   * With |x| + |y| <= 2^61 sqrt(2) (the components of one value, or two terms of one sum) the
//     low part of a two-term product (fx_mul2) stays below 2^62 (|c| + |s|) + 2^60.5 < 2^63.
// The scale of the inverse transforms follows from sum_G |C(G)| <= 2^61 (every partial result
// is a combination of the inputs with coefficients of modulus <= 1); a forward line is shifted
// right, rounded to nearest, by what its largest value needs for the N-term sum, and the shift
// is recorded per line (fx_cap, fx_shift; the kernels align the lines of the next pass).
#pragma once
#include <cuda_runtime.h>

#define PWK_FX_HD __host__ __device__ __forceinline__

namespace pwk {

constexpr int kFxBits = 61;   // |x| <= 2^kFxBits through the transforms
// exponent of a field with a value that is not finite (every result becomes NaN, as the product
// and the transform would make it)
constexpr int kFxBadField = 0x7fffffff;

// cos(2 pi e / n) 2^63 to a few units in the last place, |cos| < 1: the angle reduced to an
// octant as an exact fraction, then the Taylor series with 128-bit products.
__host__ __device__ constexpr long long fx_cos2pi(long e, long n) {
  e %= n;
  if (e < 0) e += n;
  if (2 * e > n) e = n - e;
  long long sgn = 1;
  if (4 * e > n) {
    sgn = -1;
    e = n - 2 * e;
    n = 2 * n;
  }
  const bool odd = 8 * e > n;   // sin of the complement
  if (odd) {
    e = n - 4 * e;
    n = 4 * n;
  }
  const __int128 x = (__int128)14488038916154245685ull * 2 * e / n;   // pi 2^62 times 2 e / n
  const __int128 x2 = (x * x) >> 62;
  __int128 term = odd ? x : (__int128)1 << 62, sum = term;
  for (int k = 1; k < 14; ++k) {
    term = -((term * x2) >> 62) / (odd ? 2 * k * (2 * k + 1) : (2 * k - 1) * (2 * k));
    sum += term;
  }
  return sgn * (long long)(2 * sum);
}
__host__ __device__ constexpr long long fx_sin2pi(long e, long n) { return fx_cos2pi(4 * e - n, 4 * n); }
__host__ __device__ constexpr int fx_ch(long long q) { return (int)((q + 0x80000000LL) >> 32); }
__host__ __device__ constexpr int fx_cl(long long q) {
  return (int)(q - (((q + 0x80000000LL) >> 32) * 4294967296LL));
}

struct FxLimbs {
  int hp, ls;   // x = hp 2^32 + ls
};
PWK_FX_HD FxLimbs fx_limbs(long long x) {
  const int ls = (int)(unsigned)(unsigned long long)x;
  return FxLimbs{(int)(x >> 32) + (int)((unsigned)ls >> 31), ls};
}
PWK_FX_HD long long fx_wide(int a, int b) { return (long long)a * (long long)b; }

// x q / 2^63 for a limb pair (qh, ql) with |q| < 2^63
PWK_FX_HD long long fx_mul(long long x, int qh, int ql) {
  const FxLimbs a = fx_limbs(x);
  const long long t = fx_wide(a.hp, ql) + fx_wide(a.ls, qh) + 0x40000000LL;
  return fx_wide(2 * a.hp, qh) + (t >> 31);
}
// (x p + y q) / 2^63
PWK_FX_HD long long fx_mul2(long long x, int ph, int pl, long long y, int qh, int ql) {
  const FxLimbs a = fx_limbs(x), b = fx_limbs(y);
  const long long t = fx_wide(a.hp, pl) + fx_wide(a.ls, ph) + fx_wide(b.hp, ql) + fx_wide(b.ls, qh) + 0x40000000LL;
  return fx_wide(2 * a.hp, ph) + fx_wide(2 * b.hp, qh) + (t >> 31);
}
// the same with compile-time constants
template <long long Q>
PWK_FX_HD long long fx_mulc(long long x) {
  return fx_mul(x, fx_ch(Q), fx_cl(Q));
}
template <long long P, long long Q>
PWK_FX_HD long long fx_mulc2(long long x, long long y) {
  return fx_mul2(x, fx_ch(P), fx_cl(P), y, fx_ch(Q), fx_cl(Q));
}

// A coefficient v (|v| < 2^63 - 2^31) as the limb pair fx_mul takes; fx_mul2 takes two with
// |p| + |q| <= sqrt(2) 2^63
PWK_FX_HD int2 fx_pair(long long v) {
  const FxLimbs l = fx_limbs(v);
  return int2{l.hp, l.ls};
}

// Largest bit length a value may have before a forward transform of length n: the sums of n
// terms of modulus sqrt(2) |component| stay below 2^kFxBits.
__host__ __device__ constexpr int fx_cap(int n) {
  int b = 0;
  while ((1LL << (2 * b)) < 2LL * n * n) ++b;   // 2^b >= n sqrt(2)
  return kFxBits - b;
}

// OR of (h ^ sign) over the high words of a line: its bit length bounds every |component|
PWK_FX_HD unsigned fx_magnitude(unsigned acc, long long v) {
  const int h = (int)(v >> 32);
  return acc | (unsigned)(h ^ (h >> 31));
}

}  // namespace pwk
