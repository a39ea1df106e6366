// Nonlocal projector terms inside the fused H|psi> kernels (paper Sec. 2.2, "Non local
// pseudopotential and overlap matrix"), so that one band-k work item reads C(G) and writes
// H C(G) (and S C(G)) once from and to HBM:
//
//   prologue  lambda_m = sum_G conj(beta_m(k+G)) C(G)           (Eq. lambdah)
//             gamma_m  = sum_n D_mn lambda_n                    (Eq. gamma)
//             delta_m  = sum_n q_mn lambda_n                    (Eq. delta_eq, with q)
//   epilogue  H C(G)  += sum_m gamma_m beta_m(k+G)              (Eq. finalnl)
//             S C(G)   = C(G) + sum_m delta_m beta_m(k+G)       (Eq. finals, with q)
//
// beta(k) is read through L1/L2 (the bands of a k-point run in neighbouring CTAs, so it
// crosses HBM about once per k-point).  The projections are computed by warps, one group of
// G projectors per warp at a time: lane l sums G = l, l + 32, ... in ascending order and the
// lanes are combined by a fixed xor tree, so lambda does not depend on the number of warps
// (every launch shape gives the same bits); gamma, delta and the add-back sum the projectors
// in ascending order.  The coefficients live in shared memory at byte offset a.nl_off:
// [0, nkb) lambda, [nkb, 2 nkb) gamma, [2 nkb, 3 nkb) delta.
#pragma once
#include "fft_line.cuh"
#include "fixed_block.cuh"
#include "pwk_internal.h"

namespace pwk {

// Prologue, part 1: lambda of every projector into nls[0, nkb).  C(G) is read through
// `cin`, beta(k) through `bk` ([nkb][ldb]); either may be global or shared memory.
template <typename T, typename CV>
__device__ __forceinline__ void nl_fused_project(const FusedArgs& a, const c2_t<T>* bk, int ldb,
                                                 const CV* cin, int np, c2_t<T>* nls) {
  using V = c2_t<T>;
  constexpr int G = sizeof(T) == 4 ? 4 : 3;   // projectors per warp group (accumulators held in registers)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int ngroups = (a.nkb + G - 1) / G;
  for (int grp = warp; grp < ngroups; grp += nw) {
    const int m0 = grp * G;
    const int nc = min(G, a.nkb - m0);
    T ar[G], ai[G];
#pragma unroll
    for (int j = 0; j < G; ++j) ar[j] = ai[j] = T(0);
    const V* bg = bk + (size_t)m0 * ldb;
    for (int g = lane; g < np; g += 32) {
      const CV cv = cin[g];
      const T cr = T(cv.x), ci = T(cv.y);
#pragma unroll
      for (int j = 0; j < G; ++j) {
        if (j < nc) {
          const V b = bg[(size_t)j * ldb + g];
          ar[j] += b.x * cr + b.y * ci;   // conj(beta) C
          ai[j] += b.x * ci - b.y * cr;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < G; ++j) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        ar[j] += __shfl_xor_sync(0xffffffffu, ar[j], o);
        ai[j] += __shfl_xor_sync(0xffffffffu, ai[j], o);
      }
    }
    if (lane == 0) {
#pragma unroll
      for (int j = 0; j < G; ++j)
        if (j < nc) nls[m0 + j] = V{ar[j], ai[j]};
    }
  }
}

// Prologue, part 2 (after a barrier): gamma = D lambda into nls[nkb, 2 nkb) and, with q,
// delta = q lambda into nls[2 nkb, 3 nkb).
template <typename T>
__device__ __forceinline__ void nl_fused_coef(const FusedArgs& a, c2_t<T>* nls) {
  using V = c2_t<T>;
  const int nkb = a.nkb;
  const int rows = a.qm != nullptr ? 2 * nkb : nkb;
  for (int i = threadIdx.x; i < rows; i += blockDim.x) {
    const bool del = i >= nkb;
    const T* M = static_cast<const T*>(del ? a.qm : a.Dm) + (size_t)(del ? i - nkb : i) * nkb;
    T gr = T(0), gi = T(0);
    for (int j = 0; j < nkb; ++j) {
      const T d = M[j];
      const V l = nls[j];
      gr += d * l.x;
      gi += d * l.y;
    }
    nls[nkb + i] = V{gr, gi};
  }
}

// Epilogue for one plane wave g: the add-back sums h = sum gamma beta and, when with_q (the
// plan has q and S C is wanted), s = sum delta beta (else s = 0: S C = C).  beta(k) through
// `bk` ([nkb][ldb], global or shared memory).
template <typename T>
__device__ __forceinline__ void nl_fused_addback(const FusedArgs& a, const c2_t<T>* bk, int ldb, int g,
                                                 const c2_t<T>* nls, bool with_q, c2_t<T>& h, c2_t<T>& s) {
  using V = c2_t<T>;
  const int nkb = a.nkb;
  const V* bg = bk + g;
  T hr = T(0), hi = T(0), sr = T(0), si = T(0);
#pragma unroll 4
  for (int m = 0; m < nkb; ++m) {
    const V b = bg[(size_t)m * ldb];
    const V gm = nls[nkb + m];
    hr += gm.x * b.x - gm.y * b.y;
    hi += gm.x * b.y + gm.y * b.x;
    if (with_q) {
      const V dl = nls[2 * nkb + m];
      sr += dl.x * b.x - dl.y * b.y;
      si += dl.x * b.y + dl.y * b.x;
    }
  }
  h = V{hr, hi};
  s = V{sr, si};
}

// beta(k) ([nkb][npw_beta] contiguous) into shared memory at dst by asynchronous copies from
// every thread of the CTA (16-byte copies when the block is 16-byte aligned and sized, else one
// complex element per copy); returns once every copy has landed and the CTA has synchronised.
template <typename T>
__device__ __forceinline__ void nl_stage_beta(const FusedArgs& a, int k, c2_t<T>* dst) {
  using V = c2_t<T>;
  const V* src = static_cast<const V*>(a.beta) + (size_t)k * a.nkb * a.npw_beta;
  const size_t n = (size_t)a.nkb * a.npw_beta, bytes = n * sizeof(V);
  const unsigned d0 = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  if ((reinterpret_cast<size_t>(src) & 15) == 0 && (bytes & 15) == 0) {
    const char* s = reinterpret_cast<const char*>(src);
    for (size_t i = (size_t)threadIdx.x * 16; i < bytes; i += (size_t)blockDim.x * 16)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d0 + (unsigned)i), "l"(s + i) : "memory");
  } else {
    for (size_t i = threadIdx.x; i < n; i += blockDim.x) {
      if constexpr (sizeof(V) == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d0 + (unsigned)(i * 16)), "l"(src + i)
                     : "memory");
      else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d0 + (unsigned)(i * 8)), "l"(src + i)
                     : "memory");
    }
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
}

// ------------------------------------------------------------------ FP64 projector terms of H
// The same sums for FP64 vectors on the integer pipe, where S C is not asked for: beta_m(k), C and
// the coefficients as
// integers of 57 bits (scaled by the largest component of the projector, of the vector, of all
// coefficients), split X = h 2^29 + l, so that a complex multiply-add is 12 wide integer
// multiply-adds (the l l products, below 2^-56 of the largest product, are left out) instead
// of 4 FP64 instructions at a fifteenth of their rate.  Sums are exact up to that; they return
// to double once per lane and projector, and once per plane wave.  1280 band-k at N = 24 with 9
// projectors: 0.48 -> 0.44 ms for the whole application, error against long double unchanged
// (1.9e-16).  What the sums lose below 2^-57 of the largest component stays under the rounding of
// the local term, which spreads over all components alike; a plan whose V is weaker than its
// projectors (choose_projector_sums in plan.cu) takes the sums in doubles.  S C = C + sum delta beta
// has no such term and is exact to rounding in every component with sums in doubles, so a call
// that wants S with q takes those (nl_fused_project and so on) for H too.
// kNlFlush: terms an accumulator holds before it is taken over into double (|h| <= 2^28: a
// complex term adds at most 4 2^56 to the middle sum).
constexpr int kNlFlush = 31;

// v 2^(57 - R) rounded, as the pair (h, l); |v| < 2^R
__device__ __forceinline__ int2 nl_limbs(double v, int R) {
  const long long b = __double_as_longlong(v);
  const int e = (int)((unsigned long long)b >> 52) & 0x7ff;
  long long m = (b & 0xfffffffffffffLL) | (e != 0 ? 1LL << 52 : 0LL);
  const int d = min(R + 1022 - max(e, 1), 62);   // v = m 2^(e - 1075): X = 16 m / 2^d (d < 0: a
  m <<= 4;                                         // vector or projector of subnormal numbers)
  m = d < 0 ? m << -d : (m + ((1LL << d) >> 1)) >> d;
  if (b < 0) m = -m;
  const int h = (int)((m + (1LL << 28)) >> 29);
  return int2{h, (int)(m - ((long long)h << 29))};
}
__device__ __forceinline__ int4 nl_limbs(double2 v, int R) {
  const int2 x = nl_limbs(v.x, R), y = nl_limbs(v.y, R);
  return int4{x.x, x.y, y.x, y.y};
}

struct NlSum {   // sum of complex products in integers: h h and (h l + l h) parts
  long long hx = 0, mx = 0, hy = 0, my = 0;
  // += b c, or conj(b) c
  template <bool CONJ>
  __device__ __forceinline__ void add(int4 b, int4 c) {
    const int ih = CONJ ? b.z : -b.z, il = CONJ ? b.w : -b.w;   // the sign of b.y c.y
    hx += fx_wide(b.x, c.x) + fx_wide(ih, c.z);
    mx += fx_wide(b.x, c.y) + fx_wide(b.y, c.x) + fx_wide(ih, c.w) + fx_wide(il, c.z);
    hy += fx_wide(b.x, c.z) + fx_wide(-ih, c.x);
    my += fx_wide(b.x, c.w) + fx_wide(b.y, c.z) + fx_wide(-ih, c.y) + fx_wide(-il, c.x);
  }
  // the sum so far, in units of 2^29, added to s; cleared
  __device__ __forceinline__ void flush(double2& s) {
    s.x += fma(__ll2double_rn(hx), 536870912.0, __ll2double_rn(mx));
    s.y += fma(__ll2double_rn(hy), 536870912.0, __ll2double_rn(my));
    hx = mx = hy = my = 0;
  }
};
__device__ __forceinline__ double nl_scaled(double v, int e) {   // v 2^e
  return fx_plain_scale(e) ? v * fx_factor(1.0, e) : ldexp(v, e);
}

// Prologue, part 1 (nl_fused_project): load_b(m, g), load_c(g) give the limbs of beta_m and C
// (C below 2^ce; ce = kFxBadField: C has a component that is not finite, and lambda is NaN); bexp:
// exponents of the projectors of this k-point.
template <typename LB, typename LC>
__device__ __forceinline__ void nl_fx_project(int nkb, int np, const int* bexp, int ce, const LB& load_b,
                                              const LC& load_c, double2* nls) {
  constexpr int G = 3;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int ngroups = (nkb + G - 1) / G;
  for (int grp = warp; grp < ngroups; grp += nw) {
    const int m0 = grp * G, nc = min(G, nkb - m0);
    NlSum acc[G];
    double2 tot[G];
#pragma unroll
    for (int j = 0; j < G; ++j) tot[j] = make_double2(0.0, 0.0);
    for (int g0 = 0; g0 < np; g0 += 32 * kNlFlush) {
      const int g1 = min(np, g0 + 32 * kNlFlush);
      for (int g = g0 + lane; g < g1; g += 32) {
        const int4 c = load_c(g);
#pragma unroll
        for (int j = 0; j < G; ++j)
          if (j < nc) acc[j].template add<true>(load_b(m0 + j, g), c);
      }
#pragma unroll
      for (int j = 0; j < G; ++j) acc[j].flush(tot[j]);
    }
#pragma unroll
    for (int j = 0; j < G; ++j) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        tot[j].x += __shfl_xor_sync(0xffffffffu, tot[j].x, o);
        tot[j].y += __shfl_xor_sync(0xffffffffu, tot[j].y, o);
      }
      if (lane == 0 && j < nc) {
        const int be = bexp[m0 + j];
        const bool bad = be == kFxBadField || ce == kFxBadField;
        if (bad) tot[j] = make_double2(nan(""), nan(""));
        const int e = bad ? 0 : be + ce - 85;   // 2^29 / 2^114
        nls[m0 + j] = make_double2(nl_scaled(tot[j].x, e), nl_scaled(tot[j].y, e));
      }
    }
  }
}

// After nl_fused_coef and a barrier, by warp 0: gamma turned into limbs in place, scaled so that
// with beta_m's scale every product has one unit; the exponent to *ex (kFxBadField: a coefficient
// is not finite).
__device__ __forceinline__ void nl_fx_coef(int nkb, const int* bexp, double2* nls, int* ex) {
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  double2* c = nls + nkb;
  int top = -100000;
  for (int m = lane; m < nkb; m += 32) {
    const unsigned h = max(fx_abs_hi(c[m].x), fx_abs_hi(c[m].y));
    const int be = bexp[m];
    if ((h >> 20) == 0x7ff || be == kFxBadField) top = kFxBadField;
    else if (c[m].x != 0.0 || c[m].y != 0.0) top = max(top, (int)max(h >> 20, 1u) - 1022 + be);
  }
  top = __reduce_max_sync(0xffffffffu, top);
  if (top == -100000) top = 0;   // every coefficient is zero
  if (lane == 0) *ex = top;
  for (int m = lane; m < nkb; m += 32) {
    const bool zero = top == kFxBadField || (c[m].x == 0.0 && c[m].y == 0.0);
    reinterpret_cast<int4*>(c)[m] = zero ? int4{0, 0, 0, 0} : nl_limbs(c[m], top - bexp[m]);
  }
}

// Epilogue for one plane wave (nl_fused_addback): sum_m gamma_m beta_m; coef: the limbs of gamma
template <typename LB>
__device__ __forceinline__ double2 nl_fx_addback(int nkb, int g, const int4* coef, int ex, const LB& load_b) {
  double2 h = make_double2(0.0, 0.0);
  NlSum ah;
  for (int m0 = 0; m0 < nkb; m0 += kNlFlush) {
    const int m1 = min(nkb, m0 + kNlFlush);
#pragma unroll 3
    for (int m = m0; m < m1; ++m) ah.add<false>(load_b(m, g), coef[m]);
    ah.flush(h);
  }
  if (ex == kFxBadField) return make_double2(nan(""), nan(""));
  return make_double2(nl_scaled(h.x, ex - 85), nl_scaled(h.y, ex - 85));
}

// shared-memory bytes of the coefficients (lambda, gamma, delta) for nkb projectors; FP64: then
// the exponent of gamma
inline size_t nl_fused_bytes(int nkb, int elem_bytes) {
  return nkb > 0 ? (((size_t)3 * nkb * elem_bytes + 15) & ~(size_t)15) + (elem_bytes == 16 ? 16 : 0) : 0;
}

}  // namespace pwk
