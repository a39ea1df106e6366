// Induced charge density of a perturbation (paper Sec. 2.3, Eq. drho):
//
//   drho(r) = 4 sum_k w_k sum_nu conj(u_{k,nu}(r)) [P_c du_{k,nu}](r)
//
// u_{k,nu} on the k sphere (plan_k), du on the k+q sphere (plan_kq), both brought to the real-
// space grid by the inverse transform of Sec. 2.2.2 (no normalisation); P_c du = du -
// sum_v u_{k+q,v} <S u_{k+q,v}|du> (S = 1 without q).  The augmentation term is not included
// (the paper did not accelerate it).
//
// The paper keeps two full FFT grids per band in HBM for this step (Sec. 3).  Here one CTA
// takes one (k, nu) pair at a time: both coefficient sets are scattered onto the union of the
// two spheres' z-sticks in shared memory (the transfer maps of the k -> k+q pair), both are
// transformed z on the sticks, y on the carried m1 planes, x on every line, and the product
// of an x line pair is added at once to the CTA's own partial grid (FP64, in global memory,
// L2-resident).  The CTAs take the pairs in a fixed grid-stride order and the partial grids
// are summed in a fixed order by a second kernel: the result does not depend on timing.
#include <algorithm>

#include "fft_line.cuh"
#include "fixed_block.cuh"
#include "fused_kernel.cuh"
#include "nl_fused.cuh"
#include "pwk_internal.h"
#include "solvers.h"

namespace pwk {

namespace {

constexpr int kDrhoParts = 256;   // partial grids (CTAs) of the accumulation

struct DrhoArgs {
  const void* uk = nullptr;      // [nk][nocc][npw_k] complex128
  const double2* du = nullptr;   // [nk][nocc][npw_kq] complex128 (already projected)
  const double* w = nullptr;     // [nk] weights
  double2* part = nullptr;       // [kDrhoParts][N^3]
  int nk = 0, nocc = 0, npw_k = 0, npw_kq = 0;
  const int* npwk = nullptr;
  const int* npwq = nullptr;
  const int* nstick = nullptr;
  const int* gin = nullptr;      // k sphere -> sticks
  const int* gout = nullptr;     // k+q sphere -> sticks
  const short* sid = nullptr;
  int nstick_max = 0, m1lo = 0, P = 0, L = 0, zs = 0;
};

// v 2^e for an integer value v (0, or 1 <= |v| < 2^62) and fx_plain_scale(e): on the exponent field
__device__ __forceinline__ double times_pow2(double v, int e) {
  const int h = __double2hiint(v);
  return h == 0 ? v : __hiloint2double(h + (e << 20), __double2loint(v));
}

// CTAs per SM the registers allow for: an FP64 line of N <= 20 fits 128 registers
template <typename T, int N>
constexpr int drho_ctas() { return sizeof(T) == 4 || N <= 20 ? 2 : 1; }

template <typename V>
__device__ __forceinline__ V drho_value(float2 q) { return q; }
template <typename V>
__device__ __forceinline__ V drho_value(longlong2 q) { return V{__ll2double_rn(q.x), __ll2double_rn(q.y)}; }

// FP64 transforms run in the fixed point of fixed.cuh (inverse only, so each field keeps the one
// scale of its vector); the values come back to double at the product.  768 pairs at N = 20: 1.05
// ms with FP64 transforms, 0.42 with these; then bound by the conversions and the product (eight FP64
// instructions per grid point, 53 % of that pipe) and the barriers between the passes.
template <typename T, int N>
__global__ void __launch_bounds__(256, drho_ctas<T, N>()) drho_kernel(DrhoArgs a) {
  using V = c2_t<T>;
  using A = fft_arith_t<T>;
  using VA = c2_t<A>;
  constexpr bool FX = std::is_same<A, long long>::value;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int zs = a.zs, P = a.P, L = a.L;
  VA* ZA = reinterpret_cast<VA*>(smem_raw);                // [nstick_max][zs]  u
  VA* ZB = ZA + (size_t)a.nstick_max * zs;                 // [nstick_max][zs]  du
  VA* YA = ZB + (size_t)a.nstick_max * zs;                 // [P][N][L]
  VA* YB = YA + (size_t)P * N * L;
  V* XA = reinterpret_cast<V*>(YB + (size_t)P * N * L);    // [N (l1)][N (l2)][L]
  short* sid = reinterpret_cast<short*>(XA + (size_t)N * N * L);   // [P][N]
  const int tid = threadIdx.x, nth = blockDim.x;
  double2* acc = a.part + (size_t)blockIdx.x * N * N * N;
  for (int i = tid; i < N * N * N; i += nth) acc[i] = make_double2(0.0, 0.0);
  const int npairs = a.nk * a.nocc;
  for (int pr = blockIdx.x; pr < npairs; pr += gridDim.x) {
    const int k = pr / a.nocc, v = pr - k * a.nocc;
    const int ns = a.nstick[k];
    const int nka = a.npwk[k], nkb = a.npwq[k];
    const double wk = 4.0 * a.w[k];
    const double2* pu = static_cast<const double2*>(a.uk) + ((size_t)k * a.nocc + v) * a.npw_k;
    const double2* pd = a.du + ((size_t)k * a.nocc + v) * a.npw_kq;
    __syncthreads();   // the previous pair is done with the buffers
    for (int i = tid; i < ns * zs; i += nth) ZA[i] = ZB[i] = VA{A(0), A(0)};
    {
      const short* sk = a.sid + (size_t)k * P * N;
      for (int i = tid; i < P * N; i += nth) sid[i] = sk[i];
    }
    FxScale su{1.0, 0.0, 0, false, 0}, sd = su;
    int eu = 0, ed = 0;          // powers of two that u and du take at the product
    bool plain = true;
    if constexpr (FX) {
      FxScratch* scratch = fx_scratch_at(reinterpret_cast<unsigned char*>(sid + P * N));
      su = fx_block_scale(pu, nka, scratch);
      __syncthreads();
      sd = fx_block_scale(pd, nkb, scratch);
      // the weight goes into the scale of du (its mantissa, in [1/2, 1)) and of u (a power of two),
      // so that a grid point takes two multiply-adds per component
      int we = 0;
      sd.in *= frexp(wk, &we);
      if (su.bad || sd.bad || !isfinite(wk)) sd.in = 0.0;
      eu = we - su.exp - sd.exp;
      plain = fx_plain_scale(eu) && !su.bad && !sd.bad && isfinite(wk);
      if (!plain) {
        eu = -su.exp;
        ed = su.bad || sd.bad || !isfinite(wk) ? kFxBadField : we - sd.exp;
      }
    }
    __syncthreads();
    {
      const int* gi = a.gin + (size_t)k * a.npw_k;
      const int* go = a.gout + (size_t)k * a.npw_kq;
      for (int g = tid; g < nka; g += nth) {
        const int m = gi[g];
        const double2 c = pu[g];
        if constexpr (FX) ZA[(m >> 8) * zs + (m & 255)] = fx_from(su, c);
        else ZA[(m >> 8) * zs + (m & 255)] = VA{A(c.x), A(c.y)};
      }
      for (int g = tid; g < nkb; g += nth) {
        const int m = go[g];
        const double2 c = pd[g];
        if constexpr (FX) ZB[(m >> 8) * zs + (m & 255)] = fx_from(sd, c);
        else ZB[(m >> 8) * zs + (m & 255)] = VA{A(c.x), A(c.y)};
      }
    }
    __syncthreads();
    // inverse z transforms of both fields on the sticks (Eq. zfft)
    for (int s = tid; s < 2 * ns; s += nth) {
      VA x[N];
      VA* zr = (s < ns ? ZA + s * zs : ZB + (s - ns) * zs);
      PWK_SFOR(N, j, x[j] = zr[j]);
      LineFFT<A, N, +1>::run(x);
      PWK_SFOR(N, j, zr[j] = x[OutSlot<N, j>::value]);
    }
    __syncthreads();
    for (int l0 = 0; l0 < N; l0 += L) {
      const int lc = min(L, N - l0);
      // inverse y transforms of the carried m1 planes (Eq. yfft), both fields
      for (int t = tid; t < 2 * P * lc; t += nth) {
        const int f = t / (P * lc), r = t - f * P * lc;
        const int p = r / lc, c = r - p * lc;
        const VA* Z = f ? ZB : ZA;
        VA x[N];
        PWK_SFOR(N, j, {
          const int s = sid[p * N + j];
          x[j] = s >= 0 ? Z[s * zs + l0 + c] : VA{A(0), A(0)};
        });
        LineFFT<A, N, +1>::run(x);
        VA* yp = (f ? YB : YA) + (size_t)p * N * L + c;
        PWK_SFOR(N, l2, yp[l2 * L] = x[OutSlot<N, l2>::value]);
      }
      __syncthreads();
      // x lines (Eq. xfft): those of u kept in shared memory, then those of du with the product
      // conj(u) du added to this CTA's grid
      for (int f = 0; f < 2; ++f) {
        const VA* Y = f ? YB : YA;
        for (int t = tid; t < N * lc; t += nth) {   // the same thread takes a line of both fields
          const int l2 = t / lc, c = t - l2 * lc;
          VA x[N];
          PWK_SFOR(N, i, {
            const int p = plane_of_slot<N>(i, a.m1lo);
            x[i] = (unsigned)p < (unsigned)P ? Y[((size_t)p * N + l2) * L + c] : VA{A(0), A(0)};
          });
          LineFFT<A, N, +1>::run(x);
          V* xa = XA + (size_t)l2 * L + c;
          if (f == 0) {
            PWK_SFOR(N, l1, {
              V z = drho_value<V>(x[OutSlot<N, l1>::value]);
              if constexpr (FX) z = plain ? V{times_pow2(z.x, eu), times_pow2(z.y, eu)} : V{ldexp(z.x, eu), ldexp(z.y, eu)};
              xa[(size_t)l1 * N * L] = z;
            });
          } else {
            double2* ag = acc + (size_t)l2 * N + l0 + c;
            PWK_SFOR(N, l1, {
              const V ua = xa[(size_t)l1 * N * L];
              V ub = drho_value<V>(x[OutSlot<N, l1>::value]);
              double2& d = ag[(size_t)l1 * N * N];   // += conj(u) du (times the weight, FP64: in the scales)
              if constexpr (FX) {
                if (!plain) {   // uniform
                  const double bad = __longlong_as_double(0x7ff8000000000000LL);
                  ub = ed == kFxBadField ? V{bad, bad} : V{ldexp(ub.x, ed), ldexp(ub.y, ed)};
                }
                d.x = fma(ua.x, ub.x, fma(ua.y, ub.y, d.x));
                d.y = fma(ua.x, ub.y, fma(-ua.y, ub.x, d.y));
              } else {
                const double re = (double)ua.x * ub.x + (double)ua.y * ub.y;
                const double im = (double)ua.x * ub.y - (double)ua.y * ub.x;
                d.x += wk * re;
                d.y += wk * im;
              }
            });
          }
        }
      }
      __syncthreads();
    }
  }
}

// (One thread per point left most SMs idle: 57 us for 256 grids of 20^3, 15 with this split.)
// drho[l] = sum_p part[p][l]: 32 points per CTA, each of its 8 warps sums every eighth partial
// grid in ascending order, and the eight sums are added in ascending order.
__global__ void __launch_bounds__(256) drho_reduce_kernel(int nr, int nparts, const double2* part, double2* out) {
  __shared__ double2 sums[8][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l = blockIdx.x * 32 + lane;
  double sx = 0.0, sy = 0.0;
  if (l < nr)
    for (int p = warp; p < nparts; p += 8) {
      const double2 v = part[(size_t)p * nr + l];
      sx += v.x;
      sy += v.y;
    }
  sums[warp][lane] = make_double2(sx, sy);
  __syncthreads();
  if (warp != 0 || l >= nr) return;
  for (int w = 1; w < 8; ++w) {
    sx += sums[w][lane].x;
    sy += sums[w][lane].y;
  }
  out[l] = make_double2(sx, sy);
}

// Exponent of a vector of np complex numbers by one warp: every |component| < 2^exponent
// (kFxBadField: one is not finite)
__device__ __forceinline__ int warp_exponent(const double2* v, int np) {
  unsigned h = 0;
  for (int g = threadIdx.x & 31; g < np; g += 32) h = max(h, max(fx_abs_hi(v[g].x), fx_abs_hi(v[g].y)));
  h = __reduce_max_sync(0xffffffffu, h);
  return (h >> 20) == 0x7ff ? kFxBadField : (int)(h >> 20) - 1022;
}

// P_c du = du - sum_v u_v <su_v|du> (su = S u, or u when S = 1), one CTA per (k, nu).  The two
// contractions are the projector sums of nl_fused.cuh with the valence states as projectors, on
// the integer pipe: with FP64 multiply-adds they held that pipe (85 % busy) for 113 us on 768 pairs
// of 12 valence states; now 83 us (21 %).  The components of P_c du carry 57 bits of the largest;
// the transform that follows spreads its rounding over all of them alike.  drho against long double,
// limbs (doubles), 3 and 12 valence states: flat vectors 3.3e-16 (3.4), 3.4 (3.8); falling off with
// the kinetic energy 3.2 (3.3), 3.4 (3.8).
__global__ void __launch_bounds__(256) conduction_kernel(int nocc, int np, const int* npw,
                                                         const double2* u, const double2* su,
                                                         const double2* du, double2* out) {
  const int k = blockIdx.x / nocc;
  const int npk = npw[k];
  __shared__ double2 buf[2 * 64];   // the second half: <su_v|du>, then its limbs
  __shared__ int eu[64], es[64], ex, ed;
  const double2* D = du + (size_t)blockIdx.x * np;
  const double2* U = u + (size_t)k * nocc * np;
  const double2* SU = su + (size_t)k * nocc * np;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int v = warp; v <= nocc; v += nw) {
    const int e = warp_exponent(v < nocc ? U + (size_t)v * np : D, npk);
    const int e2 = v < nocc && su != u ? warp_exponent(SU + (size_t)v * np, npk) : e;
    if (lane == 0) {
      if (v < nocc) {
        eu[v] = e;
        es[v] = e2;
      } else {
        ed = e;
      }
    }
  }
  __syncthreads();
  double2* O = out + (size_t)blockIdx.x * np;
  const int ce = ed;
  if (ce == kFxBadField) {   // uniform: a component of du is not finite
    for (int g = threadIdx.x; g < np; g += blockDim.x) O[g] = g < npk ? make_double2(nan(""), nan("")) : make_double2(0.0, 0.0);
    return;
  }
  auto limbs = [&](const double2* base, const int* e, int v, int g) {
    return nl_limbs(base[(size_t)v * np + g], e[v] == kFxBadField ? 0 : e[v]);
  };
  nl_fx_project(nocc, npk, es, ce, [&](int v, int g) { return limbs(SU, es, v, g); },
                [&](int g) { return nl_limbs(D[g], ce); }, buf + nocc);
  __syncthreads();
  nl_fx_coef(nocc, eu, buf, &ex);
  __syncthreads();
  const int4* mu = reinterpret_cast<const int4*>(buf + nocc);
  for (int g = threadIdx.x; g < np; g += blockDim.x) {
    if (g >= npk) {
      O[g] = make_double2(0.0, 0.0);
      continue;
    }
    const double2 h = nl_fx_addback(nocc, g, mu, ex, [&](int v, int i) { return limbs(U, eu, v, i); });
    O[g] = make_double2(D[g].x - h.x, D[g].y - h.y);
  }
}

// work list (k, nu, nu) of every pair
__global__ void pair_items_kernel(int npairs, int nocc, int* items) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= npairs) return;
  items[3 * i] = i / nocc;
  items[3 * i + 1] = items[3 * i + 2] = i % nocc;
}

size_t drho_smem(int N, int elem_bytes, const SphereMap& sm, int L) {
  const int zs = (N % 2 == 0) ? N + 1 : N;
  return ((size_t)2 * sm.nstick_max * zs + (size_t)2 * sm.P * N * L + (size_t)N * N * L) * elem_bytes +
         (size_t)sm.P * N * sizeof(short) + 16;
}

template <typename T>
int launch_drho_typed(int N, const DrhoArgs& a, int nparts, size_t smem, cudaStream_t st) {
  switch (N) {
#define PWK_DCASE(n)                                                                             \
  case n: {                                                                                      \
    auto kern = drho_kernel<T, n>;                                                               \
    cudaError_t e = allow_full_smem(kern);                                                       \
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(drho)");                     \
    kern<<<nparts, 256, smem, st>>>(a); note_launch();                                                          \
    e = cudaGetLastError();                                                                      \
    return e == cudaSuccess ? PWK_OK : cuda_fail(e, "drho_kernel");                              \
  }
    PWK_FOR_EACH_N(PWK_DCASE)
#undef PWK_DCASE
    default:
      set_error("unsupported grid size");
      return PWK_ERR_UNSUPPORTED;
  }
}

}  // namespace

}  // namespace pwk

using namespace pwk;

extern "C" int pwk_drho_batched(pwk_plan* pq, pwk_plan* pk, int precision, const void* psi_k,
                                const void* psi_kq, const void* dpsi, int nocc, const double* weights,
                                void* drho, void* stream) {
  if (pq == nullptr || pk == nullptr || psi_k == nullptr || psi_kq == nullptr || dpsi == nullptr ||
      weights == nullptr || drho == nullptr || nocc < 1) {
    set_error("null pointer or nocc < 1");
    return PWK_ERR_INVALID;
  }
  if (precision != PWK_FP64 && precision != PWK_FP32_C128) {
    set_error("precision must be PWK_FP64 or PWK_FP32_C128");
    return PWK_ERR_INVALID;
  }
  if (nocc > 64) {
    set_error("nocc > 64");
    return PWK_ERR_UNSUPPORTED;
  }
  if (pq->nk != pk->nk || pq->N != pk->N) {
    set_error("plan_k and plan_kq must have the same nk and grid");
    return PWK_ERR_INVALID;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int rc;
  if ((rc = ensure_xfer(pq, pk))) return rc;
  const int N = pq->N, nk = pq->nk, npq = pq->npw_max, npairs = nk * nocc;
  const SphereMap& sm = pq->xfer;
  const int elem = precision == PWK_FP64 ? 16 : 8;
  int L = N;
  while (L > 1 && drho_smem(N, elem, sm, L) > 100 * 1024) --L;
  const size_t smem = drho_smem(N, elem, sm, L);
  if (smem > 227 * 1024) {
    set_error("induced-density kernel does not fit in shared memory");
    return PWK_ERR_UNSUPPORTED;
  }
  const int nparts = std::min(npairs, kDrhoParts);
  const size_t nr = (size_t)N * N * N;
  // scratch: P_c du [nk][nocc][npw_kq], S u (with q), the work list and the partial grids
  double2 *duc = nullptr, *su = nullptr, *part = nullptr;
  int* items = nullptr;
  const size_t nv = (size_t)npairs * npq;
  cudaError_t e = scratch_alloc((void**)&duc, nv * sizeof(double2), st);
  if (e == cudaSuccess) e = scratch_alloc((void**)&part, (size_t)nparts * nr * sizeof(double2), st);
  if (e == cudaSuccess && pq->d_q != nullptr) e = scratch_alloc((void**)&su, nv * sizeof(double2), st);
  if (e == cudaSuccess && pq->d_q != nullptr)
    e = scratch_alloc((void**)&items, (size_t)npairs * 3 * sizeof(int), st);
  if (e != cudaSuccess) {
    for (void* q : {(void*)duc, (void*)part, (void*)su, (void*)items})
      if (q) cudaFreeAsync(q, st);
    return cuda_fail(e, "scratch_alloc(drho)");
  }
  const double2* suv = static_cast<const double2*>(psi_kq);
  if (pq->d_q != nullptr) {   // S u_{k+q,v}: the projector terms alone
    pair_items_kernel<<<(npairs + 255) / 256, 256, 0, st>>>(npairs, nocc, items); note_launch();
    e = cudaGetLastError();
    rc = e == cudaSuccess ? run_hpsi(pq, PWK_FP64, psi_kq, nullptr, items, nullptr, npairs, nocc, nocc, st, su)
                          : cuda_fail(e, "pair_items_kernel");
    suv = su;
  }
  if (rc == PWK_OK) {
    conduction_kernel<<<npairs, 256, 0, st>>>(nocc, npq, pq->d_npw, static_cast<const double2*>(psi_kq), suv,
                                              static_cast<const double2*>(dpsi), duc); note_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) rc = cuda_fail(e, "conduction_kernel");
  }
  if (rc == PWK_OK) {
    DrhoArgs a;
    a.uk = psi_k;
    a.du = duc;
    a.w = weights;
    a.part = part;
    a.nk = nk;
    a.nocc = nocc;
    a.npw_k = pk->npw_max;
    a.npw_kq = npq;
    a.npwk = pk->d_npw;
    a.npwq = pq->d_npw;
    a.nstick = sm.d_nstick;
    a.gin = sm.d_gin;
    a.gout = sm.d_gout;
    a.sid = sm.d_sid;
    a.nstick_max = sm.nstick_max;
    a.m1lo = sm.m1lo;
    a.P = sm.P;
    a.L = L;
    a.zs = (N % 2 == 0) ? N + 1 : N;
    rc = precision == PWK_FP64 ? launch_drho_typed<double>(N, a, nparts, smem, st)
                               : launch_drho_typed<float>(N, a, nparts, smem, st);
  }
  if (rc == PWK_OK) {
    drho_reduce_kernel<<<(int)((nr + 31) / 32), 256, 0, st>>>((int)nr, nparts, part,
                                                                static_cast<double2*>(drho)); note_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) rc = cuda_fail(e, "drho_reduce_kernel");
  }
  cudaFreeAsync(duc, st);
  cudaFreeAsync(part, st);
  if (su) cudaFreeAsync(su, st);
  if (items) cudaFreeAsync(items, st);
  return rc;
}
