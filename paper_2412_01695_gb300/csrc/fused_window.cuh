// Window-specialised fused H|psi> kernel.
//
// Same operator (kinetic and local terms) and the same one-HBM-round-trip structure as
// fused_kernel (paper Sec. 2.2 and Sec. 4; see fused_kernel.cuh), for spheres whose Miller indices all satisfy |m_i| <= W with
// W = N/4: a grid chosen to hold the differences G - G' of the basis (Sec. 4: "N_i large
// enough"), N >= 4 max|m|, always satisfies it.  With the window known at compile time:
//   * the z-sticks live in a dense (2W+1) x (2W+1) square of rows [m1][m2] (rows without a
//     stick of this k stay zero), so the y pass reads and writes them without a stick table; on
//     grids of N >= 30 (window_lists) they lie one row after another instead, m1 fastest, found
//     from the y pass by a table over the window (a row of zeros stands for a missing stick):
//     half the square is empty there, and the shared memory it takes costs a CTA per SM;
//   * every transform reads only the 2W+1 window inputs (the others are literal zeros) and
//     stores only the outputs that are used later; no per-element index arithmetic or
//     predicated shared-memory access remains.
// The rows of the sticks (or the table) and the packed (row, m3) place of every basis vector
// come from the plan's window tables.
#pragma once
#include <type_traits>

#include "fft_line.cuh"
#include "fixed_block.cuh"
#include "fused_kernel.cuh"
#include "nl_fused.cuh"
#include "pwk_internal.h"

namespace pwk {

template <int N, int W>
struct Win {
  static constexpr int NW = 2 * W + 1;
  __host__ __device__ static constexpr bool in(int i) { return i <= W || i >= N - W; }
  __host__ __device__ static constexpr int idx(int i) { return i <= W ? i + W : i - N + W; }  // 0 .. 2W
};

// inputs outside the window, known zero in the inverse transforms (LineFFTZ prunes them)
template <int N, int W>
struct OutOfWin {
  __host__ __device__ static constexpr bool zero(int i) { return !Win<N, W>::in(i); }
};

// MODE 0: the CTA takes the l3 planes in chunks of L, with block barriers between the y, x
//         and y passes of a chunk.
// MODE 1: each warp takes its own L planes at a time (planes w L, w L + 1, ... in rounds of
//         nwarps L) through the y, x and y passes with warp-level synchronisation only; block
//         barriers remain only around the z passes.  The arithmetic of every line is the same
//         in both modes (the results are bitwise equal); only the thread mapping differs.
// The work of one band-k item (k, input slot vin, output slot vout) of the plan described
// by `a`; the kernels below decode the item and call it.
// NL: the nonlocal projector terms are applied in the epilogue (nl_fused.cuh) when the plan
//     has projectors (a.nkb > 0); the kernel without them (NL false) is compiled apart, so the
//     projector code costs it nothing.
// FP64 (T = double): the transforms run in the 64-bit fixed point of fixed.cuh; C is scaled
// into it by the scatter, and the gather returns to double with the shift of its z line.  What
// bounds it now (N = 24): about 2500 integer instructions per line at two to three warps per
// scheduler (the line takes 168 registers; ALU pipe 36 % busy, FMA pipe 22 %, FP64 pipe 12 %), with
// barriers and instruction fetch between them.  Two CTAs of 192
// threads (168 registers) ran 1280 band-k in 0.48 ms, of 128 threads (222 registers) in 0.56.
template <typename T, typename TI, int N, int W, int MODE, bool NL>
__device__ __forceinline__ void window_body(const FusedArgs& a, int k, int vin, int vout) {
  using V = c2_t<T>;
  using VI = c2_t<TI>;
  using A = fft_arith_t<T>;
  using VA = c2_t<A>;
  constexpr bool FX = std::is_same<A, long long>::value;
  using Wn = Win<N, W>;
  constexpr int NW = Wn::NW;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, nth = blockDim.x;
  const int np = a.npw_in[k];
  const int ns = a.nstick[k];
  const int zs = a.zs, L = a.L, yps = a.yps;

  constexpr bool LIST = window_lists(N);
  const int nz = a.nstick_max;                          // LIST: the row of zeros
  const int nrows = LIST ? nz + 1 : NW * NW;
  VA* Z = reinterpret_cast<VA*>(smem_raw);              // [nrows][zs]
  // fixed point: the shifts of the z lines next to the sticks (the gather reads them while the
  // projector terms reuse what follows), those of the x lines [ycopies][N][L] and y lines
  // [NW][N] at the end
  unsigned char* sz = reinterpret_cast<unsigned char*>(Z + (size_t)nrows * zs);   // [nrows]
  VA* Y = Z + (size_t)nrows * zs + (FX ? window_shift_elems(nrows) : 0);   // [NW][yps] (N x L used per plane)
  // plane buffers: one [NW][yps] for the CTA (MODE 0) or one per warp (MODE 1), then the rows of
  // the sticks, or the table [NW (m2)][NW (m1)]
  const int ycopies = MODE == 1 ? (int)(blockDim.x >> 5) : 1;
  short* tab = reinterpret_cast<short*>(Y + (size_t)ycopies * NW * yps);
  unsigned char* sx = reinterpret_cast<unsigned char*>(tab + (LIST ? NW * NW : nz));
  unsigned char* sy = sx + (size_t)ycopies * N * L;
  auto stick_row = [&](int s) { return LIST ? s : (int)tab[s]; };
  auto window_row = [&](int p, int i) { return LIST ? (int)tab[i * NW + p] : p * NW + i; };   // plane p, m2 index i
  // the same in two parts: on the square the rows of a plane lie at fixed steps from its first
  auto plane_at = [&](int p) { return LIST ? Z : Z + (size_t)p * NW * zs; };
  auto plane_row = [&](int p, int i) { return LIST ? (int)tab[i * NW + p] : i; };

  const VI* pin = static_cast<const VI*>(a.in) + ((size_t)k * a.nvec_in + vin) * a.npw_in_max;
  VI* pout = static_cast<VI*>(a.out) + ((size_t)k * a.nvec_out + vout) * a.npw_out_max;

  // C(G) is read from global memory by the two stages that need it (scatter, kinetic term):
  // the second read hits L1/L2, and the shared memory a staged copy would take buys occupancy.
  // ---- 0: zero the rows, stage the table
  for (int i = tid; i < (LIST ? ns : nrows) * zs; i += nth) Z[i] = VA{A(0), A(0)};
  if constexpr (LIST) {
    for (int i = tid; i < zs; i += nth) Z[(size_t)nz * zs + i] = VA{A(0), A(0)};
    const short* rk = a.sid + (size_t)k * NW * NW;
    for (int i = tid; i < NW * NW; i += nth) {
      const int r = rk[i];
      tab[i] = (short)(r < 0 ? nz : r);
      if (FX && r >= 0) sz[r] = (unsigned char)(i % NW);   // the stick's m1 plane, until its shift
    }
  } else {
    const short* rk = a.sid + (size_t)k * nz;
    for (int i = tid; i < ns; i += nth) {
      tab[i] = rk[i];
      if (FX) sz[rk[i]] = (unsigned char)(rk[i] / NW);
    }
  }
  FxScale scale{1.0, 0.0, 0, false, 0};
  if constexpr (FX) {
    scale = fx_block_scale(pin, np, fx_scratch_at(sy + NW * N));   // synchronises the block
  }
  __syncthreads();

  // ---- 1: scatter
  {
    const int* gin = a.gin + (size_t)k * a.npw_in_max;
    for (int g = tid; g < np; g += nth) {
      const int m = gin[g];
      const VI v = pin[g];
      if constexpr (FX) Z[(m >> 8) * zs + (m & 255)] = fx_from(scale, v);
      else Z[(m >> 8) * zs + (m & 255)] = VA{A(v.x), A(v.y)};
    }
  }
  __syncthreads();

  // ---- 2-4: the line passes.  Inverse z on the real sticks; per chunk of L planes inverse y on
  // the m2 window of plane p, the x lines (inverse, V(r) product, forward, window outputs only)
  // and forward y, window outputs back to the stick square; forward z.  MODE 1: a warp's chunks
  // are its own.
  const int warp = MODE == 1 ? tid >> 5 : 0, nw = MODE == 1 ? nth >> 5 : 1;
  const int lane0 = MODE == 1 ? tid & 31 : tid, step0 = MODE == 1 ? 32 : nth;
  VA* Yc = Y + (size_t)warp * NW * yps;        // [NW][yps]: plane p row, (l2, cc) at l2 L + cc
  auto sync_pass = [&]() {
    if constexpr (MODE == 1) __syncwarp();
    else __syncthreads();
  };
  if constexpr (!FX) {
    for (int s = tid; s < ns; s += nth) {
      VA x[N];
      VA* zr = Z + stick_row(s) * zs;
      PWK_SFOR(N, j, x[j] = Wn::in(j) ? zr[j] : VA{A(0), A(0)});
      LineFFTZ<A, N, +1, OutOfWin<N, W>>::run(x);
      PWK_SFOR(N, j, zr[j] = x[OutSlot<N, j>::value]);
    }
    __syncthreads();
    for (int l0 = warp * L; l0 < N; l0 += nw * L) {
      const int lc = min(L, N - l0);
      for (int t = lane0; t < NW * lc; t += step0) {
        const int c = t / NW, p = t - c * NW;   // plane fastest: see window_strides
        VA x[N];
        const VA* zp = plane_at(p) + l0 + c;
        PWK_SFOR(N, j, {
          if constexpr (Wn::in(j)) x[j] = zp[plane_row(p, Wn::idx(j)) * zs];
          else x[j] = VA{A(0), A(0)};
        });
        LineFFTZ<A, N, +1, OutOfWin<N, W>>::run(x);
        VA* yp = Yc + (size_t)p * yps + c;
        PWK_SFOR(N, l2, yp[l2 * L] = x[OutSlot<N, l2>::value]);
      }
      sync_pass();
      for (int t = lane0; t < N * lc; t += step0) {
        const int l2 = t / lc, c = t - l2 * lc;
        // V(r) of the line is requested first: its latency hides behind the inverse transform
        A w[N];
        load_vline<N>(static_cast<const float*>(a.V) + ((size_t)l2 * N + l0 + c) * N, w);
        VA x[N], y[N];
        VA* yl = Yc + (size_t)l2 * L + c;
        PWK_SFOR(N, i, x[i] = Wn::in(i) ? yl[(size_t)Wn::idx(i) * yps] : VA{A(0), A(0)});
        LineFFTZ<A, N, +1, OutOfWin<N, W>>::run(x);
        PWK_SFOR(N, l1, {
          const VA u = x[OutSlot<N, l1>::value];
          y[l1] = VA{u.x * w[l1], u.y * w[l1]};
        });
        LineFFT<A, N, -1>::run(y);
        PWK_SFOR(N, i, {
          if constexpr (Wn::in(i)) yl[(size_t)Wn::idx(i) * yps] = y[OutSlot<N, i>::value];
        });
      }
      sync_pass();
      for (int t = lane0; t < NW * lc; t += step0) {
        const int c = t / NW, p = t - c * NW;
        VA x[N];
        const VA* yp = Yc + (size_t)p * yps + c;
        PWK_SFOR(N, l2, x[l2] = yp[l2 * L]);
        LineFFT<A, N, -1>::run(x);
        VA* zp = plane_at(p) + l0 + c;
        PWK_SFOR(N, j, {
          if constexpr (Wn::in(j)) {
            const int row = plane_row(p, Wn::idx(j));
            if (!LIST || row != nz) zp[row * zs] = x[OutSlot<N, j>::value];
          }
        });
      }
      sync_pass();
    }
    __syncthreads();
    for (int s = tid; s < ns; s += nth) {
      VA x[N];
      VA* zr = Z + stick_row(s) * zs;
      PWK_SFOR(N, j, x[j] = zr[j]);
      LineFFT<A, N, -1>::run(x);
      PWK_SFOR(N, j, {
        if constexpr (Wn::in(j)) zr[j] = x[OutSlot<N, j>::value];
      });
    }
    __syncthreads();
  } else {
    // fixed point: one copy of the inverse and of the forward code for the z and y lines
    // (unrolled over a line it is thousands of instructions, and the instruction cache holds
    // few): stages inverse z, the chunks' y, x, y, forward z, with one block barrier that ends
    // each stage for every warp, also one without a chunk of its own.
    // z: the line is stick t; y: plane t % NW of column l0 + t / NW, its window elements in the
    // rows of the table.
    unsigned char* sxc = sx + (size_t)warp * N * L;
    auto inverse_line = [&](bool z, int t, int l0) {
      VA x[N];
      VA* zp = z ? Z + stick_row(t) * zs : Z + l0 + t / NW;
      PWK_SFOR(N, j, {
        if constexpr (!Wn::in(j)) {
          x[j] = VA{A(0), A(0)};
        } else {
          const int o = z ? j : window_row(t % NW, Wn::idx(j)) * zs;
          x[j] = zp[o];
        }
      });
      LineFFTZ<A, N, +1, OutOfWin<N, W>>::run(x);
      VA* out = z ? zp : Yc + (size_t)(t % NW) * yps + t / NW;
      const int os = z ? 1 : L;
      PWK_SFOR(N, j, out[j * os] = x[OutSlot<N, j>::value]);
    };
    auto forward_line = [&](bool z, int t, int l0) {
      VA x[N];
      const int srow = z ? stick_row(t) : 0;
      VA* zp = z ? Z + srow * zs : Z + l0 + t / NW;
      const VA* in = z ? zp : Yc + (size_t)(t % NW) * yps + t / NW;
      const int is = z ? 1 : L;
      PWK_SFOR(N, j, x[j] = in[j * is]);
      const int sh = fx_align<N>(x, z ? sy + sz[srow] * N : sxc + t / NW, is);
      (z ? sz + srow : sy + t % NW * N + l0 + t / NW)[0] = (unsigned char)sh;
      LineFFT<A, N, -1>::run(x);
      PWK_SFOR(N, j, {
        if constexpr (Wn::in(j)) {
          const int row = z ? 0 : window_row(t % NW, Wn::idx(j));
          if (!LIST || z || row != nz) zp[z ? j : row * zs] = x[OutSlot<N, j>::value];
        }
      });
    };
    auto x_line = [&](int t, int l0, int lc) {
      const int l2 = t / lc, c = t - l2 * lc;
      VA x[N], y[N];
      VA* yl = Yc + (size_t)l2 * L + c;
      PWK_SFOR(N, i, x[i] = Wn::in(i) ? yl[(size_t)Wn::idx(i) * yps] : VA{A(0), A(0)});
      LineFFTZ<A, N, +1, OutOfWin<N, W>>::run(x);
      sxc[l2 * L + c] = (unsigned char)fx_v_product<N>(x, static_cast<const int2*>(a.V) + ((size_t)l2 * N + l0 + c) * N, y);
      LineFFT<A, N, -1>::run(y);
      PWK_SFOR(N, i, {
        if constexpr (Wn::in(i)) yl[(size_t)Wn::idx(i) * yps] = y[OutSlot<N, i>::value];
      });
    };
#pragma unroll 1
    for (int stage = 0; stage < 3; ++stage) {   // uniform: every warp meets the barrier below three times
      const bool first = stage == 0, last = stage == 2;
      // the chunks of stage 1; the z stages take the body once
#pragma unroll 1
      for (int l0 = stage == 1 ? warp * L : 0; l0 < (stage == 1 ? N : 1); l0 += nw * L) {
        const int lc = min(L, N - l0);
        const int n = stage == 1 ? NW * lc : ns, t0 = stage == 1 ? lane0 : tid, step = stage == 1 ? step0 : nth;
        if (!last)
          for (int t = t0; t < n; t += step) inverse_line(first, t, l0);
        if (stage == 1) {
          sync_pass();
          for (int t = lane0; t < N * lc; t += step0) x_line(t, l0, lc);
          sync_pass();
        }
        if (!first)
          for (int t = t0; t < n; t += step) forward_line(last, t, l0);
        if (stage == 1 && l0 + nw * L < N) sync_pass();   // another chunk reuses the planes
      }
      __syncthreads();
    }
  }

  // ---- 5: gather with 1/N_r; kinetic term
  const int vexp = a.vexp == kFxBadField ? 0 : a.vexp;
  const double scd = FX && (scale.bad || a.vexp == kFxBadField) ? __longlong_as_double(0x7ff8000000000000LL) : a.scale;
  const T sc = T(scd);
  // the local term of the basis vector at packed place m, with the kinetic term t2 c
  auto local = [&](int m, T t2, VI c) -> V {
    const VA z = Z[(m >> 8) * zs + (m & 255)];
    if constexpr (FX) {
      const int e = sz[m >> 8] + vexp - scale.exp;
      const double f = fx_factor(scd, e);
      return V{fx_scaled(z.x, f, e) + t2 * c.x, fx_scaled(z.y, f, e) + t2 * c.y};
    } else {
      return V{z.x * sc + t2 * T(c.x), z.y * sc + t2 * T(c.y)};
    }
  };
  if (!NL || a.nkb == 0) {
    const int* gout = a.gout + (size_t)k * a.npw_out_max;
    const double* g2k = a.g2 + (size_t)k * a.npw_out_max;
    for (int g = tid; g < np; g += nth) {
      const V acc = local(gout[g], T(g2k[g]), pin[g]);
      pout[g] = VI{TI(acc.x), TI(acc.y)};
    }
    for (int g = np + tid; g < a.npw_out_max; g += nth) pout[g] = VI{TI(0), TI(0)};
  } else if constexpr (NL) {
    // With projectors (nl_fused.cuh): the local result and C go to shared memory past the
    // stick square; once the square is read, beta(k) is staged over it, and the projections,
    // gamma (delta) and the add-back (S C) run from shared memory.
    const int* gout = a.gout + (size_t)k * a.npw_out_max;
    const double* g2k = a.g2 + (size_t)k * a.npw_out_max;
    V* LOC = reinterpret_cast<V*>(smem_raw + a.loc_off);   // [npw_out_max] local + kinetic
    V* Cs = LOC + a.npw_out_max;                             // [npw_out_max] C in T, or its limbs
    V* nls = reinterpret_cast<V*>(smem_raw + a.nl_off);
    const bool with_s = a.sout != nullptr;
    const bool with_q = with_s && a.qm != nullptr;
    VI* sout = with_s ? static_cast<VI*>(a.sout) + ((size_t)k * a.nvec_out + vout) * a.npw_out_max : nullptr;
    const bool ints = FX && a.nl_ints && !with_q;            // the integer sums of nl_fused.cuh
    for (int g = tid; g < np; g += nth) {
      const VI cv = pin[g];
      LOC[g] = local(gout[g], T(g2k[g]), cv);
      if constexpr (FX) {
        if (ints) {
          reinterpret_cast<int4*>(Cs)[g] = scale.bad ? int4{0, 0, 0, 0} : nl_limbs(cv, scale.top);
          continue;
        }
      }
      Cs[g] = V{T(cv.x), T(cv.y)};
    }
    __syncthreads();
    V* Bs = reinterpret_cast<V*>(smem_raw);                  // [nkb][npw_beta] in T, or limbs
    if constexpr (FX) {
      if (ints) {
        int4* Bl = reinterpret_cast<int4*>(Bs);
        const int4* Cl = reinterpret_cast<const int4*>(Cs);
        const int* be = a.bexp + (size_t)k * a.nkb;
        int* ex = reinterpret_cast<int*>(nls + 3 * (size_t)a.nkb);
        const double2* bk = static_cast<const double2*>(a.beta) + (size_t)k * a.nkb * a.npw_beta;
        for (int m = 0; m < a.nkb; ++m) {
          const int R = be[m] == kFxBadField ? 0 : be[m];
          for (int g = tid; g < np; g += nth) {
            const size_t i = (size_t)m * a.npw_beta + g;
            Bl[i] = nl_limbs(bk[i], R);
          }
        }
        __syncthreads();
        auto load_b = [&](int m, int g) { return Bl[(size_t)m * a.npw_beta + g]; };
        nl_fx_project(a.nkb, np, be, scale.top, load_b, [&](int g) { return Cl[g]; }, nls);
        __syncthreads();
        nl_fused_coef<T>(a, nls);
        __syncthreads();
        nl_fx_coef(a.nkb, be, nls, ex);
        __syncthreads();
        const int4* gl = reinterpret_cast<const int4*>(nls) + a.nkb;
        for (int g = tid; g < np; g += nth) {
          const double2 h = nl_fx_addback(a.nkb, g, gl, *ex, load_b);
          const V l = LOC[g];
          if (with_s) sout[g] = pin[g];
          pout[g] = VI{l.x + h.x, l.y + h.y};
        }
      }
    }
    if (!ints) {
      nl_stage_beta<T>(a, k, Bs);
      nl_fused_project<T>(a, Bs, a.npw_beta, Cs, np, nls);
      __syncthreads();
      nl_fused_coef<T>(a, nls);
      __syncthreads();
      for (int g = tid; g < np; g += nth) {
        V h, sv;
        nl_fused_addback<T>(a, Bs, a.npw_beta, g, nls, with_q, h, sv);
        const V l = LOC[g];
        pout[g] = VI{TI(l.x + h.x), TI(l.y + h.y)};
        if (with_s) {
          const VI cv = pin[g];
          sout[g] = with_q ? VI{cv.x + TI(sv.x), cv.y + TI(sv.y)} : cv;
        }
      }
    }
    for (int g = np + tid; g < a.npw_out_max; g += nth) {
      pout[g] = VI{TI(0), TI(0)};
      if (with_s) sout[g] = VI{TI(0), TI(0)};
    }
  }
}

// Threads the register budget allows for: an FP64 line of N <= 27 fits the 168 registers of 384
// threads per SM (a few words spilled at N = 24, 27), which lets two CTAs of 192 run on an SM.
template <typename T, int N>
constexpr int window_max_threads() { return sizeof(T) == 8 && N <= 27 ? 384 : 256; }

// One CTA per work item of one plan: item = (k - k0) * nvec + band of a batched call, or the
// (k, in_slot, out_slot) entry of a work list.
template <typename T, typename TI, int N, int W, int MODE, bool NL>
__global__ void __launch_bounds__(window_max_threads<T, N>()) fused_window_kernel(FusedArgs a) {
  const int item = blockIdx.x;
  if (a.d_count != nullptr && item >= *a.d_count) return;
  int k, vin, vout;
  if (a.items != nullptr) {
    k = a.items[3 * item];
    vin = a.items[3 * item + 1];
    vout = a.items[3 * item + 2];
    if (k == -1) return;
    if (k < 0 || k >= a.nk || vin < 0 || vin >= a.nvec_in || vout < 0 || vout >= a.nvec_out) {
      if (threadIdx.x == 0 && a.err != nullptr) atomicOr(a.err, 1);
      return;
    }
  } else {
    const int kr = item / a.nvec_in;
    vin = vout = item - kr * a.nvec_in;
    k = a.k0 + kr;
  }
  window_body<T, TI, N, W, MODE, NL>(a, k, vin, vout);
}

// One CTA per work item of a list that spans several plans of the same grid (cells with their
// own atoms, projectors, V(r), spheres and k-points): entry (plan, k, in_slot, out_slot) of
// a.items, the plan's arguments at a.multi[plan] (in device memory).  An entry with plan = -1
// is an empty slot; one outside the plans or the plan's k-points and slots is skipped and
// flagged in the first plan's error word.
template <typename T, typename TI, int N, int W, int MODE>
__global__ void __launch_bounds__(window_max_threads<T, N>()) fused_window_multi_kernel(FusedArgs a0) {
  const int item = blockIdx.x;
  const int* it = a0.items + 4 * (size_t)item;
  const int p = it[0], k = it[1], vin = it[2], vout = it[3];
  if (p == -1) return;
  if (p < 0 || p >= a0.nmulti) {
    if (threadIdx.x == 0 && a0.err != nullptr) atomicOr(a0.err, 1);
    return;
  }
  const FusedArgs& a = a0.multi[p];
  if (k < 0 || k >= a.nk || vin < 0 || vin >= a.nvec_in || vout < 0 || vout >= a.nvec_out) {
    if (threadIdx.x == 0 && a0.err != nullptr) atomicOr(a0.err, 1);
    return;
  }
  window_body<T, TI, N, W, MODE, true>(a, k, vin, vout);
}

// window half-width instantiated for a grid of size N
__host__ __device__ constexpr int window_of(int N) { return N / 4; }

template <typename T, typename TI>
int launch_window_multi(int N, const FusedArgs& a, int nblocks, const LaunchShape& s, cudaStream_t st) {
  if (nblocks <= 0) return PWK_OK;
  switch (N) {
#define PWK_WMCASE(n)                                                                           \
  case n: {                                                                                     \
    auto kern = s.kind == 2 ? fused_window_multi_kernel<T, TI, n, window_of(n), 1>              \
                            : fused_window_multi_kernel<T, TI, n, window_of(n), 0>;             \
    cudaError_t e = allow_full_smem(kern);                                                      \
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(window multi)");            \
    kern<<<nblocks, s.threads, s.smem, st>>>(a); note_launch();                                                \
    e = cudaGetLastError();                                                                     \
    if (e != cudaSuccess) return cuda_fail(e, "window multi kernel launch");                    \
    return PWK_OK;                                                                              \
  }
    PWK_FOR_EACH_N(PWK_WMCASE)
#undef PWK_WMCASE
    default:
      set_error("unsupported grid size");
      return PWK_ERR_UNSUPPORTED;
  }
}

template <typename T, typename TI, bool NL>
int launch_window(int N, const FusedArgs& a, int nblocks, const LaunchShape& s, cudaStream_t st) {
  if (nblocks <= 0) return PWK_OK;
  switch (N) {
#define PWK_WCASE(n)                                                                            \
  case n: {                                                                                     \
    auto kern = s.kind == 2 ? fused_window_kernel<T, TI, n, window_of(n), 1, NL>                \
                            : fused_window_kernel<T, TI, n, window_of(n), 0, NL>;               \
    cudaError_t e = allow_full_smem(kern);                                                      \
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(window)");                  \
    kern<<<nblocks, s.threads, s.smem, st>>>(a); note_launch();                                                \
    e = cudaGetLastError();                                                                     \
    if (e != cudaSuccess) return cuda_fail(e, "window kernel launch");                          \
    return PWK_OK;                                                                              \
  }
    PWK_FOR_EACH_N(PWK_WCASE)
#undef PWK_WCASE
    default:
      set_error("unsupported grid size");
      return PWK_ERR_UNSUPPORTED;
  }
}

}  // namespace pwk
