// Rows of the stored Galerkin operators (Sec. 2.2 eq. coarseGridMatrix): the
// table element loads and the compile-time unrolled row sums shared by the
// Galerkin-level kernels (k_stencil.cu) and the persistent MG-DD coarsest solve
// (k_coarse_persist.cu).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "kernels.h"

namespace ehs {

// Stencil-table element load: complex64/complex128 tables as stored, and the
// half-precision table formats (FP16 or BF16 real/imag pairs) widened to
// complex64 so that accumulation stays in FP32.
template <typename T> __device__ __forceinline__ typename CT<T>::type ldtab(const typename CT<T>::type* p) {
  return __ldg(p);
}
template <typename T> __device__ __forceinline__ float2 ldtab(const __half2* p) {
  return __half22float2(__ldg(p));
}
template <typename T> __device__ __forceinline__ float2 ldtab(const __nv_bfloat162* p) {
  return __bfloat1622float2(__ldg(p));
}

namespace rows {

// Compact slot and mirror flag of box position ti of pair Q in a half table
// (half_index in common.cuh with the pair's constants folded).
template <int D, int LV, int Q>
__device__ __forceinline__ int half_slot_of(int ti, bool& mir) {
  constexpr StencilLayout L = level_layout(D, LV);
  constexpr int a = L.p[Q].a, b = L.p[Q].b;
  constexpr int ne = L.p[Q].ext[0] * L.p[Q].ext[1] * L.p[Q].ext[2];
  constexpr int hb = half_base(L, Q);
  if constexpr (a < b) {
    mir = false;
    return hb + ti;
  } else if constexpr (a == b) {
    constexpr int tc = (ne - 1) / 2;
    mir = ti < tc;
    return hb + (mir ? tc - ti : ti - tc);
  } else {
    constexpr int hbm = half_base(L, L.pidx[b][a]);
    mir = true;
    return hbm + (ne - 1 - ti);
  }
}

// Row a of the stored operator at cell c (coords i), with the stencil box of
// Galerkin level variant LV (1 = first coarse level, 2 = all coarser ones)
// known at compile time so that every table and vector load of the row is
// issued back to back.  SYM: the table is stored half (common.cuh HalfMap), an
// unstored coefficient read from its mirror at the neighbour cell.
// XCG: x is read through L2 only (x written earlier by the same launch on other SMs).  PLAIN: the kernel is launched
// plainly and reads x as data that does not change.
// NS > 1: only the coefficients whose slot index is SI modulo NS (a share of the row, the
// rest summed by NS - 1 other threads).
template <typename T, typename TT, int D, int LV, bool SYM, int Q, int QE, bool XCG = false, int NS = 1, int SI = 0,
          bool PLAIN = false>
__device__ __forceinline__ void row_acc(typename CT<T>::type& y, const Grid& g,
                                        const TT* __restrict__ tab,
                                        long long c, const int i[3],
                                        const typename CT<T>::type* x) {
  if constexpr (Q < QE) {
    constexpr StencilLayout L = level_layout(D, LV);
    constexpr int b = L.p[Q].b, base = L.p[Q].base;
    constexpr int lo0 = L.p[Q].lo[0], lo1 = L.p[Q].lo[1], lo2 = L.p[Q].lo[2];
    constexpr int e0 = L.p[Q].ext[0], e1 = L.p[Q].ext[1], e2 = L.p[Q].ext[2];
    const long long N = g.ncell;
    const long long sy = g.n[0], sz = (long long)g.n[0] * g.n[1];
    const typename CT<T>::type* xb = x + (long long)b * N;
#pragma unroll
    for (int oz = 0; oz < e2; ++oz) {
      const int jz = i[2] + lo2 + oz;
#pragma unroll
      for (int oy = 0; oy < e1; ++oy) {
        const int jy = i[1] + lo1 + oy;
        const bool rin = (D < 3 || (jz >= 0 && jz < g.n[2])) && jy >= 0 && jy < g.n[1];
#pragma unroll
        for (int ox = 0; ox < e0; ++ox) {
          if (NS == 1 || (base + (oz * e1 + oy) * e0 + ox) % NS == SI) {
            // only the loads of a neighbour are conditional, not the sum: with the whole term under one
            // condition its loads wait for the terms before it (gather of the 512x512 line 13.2 -> 10.1 us)
            const int jx = i[0] + lo0 + ox;
            const bool in = rin && jx >= 0 && jx < g.n[0];
            const int ti = (oz * e1 + oy) * e0 + ox;
            const long long cj = c + (lo2 + oz) * sz + (lo1 + oy) * sy + (lo0 + ox);
            typedef typename CT<T>::type Cx;
            if constexpr (PLAIN && sizeof(T) == 4 && !SYM) {
              // loads of data that does not change run ahead under the condition too (four media of 128^2, level 2:
              // a sweep 33 us, 37 with the loads alone conditional)
              if (in) y = cfma(ldtab<T>(tab + (long long)(base + ti) * N + c), ld_vec<PLAIN>(xb + cj), y);
              continue;
            }
            Cx tv = czero<Cx>(), xv = czero<Cx>();
            if constexpr (SYM) {
              bool mir = false;
              const int hs = half_slot_of<D, LV, Q>(ti, mir);
              const TT* tp = tab + (long long)hs * N;
              if (!mir) tv = ldtab<T>(tp + c);
              else if (in) tv = ldtab<T>(tp + cj);
            } else {
              tv = ldtab<T>(tab + (long long)(base + ti) * N + c);
            }
            if (in) xv = XCG ? __ldcg(xb + cj) : ld_vec<PLAIN>(xb + cj);
            y = cfma(tv, xv, y);
          }
        }
      }
    }
    row_acc<T, TT, D, LV, SYM, Q + 1, QE, XCG, NS, SI, PLAIN>(y, g, tab, c, i, x);
  }
}

template <typename T, typename TT, int D, int LV, bool SYM, int A, bool XCG = false, int NS = 1, int SI = 0,
          bool PLAIN = false>
__device__ __forceinline__ typename CT<T>::type st_row_ct(const Grid& g, const TT* tab,
                                                           long long c, const int i[3],
                                                           const typename CT<T>::type* x) {
  constexpr StencilLayout L = level_layout(D, LV);
  typename CT<T>::type y = czero<typename CT<T>::type>();
  row_acc<T, TT, D, LV, SYM, L.row_first[A], L.row_first[A + 1], XCG, NS, SI, PLAIN>(y, g, tab, c, i, x);
  return y;
}

// Coefficient (row A, column B, offset O) of the row at cell c from a full table
// (slot of the layout at cell c) or a half table (compact slot at c, or its
// mirror's at c + O; off = the linear cell offset of O), slots folded at
// compile time.
template <typename T, typename TT, int D, int LV, bool SYM, int A, int B, int OX, int OY, int OZ>
__device__ __forceinline__ typename CT<T>::type tab_coef(const TT* ts, long long N, long long c, long long off) {
  constexpr StencilLayout L = level_layout(D, LV);
  constexpr int sl = st_slot(L, A, B, OX, OY, OZ);
  static_assert(sl >= 0, "coefficient outside the stored box");
  if constexpr (SYM) {
    constexpr int q = L.pidx[A][B];
    constexpr bool mir = half_mir_c(L, q, sl - L.p[q].base);
    constexpr int hs = half_slot_c(L, q, sl - L.p[q].base);
    return ldtab<T>(ts + (long long)hs * N + (mir ? c + off : c));
  } else {
    return ldtab<T>(ts + (long long)sl * N + c);
  }
}

// The block coefficients of component K of the economic cell update: couplings of the low and high face to the
// cell's pressure (gr) and back (gc), and the inverses of the two diagonals (dinv), from the setup-time table vt
// ([D + 1][ncell] of one medium: inverse diagonals of the low face rows, then the blocks' inverse Schur
// complements; launch_vupd_tab).
template <typename T, typename TT, int D, int LV, bool SYM, int K>
__device__ __forceinline__ void vupd_coefs(const TT* ts, const typename CT<T>::type* vt, long long N, long long c,
                                           long long sk, bool lo_ok, bool hi_ok, typename CT<T>::type* dinv,
                                           typename CT<T>::type* gr, typename CT<T>::type* gc) {
  constexpr int E0 = K == 0, E1 = K == 1, E2 = K == 2;
  if (lo_ok) {
    dinv[K] = __ldg(vt + (long long)K * N + c);
    gr[K] = tab_coef<T, TT, D, LV, SYM, K, D, 0, 0, 0>(ts, N, c, 0);
    gc[K] = tab_coef<T, TT, D, LV, SYM, D, K, 0, 0, 0>(ts, N, c, 0);
  }
  if (hi_ok) {
    dinv[D + K] = __ldg(vt + (long long)K * N + c + sk);
    gr[D + K] = tab_coef<T, TT, D, LV, SYM, K, D, -E0, -E1, -E2>(ts, N, c + sk, -sk);
    gc[D + K] = tab_coef<T, TT, D, LV, SYM, D, K, E0, E1, E2>(ts, N, c, sk);
  }
}

}  // namespace rows
using rows::st_row_ct;
using rows::tab_coef;
using rows::vupd_coefs;
using rows::half_slot_of;

}  // namespace ehs
