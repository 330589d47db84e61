// Fine-level relaxation and operator from setup-time tables of the terms that depend on
// the medium alone (Sec. 3 and Sec. 4.2; the arithmetic of k_fine.cu, whose kernels form
// them anew in every row: five complex inverses a cell and up to ten neighbouring cells'
// coefficients a row).
//
// k_fine_vanka_tab: one colour of the economic cell relaxation (eq. RelaxationMatrix) for
//   contexts' fine levels outside the fused 2D complex64 tiles (k_fine_fused.cu): the FP64
//   form, 3D, and 2D grids that do not split into tiles.  The FP64 form is bound by the FP64
//   pipe: 435 FP64 operations a 2D cell with the terms formed in place, about 130 from the
//   tables.  3D complex64 is bound by its loads, six rows of ten coefficient gathers each.
// k_fine_apply_tab: K x or K_s x (and b - K x) of the FP64 form: about 105 -> 50 FP64
//   operations a 2D cell.
//
// Tables, [nsets][ncell] each, formed in FP64: dv[k] the inverse diagonal of the low u_k
// face row of K_s and dg[k], rf[k] its unshifted diagonal and face mean of omega^2 rho (the
// shift adds i alpha rf); sinv the inverse pressure Schur complement of the cell's block;
// muh = mu / h^2; kap = 1 / (lambda + mu); em[pair] the mean of mu / h^2 over the four cells
// around the edge at the cell's low corner in the two directions of the pair ((0,1), (0,2),
// (1,2)): the tangential weight of both components there.  Off-diagonal weights are only used
// towards unknowns inside the grid, so the arrays need no halo.
#include "kernels.h"

namespace ehs {
namespace {

__host__ __device__ constexpr int pair_of(int k, int j) { return k + j - 1; }   // (0,1) 0, (0,2) 1, (1,2) 2

// a + w v, w real
template <typename T, typename C> __device__ __forceinline__ C rfma(T w, C v, C a) {
  a.x = fma(w, v.x, a.x);
  a.y = fma(w, v.y, a.y);
  return a;
}
template <typename T, typename C> __device__ __forceinline__ C cmulf(C a, C b) {
  C r;
  r.x = fma(-a.y, b.y, a.x * b.x);
  r.y = fma(a.y, b.x, a.x * b.y);
  return r;
}

__device__ __forceinline__ double mu_at(const Coef4<double>* cf, const Grid& g, const int i[3]) {   // clamped
  int q[3];
  for (int k = 0; k < 3; ++k) q[k] = min(max(i[k], 0), g.n[k] - 1);
  return cf[cell_index(g, q)].mu;
}

template <typename T, int D>
__global__ void k_fine_tab_faces(Grid g, const Coef4<double>* __restrict__ cf, double h2inv, double alpha,
                                 FineTab<T> F) {
  typedef typename CT<T>::type C;
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  const Coef4<double>* cs = cf + (long long)blockIdx.y * g.ncell;
  const long long o = (long long)blockIdx.y * g.ncell + c;
  int i[3];
  cell_coords(g, c, i);
  const Coef4<double> c0 = cs[c];
  F.muh[o] = (T)(c0.mu * h2inv);
  F.kap[o] = (T)c0.kap;
  for (int k = 0; k < D; ++k) {
    for (int j = k + 1; j < D; ++j) {
      int q[3] = {i[0], i[1], i[2]};
      double s = c0.mu;
      --q[k]; s += mu_at(cs, g, q);
      --q[j]; s += mu_at(cs, g, q);
      ++q[k]; s += mu_at(cs, g, q);
      F.em[pair_of(k, j)][o] = (T)(0.25 * s * h2inv);
    }
    C dg = mk<T>(1, 0), dv = mk<T>(0, 0);
    T rft = 0;
    if (i[k] >= 1) {
      const Coef4<double> c1 = cs[c - stride_of(g, k)];
      const double base = c0.mu + c1.mu;
      double w = base;
      for (int j = 0; j < D; ++j) {
        if (j == k) continue;
        for (int sgn = -1; sgn <= 1; sgn += 2) {
          int q[3] = {i[0], i[1], i[2]};
          q[j] += sgn;
          const double a = mu_at(cs, g, q);
          --q[k];
          w += 0.25 * (base + a + mu_at(cs, g, q));
        }
      }
      const double rf = 0.5 * (c0.mr + c1.mr), gf = 0.5 * (c0.mi + c1.mi);
      const double2 d = make_double2(w * h2inv - rf, gf), v = cinv(make_double2(d.x, gf + alpha * rf));
      dg = mk<T>((T)d.x, (T)d.y);
      dv = mk<T>((T)v.x, (T)v.y);
      rft = (T)rf;
    }
    F.dv[k][o] = dv;
    if (F.dg[k]) {
      F.dg[k][o] = dg;
      F.rf[k][o] = rft;
    }
  }
}
template <typename T, int D>
__global__ void k_fine_tab_schur(Grid g, const Coef4<double>* __restrict__ cf, double h2inv, FineTab<T> F) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  const long long o = (long long)blockIdx.y * g.ncell + c;
  int i[3];
  cell_coords(g, c, i);
  double2 s = make_double2(-cf[o].kap, 0.0);   // dv is zero on faces that are not unknowns
  for (int k = 0; k < D; ++k) {
    const typename CT<T>::type a = F.dv[k][o];
    s.x -= h2inv * (double)a.x;
    s.y -= h2inv * (double)a.y;
    if (i[k] + 1 < g.n[k]) {
      const typename CT<T>::type b = F.dv[k][o + stride_of(g, k)];
      s.x -= h2inv * (double)b.x;
      s.y -= h2inv * (double)b.y;
    }
  }
  const double2 v = cinv(s);
  F.sinv[o] = mk<T>((T)v.x, (T)v.y);
}

// weights of the u_k row's neighbours at face (cell) c with coordinates i (zero towards what is no unknown)
template <typename T, int D> struct RowW {
  T p, m, tp[D], tm[D];
};
template <typename T, int D>
__device__ __forceinline__ RowW<T, D> row_weights(const Grid& g, int k, int c, const int i[3], const FineTab<T>& F,
                                                  long long so) {
  RowW<T, D> w;
  const T* mu = F.muh + so;
  w.p = i[k] + 1 < g.n[k] ? __ldg(mu + c) : T(0);
  w.m = __ldg(mu + c - (int)stride_of(g, k));
#pragma unroll
  for (int j = 0; j < D; ++j) {
    w.tp[j] = w.tm[j] = 0;
    if (j == k) continue;
    const T* em = F.em[k < j ? pair_of(k, j) : pair_of(j, k)] + so;
    if (i[j] + 1 < g.n[j]) w.tp[j] = __ldg(em + c + (int)stride_of(g, j));
    if (i[j] >= 1) w.tm[j] = __ldg(em + c);
  }
  return w;
}
// s + sum of weights * neighbours - (p_c - p_{c - e_k}) / h: minus the row's off-diagonal part
template <typename T, int D>
__device__ __forceinline__ typename CT<T>::type off_row(const Grid& g, int k, int c, const int i[3],
                                                        const RowW<T, D>& w, const typename CT<T>::type* x, long long N,
                                                        T hinv, typename CT<T>::type s) {
  typedef typename CT<T>::type C;
  const int sk = (int)stride_of(g, k);
  const C* xk = x + (long long)k * N;
  const C* p = x + (long long)D * N;
  C xp = czero<C>(), xm = czero<C>(), tp[D], tm[D];
  if (i[k] + 1 < g.n[k]) xp = xk[c + sk];
  if (i[k] - 1 >= 1) xm = xk[c - sk];
  const C pc = p[c], pm = p[c - sk];
#pragma unroll
  for (int j = 0; j < D; ++j) {
    tp[j] = tm[j] = czero<C>();
    if (j == k) continue;
    const int sj = (int)stride_of(g, j);
    if (i[j] + 1 < g.n[j]) tp[j] = xk[c + sj];
    if (i[j] >= 1) tm[j] = xk[c - sj];
  }
  s = rfma(w.p, xp, s);
  s = rfma(w.m, xm, s);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    if (j == k) continue;
    s = rfma(w.tp[j], tp[j], s);
    s = rfma(w.tm[j], tm[j], s);
  }
  return rfma(-hinv, csub(pc, pm), s);
}

// Thread = pair of cells along x; the cell of the colour is relaxed, the other one's pressure copied (as k_fine_vanka).
// With t_a = (b_a - offdiag_a) / dg_a - x_a: dp = (r_p - sum_a g_a t_a) / S, du_a = t_a - g_a dp / dg_a,
// g = +1/h on the low faces, -1/h on the high ones.  Everything the tables hold is loaded before the wait for the
// launch before (launch_pdl).
template <typename T, int D>
__global__ void k_fine_vanka_tab(Grid g, int nrhs, FineTab<T> F, T hinv, T wu, T wp, int colour,
                                 const typename CT<T>::type* b, const typename CT<T>::type* xi,
                                 typename CT<T>::type* __restrict__ xo, const int* il) {
  pdl_trigger();
  typedef typename CT<T>::type C;
  const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long N = g.ncell;
  const bool live = t0 < N / 2;
  const int item = il ? il[blockIdx.y] : blockIdx.y;   // not changed while a cycle runs
  const long long vo = (long long)item * (D + 1) * N, so = (long long)(item / nrhs) * N;
  int c = (int)(2 * t0);
  int i[3] = {0, 0, 0};
  RowW<T, D> w[2 * D];
  C dv[2 * D], sinv = czero<C>();
  T kap = 0;
  bool ok[2 * D];
  if (live) {
    cell_coords(g, c, i);
    if (((i[0] + i[1] + i[2]) & 1) != colour) { ++c; ++i[0]; }
#pragma unroll
    for (int a = 0; a < 2 * D; ++a) {
      const int k = a % D, hi = a >= D, cc = c + (hi ? (int)stride_of(g, k) : 0);
      int ia[3] = {i[0], i[1], i[2]};
      ia[k] += hi;
      ok[a] = ia[k] >= 1 && ia[k] < g.n[k];
      dv[a] = czero<C>();
      if (ok[a]) {
        dv[a] = __ldg(F.dv[k] + so + cc);
        w[a] = row_weights<T, D>(g, k, cc, ia, F, so);
      }
    }
    kap = __ldg(F.kap + so + c);
    sinv = __ldg(F.sinv + so + c);
  }
  pdl_wait();
  if (!live) return;
  const C* x = xi + vo;
  const C* bb = b + vo;
  C* xout = xo + vo;
  const int co = (c & 1) ? c - 1 : c + 1;
  xout[(long long)D * N + co] = x[(long long)D * N + co];
  const C pc = x[(long long)D * N + c];
  C t[2 * D], xv[2 * D];
  C dsum = czero<C>();                              // sum over the faces of (low - high) x
#pragma unroll
  for (int a = 0; a < 2 * D; ++a) {
    const int k = a % D, hi = a >= D, cc = c + (hi ? (int)stride_of(g, k) : 0);
    int ia[3] = {i[0], i[1], i[2]};
    ia[k] += hi;
    t[a] = xv[a] = czero<C>();
    if (ok[a]) {
      xv[a] = x[(long long)k * N + cc];
      const C s = off_row<T, D>(g, k, cc, ia, w[a], x, N, hinv, bb[(long long)k * N + cc]);
      t[a] = csub(cmulf<T>(dv[a], s), xv[a]);
    }
    dsum = hi ? csub(dsum, xv[a]) : cadd(dsum, xv[a]);
  }
  // pressure row residual and the block's Schur complement; t is zero on faces that are not unknowns
  C rp = bb[(long long)D * N + c];
  rp = rfma(kap, pc, rfma(-hinv, dsum, rp));
#pragma unroll
  for (int a = 0; a < 2 * D; ++a) rp = rfma(a >= D ? hinv : -hinv, t[a], rp);
  const C dp = cmulf<T>(rp, sinv);
  xout[(long long)D * N + c] = rfma(wp, dp, pc);
#pragma unroll
  for (int a = 0; a < 2 * D; ++a) {
    if (!ok[a]) continue;
    const int k = a % D;
    const C du = rfma(a >= D ? hinv : -hinv, cmulf<T>(dp, dv[a]), t[a]);
    xout[(long long)k * N + c + (a >= D ? stride_of(g, k) : 0)] = rfma(wu, du, xv[a]);
  }
}

// y = K x (mode 0) or b - K x (mode 1), alpha = shift
template <typename T, int D>
__global__ void k_fine_apply_tab(Grid g, int nrhs, FineTab<T> F, T hinv, T alpha,
                                 const typename CT<T>::type* xi, const typename CT<T>::type* b,
                                 typename CT<T>::type* __restrict__ y, int mode, const int* il) {
  pdl_enter();
  typedef typename CT<T>::type C;
  const long long c0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long N = g.ncell;
  if (c0 >= N) return;
  const int c = (int)c0, item = il ? il[blockIdx.y] : blockIdx.y;
  const long long vo = (long long)item * (D + 1) * N, so = (long long)(item / nrhs) * N;
  const C* x = xi + vo;
  int i[3];
  cell_coords(g, c, i);
  C dsum = czero<C>();
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const long long o = (long long)k * N + c;
    C r = czero<C>();
    if (i[k] >= 1) {
      const C xc = *(x + o);
      C dg = __ldg(F.dg[k] + so + c);
      dg.y = fma(alpha, __ldg(F.rf[k] + so + c), dg.y);
      dsum = cadd(dsum, xc);
      const C off = off_row<T, D>(g, k, c, i, row_weights<T, D>(g, k, c, i, F, so), x, N, hinv, mode ? *(b + vo + o) : czero<C>());
      const C dx = cmulf<T>(dg, xc);
      r = mode ? csub(off, dx) : csub(dx, off);
    }
    if (i[k] + 1 < g.n[k]) dsum = csub(dsum, *(x + o + stride_of(g, k)));
    y[vo + o] = r;
  }
  const long long o = (long long)D * N + c;
  C r = rfma(-__ldg(F.kap + so + c), *(x + o), czero<C>());
  r = rfma(hinv, dsum, r);
  if (mode) r = csub(*(b + vo + o), r);
  y[vo + o] = r;
}

}  // namespace

template <typename T>
void launch_fine_tab(const Grid& g, int nsets, const Coef4<double>* cf, double h, double alpha, const FineTab<T>& F,
                     cudaStream_t s) {
  const dim3 gr((unsigned)((g.ncell + 127) / 128), nsets);
  const double h2 = 1.0 / (h * h);
  if (g.d == 2) {
    k_fine_tab_faces<T, 2><<<gr, 128, 0, s>>>(g, cf, h2, alpha, F);
    k_fine_tab_schur<T, 2><<<gr, 128, 0, s>>>(g, cf, h2, F);
  } else {
    k_fine_tab_faces<T, 3><<<gr, 128, 0, s>>>(g, cf, h2, alpha, F);
    k_fine_tab_schur<T, 3><<<gr, 128, 0, s>>>(g, cf, h2, F);
  }
}

template <typename T>
void launch_fine_vanka_tab(const Grid& g, int items, int nrhs, const FineTab<T>& F, double h, T wu, T wp, int colour,
                           const typename CT<T>::type* b, const typename CT<T>::type* xi, typename CT<T>::type* xo,
                           cudaStream_t s) {
  const int bs = spread_bs(g.ncell / 2, items, 128);
  const dim3 gr((unsigned)((g.ncell / 2 + bs - 1) / bs), sel_items(items));
  const T hinv = (T)(1.0 / h);
  if (g.d == 2) launch_pdl(gr, bs, 0, s, k_fine_vanka_tab<T, 2>, g, nrhs, F, hinv, wu, wp, colour, b, xi, xo, g_sel.list);
  else launch_pdl(gr, bs, 0, s, k_fine_vanka_tab<T, 3>, g, nrhs, F, hinv, wu, wp, colour, b, xi, xo, g_sel.list);
}

void launch_fine_apply_tab(const Grid& g, int items, int nrhs, const FineTab<double>& F, double h, double alpha,
                           const double2* x, const double2* b, double2* y, int mode, cudaStream_t s) {
  const int bs = spread_bs(g.ncell, items, 128);
  const dim3 gr((unsigned)((g.ncell + bs - 1) / bs), sel_items(items));
  const double hinv = 1.0 / h;
  if (g.d == 2) launch_pdl(gr, bs, 0, s, k_fine_apply_tab<double, 2>, g, nrhs, F, hinv, alpha, x, b, y, mode, g_sel.list);
  else launch_pdl(gr, bs, 0, s, k_fine_apply_tab<double, 3>, g, nrhs, F, hinv, alpha, x, b, y, mode, g_sel.list);
}

#define INST(T)                                                                                                       \
  template void launch_fine_tab<T>(const Grid&, int, const Coef4<double>*, double, double, const FineTab<T>&,           \
                                   cudaStream_t);                                                                      \
  template void launch_fine_vanka_tab<T>(const Grid&, int, int, const FineTab<T>&, double, T, T, int,                   \
                                         const CT<T>::type*, const CT<T>::type*, CT<T>::type*, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace ehs
