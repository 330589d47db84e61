// Galerkin-level kernels for levels too small (or rows too long) for one thread per
// row: a row's sum is split over several warps.
//
// A row of a Galerkin operator has 29 to 45 coefficients in 2D and up to 285 in 3D.
// With one thread per row (k_stencil_rows.cu) a 64^2 or 16^3 level is a few thousand
// threads that each wait for a long chain of loads.  Here a block covers 32 rows (lane =
// cell), each of its NS warps sums a share of the coefficients, and the partial sums
// meet in shared memory.  In 2D a warp takes the slots of one residue modulo NS, unrolled
// at compile time.  In 3D the unrolled rows are 50 KB of code each that a small level runs
// once, and fetching it is what bounds it (16^3, complex64 table: 40 us with one thread
// per row, 33 us with the unrolled rows split over 8 warps); there a warp loops over
// lines of the stencil box (up to 5 coefficients along x) described in constant memory:
// 12 us, 24^3 101 -> 27 us.
//
// k_st_rows_split: y = A x or b - A x, as k_st_rows.
// k_st_colour (2D): one colour of the red-black economic cell relaxation in one launch.
//   A colour's cells own their faces (every face belongs to exactly one cell of each
//   colour), so the residual rows a cell needs are needed by no other cell of that
//   colour: NS warps per block row form them, and the block's first warp solves the
//   cell's arrowhead block (eq. RelaxationMatrix) from shared memory, with its
//   coefficients loaded before the rows are summed.  The residual never goes through
//   memory and the second launch goes (64^2, complex64: a whole sweep 24.6 -> 12.4 us,
//   its launches included).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "kernels.h"
#include "stencil_rows.cuh"

namespace ehs {
namespace {

// A stencil line of a 3D row: the coefficients at x offsets ox0 .. ox0 + len - 1 of column component b and
// offsets oy, oz, in slots slot0, slot0 + 1, ...
struct Line {
  int slot0, b, ox0, len, oy, oz;
};
constexpr int MAXLINE = 224, MAXLEN = 5;
struct LineTab {
  int first[5];      // lines of row a: first[a] .. first[a + 1] - 1
  Line l[MAXLINE];
};
__host__ __device__ constexpr LineTab make_lines(int lv) {
  const StencilLayout L = level_layout(3, lv);
  LineTab T{};
  int n = 0;
  for (int a = 0; a <= 3; ++a) {
    T.first[a] = n;
    for (int q = L.row_first[a]; q < L.row_first[a + 1]; ++q) {
      const PairBox& P = L.p[q];
      for (int z = 0; z < P.ext[2]; ++z)
        for (int y = 0; y < P.ext[1]; ++y)
          T.l[n++] = Line{P.base + (z * P.ext[1] + y) * P.ext[0], P.b, P.lo[0], P.ext[0], P.lo[1] + y, P.lo[2] + z};
    }
  }
  T.first[4] = n;
  return T;
}
__host__ __device__ constexpr bool lines_ok(const LineTab& T) {
  for (int l = 0; l < T.first[4]; ++l)
    if (T.l[l].len < 1 || T.l[l].len > MAXLEN) return false;
  return T.first[4] <= MAXLINE;
}
static_assert(lines_ok(make_lines(1)) && lines_ok(make_lines(2)), "line tables");
__constant__ LineTab kLines[2] = {make_lines(1), make_lines(2)};   // level 1, level 2 on

// lines part, part + NS, ... of row a at cell c for NI vectors: a loop over the lines (read from constant memory, the
// same for the whole warp), each line's loads in flight together
template <typename T, typename TT, int NS, int NI>
__device__ __forceinline__ void row_lines(const Grid& g, const LineTab& LT, const TT* __restrict__ ts, long long c,
                                          const int i[3], const typename CT<T>::type* const (&x)[NI], int a, int part,
                                          typename CT<T>::type (&y)[NI]) {
  typedef typename CT<T>::type Cx;
  const long long N = g.ncell, sy = g.n[0], sz = (long long)g.n[0] * g.n[1];
#pragma unroll
  for (int q = 0; q < NI; ++q) y[q] = czero<Cx>();
#pragma unroll 2
  for (int l = LT.first[a] + part; l < LT.first[a + 1]; l += NS) {
    const Line& R = LT.l[l];
    const int jy = i[1] + R.oy, jz = i[2] + R.oz, jx = i[0] + R.ox0;
    const bool rin = jy >= 0 && jy < g.n[1] && jz >= 0 && jz < g.n[2];
    const long long xo = R.b * N + (c + R.oz * sz + R.oy * sy + R.ox0);
    const TT* tp = ts + R.slot0 * N + c;
    Cx tv[MAXLEN], xv[NI][MAXLEN];
#pragma unroll
    for (int k = 0; k < MAXLEN; ++k) {
      tv[k] = czero<Cx>();
#pragma unroll
      for (int q = 0; q < NI; ++q) xv[q][k] = czero<Cx>();
      if (k < R.len && rin && jx + k >= 0 && jx + k < g.n[0]) {
        tv[k] = ldtab<T>(tp + k * N);
#pragma unroll
        for (int q = 0; q < NI; ++q) xv[q][k] = x[q][xo + k];
      }
    }
#pragma unroll
    for (int k = 0; k < MAXLEN; ++k)
#pragma unroll
      for (int q = 0; q < NI; ++q) y[q] = cfma(tv[k], xv[q][k], y[q]);
  }
}

// the share `part` of NS of row a at cell c, unrolled (2D)
template <typename T, typename TT, int LV, bool SYM, int NS, int A, int SI = 0>
__device__ __forceinline__ typename CT<T>::type row_part(const Grid& g, const TT* ts, long long c, const int i[3],
                                                         const typename CT<T>::type* x, int part) {
  if constexpr (SI < NS) {
    if (part == SI) return st_row_ct<T, TT, 2, LV, SYM, A, false, NS, SI>(g, ts, c, i, x);
    return row_part<T, TT, LV, SYM, NS, A, SI + 1>(g, ts, c, i, x, part);
  } else {
    return czero<typename CT<T>::type>();
  }
}
template <typename T, typename TT, int LV, bool SYM, int NS>
__device__ __forceinline__ typename CT<T>::type row_share(const Grid& g, const TT* ts, long long c, const int i[3],
                                                          const typename CT<T>::type* x, int a, int part) {
  if (a == 0) return row_part<T, TT, LV, SYM, NS, 0>(g, ts, c, i, x, part);
  if (a == 1) return row_part<T, TT, LV, SYM, NS, 1>(g, ts, c, i, x, part);
  return row_part<T, TT, LV, SYM, NS, 2>(g, ts, c, i, x, part);
}

template <typename T, typename TT, int D, int LV, bool SYM, int NS>
__global__ void __launch_bounds__(32 * NS) k_st_rows_split(Grid g, int nit, int nrhs, const TT* __restrict__ tab,
                                                           const typename CT<T>::type* x,
                                                           const typename CT<T>::type* b,
                                                           typename CT<T>::type* __restrict__ y, int mode, int colour,
                                                           const int* il) {
  pdl_enter();
  typedef typename CT<T>::type Cx;
  constexpr StencilLayout L = level_layout(D, LV);
  constexpr int nslot = SYM ? half_base(L, L.npair) : L.nslot;
  __shared__ Cx sp[NS][32];
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5, a = blockIdx.z;
  const unsigned blk = blockIdx.x / (unsigned)nit, it = blockIdx.x - blk * (unsigned)nit;
  const long long c = (long long)blk * 32 + lane, N = g.ncell;
  const int item = il ? il[it] : it;
  const long long vo = (long long)item * (D + 1) * N;
  const TT* ts = tab + (long long)(item / nrhs) * nslot * N;
  int i[3] = {0, 0, 0};
  bool run = c < N;
  if (run) {
    cell_coords(g, c, i);
    run = !(a == D && colour >= 0 && ((i[0] + i[1] + i[2]) & 1) != colour);
  }
  const bool row = run && slot_valid(a, D, i);
  sp[part][lane] = row ? row_share<T, TT, LV, SYM, NS>(g, ts, c, i, x + vo, a, part) : czero<Cx>();
  __syncthreads();
  if (part || !run) return;
  Cx r = sp[0][lane];
#pragma unroll
  for (int q = 1; q < NS; ++q) r = cadd(r, sp[q][lane]);
  if (mode && row) r = csub(*(b + vo + (long long)a * N + c), r);
  y[vo + (long long)a * N + c] = r;
}

// The 3D form: NI items of the list per block, one read of the table for all of them where they are of one medium
// (its coefficients are nine tenths of the bytes; 64^3, complex64 tables, two sources, mean of levels 1 and 2: 43 us with an
// item a block, the table read once per item -> 30 us).  The FP64 form keeps an item a block: its pipe bounds it, not the
// table (16^3 from level 2 on, three items: 94 us, 143 with two items a block).
template <typename T, typename TT, int LV, int NS, int NI>
__global__ void __launch_bounds__(32 * NS) k_st_rows_split3(Grid g, int nit, int nrhs, const TT* __restrict__ tab,
                                                            const typename CT<T>::type* x,
                                                            const typename CT<T>::type* b,
                                                            typename CT<T>::type* __restrict__ y, int mode, int colour,
                                                            const int* il) {
  pdl_enter();
  typedef typename CT<T>::type Cx;
  constexpr int nslot = level_layout(3, LV).nslot;
  __shared__ Cx sp[NI][NS][32];
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5, a = blockIdx.z;
  const unsigned ng = (nit + NI - 1) / NI, blk = blockIdx.x / ng, it0 = (blockIdx.x - blk * ng) * NI;
  const long long c = (long long)blk * 32 + lane, N = g.ncell;
  int item[NI], live = 0;
  bool same = true;
#pragma unroll
  for (int q = 0; q < NI; ++q) {
    item[q] = item[0];
    if ((int)it0 + q < nit) { item[q] = il ? il[it0 + q] : it0 + q; ++live; }
    same = same && item[q] / nrhs == item[0] / nrhs;
  }
  int i[3] = {0, 0, 0};
  bool run = c < N;
  if (run) {
    cell_coords(g, c, i);
    run = !(a == 3 && colour >= 0 && ((i[0] + i[1] + i[2]) & 1) != colour);
  }
  const bool row = run && slot_valid(a, 3, i);
  const Cx* xs[NI];
#pragma unroll
  for (int q = 0; q < NI; ++q) xs[q] = x + (long long)item[q] * 4 * N;
  Cx v[NI];
#pragma unroll
  for (int q = 0; q < NI; ++q) v[q] = czero<Cx>();
  if (row) {
    if (same) {
      row_lines<T, TT, NS, NI>(g, kLines[LV - 1], tab + (long long)(item[0] / nrhs) * nslot * N, c, i, xs, a, part, v);
    } else {
      for (int q = 0; q < live; ++q) {
        const Cx* x1[1] = {x + (long long)item[q] * 4 * N};
        Cx y1[1];
        row_lines<T, TT, NS, 1>(g, kLines[LV - 1], tab + (long long)(item[q] / nrhs) * nslot * N, c, i, x1, a, part, y1);
#pragma unroll
        for (int p = 0; p < NI; ++p)
          if (p == q) v[p] = y1[0];
      }
    }
  }
#pragma unroll
  for (int q = 0; q < NI; ++q) sp[q][part][lane] = v[q];
  __syncthreads();
  if (part >= live || !run) return;      // warp q finishes item q
  Cx r = sp[part][0][lane];
#pragma unroll
  for (int q = 1; q < NS; ++q) r = cadd(r, sp[part][q][lane]);
  int it = item[0];
#pragma unroll
  for (int q = 1; q < NI; ++q)
    if (part == q) it = item[q];
  const long long o = ((long long)it * 4 + a) * N + c;
  if (mode && row) r = csub(b[o], r);
  y[o] = r;
}

template <typename T, typename TT, int LV, bool SYM, int NS>
__global__ void __launch_bounds__(32 * 5 * NS) k_st_colour(Grid g, int nit, int nrhs, const TT* __restrict__ tab,
                                                           const typename CT<T>::type* __restrict__ vtab,
                                                           T wu, T wp, int colour,
                                                           const typename CT<T>::type* b,
                                                           const typename CT<T>::type* xi,
                                                           typename CT<T>::type* __restrict__ xo,
                                                           const int* il) {
  pdl_trigger();
  typedef typename CT<T>::type Cx;
  constexpr int D = 2;
  constexpr StencilLayout L = level_layout(D, LV);
  constexpr int NB = 2 * D + 1;
  __shared__ Cx sp[NB][NS][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, row = wid / NS, part = wid % NS;
  const unsigned blk = blockIdx.x / (unsigned)nit, it = blockIdx.x - blk * (unsigned)nit;
  const long long t = (long long)blk * 32 + lane, N = g.ncell;
  const int item = il ? il[it] : it;
  const long long vo = (long long)item * (D + 1) * N;
  constexpr int nslot = SYM ? half_base(L, L.npair) : L.nslot;
  const TT* ts = tab + (long long)(item / nrhs) * nslot * N;
  const Cx* x = xi + vo;
  const bool live = t < N / 2;
  long long c = 2 * t;
  int i[3] = {0, 0, 0};
  if (live) {
    cell_coords(g, c, i);
    if (((i[0] + i[1] + i[2]) & 1) != colour) { ++c; ++i[0]; }
  }
  // the first warp: block coefficients (setup-time data, before the wait), then right-hand sides and the old
  // iterate, in flight while the rows are summed
  const Cx* vt = vtab + (long long)(item / nrhs) * (D + 1) * N;
  Cx r[NB], dinv[2 * D], gr[2 * D], gc[2 * D], sinv = czero<Cx>(), xv[NB], po = czero<Cx>();
  bool ok[2 * D];
  const long long co = (c & 1) ? c - 1 : c + 1;
  if (wid == 0 && live) {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      ok[k] = i[k] >= 1;
      ok[D + k] = i[k] + 1 < g.n[k];
    }
    vupd_coefs<T, TT, D, LV, SYM, 0>(ts, vt, N, c, stride_of(g, 0), ok[0], ok[D], dinv, gr, gc);
    vupd_coefs<T, TT, D, LV, SYM, 1>(ts, vt, N, c, stride_of(g, 1), ok[1], ok[D + 1], dinv, gr, gc);
    sinv = __ldg(vt + (long long)D * N + c);
  }
  pdl_wait();
  if (wid == 0 && live) {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const long long lo = (long long)k * N + c, hi = lo + stride_of(g, k);
      if (ok[k]) { r[k] = b[vo + lo]; xv[k] = x[lo]; }
      if (ok[D + k]) { r[D + k] = b[vo + hi]; xv[D + k] = x[hi]; }
    }
    r[2 * D] = b[vo + (long long)D * N + c];
    xv[2 * D] = x[(long long)D * N + c];
    po = x[(long long)D * N + co];
  }
  {  // this warp's share of one row of the cell's block
    const int k = row % D;
    const bool high = row >= D && row < 2 * D;
    int ir[3] = {i[0], i[1], i[2]};
    long long cr = c;
    bool in = live;
    if (row < 2 * D) {
      if (high) { ir[k] += 1; cr += stride_of(g, k); }
      in = in && ir[k] >= 1 && ir[k] < g.n[k];
    }
    sp[row][part][lane] =
        in ? row_share<T, TT, LV, SYM, NS>(g, ts, cr, ir, x, row < 2 * D ? k : D, part) : czero<Cx>();
  }
  __syncthreads();
  if (wid || !live) return;
  Cx* xout = xo + vo;
  xout[(long long)D * N + co] = po;
  Cx rp = r[2 * D];
#pragma unroll
  for (int a = 0; a < NB; ++a) {
    Cx s = sp[a][0][lane];
#pragma unroll
    for (int q = 1; q < NS; ++q) s = cadd(s, sp[a][q][lane]);
    if (a == 2 * D) rp = csub(rp, s);
    else if (ok[a]) r[a] = csub(r[a], s);
  }
#pragma unroll
  for (int a = 0; a < 2 * D; ++a)
    if (ok[a]) rp = csub(rp, cmul(cmul(gc[a], dinv[a]), r[a]));
  const Cx dp = cmul(rp, sinv);
  xout[(long long)D * N + c] = cfma(mk<T>(wp, 0), dp, xv[2 * D]);
#pragma unroll
  for (int a = 0; a < 2 * D; ++a) {
    if (!ok[a]) continue;
    const int k = a % D;
    const long long idx = (long long)k * N + c + (a >= D ? stride_of(g, k) : 0);
    const Cx du = cmul(csub(r[a], cmul(gr[a], dp)), dinv[a]);
    xout[idx] = cfma(mk<T>(wu, 0), du, xv[a]);
  }
}

// 3D MG-DD colour residual at the box unknowns, as k_st_resid_gather (k_stencil.cu; 2D), with 8 warps
// looping over the lines of 32 unknowns' rows: the unrolled rows were bound by fetching their code (one box of
// 8^3 coarsest cells, 36 us).
template <typename T, typename TT, int LV>
__global__ void __launch_bounds__(256) k_st_gather3(Grid g, int nrhs, int nsub, int nloc, const int* __restrict__ map,
                                                    const TT* __restrict__ tab,
                                                    const typename CT<T>::type* x,
                                                    const typename CT<T>::type* b,
                                                    typename CT<T>::type* __restrict__ out,
                                                    const int* il) {
  pdl_enter();
  typedef typename CT<T>::type Cx;
  constexpr int nslot = level_layout(3, LV).nslot;
  constexpr int NS = 8;
  __shared__ Cx sp[NS][32];
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  const int bl = il ? il[blockIdx.y] : blockIdx.y;
  const int r = bl % nrhs, s = (bl / nrhs) % nsub, m = bl / (nrhs * nsub);
  const long long N = g.ncell, vo = (long long)(m * nrhs + r) * 4 * N;
  const int gs = e < nloc ? map[(long long)s * nloc + e] : -1;
  Cx v = czero<Cx>();
  if (gs >= 0) {
    const int a = gs / (int)N, c = gs - a * (int)N;
    int i[3];
    cell_coords(g, c, i);
    const Cx* xs[1] = {x + vo};
    Cx y[1];
    row_lines<T, TT, NS, 1>(g, kLines[LV - 1], tab + (long long)m * nslot * N, c, i, xs, a, part, y);
    v = y[0];
  }
  sp[part][lane] = v;
  __syncthreads();
  if (part || e >= nloc) return;
#pragma unroll
  for (int q = 1; q < NS; ++q) v = cadd(v, sp[q][lane]);
  if (gs >= 0) v = csub(*(b + vo + gs), v);
  out[(long long)bl * nloc + e] = v;
}

// warps per row
template <int D> struct Ns;
template <> struct Ns<2> { static const int rows = 4, colour = 2; };
template <> struct Ns<3> { static const int rows = 8; };

// dispatch on dimension, layout variant and table storage (st_apply_any in k_stencil_rows.cu: half
// formats are stored half by symmetry in 2D, whole in 3D)
#define EHS_ST_FORMATS(FN, ...)                                                                       \
  do {                                                                                                \
    if constexpr (sizeof(T) == 4) {                                                                   \
      if (fmt == 1 && g.d == 2) return FN<T, __half2, true>(v, (const __half2*)tab, __VA_ARGS__);     \
      if (fmt == 2 && g.d == 2)                                                                       \
        return FN<T, __nv_bfloat162, true>(v, (const __nv_bfloat162*)tab, __VA_ARGS__);               \
      if (fmt == 1) return FN<T, __half2, false>(v, (const __half2*)tab, __VA_ARGS__);                \
      if (fmt == 2) return FN<T, __nv_bfloat162, false>(v, (const __nv_bfloat162*)tab, __VA_ARGS__);  \
    }                                                                                                 \
    FN<T, typename CT<T>::type, false>(v, (const typename CT<T>::type*)tab, __VA_ARGS__);             \
  } while (0)

template <typename T, typename TT, int D, int LV, bool SYM>
void rows_split_t(const Grid& g, int items, int nrhs, const TT* tab, const typename CT<T>::type* x,
                  const typename CT<T>::type* b, typename CT<T>::type* y, int mode, int colour, cudaStream_t s) {
  constexpr int NS = Ns<D>::rows;
  const int nit = (int)sel_items(items);
  const unsigned nb = (unsigned)((g.ncell + 31) / 32);
  if constexpr (D == 3) {
    if constexpr (sizeof(T) == 4) {
      if (nrhs > 1) {
        launch_pdl(dim3(nb * ((nit + 1) / 2), 1, 4), 32 * NS, 0, s, k_st_rows_split3<T, TT, LV, NS, 2>, g, nit, nrhs,
                   tab, x, b, y, mode, colour, g_sel.list);
        return;
      }
    }
    launch_pdl(dim3(nb * nit, 1, 4), 32 * NS, 0, s, k_st_rows_split3<T, TT, LV, NS, 1>, g, nit, nrhs, tab, x, b, y, mode,
               colour, g_sel.list);
  } else {
    launch_pdl(dim3(nb * nit, 1, 3), 32 * NS, 0, s, k_st_rows_split<T, TT, D, LV, SYM, NS>, g, nit, nrhs, tab, x, b, y,
               mode, colour, g_sel.list);
  }
}
template <typename T, typename TT, bool SYM>
void rows_split_d(int v, const TT* tab, const Grid& g, int items, int nrhs, const typename CT<T>::type* x,
                  const typename CT<T>::type* b, typename CT<T>::type* y, int mode, int colour, cudaStream_t s) {
  if (g.d == 2) {
    if (v == 1) rows_split_t<T, TT, 2, 1, SYM>(g, items, nrhs, tab, x, b, y, mode, colour, s);
    else rows_split_t<T, TT, 2, 2, SYM>(g, items, nrhs, tab, x, b, y, mode, colour, s);
  } else if constexpr (!SYM) {
    if (v == 1) rows_split_t<T, TT, 3, 1, SYM>(g, items, nrhs, tab, x, b, y, mode, colour, s);
    else rows_split_t<T, TT, 3, 2, SYM>(g, items, nrhs, tab, x, b, y, mode, colour, s);
  }
}
template <typename T, typename TT, bool SYM>
void gather3_d(int v, const TT* tab, const Grid& g, int items_l, int nrhs, int nsub, int nloc, const int* map,
               const typename CT<T>::type* x, const typename CT<T>::type* b, typename CT<T>::type* out, cudaStream_t s) {
  if constexpr (!SYM) {
    const dim3 gr((unsigned)((nloc + 31) / 32), sel_items(items_l));
    if (v == 1) launch_pdl(gr, 256, 0, s, k_st_gather3<T, TT, 1>, g, nrhs, nsub, nloc, map, tab, x, b, out, g_sel.list);
    else launch_pdl(gr, 256, 0, s, k_st_gather3<T, TT, 2>, g, nrhs, nsub, nloc, map, tab, x, b, out, g_sel.list);
  }
}
template <typename TT, int LV, bool SYM>
void colour_t(const Grid& g, int items, int nrhs, const TT* tab, const float2* vt, float wu, float wp, int colour, const float2* b,
              const float2* xi, float2* xo, cudaStream_t s) {
  constexpr int NS = Ns<2>::colour;
  const int nit = (int)sel_items(items);
  const dim3 gr((unsigned)((g.ncell / 2 + 31) / 32) * nit);
  launch_pdl(gr, 32 * 5 * NS, 0, s, k_st_colour<float, TT, LV, SYM, NS>, g, nit, nrhs, tab, vt, wu, wp, colour, b, xi, xo,
                                                                    g_sel.list);
}
template <typename T, typename TT, bool SYM>
void colour_d(int v, const TT* tab, const Grid& g, int items, int nrhs, const float2* vt, float wu, float wp, int colour,
              const float2* b, const float2* xi, float2* xo, cudaStream_t s) {
  if (v == 1) colour_t<TT, 1, SYM>(g, items, nrhs, tab, vt, wu, wp, colour, b, xi, xo, s);
  else colour_t<TT, 2, SYM>(g, items, nrhs, tab, vt, wu, wp, colour, b, xi, xo, s);
}

}  // namespace

// Where the split rows are the faster ones, by the cells of the whole batch (the context's items, so that a
// batch keeps its summation order while items converge).  us per residual pass, one thread per row -> split:
//   2D, 128^2: 8.4 -> 6.3 (complex64 table, level 1), 12.7 -> 8.4 (level 2 on), 6.3 -> 6.2 (FP16 half table);
//   32^2: 6.4 -> 4.2; above, 256^2: 8.5 -> 12.5
//   3D, from level 2 on: every size measured (16^3 40 -> 12, two items of 24^3 158 -> 43, FP16 tables 62 -> 39);
//   3D, level 1 (rows half as long): 16^3 21 -> 8, 32^3 with complex64 tables 52 -> 35 and two items 66 -> 62, but
//   with FP16 tables 21 -> 31; 48^3 97 -> 105; an odd batch fills only half of its last pair of items (three of
//   24 x 20 x 28: 25 -> 29).  FP64: 16^3 39 -> 27, but two items 41 -> 44, 24 x 20 x 28 64 -> 64, 32^3 128 -> 149.
// and a sweep of the 2D complex64 cycle with one launch per colour instead of two: 128^2 24.8 -> 16.9 us (complex64
// table), 28.9 -> 20.4 (FP16, level 2 on), 64^2 24.8 -> 12.4; not at 256^2 (31 -> 33 to 50) nor for 16 items of 64^2
// (40 -> 49).  The FP64 cycle keeps two launches (53 -> 62 at 128^2: one warp of the block would do all of the
// block solve's FP64 arithmetic).
bool st_split(const Grid& g, int items, int nrhs, int v, int fmt, bool fp64) {
  const long long cells = (long long)items * g.ncell;
  if (g.d == 2) return cells <= 16384;
  return v != 1 || cells <= (fp64 ? 4096 : fmt ? 16384 : nrhs > 1 && nrhs % 2 ? 32768 : 65536);
}
template <typename T>
void launch_st_rows_split(const Grid& g, int items, int nrhs, int v, const void* tab, int fmt,
                          const typename CT<T>::type* x, const typename CT<T>::type* b, typename CT<T>::type* y,
                          int mode, int colour, cudaStream_t s) {
  EHS_ST_FORMATS(rows_split_d, g, items, nrhs, x, b, y, mode, colour, s);
}
void launch_st_colour(const Grid& g, int items, int nrhs, int v, const void* tab, int fmt, const float2* vt, float wu,
                      float wp, int colour, const float2* b, const float2* xi, float2* xo, cudaStream_t s) {
  typedef float T;
  EHS_ST_FORMATS(colour_d, g, items, nrhs, vt, wu, wp, colour, b, xi, xo, s);
}

template <typename T>
void launch_st_gather3(const Grid& g, int items_l, int nrhs, int nsub, int nloc, const int* map, int v, const void* tab,
                       int fmt, const typename CT<T>::type* x, const typename CT<T>::type* b,
                       typename CT<T>::type* out, cudaStream_t s) {
  EHS_ST_FORMATS(gather3_d, g, items_l, nrhs, nsub, nloc, map, x, b, out, s);
}

#define INST(T)                                                                                                \
  template void launch_st_gather3<T>(const Grid&, int, int, int, int, const int*, int, const void*, int,         \
                                     const CT<T>::type*, const CT<T>::type*, CT<T>::type*, cudaStream_t);       \
  template void launch_st_rows_split<T>(const Grid&, int, int, int, const void*, int, const CT<T>::type*,        \
                                        const CT<T>::type*, CT<T>::type*, int, int, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace ehs
