// Coarsest level: the Galerkin operator is assembled densely, inverted once in
// FP64 at setup (k_invert.cu), and every cycle applies
// the stored inverse (Algorithm TwoCycle step 3 solved exactly, as the paper's
// coarsest LU does).  Boundary slots are identity rows so the dense index is
// simply comp * ncell + cell.
//
// The matrices are assembled equilibrated, D A D with D a diagonal of powers of two (k_dense_scale), and the
// inverse is scaled back by D from both sides (k_invert.cu): exact scalings, and what is inverted no longer depends
// on the units of the medium.  Displacements and pressures differ in scale by sqrt(mu (lambda + mu)) / h, near 1
// in km, km/s and g/cm^3 with h = 1 and about 2^30 in SI units with h = 10 m, and the inverse's digits hold the entries of a
// row to 2^-55 of the largest: without D the inverse of an SI medium (12 x 14 coarsest cells) is off by 2.7e-8, with
// it by 1.3e-15 (numpy restatement; FP64 elimination column by column 2.9e-15).
//
// MG-DD (Sec. 4): the same machinery for the subdomains of the coarsest grid.
// Each box's local matrix (the coarsest operator restricted to the box
// unknowns, padded with identity rows to nloc) is assembled from the stencil
// table and inverted in FP64 together with the others; per colour one launch
// multiplies every subdomain's stored inverse (double-float, complex64, FP16
// or BF16 pairs) with its local residuals, skipping the padding rows.
#include "kernels.h"
#include "dense_rows.cuh"

namespace ehs {
namespace {

// floor(log2 of the larger part), NONE for zero (and what is below the normal range)
constexpr int NONE = -8192;
__device__ __forceinline__ int exponent(double2 v) {
  const int h = max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff) >> 20;
  return h ? h - 1023 : NONE;
}

// Exponents ex of the equilibration D (d = 2^ex) of the coarsest unknowns, [nsets][(D + 1) ncell].  Displacements
// (pass 0): the largest entry of the row towards its own component, of size about one after scaling (the diagonal
// alone may cancel between stiffness and mass).  Pressures (pass 1): half of the same, so that pivots stay on the
// diagonal (error of the inverse in km units 1.1e-15, 2.9e-15 without that half), but no larger than what leaves the
// largest coupling to a scaled displacement in [2, 4): a nearly incompressible medium, whose pressure diagonal is
// tiny, keeps its displacement block (lambda / mu = 1e6: 2.4e-15, 6.9e-14 from the diagonal alone, and a pressure block
// ten times worse with the coupling in [1/2, 1)).  A thread per row, once per context.
template <int D>
__global__ void k_dense_scale(Grid g, StencilLayout L, const double2* __restrict__ tab, int* ex, int pass) {
  const long long N = (long long)(D + 1) * g.ncell;
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= N) return;
  const int a = (int)(r / g.ncell);
  if ((a == D) != (pass == 1)) return;
  const double2* ts = tab + (long long)blockIdx.y * L.nslot * g.ncell;
  int* es = ex + (long long)blockIdx.y * N;
  const long long c = r % g.ncell;
  int i[3];
  cell_coords(g, c, i);
  if (!slot_valid(a, D, i)) { es[r] = 0; return; }
  int own = NONE, coup = NONE;
  for (int q = L.row_first[a]; q < L.row_first[a + 1]; ++q) {
    const PairBox& P = L.p[q];
    if (P.b != a && a != D) continue;
    int s = P.base;
    for (int oz = 0; oz < P.ext[2]; ++oz)
      for (int oy = 0; oy < P.ext[1]; ++oy)
        for (int ox = 0; ox < P.ext[0]; ++ox, ++s) {
          const int j[3] = {i[0] + P.lo[0] + ox, i[1] + P.lo[1] + oy, i[2] + P.lo[2] + oz};
          bool in = true;
          for (int k = 0; k < 3; ++k) in = in && j[k] >= 0 && j[k] < g.n[k];
          if (!in || !slot_valid(P.b, D, j)) continue;
          const int e = exponent(ts[(long long)s * g.ncell + c]);
          if (e == NONE) continue;
          if (P.b == a) own = max(own, e);
          else coup = max(coup, e + es[(long long)P.b * g.ncell + cell_index(g, j)]);
        }
  }
  int e = own == NONE ? 0 : -((own + 1) >> 1);
  if (a == D) {
    e -= 1;
    if (coup != NONE) e = own == NONE ? 1 - coup : min(e, 1 - coup);
  }
  es[r] = e;
}

// A: D K_c D, zeroed before
template <int D>
__global__ void k_dense_assemble(Grid g, StencilLayout L, const double2* __restrict__ tab, const int* __restrict__ ex,
                                 double2* __restrict__ A) {
  const long long N = (long long)(D + 1) * g.ncell;
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= N) return;
  const int set = blockIdx.y;
  const double2* ts = tab + (long long)set * L.nslot * g.ncell;
  const int* es = ex + (long long)set * N;
  double2* row = A + ((long long)set * N + r) * N;
  const int a = (int)(r / g.ncell);
  const long long c = r % g.ncell;
  int i[3];
  cell_coords(g, c, i);
  if (!slot_valid(a, D, i)) { row[r] = make_double2(1, 0); return; }
  for (int q = L.row_first[a]; q < L.row_first[a + 1]; ++q) {
    const PairBox& P = L.p[q];
    int s = P.base;
    for (int oz = 0; oz < P.ext[2]; ++oz)
      for (int oy = 0; oy < P.ext[1]; ++oy)
        for (int ox = 0; ox < P.ext[0]; ++ox, ++s) {
          const int j[3] = {i[0] + P.lo[0] + ox, i[1] + P.lo[1] + oy, i[2] + P.lo[2] + oz};
          bool in = true;
          for (int k = 0; k < 3; ++k) in = in && j[k] >= 0 && j[k] < g.n[k];
          if (!in || !slot_valid(P.b, D, j)) continue;
          const long long col = (long long)P.b * g.ncell + cell_index(g, j);
          const double2 v = pow2_scaled(ts[(long long)s * g.ncell + c], es[r] + es[col]);
          row[col].x += v.x;
          row[col].y += v.y;
        }
  }
}

// x = Ainv r, one warp per dense row; input/output in the working precision.  Bound by the FP64 pipe.  PLAIN: launched
// plainly, r read as data that does not change, so that the loop's loads run ahead (N = 3072 82 us, 123 with
// launch_pdl, 100 with four of its loads issued together by hand)
template <typename T, bool PLAIN>
__global__ void k_dense_apply(int N, int nrhs, const double2* __restrict__ inv,
                              const typename CT<T>::type* r,
                              typename CT<T>::type* __restrict__ x, const int* il) {
  pdl_enter();
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int item = il ? il[blockIdx.y] : blockIdx.y;
  if (warp >= N) return;
  const double2* row = inv + ((long long)(item / nrhs) * N + warp) * N;
  const typename CT<T>::type* rv = r + (long long)item * N;
  double sx = 0.0, sy = 0.0;
  for (int j = lane; j < N; j += 32) {
    const double2 a = __ldg(row + j);
    const typename CT<T>::type b = ld_vec<PLAIN>(rv + j);
    sx = fma(a.x, (double)b.x, fma(-a.y, (double)b.y, sx));
    sy = fma(a.x, (double)b.y, fma(a.y, (double)b.x, sy));
  }
  for (int o = 16; o > 0; o >>= 1) {
    sx += __shfl_xor_sync(0xffffffffu, sx, o);
    sy += __shfl_xor_sync(0xffffffffu, sy, o);
  }
  if (lane == 0) {
    typename CT<T>::type v;
    v.x = (T)sx; v.y = (T)sy;
    x[(long long)item * N + warp] = v;
  }
}

// MG-DD local problems (Sec. 4): row e of local matrix (set, s) is the
// coarsest-level row of global slot map[s][e], restricted to the columns that
// are local unknowns of subdomain s (g2l[s][slot] >= 0); padding rows (map -1)
// are identity rows.  A comes zeroed and goes out equilibrated, as for k_dense_assemble; exl: the
// exponents of its rows.
template <int D>
__global__ void k_dense_assemble_sub(Grid g, StencilLayout L, const double2* __restrict__ tab,
                                     const int* __restrict__ ex, int nsub, int nloc, const int* __restrict__ map,
                                     const int* __restrict__ g2l, double2* __restrict__ A, int* __restrict__ exl) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nloc) return;
  const int ms = blockIdx.y;                 // set * nsub + s
  const int set = ms / nsub, sub = ms % nsub;
  const long long NG = (long long)(D + 1) * g.ncell;
  const double2* ts = tab + (long long)set * L.nslot * g.ncell;
  double2* row = A + ((long long)ms * nloc + e) * nloc;
  const int gs = map[(long long)sub * nloc + e];
  if (gs < 0) { row[e] = make_double2(1, 0); exl[(long long)ms * nloc + e] = 0; return; }
  const int* es = ex + (long long)set * NG;
  exl[(long long)ms * nloc + e] = es[gs];
  const int* gl = g2l + (long long)sub * NG;
  const int a = (int)(gs / g.ncell);
  const long long c = gs % g.ncell;
  int i[3];
  cell_coords(g, c, i);
  for (int q = L.row_first[a]; q < L.row_first[a + 1]; ++q) {
    const PairBox& P = L.p[q];
    int sl = P.base;
    for (int oz = 0; oz < P.ext[2]; ++oz)
      for (int oy = 0; oy < P.ext[1]; ++oy)
        for (int ox = 0; ox < P.ext[0]; ++ox, ++sl) {
          const int j[3] = {i[0] + P.lo[0] + ox, i[1] + P.lo[1] + oy, i[2] + P.lo[2] + oz};
          bool in = true;
          for (int k = 0; k < 3; ++k) in = in && j[k] >= 0 && j[k] < g.n[k];
          if (!in || !slot_valid(P.b, D, j)) continue;
          const long long gc = (long long)P.b * g.ncell + cell_index(g, j);
          const int lc = gl[gc];
          if (lc < 0) continue;
          const double2 v = pow2_scaled(ts[(long long)sl * g.ncell + c], es[gs] + es[gc]);
          row[lc].x += v.x;
          row[lc].y += v.y;
        }
  }
}

// x = Ainv r with Ainv stored in complex64, FP16 or BF16 pairs (FP32
// accumulation); one warp per row, four independent loads in flight per lane

template <typename TI>
__global__ void k_dense_apply_lp(int N, int nrhs, const TI* __restrict__ inv, const float2* r,
                                 float2* __restrict__ x, const int* il) {
  pdl_enter();
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int item = il ? il[blockIdx.y] : blockIdx.y;
  if (warp >= N) return;
  const TI* row = inv + ((long long)(item / nrhs) * N + warp) * N;
  const float2* rv = r + (long long)item * N;
  float sx0 = 0.f, sy0 = 0.f, sx1 = 0.f, sy1 = 0.f;
  int j = lane;
  for (; j + 96 < N; j += 128) {
    const float2 a0 = ldlp(row + j), a1 = ldlp(row + j + 32), a2 = ldlp(row + j + 64), a3 = ldlp(row + j + 96);
    const float2 b0 = *(rv + j), b1 = *(rv + j + 32), b2 = *(rv + j + 64), b3 = *(rv + j + 96);
    sx0 = fmaf(a0.x, b0.x, fmaf(-a0.y, b0.y, sx0)); sy0 = fmaf(a0.x, b0.y, fmaf(a0.y, b0.x, sy0));
    sx1 = fmaf(a1.x, b1.x, fmaf(-a1.y, b1.y, sx1)); sy1 = fmaf(a1.x, b1.y, fmaf(a1.y, b1.x, sy1));
    sx0 = fmaf(a2.x, b2.x, fmaf(-a2.y, b2.y, sx0)); sy0 = fmaf(a2.x, b2.y, fmaf(a2.y, b2.x, sy0));
    sx1 = fmaf(a3.x, b3.x, fmaf(-a3.y, b3.y, sx1)); sy1 = fmaf(a3.x, b3.y, fmaf(a3.y, b3.x, sy1));
  }
  for (; j < N; j += 32) {
    const float2 a = ldlp(row + j), b = *(rv + j);
    sx0 = fmaf(a.x, b.x, fmaf(-a.y, b.y, sx0)); sy0 = fmaf(a.x, b.y, fmaf(a.y, b.x, sy0));
  }
  float sx = sx0 + sx1, sy = sy0 + sy1;
  for (int o = 16; o > 0; o >>= 1) {
    sx += __shfl_xor_sync(0xffffffffu, sx, o);
    sy += __shfl_xor_sync(0xffffffffu, sy, o);
  }
  if (lane == 0) x[(long long)item * N + warp] = make_float2(sx, sy);
}

// The same product with 16-byte loads (dense_rows4 in dense_rows.cuh): each warp
// computes 4 consecutive rows of the matrix set (item / nrhs), whose live size is
// sizes[set % nsub]; groups of rows at or beyond it are skipped.
template <typename TI>
__global__ void __launch_bounds__(256) k_dense_apply_v(int N, int nrhs, int nsub, const int* __restrict__ sizes,
                                                       const TI* __restrict__ inv, const float2* r,
                                                       float2* __restrict__ x, const int* il) {
  pdl_enter();
  const int row0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4;
  const int item = il ? il[blockIdx.y] : blockIdx.y;
  const int set = item / nrhs;
  const int n = sizes ? sizes[set % nsub] : N;
  if (row0 >= n) return;
  dense_rows4<TI>(N, n, row0, inv + (long long)set * N * N, r + (long long)item * N, x + (long long)item * N);
}

// The inverses are setup-time data, so a block that is resident while its predecessor still runs (launch_pdl: the
// colour's residual gather, latency-bound and nearly idle on HBM) asks for the first `pre` bytes of each of its
// rows before it waits.  The budget is 64 MB a launch over all its warps: half of L2, about what HBM delivers in
// the time of a gather.  In the 512^2 cycle (one medium, four
// colours) with the other kernels' early loads: 245 -> 239 us.
__device__ __forceinline__ void prefetch_rows(const void* row, long long row_bytes, int rows, int pre) {
  const int lane = threadIdx.x & 31;
  if (lane < rows && pre > 0) {
    const char* p = (const char*)row + lane * row_bytes;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(pre) : "memory");
  }
}

// The MG-DD form that also scatters: sub-item = ((m * nsub) + s) * nrhs + r, its four results
// added to the coarsest vector xg of item m * nrhs + r at the subdomain's unknowns map[s][row]
// (subdomains of one colour are disjoint, so no two threads add to the same entry).
template <typename TI>
__global__ void __launch_bounds__(256) k_dense_apply_vs(int N, int nrhs, int nsub, const int* __restrict__ sizes,
                                                        const TI* __restrict__ inv, const float2* r,
                                                        const int* __restrict__ map, long long NG, float2* xg,
                                                        const int* il, int pre) {
  pdl_trigger();
  const int row0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4;
  if (row0 < N) {
    // il may be from the launch before this one and not yet written: then it holds older items of the batch (zeros
    // from setup at first), and what is asked for early is of no use, no more
    const int early = il ? il[blockIdx.y] : blockIdx.y;
    prefetch_rows(inv + ((long long)(early / nrhs) * N + row0) * N, (long long)N * sizeof(TI), 4, pre);
  }
  pdl_wait();
  const int item = il ? il[blockIdx.y] : blockIdx.y;
  const int set = item / nrhs, sub = set % nsub;
  const int n = sizes[sub];
  if (row0 >= n) return;
  const long long gi = (long long)(set / nsub) * nrhs + item % nrhs;
  dense_rows4<TI, false, true>(N, n, row0, inv + (long long)set * N * N, r + (long long)item * N, nullptr,
                               map + (long long)sub * N, xg + gi * NG);
}

}  // namespace

bool launch_dense_apply_scatter(int N, int items, int nrhs, int nsub, const int* sizes, const void* inv, int fmt,
                                const float2* r, const int* map, long long NG, float2* xg, cudaStream_t s) {
  const int wpb = 8;
  const int E = fmt >= 2 ? 4 : 2;
  if (N % 4 != 0 || N % E != 0 || !sizes) return false;
  const dim3 gv((N / 4 + wpb - 1) / wpb, sel_items(items));   // a warp per 4 rows
  const long long row = (long long)N * (fmt >= 2 ? 4 : 8), share = (64ll << 20) / ((long long)gv.x * gv.y * wpb * 4);
  const int pre = (int)((share < row ? share : row) / 16 * 16);
  if (fmt == 2)
    launch_pdl(gv, 32 * wpb, 0, s, k_dense_apply_vs<__half2>, N, nrhs, nsub, sizes, (const __half2*)inv, r, map, NG, xg,
                                                       g_sel.list, pre);
  else if (fmt == 3)
    launch_pdl(gv, 32 * wpb, 0, s, k_dense_apply_vs<__nv_bfloat162>, N, nrhs, nsub, sizes, (const __nv_bfloat162*)inv, r, map,
                                                              NG, xg, g_sel.list, pre);
  else
    launch_pdl(gv, 32 * wpb, 0, s, k_dense_apply_vs<float2>, N, nrhs, nsub, sizes, (const float2*)inv, r, map, NG, xg,
                                                      g_sel.list, pre);
  return true;
}

void launch_dense_scale(const Grid& g, int nsets, const StencilLayout& L, const double2* tab, int* ex,
                        cudaStream_t s) {
  const long long N = (long long)(g.d + 1) * g.ncell;
  dim3 grid((unsigned)((N + 127) / 128), nsets);
  for (int pass = 0; pass < 2; ++pass) {
    if (g.d == 2) k_dense_scale<2><<<grid, 128, 0, s>>>(g, L, tab, ex, pass);
    else k_dense_scale<3><<<grid, 128, 0, s>>>(g, L, tab, ex, pass);
  }
}

void launch_dense_assemble(const Grid& g, int nsets, const StencilLayout& L, const double2* tab, const int* ex,
                           double2* A, cudaStream_t s) {
  const long long N = (long long)(g.d + 1) * g.ncell;
  dim3 grid((unsigned)((N + 127) / 128), nsets);
  if (g.d == 2) k_dense_assemble<2><<<grid, 128, 0, s>>>(g, L, tab, ex, A);
  else k_dense_assemble<3><<<grid, 128, 0, s>>>(g, L, tab, ex, A);
}

template <typename T>
void launch_dense_apply(int N, int items, int nrhs, const double2* inv, const typename CT<T>::type* r,
                        typename CT<T>::type* x, cudaStream_t s) {
  const int wpb = 8;
  dim3 grid((N + wpb - 1) / wpb, sel_items(items));
  // from 2048 rows of the batch on the loop counts, below it the launch (N = 768: 9.8 us by launch_pdl, 10.7 plain; four
  // items of it 33.4 and 24.6)
  if ((long long)N * sel_items(items) >= 2048)
    launch_plain(grid, 32 * wpb, 0, s, k_dense_apply<T, true>, N, nrhs, inv, r, x, g_sel.list);
  else
    launch_pdl(grid, 32 * wpb, 0, s, k_dense_apply<T, false>, N, nrhs, inv, r, x, g_sel.list);
}

void launch_dense_assemble_sub(const Grid& g, int nsets, int nsub, int nloc, const StencilLayout& L,
                               const double2* tab, const int* ex, const int* map, const int* g2l, double2* A,
                               int* exl, cudaStream_t s) {
  const dim3 grid((unsigned)((nloc + 127) / 128), nsets * nsub);
  if (g.d == 2) k_dense_assemble_sub<2><<<grid, 128, 0, s>>>(g, L, tab, ex, nsub, nloc, map, g2l, A, exl);
  else k_dense_assemble_sub<3><<<grid, 128, 0, s>>>(g, L, tab, ex, nsub, nloc, map, g2l, A, exl);
}

void launch_dense_apply_lp(int N, int items, int nrhs, int nsub, const int* sizes, const void* inv, int fmt,
                           const float2* r, float2* x, cudaStream_t s) {
  const int wpb = 8;
  const dim3 grid((N + wpb - 1) / wpb, sel_items(items));
  const int E = fmt >= 2 ? 4 : 2;
  if (N % 4 == 0 && N % E == 0) {
    const dim3 gv((N / 4 + wpb - 1) / wpb, sel_items(items));   // a warp per 4 rows
    if (fmt == 2)
      launch_pdl(gv, 32 * wpb, 0, s, k_dense_apply_v<__half2>, N, nrhs, nsub, sizes, (const __half2*)inv, r, x, g_sel.list);
    else if (fmt == 3)
      launch_pdl(gv, 32 * wpb, 0, s, k_dense_apply_v<__nv_bfloat162>, N, nrhs, nsub, sizes, (const __nv_bfloat162*)inv, r, x,
                                                              g_sel.list);
    else
      launch_pdl(gv, 32 * wpb, 0, s, k_dense_apply_v<float2>, N, nrhs, nsub, sizes, (const float2*)inv, r, x, g_sel.list);
    return;
  }
  if (fmt == 2)
    launch_pdl(grid, 32 * wpb, 0, s, k_dense_apply_lp<__half2>, N, nrhs, (const __half2*)inv, r, x, g_sel.list);
  else if (fmt == 3)
    launch_pdl(grid, 32 * wpb, 0, s, k_dense_apply_lp<__nv_bfloat162>, N, nrhs, (const __nv_bfloat162*)inv, r, x, g_sel.list);
  else
    launch_pdl(grid, 32 * wpb, 0, s, k_dense_apply_lp<float2>, N, nrhs, (const float2*)inv, r, x, g_sel.list);
}

template void launch_dense_apply<float>(int, int, int, const double2*, const float2*, float2*, cudaStream_t);
template void launch_dense_apply<double>(int, int, int, const double2*, const double2*, double2*, cudaStream_t);

}  // namespace ehs
