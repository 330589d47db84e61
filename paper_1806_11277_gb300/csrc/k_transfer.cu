// Restriction r_c = P^T r_f and prolongation x_f += P e_c (Algorithm TwoCycle
// steps 2 and 4) with the bilinear staggered-grid transfer of Sec. 3: per
// component a tensor product of 1D rules (vertex-like along the component's
// own direction, cell-like with zero ghosts across it, cell-like with clamped
// ghosts for p).  One thread per cell and component (blockIdx.z), so that the small
// levels fill more of the chip and a thread's taps are few enough to be in flight
// together; weights are integer quarters until they multiply, and real (two FMAs a tap), as
// the FP64 form is bound by the FP64 pipe.  Large complex64 prolongations run a thread per cell
// (launch_prolong_add).  (The 2D complex64 fine level of the cycle uses the fused kernels of k_fine_fused.cu instead.)
#include "kernels.h"

namespace ehs {
namespace {

// weight in quarters of fine index 2 J - 1 + t in coarse index J (t = 0..3, J a valid unknown index)
__host__ __device__ constexpr int rw4(int kind, int t, int J, int nc) {
  if (kind == 0) return t == 1 ? 4 : t == 3 ? 0 : 2;
  if (t == 0) return J >= 1 ? 1 : 0;
  if (t == 3) return J + 1 < nc ? 1 : 0;
  return 3 + (kind == 2 && (t == 1 ? J == 0 : J + 1 == nc) ? 1 : 0);
}
__host__ __device__ constexpr bool rw4_agrees(int nc) {
  for (int kind = 0; kind < 3; ++kind)
    for (int J = kind == 0 ? 1 : 0; J < nc; ++J)
      for (int t = 0; t < 4; ++t)
        if (rw4(kind, t, J, nc) != pw4(kind, 2 * J - 1 + t, J, nc)) return false;
  return true;
}
static_assert(rw4_agrees(1) && rw4_agrees(2) && rw4_agrees(3) && rw4_agrees(8), "restriction weights = pw4()");

// q / 4 for q = 0..4, without an FP64 instruction
template <typename T> __device__ __forceinline__ T quarters(int q);
template <> __device__ __forceinline__ float quarters<float>(int q) { return 0.25f * (float)q; }
template <> __device__ __forceinline__ double quarters<double>(int q) {
  const int hi = q == 0 ? 0 : q == 1 ? 0x3fd00000 : q == 2 ? 0x3fe00000 : q == 3 ? 0x3fe80000 : 0x3ff00000;
  return __hiloint2double(hi, 0);
}
// a weight of 0, 1/4, .., 1 as a T, likewise
template <typename T> __device__ __forceinline__ T weight(float w) {
  if constexpr (sizeof(T) == 4) return w;
  else return quarters<T>((int)(4.0f * w));
}
// a + w v, w real
template <typename T, typename C> __device__ __forceinline__ C rfma(T w, C v, C a) {
  a.x = fma(w, v.x, a.x);
  a.y = fma(w, v.y, a.y);
  return a;
}

// thread per coarse cell and component: fine offsets -1..2 around 2 I along every direction
template <typename T, int D>
__global__ void k_restrict(Grid gf, Grid gc, const typename CT<T>::type* rf,
                           typename CT<T>::type* __restrict__ rc, const int* il) {
  pdl_enter();
  typedef typename CT<T>::type C;
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= gc.ncell) return;
  const int item = il ? il[blockIdx.y] : blockIdx.y, a = blockIdx.z;
  const C* fa = rf + ((long long)item * (D + 1) + a) * gf.ncell;
  int I[3];
  cell_coords(gc, c, I);
  C acc = czero<C>();
  if (slot_valid(a, D, I)) {
    int q[3][4];
#pragma unroll
    for (int k = 0; k < D; ++k)
#pragma unroll
      for (int t = 0; t < 4; ++t) q[k][t] = rw4(tkind(a, k, D), t, I[k], gc.n[k]);
    constexpr int NZ = D == 3 ? 4 : 1;
#pragma unroll
    for (int z = 0; z < NZ; ++z) {
      C pl = czero<C>();                            // one plane
      const bool zin = D < 3 || q[D - 1][z] != 0;
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const bool yin = zin && q[1][y] != 0;
        const C* row = fa + ((long long)(D == 3 ? 2 * I[2] - 1 + z : 0) * gf.n[1] + (2 * I[1] - 1 + y)) * gf.n[0] +
                       2 * I[0] - 1;
        C rs = czero<C>();                          // one row
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          C v = czero<C>();
          if (yin && q[0][x] != 0) v = *(row + x);
          rs = rfma(quarters<T>(q[0][x]), v, rs);
        }
        pl = rfma(quarters<T>(q[1][y]), rs, pl);
      }
      acc = D == 3 ? rfma(quarters<T>(q[D - 1][z]), pl, acc) : pl;
    }
  }
  rc[((long long)item * (D + 1) + a) * gc.ncell + c] = acc;
}

// (P e_c) of component a at the fine cell i: at most two coarse indices per direction (pw_pair)
template <typename T, int D>
__device__ __forceinline__ typename CT<T>::type prolong_one(const Grid& gc, const typename CT<T>::type* ea, int a,
                                                            const int i[3]) {
  typedef typename CT<T>::type C;
  int J[3][2] = {{0, 0}, {0, 0}, {0, 0}};
  float w[3][2];
#pragma unroll
  for (int k = 0; k < D; ++k) pw_pair<float>(tkind(a, k, D), i[k], gc.n[k], J[k][0], w[k][0], J[k][1], w[k][1]);
  constexpr int NZ = D == 3 ? 2 : 1;
  C acc = czero<C>();
#pragma unroll
  for (int z = 0; z < NZ; ++z) {
    C pl = czero<C>();
    const bool zin = D < 3 || w[D - 1][z] != 0.f;
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      const bool yin = zin && w[1][y] != 0.f;
      const C* row = ea + ((long long)J[2][z] * gc.n[1] + J[1][y]) * gc.n[0];
      C rs = czero<C>();
#pragma unroll
      for (int xx = 0; xx < 2; ++xx) {
        C v = czero<C>();
        if (yin && w[0][xx] != 0.f) v = *(row + J[0][xx]);
        rs = rfma(weight<T>(w[0][xx]), v, rs);
      }
      pl = rfma(weight<T>(w[1][y]), rs, pl);
    }
    acc = D == 3 ? rfma(weight<T>(w[D - 1][z]), pl, acc) : pl;
  }
  return acc;
}

// thread per fine cell and component
template <typename T, int D>
__global__ void k_prolong_add(Grid gf, Grid gc, const typename CT<T>::type* ec,
                              typename CT<T>::type* __restrict__ xf, const int* il) {
  pdl_enter();
  typedef typename CT<T>::type C;
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= gf.ncell) return;
  const int item = il ? il[blockIdx.y] : blockIdx.y, a = blockIdx.z;
  int i[3];
  cell_coords(gf, c, i);
  if (!slot_valid(a, D, i)) return;
  C* x = xf + ((long long)item * (D + 1) + a) * gf.ncell + c;
  const C old = *x;
  *x = cadd(old, prolong_one<T, D>(gc, ec + ((long long)item * (D + 1) + a) * gc.ncell, a, i));
}
// thread per fine cell, all components: the coordinates once, for launches that fill the chip many times over
template <int D>
__global__ void k_prolong_add_cells(Grid gf, Grid gc, const float2* ec, float2* __restrict__ xf, const int* il) {
  pdl_enter();
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= gf.ncell) return;
  const int item = il ? il[blockIdx.y] : blockIdx.y;
  int i[3];
  cell_coords(gf, c, i);
  const float2* e = ec + (long long)item * (D + 1) * gc.ncell;
  float2* x = xf + (long long)item * (D + 1) * gf.ncell + c;
  float2 old[D + 1];
#pragma unroll
  for (int a = 0; a <= D; ++a)
    if (slot_valid(a, D, i)) old[a] = x[(long long)a * gf.ncell];
#pragma unroll
  for (int a = 0; a <= D; ++a)
    if (slot_valid(a, D, i))
      x[(long long)a * gf.ncell] = cadd(old[a], prolong_one<float, D>(gc, e + (long long)a * gc.ncell, a, i));
}

}  // namespace

template <typename T>
void launch_restrict(const Grid& gf, const Grid& gc, int items, const typename CT<T>::type* rf,
                     typename CT<T>::type* rc, cudaStream_t s) {
  const int bs = spread_bs(gc.ncell * (gf.d + 1), items, 128);
  const dim3 gr((unsigned)((gc.ncell + bs - 1) / bs), sel_items(items), gf.d + 1);
  if (gf.d == 2) launch_pdl(gr, bs, 0, s, k_restrict<T, 2>, gf, gc, rf, rc, g_sel.list);
  else launch_pdl(gr, bs, 0, s, k_restrict<T, 3>, gf, gc, rf, rc, g_sel.list);
}

template <typename T>
void launch_prolong_add(const Grid& gf, const Grid& gc, int items, const typename CT<T>::type* ec,
                        typename CT<T>::type* xf, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    // complex64 above 400 K cells of the batch.  us, a thread per component -> per cell: 2D 1 M cells 19.4 -> 13.0, 524 K 10.6
    // -> 7.6, 262 K 6.1 -> 8.3; 3D 7.1 M 253 -> 177, 524 K 20.1 -> 15.0, 262 K 11.0 -> 12.3.  The FP64 form is bound by its
    // pipe and keeps the former (2D 1 M cells 82 against 140).
    if (gf.ncell * (long long)items > 400000) {
      const dim3 gr((unsigned)((gf.ncell + 255) / 256), sel_items(items));
      if (gf.d == 2) launch_pdl(gr, 256, 0, s, k_prolong_add_cells<2>, gf, gc, ec, xf, g_sel.list);
      else launch_pdl(gr, 256, 0, s, k_prolong_add_cells<3>, gf, gc, ec, xf, g_sel.list);
      return;
    }
  }
  const int bs = spread_bs(gf.ncell * (gf.d + 1), items, 256);
  const dim3 gr((unsigned)((gf.ncell + bs - 1) / bs), sel_items(items), gf.d + 1);
  if (gf.d == 2) launch_pdl(gr, bs, 0, s, k_prolong_add<T, 2>, gf, gc, ec, xf, g_sel.list);
  else launch_pdl(gr, bs, 0, s, k_prolong_add<T, 3>, gf, gc, ec, xf, g_sel.list);
}

#define INST(T)                                                                                 \
  template void launch_restrict<T>(const Grid&, const Grid&, int, const CT<T>::type*, CT<T>::type*, \
                                   cudaStream_t);                                                \
  template void launch_prolong_add<T>(const Grid&, const Grid&, int, const CT<T>::type*,          \
                                      CT<T>::type*, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace ehs
