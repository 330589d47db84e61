// Batched FP64 inverses of the coarsest level's dense matrices (the whole level or
// the MG-DD boxes, k_dense.cu assembles them): blocked Gauss-Jordan in place with
// partial pivoting, the rank-B updates on the tensor cores.
//
// Per block of B columns K = [k0, k0 + B), for all matrices at once:
//   k_inv_panel   unblocked Gauss-Jordan of the N x B panel in FP64 (pivot rows
//                 from all rows not yet used), giving W = D^{-1} on the pivot rows
//                 and -P D^{-1} elsewhere, D the pivot block, P the panel
//   k_inv_rows    the panel's row exchanges on the other columns; R = A[K, :]
//   k_inv_update  A := (A with the rows K zeroed) + W R on the other columns
// and at the end the row exchanges come back as a column permutation of A.
//
// Why blocks: column by column over the augmented [A | I] every step re-read
// and re-wrote the whole 2 N^2 entries, 4 N launches and 12 N^3 FP64 operations on
// a chip whose FP64 rate is 54x below its FP32 rate.  Here FP64 arithmetic is left
// in the panel (8 N^2 B operations), spread over a cluster of SMs per matrix, and
// the 8 N^3 operations of the updates run as exact products of small integers on the
// FP16 tensor cores (Ozaki, Ogita, Oishi and Rump, "Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication and its
// applications", Numerical Algorithms 2012): every row of W and column of R is scaled
// by a power of two and cut into six balanced 9-bit digits (55 bits with the sign),
// digit products of one weight 2^{-9 (i + j)} are summed in the FP32 accumulators (|digit| <= 2^8, 2 B products per
// pair of digits: exactly up to i + j = 3 at B = 32, four pairs of 2^22, and at B = 16 throughout; the five or six pairs of the
// lower weights could pass 2^24 with nearly every digit at its largest, and would then lose the last unit of
// 2^{-54} and below), and the sums of i + j <= 6
// are joined in 64-bit integers before one rounding to FP64.  On the line's box
// matrices the inverse's error against an 80-bit one is about half that of the
// FP64 column-by-column elimination (numpy restatement, N = 645: 4.0e-15 against
// 7.7e-15 in the 2-norm); with the sums of i + j <= 5 only it would be five times larger.
// An entry far below the largest of its row of W or column of R is cut, so this holds for
// matrices whose unknowns have one scale: they come in equilibrated by powers of two (k_dense.cu), and the last
// kernel takes the equilibration back.
#include <cuda_fp16.h>

#include "kernels.h"

namespace ehs {
namespace {

constexpr int NDIG = 6;               // digits per real number
constexpr int DBITS = 9;
constexpr int NGRP = 7;               // digit products with i + j < NGRP are kept
constexpr int NPL = 2 * NDIG;         // planes: (digit, re / im)
constexpr int CLMAX = 16;             // most CTAs (SMs) per matrix in the panel kernel
constexpr int PT = 512;               // its threads per CTA
constexpr int TM = 64;                // update tile: TM x TM entries of A
constexpr int EXP_BAD = 1 << 20;      // exponent of a row that holds Inf or NaN

__device__ __forceinline__ unsigned saddr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ unsigned cluster_addr(unsigned a, int rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(unsigned a, double2 v) {
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned a, int2 v) {
  asm volatile("st.shared::cluster.v2.s32 [%0], {%1, %2};" ::"r"(a), "r"(v.x), "r"(v.y) : "memory");
}

// exponent word of |x| as an ordered integer (a comparison on the integer pipe)
__device__ __forceinline__ int hi_abs(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ double2 shfl_d2(double2 v, int src) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// scale exponent of values whose largest exponent word is h: |x| < 2^e
__device__ __forceinline__ int scale_exp(int h) {
  const int ex = h >> 20;
  return ex == 0x7ff ? EXP_BAD : ex - 1022;
}
// x 2^{53 - e} rounded to an integer of at most 2^53 (integer arithmetic only: the FP64 pipe is
// the scarce one); |x| < 2^e, so x = v 2^{e + 1} 2^{-54}
__device__ __forceinline__ long long fix54(double x, int e) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((u >> 52) & 0x7ff);
  if (ex == 0 || e == EXP_BAD) return 0;
  unsigned long long m = (u & 0xfffffffffffffull) | 0x10000000000000ull;
  const int sh = e + 1022 - ex;                       // >= 0
  if (sh > 54) return 0;
  if (sh > 0) m = (m + (1ull << (sh - 1))) >> sh;
  return (u >> 63) ? -(long long)m : (long long)m;
}
// its balanced base-512 digits, most significant first, each in [-256, 256]
__device__ __forceinline__ void digits(long long v, int d[NDIG]) {
#pragma unroll
  for (int i = NDIG - 1; i > 0; --i) {
    d[i] = (int)((v + 256) & 511) - 256;
    v = (v - d[i]) >> DBITS;
  }
  d[0] = (int)v;
}

// One block's panel.  A cluster of cl CTAs holds the N x B panel of one matrix, rows
// split among the CTAs, in shared memory (in gp where it does not fit).  Lane = column
// (32 / B rows per warp pass), so a row update is 4 FP64 FMAs per lane with the pivot
// row in registers.  Per column: every CTA finds its pivot candidate (the warps kept
// theirs while updating), scales that row by the inverse pivot and sends it to all
// CTAs; the owner of row k sends that row; after one cluster barrier every CTA picks
// the same winner and updates its rows.  The receive slots alternate, so a CTA may send
// for the next column while another still reads this one's.  Bound by the FP64 pipe.
template <int B>
__global__ void __launch_bounds__(PT) k_inv_panel(int N, int Npad, int k0, int bb, int cl, double2* __restrict__ A,
                                                  double2* __restrict__ gp, __half* __restrict__ wd,
                                                  int* __restrict__ we, int* __restrict__ swp, int* __restrict__ err) {
  constexpr int G = 32 / B, NW = PT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double2 srow[2][CLMAX][B];   // scaled candidate rows by sender
  __shared__ double2 krow[2][B];       // row k before the exchange
  __shared__ int2 skey[2][CLMAX];         // (key, row) by sender
  __shared__ int2 wkey[NW];
  const int rank = blockIdx.x % cl, mat = blockIdx.x / cl;
  const int rp = (N + cl - 1) / cl, r0 = min(N, rank * rp), r1 = min(N, r0 + rp);
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, col = lane % B, sub = lane / B;
  double2* Am = A + (long long)mat * N * N;
  double2* P = gp ? gp + ((long long)mat * N + r0) * B : reinterpret_cast<double2*>(smem_raw);
  const int stepr = NW * G;
  int bk = -1, br = N;                 // this lane's pivot candidate for the coming column
  auto consider = [&](double2 v, int row, int t) {
    if (col == t && row >= k0 + t) {
      const int h = max(hi_abs(v.x), hi_abs(v.y));
      if (h > bk) { bk = h; br = row; }   // rows come in increasing order: the first of equals
    }
  };
  for (int rb = r0 + wid * G; rb < r1; rb += stepr) {
    const int row = rb + sub;
    if (row < r1) {
      const double2 v = col < bb ? Am[(long long)row * N + k0 + col] : make_double2(0.0, 0.0);
      P[(row - r0) * B + col] = v;
      consider(v, row, 0);
    }
  }
  __syncwarp();
  cluster_arrive();                    // every CTA has started before the first remote store
  cluster_wait();
  for (int t = 0; t < bb; ++t) {
    const int k = k0 + t, par = t & 1;
    // the warp's candidate sits in the lanes col == t
    int ck = __shfl_sync(0xffffffffu, bk, t), cr = __shfl_sync(0xffffffffu, br, t);
#pragma unroll
    for (int q = 1; q < G; ++q) {
      const int ok = __shfl_sync(0xffffffffu, bk, q * B + t), orow = __shfl_sync(0xffffffffu, br, q * B + t);
      if (ok > ck || (ok == ck && orow < cr)) { ck = ok; cr = orow; }
    }
    if (lane == 0) wkey[wid] = make_int2(ck, cr);
    __syncthreads();                   // candidates and the panel rows of the last column are in place
    if (wid == 0) {
      int2 c = lane < NW ? wkey[lane] : make_int2(-1, N);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const int ok = __shfl_xor_sync(0xffffffffu, c.x, o), orow = __shfl_xor_sync(0xffffffffu, c.y, o);
        if (ok > c.x || (ok == c.x && orow < c.y)) { c.x = ok; c.y = orow; }
      }
      double2 v = make_double2(0.0, 0.0);
      if (c.x >= 0) v = P[(c.y - r0) * B + col];
      const double2 inv = cinv(shfl_d2(v, t));
      const double2 u = col == t ? inv : cmul(v, inv);
      // the CTA's message to every CTA of the cluster
      for (int q = 0; q < cl; ++q) {
        if (lane < B) st_cluster(cluster_addr(saddr(&srow[par][rank][col]), q), u);
        if (lane == 0) st_cluster(cluster_addr(saddr(&skey[par][rank]), q), c);
      }
    } else if (wid == 1 && k >= r0 && k < r1 && lane < B) {
      const double2 v = P[(k - r0) * B + col];
      for (int q = 0; q < cl; ++q) st_cluster(cluster_addr(saddr(&krow[par][col]), q), v);
    }
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    int2 best = skey[par][0];
    int win = 0;
    for (int q = 1; q < cl; ++q) {
      const int2 c = skey[par][q];
      if (c.x > best.x || (c.x == best.x && c.y < best.y)) { best = c; win = q; }
    }
    const int p = best.y;
    if (rank == 0 && threadIdx.x == 0) {
      swp[(long long)mat * N + k] = p;
      // a pivot whose |.|^2 leaves the FP64 range (below 2^-537, from 2^511 on), or that is not finite: Inf and NaN
      // rank above every number in the search
      if (best.x < 0x1e600000 || best.x >= 0x5fe00000) atomicOr(err, EHS_DEVERR_SINGULAR);
    }
    const double2 u = srow[par][win][col];
    bk = -1;
    br = N;
    for (int rb = r0 + wid * G; rb < r1; rb += stepr) {
      const int row = rb + sub;
      const bool live = row < r1;
      double2 v = make_double2(0.0, 0.0);
      if (live) v = row == p && p != k ? krow[par][col] : P[(row - r0) * B + col];
      const double2 f = shfl_d2(v, sub * B + t);
      if (live) {
        if (row == k) {
          v = u;
        } else {
          if (col == t) v = make_double2(0.0, 0.0);
          v.x = fma(-f.x, u.x, fma(f.y, u.y, v.x));
          v.y = fma(-f.x, u.y, fma(-f.y, u.x, v.y));
        }
        P[(row - r0) * B + col] = v;
        if (t + 1 < bb) consider(v, row, t + 1);
      }
    }
  }
  // W back into the panel's columns, and its digits (the warp that updated a row writes it)
  __half* wm = wd + (long long)mat * NPL * Npad * B;
  for (int rb = r0 + wid * G; rb < r1; rb += stepr) {
    const int row = rb + sub;
    const bool live = row < r1;
    const double2 v = live ? P[(row - r0) * B + col] : make_double2(0.0, 0.0);
    int h = max(hi_abs(v.x), hi_abs(v.y));
#pragma unroll
    for (int o = B / 2; o > 0; o >>= 1) h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
    const int e = scale_exp(h);
    if (!live) continue;
    if (col < bb) Am[(long long)row * N + k0 + col] = v;
    int dx[NDIG], dy[NDIG];
    digits(fix54(v.x, e), dx);
    digits(fix54(v.y, e), dy);
#pragma unroll
    for (int i = 0; i < NDIG; ++i) {
      wm[((long long)(2 * i) * Npad + row) * B + col] = __int2half_rn(dx[i]);
      wm[((long long)(2 * i + 1) * Npad + row) * B + col] = __int2half_rn(dy[i]);
    }
    if (col == 0) we[(long long)mat * Npad + row] = e;
  }
}

// The panel's row exchanges on 32 columns outside it, and R's digits.  The exchanges
// run in shared memory: Ko holds the rows K, Lo the rows they are exchanged with
// (each distinct row once, at its first use), loaded together beforehand.
template <int B>
__global__ void __launch_bounds__(256) k_inv_rows(int N, int Npad, int k0, int bb, double2* __restrict__ A,
                                                  __half* __restrict__ rd, int* __restrict__ re,
                                                  const int* __restrict__ swp) {
  __shared__ double2 Ko[B][32], Lo[B][32];
  __shared__ int sp[B], first[B], hmax[32];
  const int mat = blockIdx.y, c = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int j = blockIdx.x * 32 + c;
  double2* Am = A + (long long)mat * N * N;
  const bool out = j < N && (j < k0 || j >= k0 + bb);
  if (threadIdx.x < 32) hmax[threadIdx.x] = 0;
  if (threadIdx.x < bb) sp[threadIdx.x] = swp[(long long)mat * N + k0 + threadIdx.x];
  __syncthreads();
  if (threadIdx.x < bb) {
    int f = threadIdx.x;
    for (int s = (int)threadIdx.x - 1; s >= 0; --s)
      if (sp[s] == sp[threadIdx.x]) f = s;
    first[threadIdx.x] = f;
  }
  __syncthreads();
  for (int t = ty; t < B; t += 8) {
    const double2 z = make_double2(0.0, 0.0);
    Ko[t][c] = out && t < bb ? Am[(long long)(k0 + t) * N + j] : z;
    if (out && t < bb && sp[t] >= k0 + bb && first[t] == t) Lo[t][c] = Am[(long long)sp[t] * N + j];
  }
  __syncthreads();
  if (ty == 0) {
    for (int t = 0; t < bb; ++t) {
      const int p = sp[t];
      double2* o = p >= k0 + bb ? &Lo[first[t]][c] : &Ko[p - k0][c];
      const double2 a = Ko[t][c], b = *o;
      *o = a;
      Ko[t][c] = b;                    // p == k0 + t: o is the same entry
    }
  }
  __syncthreads();
  for (int t = ty; t < bb; t += 8)
    if (out && sp[t] >= k0 + bb && first[t] == t) Am[(long long)sp[t] * N + j] = Lo[t][c];
  // column exponents and digits: thread (c, ty) holds rows 4 ty .. 4 ty + 3 of column c
  int h = 0;
  if (ty < B / 4)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double2 v = Ko[4 * ty + q][c];
      h = max(h, max(hi_abs(v.x), hi_abs(v.y)));
    }
  atomicMax(&hmax[c], h);
  __syncthreads();
  const int e = scale_exp(hmax[c]);
  if (j >= N) return;
  if (ty == 0) re[(long long)mat * Npad + j] = e;
  if (ty >= B / 4) return;
  int dx[4][NDIG], dy[4][NDIG];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const double2 v = Ko[4 * ty + q][c];
    digits(fix54(v.x, e), dx[q]);
    digits(fix54(v.y, e), dy[q]);
  }
  __half* rm = rd + (long long)mat * NPL * Npad * B;
#pragma unroll
  for (int i = 0; i < NDIG; ++i)
#pragma unroll
    for (int part = 0; part < 2; ++part) {
      __half2 w[2];
#pragma unroll
      for (int q = 0; q < 2; ++q)
        w[q] = part ? __halves2half2(__int2half_rn(dy[2 * q][i]), __int2half_rn(dy[2 * q + 1][i]))
                    : __halves2half2(__int2half_rn(dx[2 * q][i]), __int2half_rn(dx[2 * q + 1][i]));
      *reinterpret_cast<uint2*>(rm + ((long long)(2 * i + part) * Npad + j) * B + 4 * ty) =
          *reinterpret_cast<const uint2*>(w);
    }
}

__device__ __forceinline__ void ldsm4(unsigned r[4], unsigned a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}
__device__ __forceinline__ void mma16816(float c[4], const unsigned a[4], const unsigned b[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// sum_g G_g 2^{-9 (g + 2)} 2^s as a double: the exact integers are joined in units of 2^{-58}
// (the two lowest groups rounded to it) and rounded once; no FP64 instruction
__device__ __forceinline__ double join(const float G[NGRP], int s) {
  long long v = (long long)__float2int_rn(G[0]);
#pragma unroll
  for (int i = 1; i < 5; ++i) v = (v << DBITS) + __float2int_rn(G[i]);
  const long long lo = ((long long)__float2int_rn(G[5]) << DBITS) + __float2int_rn(G[6]);
  v = (v << 4) + ((lo + (1 << 13)) >> 14);
  if (s > 4096) return __longlong_as_double(0x7ff8000000000000ll);   // an Inf or NaN went in
  if (v == 0) return 0.0;
  const unsigned long long u = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
  const int lz = __clzll((long long)u);
  const unsigned long long m = u << lz;
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1);          // 53 bits, or 2^53
  const int E = 1028 - lz + s;                                       // biased exponent of the top bit
  const unsigned long long sg = v < 0 ? 0x8000000000000000ull : 0ull;
  if (E <= 0) return 0.0;
  if (E >= 2047) return __longlong_as_double((long long)(sg | 0x7ff0000000000000ull));
  return __longlong_as_double((long long)(sg + ((unsigned long long)(E - 1) << 52) + r));
}

// A := (A, rows K zero) + W R on one TM x TM tile.  Both operands' digit planes of the
// tile (24 x 64 x B halves, 96 KB at B = 32: 2 CTAs per SM) are staged at once; a warp
// takes 16 rows x 32 columns, 8 columns at a time: 26 digit pairs x 4 (complex) = 104 MMAs
// of 16 x 8 x 16 per step of 16 in k, into 14 accumulator tiles (7 weights, re and im).  The staged rows are XOR-swizzled so that
// ldmatrix meets no bank conflict.  Bound by the tensor pipe (56 % busy) and the joining; with the tile of A asked
// for early 16 matrices of 1408 take 0.59 ms a block instead of 0.64 (210 GFLOP of MMAs: 360 TFLOP/s).
template <int B>
__global__ void __launch_bounds__(256, 2) k_inv_update(int N, int Npad, int k0, int bb, double2* __restrict__ A,
                                                       const __half* __restrict__ wd, const __half* __restrict__ rd,
                                                       const int* __restrict__ we, const int* __restrict__ re) {
  constexpr int CH = B / 8;                       // 16-byte chunks per staged row
  constexpr int RB = B * 2;                       // bytes per staged row
  constexpr int PB = TM * RB;                     // bytes per plane
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int mat = blockIdx.z, i0 = blockIdx.y * TM, j0 = blockIdx.x * TM;
  const unsigned sb = saddr(smem_raw);
  auto swz = [](int row, int ch) { return B == 32 ? ch ^ ((row >> 1) & 3) : ch ^ ((row >> 2) & 1); };
  const __half* wm = wd + (long long)mat * NPL * Npad * B;
  const __half* rm = rd + (long long)mat * NPL * Npad * B;
#pragma unroll 4
  for (int q = threadIdx.x; q < 2 * NPL * TM * CH; q += 256) {
    const int ch = q % CH, row = (q / CH) % TM, pl = q / (CH * TM);
    const __half* src = pl < NPL ? wm + ((long long)pl * Npad + i0 + row) * B + ch * 8
                                 : rm + ((long long)(pl - NPL) * Npad + j0 + row) * B + ch * 8;
    const unsigned dst = sb + pl * PB + row * RB + swz(row, ch) * 16;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wr = (wid & 3) * 16, wc = (wid >> 2) * 32;
  const int ia = i0 + wr + (lane >> 2), ib = ia + 8;   // the two rows of this thread's accumulators
  // the tile of A, on its way to L2 while the digits are staged and multiplied
  double2* Am = A + (long long)mat * N * N;
  for (int q = threadIdx.x; q < TM * (TM / 8); q += 256) {
    const int row = i0 + q / (TM / 8), c8 = j0 + q % (TM / 8) * 8;
    if (row < N && c8 < N) asm volatile("prefetch.global.L2 [%0];" ::"l"(Am + (long long)row * N + c8));
  }
  const int ea = we[(long long)mat * Npad + ia] + 2, eb = we[(long long)mat * Npad + ib] + 2;
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
  for (int nt = 0; nt < 4; ++nt) {
    const int jn = wc + nt * 8;                        // tile column of this step
    float ac[NGRP][2][4];
#pragma unroll
    for (int g = 0; g < NGRP; ++g)
#pragma unroll
      for (int q = 0; q < 4; ++q) ac[g][0][q] = ac[g][1][q] = 0.f;
#pragma unroll
    for (int kk = 0; kk < B / 16; ++kk) {
      unsigned bf[NDIG][4];                            // (re lo, re hi, im lo, im hi) of each digit
      {
        const int row = jn + (lane & 7), ch = kk * 2 + ((lane >> 3) & 1);
        const unsigned a = sb + (NPL + (lane >> 4)) * PB + row * RB + swz(row, ch) * 16;
#pragma unroll
        for (int i = 0; i < NDIG; ++i) ldsm4(bf[i], a + 2 * i * PB);
      }
      const int row = wr + (lane & 7) + ((lane >> 3) & 1) * 8, ch = kk * 2 + (lane >> 4);
      const unsigned a = sb + row * RB + swz(row, ch) * 16;
#pragma unroll
      for (int i = 0; i < NDIG; ++i) {
        unsigned ar[4], ai[4], an[4];
        ldsm4(ar, a + (2 * i) * PB);
        ldsm4(ai, a + (2 * i + 1) * PB);
#pragma unroll
        for (int q = 0; q < 4; ++q) an[q] = ai[q] ^ 0x80008000u;
#pragma unroll
        for (int l = 0; l < NDIG && i + l < NGRP; ++l) {
          mma16816(ac[i + l][0], ar, bf[l]);
          mma16816(ac[i + l][1], ar, bf[l] + 2);
        }
#pragma unroll
        for (int l = 0; l < NDIG && i + l < NGRP; ++l) {
          mma16816(ac[i + l][0], an, bf[l] + 2);
          mma16816(ac[i + l][1], ai, bf[l]);
        }
      }
    }
    // join the weights and add to A, its entries loaded first
    double2 old[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = q < 2 ? ia : ib, j = j0 + jn + (lane & 3) * 2 + (q & 1);
      old[q] = make_double2(0.0, 0.0);
      if (i < N && j < N && (i < k0 || i >= k0 + bb)) old[q] = Am[(long long)i * N + j];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = q < 2 ? ia : ib, j = j0 + jn + (lane & 3) * 2 + (q & 1);
      if (i >= N || j >= N || (j >= k0 && j < k0 + bb)) continue;
      const int s = (q < 2 ? ea : eb) + re[(long long)mat * Npad + j];
      float gr[NGRP], gi[NGRP];
#pragma unroll
      for (int g = 0; g < NGRP; ++g) { gr[g] = ac[g][0][q]; gi[g] = ac[g][1][q]; }
      double2 v = make_double2(join(gr, s), join(gi, s));
      v.x += old[q].x;
      v.y += old[q].y;
      Am[(long long)i * N + j] = v;
    }
  }
}

// All row exchanges, in order, applied to 0 .. N-1: perm[j] = the column of the inverse that
// column j of A holds (one thread walks them in shared memory; N <= 16384).
__global__ void k_inv_perm(int N, const int* __restrict__ swp, int* __restrict__ perm) {
  extern __shared__ int sm[];
  int* pm = sm;
  int* sp = sm + N;
  const long long o = (long long)blockIdx.x * N;
  for (int j = threadIdx.x; j < N; j += blockDim.x) {
    pm[j] = j;
    sp[j] = swp[o + j];
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = 0; k < N; ++k) {
      const int p = sp[k], a = pm[k];
      pm[k] = pm[p];
      pm[p] = a;
    }
  __syncthreads();
  for (int j = threadIdx.x; j < N; j += blockDim.x) perm[o + j] = pm[j];
}
// X[i, perm[j]] = 2^ex[i] A[i, j] 2^ex[perm[j]]: the column order, and the equilibration of the matrix taken back
__global__ void k_inv_columns(int N, const double2* __restrict__ A, const int* __restrict__ perm,
                              const int* __restrict__ ex, double2* __restrict__ X) {
  const int mat = blockIdx.z, j = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
  if (j >= N) return;
  const long long o = ((long long)mat * N + i) * N;
  const int* es = ex + (long long)mat * N;
  const int p = perm[(long long)mat * N + j], e = es[i] + es[p];
  X[o + p] = pow2_scaled(A[o + j], e);
}

struct Plan {
  int B, cl, Npad;
  bool global;                          // the panel does not fit in shared memory
  size_t psm, usm;                      // dynamic shared memory of the panel and update kernels
  size_t dig, gp;                       // bytes of one operand's digits and of the global panel
};
// Function attributes are the process's, so they are always set to the same values (threads may build contexts side
// by side).
constexpr int PANEL_SMEM = 200 * 1024, PERM_SMEM = 2 * 16384 * (int)sizeof(int);
template <int B> void panel_attributes() {
  cudaFuncSetAttribute(k_inv_panel<B>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cudaFuncSetAttribute(k_inv_panel<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, PANEL_SMEM);
}
template <int B> int clusters_of(int cl, size_t sm) {   // clusters of cl CTAs the device runs at once
  panel_attributes<B>();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cl);
  cfg.blockDim = dim3(PT);
  cfg.dynamicSmemBytes = sm;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cl;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k_inv_panel<B>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  return n;
}
// B = 32 columns a block up to N = 3200, else 16 (the panel's FP64 work halves, the update's passes over A double).
// The panel is bound by the FP64 pipe of its SMs, so the cluster size is the one with the fewest rows per CTA
// times waves of clusters, at one CTA per SM (at least 110 KB of shared memory each beside 9 to 17 KB of fixed arrays:
// two to an SM, as clusters of 8 with 90 KB were placed, share its pipe).  GB300 runs 7 clusters of 16, 15 of 8, 23 of
// 6 or 36 of 4 that way.
// 16 matrices of 1408: 455 us a block with clusters of 8, two to an SM; 511 with 15 of the 16 at a time; 339 with 6.
Plan plan_for(int N, int nmat) {
  Plan p;
  const size_t lim = PANEL_SMEM, least = 110 * 1024;
  p.B = N <= 3200 ? 32 : 16;
  p.Npad = (N + TM - 1) / TM * TM;
  p.cl = 0;
  p.global = false;
  p.psm = 0;
  long long best = 0;
  const int sizes[] = {16, 12, 10, 8, 6, 5, 4};
  for (int cl : sizes) {
    const size_t rp = (N + cl - 1) / cl, need = rp * p.B * sizeof(double2), sm = need > least ? need : least;
    if (need > lim) continue;
    const int act = p.B == 32 ? clusters_of<32>(cl, sm) : clusters_of<16>(cl, sm);
    if (act < 1) continue;
    const long long cost = (long long)((nmat + act - 1) / act) * (long long)rp;
    if (!p.cl || cost < best) { best = cost; p.cl = cl; p.psm = sm; }
  }
  if (!p.cl) {                          // beyond N = 12800: the panel in global memory (L2)
    p.cl = 8;
    p.global = true;
  }
  p.usm = (size_t)2 * NPL * TM * p.B * sizeof(__half);
  p.dig = (size_t)nmat * NPL * p.Npad * p.B * sizeof(__half);
  p.gp = p.global ? (size_t)nmat * N * p.B * sizeof(double2) : 0;
  return p;
}
size_t up256(size_t b) { return (b + 255) / 256 * 256; }

template <int B>
int invert_t(const Plan& p, int N, int nmat, double2* A, double2* gp, __half* wd, __half* rd, int* we, int* re, int* swp,
             int* err, cudaStream_t s) {
  panel_attributes<B>();
  cudaFuncSetAttribute(k_inv_update<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.usm);
  int launches = 0;
  for (int k0 = 0; k0 < N; k0 += B) {
    const int bb = N - k0 < B ? N - k0 : B;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.cl * nmat);
    cfg.blockDim = dim3(PT);
    cfg.dynamicSmemBytes = p.psm;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = p.cl;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_inv_panel<B>, N, p.Npad, k0, bb, p.cl, A, gp, wd, we, swp, err);
    ++launches;
    if (bb == N) break;                 // no other columns
    k_inv_rows<B><<<dim3((N + 31) / 32, nmat), 256, 0, s>>>(N, p.Npad, k0, bb, A, rd, re, swp);
    k_inv_update<B><<<dim3(p.Npad / TM, p.Npad / TM, nmat), 256, p.usm, s>>>(N, p.Npad, k0, bb, A, wd, rd, we, re);
    launches += 2;
  }
  return launches;
}

}  // namespace

size_t dense_invert_workspace(int N, int nmat) {
  const Plan p = plan_for(N, nmat);
  return 2 * up256(p.dig) + up256(p.gp) + up256(sizeof(int) * (size_t)nmat * 2 * (p.Npad + N));
}

int dense_invert(int N, int nmat, double2* A, const int* ex, double2* inv, void* ws, int* err, cudaStream_t s) {
  const Plan p = plan_for(N, nmat);
  unsigned char* w = (unsigned char*)ws;
  __half* wd = (__half*)w;
  __half* rd = (__half*)(w + up256(p.dig));
  double2* gp = p.global ? (double2*)(w + 2 * up256(p.dig)) : nullptr;
  int* we = (int*)(w + 2 * up256(p.dig) + up256(p.gp));
  int* re = we + (size_t)nmat * p.Npad;
  int* swp = re + (size_t)nmat * p.Npad;
  int* perm = swp + (size_t)nmat * N;
  // the digits' padding rows stay zero
  cudaMemsetAsync(ws, 0, dense_invert_workspace(N, nmat), s);
  int n = p.B == 32 ? invert_t<32>(p, N, nmat, A, gp, wd, rd, we, re, swp, err, s)
                    : invert_t<16>(p, N, nmat, A, gp, wd, rd, we, re, swp, err, s);
  cudaFuncSetAttribute(k_inv_perm, cudaFuncAttributeMaxDynamicSharedMemorySize, PERM_SMEM);
  k_inv_perm<<<nmat, 256, 2 * N * sizeof(int), s>>>(N, swp, perm);
  k_inv_columns<<<dim3((N + 255) / 256, N, nmat), 256, 0, s>>>(N, A, perm, ex, inv);
  return n + 2;
}

}  // namespace ehs
