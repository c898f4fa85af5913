// Block cyclic reduction factor and solve (see bcr.cuh for the algebra).
#include <algorithm>
#include <cstring>
#include <new>
#include <vector>

#include "bcr.cuh"
#include "tc_gemm.cuh"
#include "tc_gemm64.cuh"
#include "scratch.h"

namespace {

// ===================================================================== level 0
constexpr int TRI_WARPS = 2;

template <typename T>
__host__ __device__ size_t tri_smem_per_warp(int ny) {
  return ((size_t)6 * ny * sizeof(cplx<T>) + (size_t)ny + 15) & ~(size_t)15;
}

// 1 / a for the serial elimination below, where the reciprocal is most of a step.
// FP64: one division; a is scaled by a power of two (exactly) so that |a|^2 neither overflows nor
// underflows (110 columns of 128: 248 us with crecip, 136 with this).
__device__ __forceinline__ double2 crecip1(double2 a) {
  const int e = max((__double2hiint(a.x) >> 20) & 0x7ff, (__double2hiint(a.y) >> 20) & 0x7ff) - 1023;
  const double f = __hiloint2double((1023 - max(-1000, min(1000, e))) << 20, 0);
  const double ar = a.x * f, ai = a.y * f;
  const double r = 1.0 / (ar * ar + ai * ai);
  if (ar == 0 && ai == 0) return a - a;  // 0 / 0: zero, as crecip
  return mkc((ar * r) * f, -(ai * r) * f);
}
// FP32: crecip bit for bit without its division of the larger part by itself.  (One division as above
// rounds differently, which decides on designs near the limit of the FP32 factorisation whether plain
// refinement stalls.)
__device__ __forceinline__ float2 crecip1(float2 a) {
  const bool x = fabsf(a.x) > fabsf(a.y);
  const float s = x ? fabsf(a.x) : fabsf(a.y), o = x ? a.y : a.x;
  if (s == 0.f) return mkc(0.f, 0.f);
  const float unit = s < INFINITY ? copysignf(1.f, x ? a.x : a.y) : s - s, q = o / s;
  const float ar = x ? unit : q, ai = x ? q : unit;
  const float d = __fmul_rn(__fmaf_rn(ar, ar, __fmul_rn(ai, ai)), s);
  return mkc(ar / d, -ai / d);
}

// Pivoted LU of the tridiagonal diagonal block T_r of an eliminated row r = 2k+1
// (Gaussian elimination with adjacent-row interchanges): multipliers dl, inverse
// pivots dinv, first and second superdiagonals du, du2 of U, and swap flags piv.
// One warp per row: the lanes stage the row's coefficients in shared memory, lane 0
// runs the sequential elimination there, and the lanes write the factors out.
template <typename T>
__global__ void __launch_bounds__(32 * TRI_WARPS)
tri_factor_kernel(const double2* __restrict__ dg, const double2* __restrict__ cy, int nx, int ny,
                  int m0, cplx<T>* __restrict__ tdl, cplx<T>* __restrict__ tdinv,
                  cplx<T>* __restrict__ tdu, cplx<T>* __restrict__ tdu2,
                  uint8_t* __restrict__ tpiv, int32_t* status) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * TRI_WARPS + w;
  if (k >= m0) return;  // whole warp
  cplx<T>* d = reinterpret_cast<cplx<T>*>(sm_raw + (size_t)w * tri_smem_per_warp<T>(ny));
  cplx<T>* o = d + ny;
  cplx<T>* dl = o + ny;
  cplx<T>* di = dl + ny;
  cplx<T>* du = di + ny;
  cplx<T>* du2 = du + ny;
  uint8_t* pv = reinterpret_cast<uint8_t*>(du2 + ny);
  const int64_t r = 2 * (int64_t)k + 1;
  for (int j = lane; j < ny; j += 32) {
    d[j] = ccast<T>(dg[r * ny + j]);
    o[j] = ccast<T>(cy[r * ny + j]);  // o[j] couples j and j+1
  }
  __syncwarp();
  if (lane == 0) {
    cplx<T> cur_d = d[0];
    cplx<T> cur_du = ny > 1 ? o[0] : czero<T>();
    bool sing = false;
    for (int j = 0; j < ny - 1; ++j) {
      const cplx<T> bs = o[j];
      const cplx<T> dnext = d[j + 1];
      const cplx<T> dunext = (j + 1 < ny - 1) ? o[j + 1] : czero<T>();
      if (cabs1(cur_d) >= cabs1(bs)) {
        if (cabs1(cur_d) == T(0)) sing = true;
        const cplx<T> inv = crecip1(cur_d);
        const cplx<T> m = bs * inv;
        dl[j] = m;
        di[j] = inv;
        du[j] = cur_du;
        du2[j] = czero<T>();
        pv[j] = 0;
        cur_d = dnext - m * cur_du;
        cur_du = dunext;
      } else {
        const cplx<T> inv = crecip1(bs);
        const cplx<T> m = cur_d * inv;
        dl[j] = m;
        di[j] = inv;
        du[j] = dnext;
        du2[j] = dunext;
        pv[j] = 1;
        cur_d = cur_du - m * dnext;
        cur_du = -(m * dunext);
      }
    }
    if (cabs1(cur_d) == T(0)) sing = true;
    di[ny - 1] = crecip1(cur_d);
    dl[ny - 1] = czero<T>();
    du[ny - 1] = czero<T>();
    du2[ny - 1] = czero<T>();
    pv[ny - 1] = 0;
    if (sing) atomicCAS(status, DEV_OK, DEV_SINGULAR);
  }
  __syncwarp();
  const int64_t base = (int64_t)k * ny;
  for (int j = lane; j < ny; j += 32) {
    tdl[base + j] = dl[j];
    tdinv[base + j] = di[j];
    tdu[base + j] = du[j];
    tdu2[base + j] = du2[j];
    tpiv[base + j] = pv[j];
  }
}

template <typename T>
struct TriRow {
  const cplx<T>* dl;
  const cplx<T>* dinv;
  const cplx<T>* du;
  const cplx<T>* du2;
  const uint8_t* piv;
};

// Forward sweep (row interchanges and unit lower factor) for the right-hand side
// rhs(j), writing y_j through store(j, y).
template <typename T, typename Rhs, typename Store>
__device__ __forceinline__ void tri_forward(const TriRow<T>& f, int n, Rhs rhs, Store store) {
  cplx<T> cur = rhs(0);
  for (int j = 0; j < n - 1; ++j) {
    cplx<T> nb = rhs(j + 1);
    if (f.piv[j]) {
      store(j, nb);
      cur = cfms(f.dl[j], nb, cur);
    } else {
      store(j, cur);
      cur = cfms(f.dl[j], cur, nb);
    }
  }
  store(n - 1, cur);
}

// Backward substitution with U (diag, du, du2); load(j) returns y_j, emit(j, g_j).
template <typename T, typename Load, typename Emit>
__device__ __forceinline__ void tri_backward(const TriRow<T>& f, int n, Load load, Emit emit) {
  cplx<T> g1 = czero<T>(), g2 = czero<T>();  // g_{j+1}, g_{j+2}
#pragma unroll 4
  for (int j = n - 1; j >= 0; --j) {
    cplx<T> y = load(j);
    y = cfms(f.du[j], g1, y);
    y = cfms(f.du2[j], g2, y);
    cplx<T> g = y * f.dinv[j];
    emit(j, g);
    g2 = g1;
    g1 = g;
  }
}

// Forward sweep for the unit vector e_b into column ycol (stride ny).  Rows j < b - 1 of the
// sweep are exactly zero (the carried value stays zero until the unit entry is reached), so
// the sweep starts at row max(b - 1, 0) and writes only rows from there on; readers take the
// rows above as zero.
template <typename T>
__device__ __forceinline__ void tri_forward_unit(const TriRow<T>& f, int n, int b,
                                                 cplx<T>* ycol, int ny) {
  cplx<T> cur = b == 0 ? mkc(T(1), T(0)) : czero<T>();
  for (int j = b > 0 ? b - 1 : 0; j < n - 1; ++j) {
    const cplx<T> nb = (j + 1 == b) ? mkc(T(1), T(0)) : czero<T>();
    if (f.piv[j]) {
      ycol[(int64_t)j * ny] = nb;
      cur = cfms(f.dl[j], nb, cur);
    } else {
      ycol[(int64_t)j * ny] = cur;
      cur = cfms(f.dl[j], cur, nb);
    }
  }
  ycol[(int64_t)(n - 1) * ny] = cur;
}

// Dense Schur blocks of the first reduced system, one block per kept row e = 2k:
//   D'_k = T_e - diag(cx[e-1]) T_{e-1}^{-1} diag(cx[e-1]) - diag(cx[e]) T_{e+1}^{-1} diag(cx[e])
//   L'_k = -diag(cx[e-1]) T_{e-1}^{-1} diag(cx[e-2])
// Thread b forms column b of both inverses: the forward sweeps of the unit vector e_b go to
// two scratch columns (YR, YL: the next level's free working arrays; only the rows from
// b - 1 on, the others being zero), then one backward sweep runs both recurrences side by
// side, so that every entry of D'_k is formed in one step (no read-back of a partial D'),
// with the scratch loads issued a few rows ahead.  D' and L' are symmetric (the couplings are
// products of a factor of the row and one of the column).  HALF: a thread stops at the diagonal
// and mirror_kernel fills the upper triangles.  That pays where the FP64 pipe bounds the kernel
// (2020 rows of 160: 4.70 -> 3.12 + 0.28 ms), not in FP32 (0.52 -> 0.47 + 0.19), whose threads wait
// for the longest one anyway.
template <typename T, bool HALF>
__global__ void level0_schur_kernel(const double2* __restrict__ dg, const double2* __restrict__ cx,
                                    const double2* __restrict__ cy, int nx, int ny,
                                    const cplx<T>* __restrict__ tdl, const cplx<T>* __restrict__ tdinv,
                                    const cplx<T>* __restrict__ tdu, const cplx<T>* __restrict__ tdu2,
                                    const uint8_t* __restrict__ tpiv, cplx<T>* __restrict__ Dn,
                                    cplx<T>* __restrict__ Ln, cplx<T>* __restrict__ scrR,
                                    cplx<T>* __restrict__ scrL) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  cplx<T>* sm = reinterpret_cast<cplx<T>*>(sm_raw);
  // [0,4ny): right factors, [4ny,8ny): left factors, then cxl2, cxl, cxr, dge, cye; piv bytes last
  cplx<T>* R = sm;
  cplx<T>* Lf = sm + 4 * ny;
  cplx<T>* cxl2 = sm + 8 * ny;
  cplx<T>* cxl = cxl2 + ny;
  cplx<T>* cxr = cxl + ny;
  cplx<T>* dge = cxr + ny;
  cplx<T>* cye = dge + ny;
  uint8_t* pivR = reinterpret_cast<uint8_t*>(cye + ny);
  uint8_t* pivL = pivR + ny;

  const int k = blockIdx.x;
  const int64_t e = 2 * (int64_t)k;
  const bool has_r = e + 1 < nx;   // eliminated row e+1 has index k
  const bool has_l = e >= 1;       // eliminated row e-1 has index k-1
  for (int j = threadIdx.x; j < ny; j += blockDim.x) {
    if (has_r) {
      int64_t b = (int64_t)k * ny + j;
      R[j] = tdl[b];
      R[ny + j] = tdinv[b];
      R[2 * ny + j] = tdu[b];
      R[3 * ny + j] = tdu2[b];
      pivR[j] = tpiv[b];
    }
    cxr[j] = has_r ? ccast<T>(cx[e * ny + j]) : czero<T>();
    if (has_l) {
      int64_t b = (int64_t)(k - 1) * ny + j;
      Lf[j] = tdl[b];
      Lf[ny + j] = tdinv[b];
      Lf[2 * ny + j] = tdu[b];
      Lf[3 * ny + j] = tdu2[b];
      pivL[j] = tpiv[b];
      cxl[j] = ccast<T>(cx[(e - 1) * ny + j]);
      cxl2[j] = ccast<T>(cx[(e - 2) * ny + j]);
    } else {
      cxl[j] = cxl2[j] = czero<T>();
    }
    dge[j] = ccast<T>(dg[e * ny + j]);
    cye[j] = ccast<T>(cy[e * ny + j]);
  }
  __syncthreads();
  const int b = threadIdx.x;
  if (b >= ny) return;
  const int64_t nn = (int64_t)ny * ny;
  cplx<T>* __restrict__ Dcol = Dn + (int64_t)k * nn + b;
  cplx<T>* __restrict__ Lcol = Ln + (int64_t)k * nn + b;
  cplx<T>* __restrict__ YR = scrR + (int64_t)k * nn + b;
  cplx<T>* __restrict__ YL = scrL + (int64_t)k * nn + b;
  const TriRow<T> fR{R, R + ny, R + 2 * ny, R + 3 * ny, pivR};
  const TriRow<T> fL{Lf, Lf + ny, Lf + 2 * ny, Lf + 3 * ny, pivL};
  if (has_r) tri_forward_unit<T>(fR, ny, b, YR, ny);
  if (has_l) tri_forward_unit<T>(fL, ny, b, YL, ny);
  const int a_lo = b > 0 ? b - 1 : 0;  // first row the sweeps wrote
  const cplx<T> sb = cxr[b], sl = cxl[b], sl2 = cxl2[b];
  cplx<T> r1 = czero<T>(), r2 = czero<T>(), l1 = czero<T>(), l2 = czero<T>();
  // scratch values of the next PF rows, loaded ahead of the recurrences
  constexpr int PF = 4;
  cplx<T> yr[PF], yl[PF];
#pragma unroll
  for (int q = 0; q < PF; ++q) {
    const int a = ny - 1 - q;
    yr[q] = (has_r && a >= a_lo) ? YR[(int64_t)a * ny] : czero<T>();
    yl[q] = (has_l && a >= a_lo) ? YL[(int64_t)a * ny] : czero<T>();
  }
  const int a_end = HALF ? b : 0;
  for (int a0 = ny - 1; a0 >= a_end; a0 -= PF) {
#pragma unroll
    for (int q = 0; q < PF; ++q) {
      const int a = a0 - q;
      if (a < a_end) break;
      const cplx<T> cr = yr[q], cl = yl[q];
      const int an = a - PF;  // the row PF steps ahead into the same ring slot
      yr[q] = (has_r && an >= a_lo) ? YR[(int64_t)an * ny] : czero<T>();
      yl[q] = (has_l && an >= a_lo) ? YL[(int64_t)an * ny] : czero<T>();
      // T_{e+1}^{-1} and T_{e-1}^{-1}, entry (a, b)
      cplx<T> gr = cfms(fR.du2[a], r2, cfms(fR.du[a], r1, cr)) * fR.dinv[a];
      if (!has_r) gr = czero<T>();
      r2 = r1;
      r1 = gr;
      cplx<T> gl = cfms(fL.du2[a], l2, cfms(fL.du[a], l1, cl)) * fL.dinv[a];
      if (!has_l) gl = czero<T>();
      l2 = l1;
      l1 = gl;
      const cplx<T> te = a == b ? dge[a] : (a == b - 1 ? cye[a] : (a == b + 1 ? cye[b] : czero<T>()));
      const cplx<T> cgl = cxl[a] * gl;
      Dcol[(int64_t)a * ny] = cfms(cgl, sl, cfms(cxr[a] * gr, sb, te));
      if (has_l) Lcol[(int64_t)a * ny] = -(cgl * sl2);
    }
  }
}

// M[z][b][a] = M[z][a][b] for a > b: the upper triangles of the n x n blocks of two arrays from their
// lower ones, a 32 x 32 tile per block through shared memory.
template <typename T>
__global__ void __launch_bounds__(256)
mirror_kernel(cplx<T>* __restrict__ D, cplx<T>* __restrict__ L, int n, int first_l) {
  __shared__ cplx<T> t[32][33];
  const int z = blockIdx.y;
  if (blockIdx.z == 1 && z < first_l) return;
  cplx<T>* M = (blockIdx.z == 0 ? D : L) + (int64_t)z * n * n;
  int ta = 0, tb = blockIdx.x;  // tile row ta >= tile column tb
  while (tb > ta) tb -= ++ta;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int i = ty; i < 32; i += 8) {
    const int a = 32 * ta + i, b = 32 * tb + tx;
    if (a < n && b < n) t[i][tx] = M[(int64_t)a * n + b];
  }
  __syncthreads();
  for (int i = ty; i < 32; i += 8) {
    const int b = 32 * tb + i, a = 32 * ta + tx;
    if (a < n && a > b) M[(int64_t)b * n + a] = t[tx][i];
  }
}

// shared memory of level0_schur_kernel: 13 ny complex values and 2 ny pivot flags
template <typename T>
inline size_t l0_smem(int ny) {
  return (size_t)13 * ny * sizeof(cplx<T>) + 2 * (size_t)ny;
}

// ===================================================================== Gauss-Jordan
// Blocked in-place inversion with partial pivoting (largest |re|+|im| in the column,
// ties to the lowest row).  For each panel of NB columns:
//   1. NB unblocked Gauss-Jordan steps restricted to the panel columns (row swaps of the
//      panel columns only, pivot rows scaled, other rows eliminated);
//   2. the panel's row swaps, in order, applied to every other column;
//   3. every other column updated at once by M, the product of the panel's elementary
//      Gauss-Jordan transforms: M differs from the identity only in the panel columns,
//      and the in-place algorithm leaves exactly M's columns there, so
//      A_rest <- M A_rest = A_rest + M[:, panel] A_rest[panel rows] off the panel rows and
//      M[panel, panel] A_rest[panel rows] on them (forming M - I there instead would cancel
//      catastrophically for diagonally dominant blocks, whose M_kk = 1/pivot).
// Row interchanges are undone as column interchanges on output.  One block of NT threads
// per matrix; the matrix lives in shared memory (SMEM) or in global memory (the source
// slot, which is destroyed); the panel rows of step 3 are staged in shared memory, and
// the column that feeds the next pivot search is kept contiguous (coln) so the search
// reads without bank conflicts.
constexpr size_t SMEM_LIMIT = 227 * 1024;

template <typename T>
struct GjSmem {
  // byte offsets of the shared-memory regions for an n x n matrix and panel width nb
  size_t coln, colk, rowk, tpanel, perm, idx, mat, total;
  __host__ __device__ GjSmem(int n, int nb, bool smem_matrix) {
    size_t e = sizeof(cplx<T>);
    coln = 0;
    colk = coln + (size_t)n * e;
    rowk = colk + (size_t)n * e;
    tpanel = rowk + (size_t)nb * e;
    perm = tpanel + (size_t)nb * n * e;
    idx = perm + (size_t)n * sizeof(int);
    mat = (idx + (size_t)n * sizeof(int) + 15) & ~(size_t)15;
    total = mat + (smem_matrix ? (size_t)n * n * e : 0);
  }
};

// NT threads = (NT/32) x 32; the update tiles are TR rows (stride NT/32) x TC columns
// (stride 32) per thread, so within a warp the panel-column reads broadcast and the
// staged-row reads are consecutive.
template <typename T, bool SMEM, int NB, int TR, int TC, int NT>
__global__ void __launch_bounds__(NT)
gj_inverse_kernel(cplx<T>* __restrict__ src, int64_t src_stride, cplx<T>* __restrict__ out,
                  int64_t out_stride, int n, int32_t* status) {
  static_assert((NB & (NB - 1)) == 0 && NB <= 32, "panel width: power of two <= 32");
  constexpr int TY = NT / 32;
  constexpr int LNB = NB == 32 ? 5 : NB == 16 ? 4 : NB == 8 ? 3 : NB == 4 ? 2 : NB == 2 ? 1 : 0;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const GjSmem<T> L(n, NB, SMEM);
  cplx<T>* coln = reinterpret_cast<cplx<T>*>(sm_raw + L.coln);    // column k before its swap
  cplx<T>* colk = reinterpret_cast<cplx<T>*>(sm_raw + L.colk);    // column k after the swap
  cplx<T>* rowk = reinterpret_cast<cplx<T>*>(sm_raw + L.rowk);    // scaled pivot row (panel)
  cplx<T>* tp = reinterpret_cast<cplx<T>*>(sm_raw + L.tpanel);    // panel rows, other columns
  int* perm = reinterpret_cast<int*>(sm_raw + L.perm);
  int* idx = reinterpret_cast<int*>(sm_raw + L.idx);
  __shared__ int s_p;
  __shared__ cplx<T> s_pinv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  cplx<T>* g = src + (int64_t)blockIdx.x * src_stride;
  cplx<T>* a = SMEM ? reinterpret_cast<cplx<T>*>(sm_raw + L.mat) : g;
  if (SMEM) {
    for (int e = tid; e < n * n; e += NT) a[e] = g[e];
  }
  bool sing = false;
  for (int c0 = 0; c0 < n; c0 += NB) {
    const int nb = n - c0 < NB ? n - c0 : NB;
    __syncthreads();
    for (int i = tid; i < n; i += NT) coln[i] = a[i * n + c0];
    __syncthreads();
    // ---------------- panel
    for (int k = c0; k < c0 + nb; ++k) {
      if (warp == 0) {
        T best = T(-1);
        int bi = k;
        for (int i = k + lane; i < n; i += 32) {
          T v = cabs1(coln[i]);
          if (v > best) {
            best = v;
            bi = i;
          }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
          T ob = __shfl_down_sync(0xffffffffu, best, off);
          int oi = __shfl_down_sync(0xffffffffu, bi, off);
          if (ob > best || (ob == best && oi < bi)) {
            best = ob;
            bi = oi;
          }
        }
        if (lane == 0) {
          s_p = bi;
          if (!(best > T(0))) sing = true;
          s_pinv = crecip(coln[bi]);
          perm[k] = bi;
        }
      }
      __syncthreads();
      const int p = s_p;
      const cplx<T> pinv = s_pinv;
      for (int i = tid; i < n; i += NT) colk[i] = coln[i == k ? p : (i == p ? k : i)];
      if (tid < nb) {
        const int j = c0 + tid;
        cplx<T> rk = a[k * n + j];
        cplx<T> rp = a[p * n + j];
        cplx<T> v = (j == k ? mkc(T(1), T(0)) : rp) * pinv;
        if (p != k) a[p * n + j] = rk;
        a[k * n + j] = v;
        rowk[tid] = v;
      }
      __syncthreads();
      const int knext = k + 1 - c0;  // panel column whose new values feed the next pivot search
      const int kt = k - c0;
      for (int e = tid; e < (n << LNB); e += NT) {
        const int i = e >> LNB, t = e & (NB - 1);
        if (t >= nb) continue;
        const int j = c0 + t;
        if (i != k) {
          cplx<T> base = (t == kt) ? czero<T>() : a[i * n + j];
          cplx<T> v = cfms(colk[i], rowk[t], base);
          a[i * n + j] = v;
          if (t == knext) coln[i] = v;
        } else if (t == knext) {
          coln[i] = rowk[t];
        }
      }
      __syncthreads();
    }
    const int m = n - nb;
    if (m == 0) continue;
    // ---------------- panel row swaps on the other columns, in order; stage panel rows
    for (int jj = tid; jj < m; jj += NT) {
      const int j = jj < c0 ? jj : jj + nb;
      for (int t = 0; t < nb; ++t) {
        const int r = c0 + t, p = perm[r];
        if (p != r) {
          cplx<T> x = a[r * n + j];
          a[r * n + j] = a[p * n + j];
          a[p * n + j] = x;
        }
      }
    }
    __syncthreads();
    for (int t = 0; t < nb; ++t)
      for (int jj = tid; jj < m; jj += NT) {
        const int j = jj < c0 ? jj : jj + nb;
        tp[t * m + jj] = a[(c0 + t) * n + j];
      }
    __syncthreads();
    // ---------------- other columns (register tiles TR x TC)
    const int ty = warp, tx = lane;
    for (int r0 = 0; r0 < n; r0 += TY * TR) {
      for (int q0 = 0; q0 < m; q0 += 32 * TC) {
        cplx<T> acc[TR][TC];
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
          for (int c = 0; c < TC; ++c) {
            const int i = r0 + ty + TY * r, jj = q0 + tx + 32 * c;
            const int j = jj < c0 ? jj : jj + nb;
            const bool panel_row = i >= c0 && i < c0 + nb;
            acc[r][c] = (i < n && jj < m && !panel_row) ? a[i * n + j] : czero<T>();
          }
        for (int t = 0; t < nb; ++t) {
          cplx<T> zv[TR], tv[TC];
#pragma unroll
          for (int r = 0; r < TR; ++r) {
            const int i = r0 + ty + TY * r;
            zv[r] = i < n ? a[i * n + c0 + t] : czero<T>();
          }
#pragma unroll
          for (int c = 0; c < TC; ++c) {
            const int jj = q0 + tx + 32 * c;
            tv[c] = jj < m ? tp[t * m + jj] : czero<T>();
          }
#pragma unroll
          for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < TC; ++c) acc[r][c] = cfma(zv[r], tv[c], acc[r][c]);
        }
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
          for (int c = 0; c < TC; ++c) {
            const int i = r0 + ty + TY * r, jj = q0 + tx + 32 * c;
            const int j = jj < c0 ? jj : jj + nb;
            if (i < n && jj < m) a[i * n + j] = acc[r][c];
          }
      }
    }
  }
  __syncthreads();
  if (tid == 0) {
    for (int j = 0; j < n; ++j) idx[j] = j;
    for (int k = n - 1; k >= 0; --k) {
      int p = perm[k];
      int t = idx[k];
      idx[k] = idx[p];
      idx[p] = t;
    }
    if (sing) atomicCAS(status, DEV_OK, DEV_SINGULAR);
  }
  __syncthreads();
  cplx<T>* o = out + (int64_t)blockIdx.x * out_stride;
  for (int i = 0; i < n; ++i)
    for (int j = tid; j < n; j += NT) o[i * n + j] = a[i * n + idx[j]];
}

// Register-panel variant: the panel is NB = NT/32 columns wide and warp t holds panel
// column t in registers (lane L keeps rows L, L+32, ..., R slots).  A pivot step then
// costs one block barrier: after its own update, the warp that holds the next pivot
// column searches it (shuffles), publishes the swapped column, the pivot row index and
// 1/pivot to a double-buffered shared slot, and every warp updates its column from that
// slot and from shuffles of its own registers (rows k and p).  The update of the other
// columns after each panel is the one of gj_inverse_kernel.
template <typename T, int R>
__device__ __forceinline__ cplx<T> reg_select(const cplx<T> (&x)[R], int s) {
  cplx<T> v = x[0];
#pragma unroll
  for (int r = 1; r < R; ++r)
    if (s == r) v = x[r];
  return v;
}

template <typename T>
__device__ __forceinline__ cplx<T> shfl_c(cplx<T> v, int src) {
  return mkc(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// value held for row `row` by the warp (row = slot * 32 + lane)
template <typename T, int R>
__device__ __forceinline__ cplx<T> warp_row(const cplx<T> (&x)[R], int row) {
  return shfl_c<T>(reg_select<T, R>(x, row >> 5), row & 31);
}

// Pivot search on the warp's column (rows k..n-1), ties to the lowest row; publishes the
// column after the swap of rows k and p, p and 1/pivot.  Returns false if singular.
template <typename T, int R>
__device__ __forceinline__ bool gj_pivot(const cplx<T> (&x)[R], int k, int n, int lane,
                                         cplx<T>* colk, int* s_p, cplx<T>* s_pinv, int* perm) {
  T best = T(-1);
  int bi = k;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = lane + 32 * r;
    if (i >= k && i < n) {
      T v = cabs1(x[r]);
      if (v > best) {
        best = v;
        bi = i;
      }
    }
  }
  if constexpr (sizeof(T) == 4) {
    // |re| + |im| >= 0, so its bit pattern orders like the value: the largest key over the
    // warp, then the lowest row holding it (a lane without rows has key 0 and row k, which
    // changes nothing: row k itself is a candidate whenever the maximum is 0)
    const uint32_t key = best >= T(0) ? __float_as_uint(best) : 0u;
    const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
    bi = (int)__reduce_min_sync(0xffffffffu, key == kmax ? (uint32_t)bi : 0xffffffffu);
    best = __uint_as_float(kmax);
  } else {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      T ob = __shfl_xor_sync(0xffffffffu, best, off);
      int oi = __shfl_xor_sync(0xffffffffu, bi, off);
      if (ob > best || (ob == best && oi < bi)) {
        best = ob;
        bi = oi;
      }
    }
  }
  const int p = bi;
  const cplx<T> vp = warp_row<T, R>(x, p), vk = warp_row<T, R>(x, k);
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = lane + 32 * r;
    if (i < n) colk[i] = i == k ? vp : (i == p ? vk : x[r]);
  }
  if (lane == 0) {
    *s_p = p;
    *s_pinv = crecip(vp);
    perm[k] = p;
  }
  return best > T(0);
}

template <typename T, bool SMEM, int R, int TR, int TC, int NT>
__global__ void __launch_bounds__(NT)
gj_regpanel_kernel(cplx<T>* __restrict__ src, int64_t src_stride, cplx<T>* __restrict__ out,
                   int64_t out_stride, int n, int32_t* status, const int32_t* __restrict__ only) {
  dep_begin();
  if (only && only[blockIdx.x] == 0) return;  // (only: the blocks to invert, null for all)
  constexpr int NB = NT / 32;
  constexpr int TY = NT / 32;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const GjSmem<T> L(n, NB, SMEM);
  cplx<T>* const cbuf0 = reinterpret_cast<cplx<T>*>(sm_raw + L.coln);  // published pivot
  cplx<T>* const cbuf1 = reinterpret_cast<cplx<T>*>(sm_raw + L.colk);  // columns, alternating
  cplx<T>* tp = reinterpret_cast<cplx<T>*>(sm_raw + L.tpanel);
  int* perm = reinterpret_cast<int*>(sm_raw + L.perm);
  int* idx = reinterpret_cast<int*>(sm_raw + L.idx);
  __shared__ int s_p[2];
  __shared__ cplx<T> s_pinv[2];
  __shared__ int s_sing;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  cplx<T>* g = src + (int64_t)blockIdx.x * src_stride;
  cplx<T>* a = SMEM ? reinterpret_cast<cplx<T>*>(sm_raw + L.mat) : g;
  if (tid == 0) s_sing = 0;
  if (SMEM) {
    for (int e = tid; e < n * n; e += NT) a[e] = g[e];
  }
  for (int c0 = 0; c0 < n; c0 += NB) {
    const int nb = n - c0 < NB ? n - c0 : NB;
    const int t = warp, j = c0 + t;
    __syncthreads();
    cplx<T> x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = lane + 32 * r;
      x[r] = (t < nb && i < n) ? a[i * n + j] : czero<T>();
    }
    if (warp == 0 && !gj_pivot<T, R>(x, c0, n, lane, cbuf0, &s_p[0], &s_pinv[0], perm))
      s_sing = 1;
    __syncthreads();
    // ---------------- panel: one barrier per pivot
    for (int kt = 0; kt < nb; ++kt) {
      const int k = c0 + kt, b = kt & 1;
      if (t < nb) {
        const int p = s_p[b];
        const cplx<T> pinv = s_pinv[b];
        const cplx<T>* colk = b ? cbuf1 : cbuf0;
        const cplx<T> vp = warp_row<T, R>(x, p), vk = warp_row<T, R>(x, k);
        const cplx<T> rk = (t == kt ? mkc(T(1), T(0)) : vp) * pinv;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int i = lane + 32 * r;
          if (i < n) {
            const cplx<T> old = i == k ? vp : (i == p ? vk : x[r]);
            const cplx<T> base = t == kt ? czero<T>() : old;
            x[r] = i == k ? rk : cfms(colk[i], rk, base);
          }
        }
        if (t == kt + 1 &&
            !gj_pivot<T, R>(x, k + 1, n, lane, b ? cbuf0 : cbuf1, &s_p[b ^ 1], &s_pinv[b ^ 1],
                            perm))
          s_sing = 1;
      }
      __syncthreads();
    }
    if (t < nb) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = lane + 32 * r;
        if (i < n) a[i * n + j] = x[r];
      }
    }
    const int m = n - nb;
    if (m == 0) continue;
    // ---------------- panel row swaps on the other columns, in order; stage panel rows
    for (int jj = tid; jj < m; jj += NT) {
      const int jc = jj < c0 ? jj : jj + nb;
      for (int u = 0; u < nb; ++u) {
        const int rr = c0 + u, p = perm[rr];
        if (p != rr) {
          cplx<T> y = a[rr * n + jc];
          a[rr * n + jc] = a[p * n + jc];
          a[p * n + jc] = y;
        }
      }
    }
    __syncthreads();
    for (int u = 0; u < nb; ++u)
      for (int jj = tid; jj < m; jj += NT) {
        const int jc = jj < c0 ? jj : jj + nb;
        tp[u * m + jj] = a[(c0 + u) * n + jc];
      }
    __syncthreads();
    // ---------------- other columns (register tiles TR x TC)
    const int ty = warp, tx = lane;
    for (int r0 = 0; r0 < n; r0 += TY * TR) {
      for (int q0 = 0; q0 < m; q0 += 32 * TC) {
        cplx<T> acc[TR][TC];
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
          for (int c = 0; c < TC; ++c) {
            const int i = r0 + ty + TY * r, jj = q0 + tx + 32 * c;
            const int jc = jj < c0 ? jj : jj + nb;
            const bool panel_row = i >= c0 && i < c0 + nb;
            acc[r][c] = (i < n && jj < m && !panel_row) ? a[i * n + jc] : czero<T>();
          }
        for (int u = 0; u < nb; ++u) {
          cplx<T> zv[TR], tv[TC];
#pragma unroll
          for (int r = 0; r < TR; ++r) {
            const int i = r0 + ty + TY * r;
            zv[r] = i < n ? a[i * n + c0 + u] : czero<T>();
          }
#pragma unroll
          for (int c = 0; c < TC; ++c) {
            const int jj = q0 + tx + 32 * c;
            tv[c] = jj < m ? tp[u * m + jj] : czero<T>();
          }
#pragma unroll
          for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < TC; ++c) acc[r][c] = cfma(zv[r], tv[c], acc[r][c]);
        }
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
          for (int c = 0; c < TC; ++c) {
            const int i = r0 + ty + TY * r, jj = q0 + tx + 32 * c;
            const int jc = jj < c0 ? jj : jj + nb;
            if (i < n && jj < m) a[i * n + jc] = acc[r][c];
          }
      }
    }
  }
  __syncthreads();
  if (tid == 0) {
    for (int jx = 0; jx < n; ++jx) idx[jx] = jx;
    for (int k = n - 1; k >= 0; --k) {
      int p = perm[k];
      int y = idx[k];
      idx[k] = idx[p];
      idx[p] = y;
    }
    if (s_sing) atomicCAS(status, DEV_OK, DEV_SINGULAR);
  }
  __syncthreads();
  cplx<T>* o = out + (int64_t)blockIdx.x * out_stride;
  for (int i = 0; i < n; ++i)
    for (int jx = tid; jx < n; jx += NT) o[i * n + jx] = a[i * n + idx[jx]];
}

// Look-ahead variant for FP32 blocks held in shared memory (n <= 160), 1024 threads in
// two groups of 16 warps.  While the panel group factors panel P+1 (one named barrier per
// pivot), the trailing group applies the rank-nb update of panel P to every column outside
// panels P and P+1; the panel group has applied that update to its own columns first.
// Rows are never swapped: the pivot of column k is physical row piv[k], chosen among the
// rows not yet used as pivots, and the permutations are applied when the inverse is
// written out (inverse[i][j] = M[piv[i]][pinv[j]] for the in-place result M).  Every entry
// is formed by the same operations as with explicit swaps, so the result equals that of
// gj_regpanel_kernel whenever no two pivot candidates tie.  The matrix row stride is odd
// (n | 1 entries), so that a warp reading one column (rows lane, lane + 32, ...) meets no
// bank conflict.
constexpr int GJLA_THREADS = 1024, GJLA_NB = 16, GJLA_R = 5, GJLA_TR = 5, GJLA_TC = 2;

struct GjLaSmem {
  // byte offsets for an n x n complex-FP32 matrix (odd row stride n | 1)
  size_t cb0, cb1, tpanel, piv, rowpanel, pinv, mat, total;
  __host__ __device__ GjLaSmem(int n) {
    const size_t e = sizeof(float2);
    const size_t tmax = (size_t)GJLA_NB * (n > GJLA_NB ? n - GJLA_NB : 1);
    cb0 = 0;
    cb1 = cb0 + (size_t)n * e;
    tpanel = cb1 + (size_t)n * e;
    piv = tpanel + tmax * e;
    rowpanel = piv + (size_t)n * sizeof(int);
    pinv = rowpanel + (size_t)n * sizeof(int);
    mat = (pinv + (size_t)n * sizeof(int) + 15) & ~(size_t)15;
    total = mat + (size_t)n * (n | 1) * e;
  }
};

__device__ __forceinline__ void group_bar(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(GJLA_THREADS / 2) : "memory");
}

// Pivot of column k held by this warp (rows lane + 32 r, `used` marks rows already taken):
// the largest |re| + |im| among unused rows, ties to the lowest row; publishes the column,
// the row, 1/pivot, piv[k] and rowpanel[row] = c0.  Returns false if the column is zero
// on every unused row (or holds no number there).
__device__ __forceinline__ bool gjla_pivot(const float2 (&x)[GJLA_R], unsigned used, int k,
                                           int c0, int n, int lane, float2* colk, int* s_p,
                                           float2* s_pinv, int* piv, volatile int* rowpanel) {
  constexpr int R = GJLA_R;
  float best = -1.f;
  int bi = 0x7fffffff, first = 0x7fffffff;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = lane + 32 * r;
    if (i < n) {
      colk[i] = x[r];
      if (!((used >> r) & 1u)) {
        const float v = cabs1(x[r]);
        if (first == 0x7fffffff) first = i;
        if (v > best) {
          best = v;
          bi = i;
        }
      }
    }
  }
  // |re| + |im| >= 0 orders like its bit pattern: the largest key over the warp, then the
  // lowest row holding it; a lane without a candidate offers key 0 and its first unused row
  if (best < 0.f) bi = first;
  const uint32_t key = best >= 0.f ? __float_as_uint(best) : 0u;
  const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
  const int p = (int)__reduce_min_sync(0xffffffffu, key == kmax ? (uint32_t)bi : 0xffffffffu);
  const float2 vp = warp_row<float, R>(x, p);
  if (lane == 0) {
    *s_p = p;
    *s_pinv = crecip(vp);
    piv[k] = p;
    rowpanel[p] = c0;
  }
  return __uint_as_float(kmax) > 0.f;
}

// Panel group: Gauss-Jordan steps on columns c0 .. c0+nb-1, warp t holding column c0 + t
// in x (rows lane + 32 r); the columns are written back to the matrix at the end.
__device__ __forceinline__ void gjla_panel(float2 (&x)[GJLA_R], int c0, int nb, int n, int ld,
                                           float2* a, float2* cbuf0, float2* cbuf1, int* s_p,
                                           float2* s_pinv, int* piv, volatile int* rowpanel,
                                           int* s_sing) {
  constexpr int R = GJLA_R;
  const int lane = threadIdx.x & 31, t = threadIdx.x >> 5;
  unsigned used = 0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = lane + 32 * r;
    if (i >= n || rowpanel[i] >= 0) used |= 1u << r;
  }
  if (t == 0 && !gjla_pivot(x, used, c0, c0, n, lane, cbuf0, &s_p[0], &s_pinv[0], piv, rowpanel))
    *s_sing = 1;
  group_bar(1);
  for (int kt = 0; kt < nb; ++kt) {
    const int b = kt & 1;
    if (t < nb) {
      const int p = s_p[b];
      const float2 pinv = s_pinv[b];
      const float2* colk = b ? cbuf1 : cbuf0;
      if (lane == (p & 31)) used |= 1u << (p >> 5);
      if (t == kt) {
        // the pivot column becomes -column / pivot, and 1 / pivot on the pivot row
        const float2 rk = mkc(1.f, 0.f) * pinv;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int i = lane + 32 * r;
          if (i < n) x[r] = i == p ? rk : cfms(colk[i], rk, czero<float>());
        }
      } else {
        const float2 rk = warp_row<float, R>(x, p) * pinv;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int i = lane + 32 * r;
          if (i < n) x[r] = i == p ? rk : cfms(colk[i], rk, x[r]);
        }
      }
      if (t == kt + 1 && !gjla_pivot(x, used, c0 + kt + 1, c0, n, lane, b ? cbuf0 : cbuf1,
                                     &s_p[b ^ 1], &s_pinv[b ^ 1], piv, rowpanel))
        *s_sing = 1;
    }
    group_bar(1);
  }
  if (t < nb) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = lane + 32 * r;
      if (i < n) a[i * ld + c0 + t] = x[r];
    }
  }
}

__global__ void __launch_bounds__(GJLA_THREADS)
gj_lookahead_kernel(const float2* __restrict__ src, int64_t src_stride, float2* __restrict__ out,
                    int64_t out_stride, int n, int32_t* status) {
  constexpr int R = GJLA_R, NB = GJLA_NB, TR = GJLA_TR, TC = GJLA_TC, TY = 16;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const GjLaSmem L(n);
  float2* const cbuf0 = reinterpret_cast<float2*>(sm_raw + L.cb0);
  float2* const cbuf1 = reinterpret_cast<float2*>(sm_raw + L.cb1);
  float2* const tp = reinterpret_cast<float2*>(sm_raw + L.tpanel);
  int* const piv = reinterpret_cast<int*>(sm_raw + L.piv);
  // panel start at which the row became a pivot, -1 before: the trailing group reads it for
  // the rows of panel P while the panel group sets it for rows of panel P+1 (from -1 to
  // c0 + nb); either value differs from c0 of panel P, so the reading does not depend on
  // the order.  All accesses are volatile (relaxed), which makes the overlap well defined.
  volatile int* const rowpanel = reinterpret_cast<volatile int*>(sm_raw + L.rowpanel);
  int* const pinv = reinterpret_cast<int*>(sm_raw + L.pinv);
  float2* const a = reinterpret_cast<float2*>(sm_raw + L.mat);
  __shared__ int s_p[2];
  __shared__ float2 s_pinv[2];
  __shared__ int s_sing;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ld = n | 1;
  const bool panel_group = warp < 16;
  const float2* g = src + (int64_t)blockIdx.x * src_stride;
  if (tid == 0) s_sing = 0;
  for (int i = tid; i < n; i += GJLA_THREADS) rowpanel[i] = -1;
  for (int e = tid; e < n * n; e += GJLA_THREADS) {
    const int i = e / n, j = e - i * n;
    a[i * ld + j] = g[e];
  }
  __syncthreads();
  float2 x[R];
  if (panel_group) {
    const int nb0 = n < NB ? n : NB;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = lane + 32 * r;
      x[r] = (warp < nb0 && i < n) ? a[i * ld + warp] : czero<float>();
    }
    gjla_panel(x, 0, nb0, n, ld, a, cbuf0, cbuf1, s_p, s_pinv, piv, rowpanel, &s_sing);
  }
  __syncthreads();
  for (int c0 = 0; c0 < n; c0 += NB) {
    const int nb = n - c0 < NB ? n - c0 : NB;
    const int c1 = c0 + nb;                                 // next panel
    const int nb1 = n - c1 < NB ? n - c1 : NB;              // its width (0: none)
    if (n - nb == 0) break;
    if (panel_group) {
      if (nb1 > 0) {
        const int j = c1 + warp;
        if (warp < nb1) {
          // this column: the rank-nb update of panel P (its pivot rows start from zero)
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int i = lane + 32 * r;
            x[r] = (i < n && rowpanel[i] != c0) ? a[i * ld + j] : czero<float>();
          }
          for (int u = 0; u < nb; ++u) {
            const float2 tv = a[piv[c0 + u] * ld + j];
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const int i = lane + 32 * r;
              if (i < n) x[r] = cfma(a[i * ld + c0 + u], tv, x[r]);
            }
          }
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) x[r] = czero<float>();
        }
        gjla_panel(x, c1, nb1, n, ld, a, cbuf0, cbuf1, s_p, s_pinv, piv, rowpanel, &s_sing);
      }
    } else {
      // trailing group: columns q = 0 .. mt-1, matrix column jc(q), outside panels P, P+1
      const int tt = tid - GJLA_THREADS / 2, ty = warp - 16, tx = lane;
      const int mt = n - nb - nb1;
      for (int u = 0; u < nb; ++u) {
        const int pr = piv[c0 + u];
        for (int q = tt; q < mt; q += GJLA_THREADS / 2) {
          const int jc = q < c0 ? q : q + nb + nb1;
          tp[u * mt + q] = a[pr * ld + jc];
        }
      }
      group_bar(2);
      for (int r0 = 0; r0 < n; r0 += TY * TR) {
        bool prow[TR];
#pragma unroll
        for (int r = 0; r < TR; ++r) {
          const int i = r0 + ty + TY * r;
          prow[r] = i < n && rowpanel[i] == c0;
        }
        for (int q0 = 0; q0 < mt; q0 += 32 * TC) {
          float2 acc[TR][TC];
#pragma unroll
          for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < TC; ++c) {
              const int i = r0 + ty + TY * r, q = q0 + tx + 32 * c;
              const int jc = q < c0 ? q : q + nb + nb1;
              acc[r][c] = (i < n && q < mt && !prow[r]) ? a[i * ld + jc] : czero<float>();
            }
          for (int u = 0; u < nb; ++u) {
            float2 zv[TR], tv[TC];
#pragma unroll
            for (int r = 0; r < TR; ++r) {
              const int i = r0 + ty + TY * r;
              zv[r] = i < n ? a[i * ld + c0 + u] : czero<float>();
            }
#pragma unroll
            for (int c = 0; c < TC; ++c) {
              const int q = q0 + tx + 32 * c;
              tv[c] = q < mt ? tp[u * mt + q] : czero<float>();
            }
#pragma unroll
            for (int r = 0; r < TR; ++r)
#pragma unroll
              for (int c = 0; c < TC; ++c) acc[r][c] = cfma(zv[r], tv[c], acc[r][c]);
          }
#pragma unroll
          for (int r = 0; r < TR; ++r)
#pragma unroll
            for (int c = 0; c < TC; ++c) {
              const int i = r0 + ty + TY * r, q = q0 + tx + 32 * c;
              const int jc = q < c0 ? q : q + nb + nb1;
              if (i < n && q < mt) a[i * ld + jc] = acc[r][c];
            }
        }
      }
    }
    __syncthreads();
  }
  for (int l = tid; l < n; l += GJLA_THREADS) pinv[piv[l]] = l;
  if (tid == 0 && s_sing) atomicCAS(status, DEV_OK, DEV_SINGULAR);
  __syncthreads();
  float2* o = out + (int64_t)blockIdx.x * out_stride;
  for (int e = tid; e < n * n; e += GJLA_THREADS) {
    const int i = e / n, jx = e - i * n;
    o[e] = a[piv[i] * ld + pinv[jx]];
  }
}

cudaError_t launch_gj_lookahead(const float2* src, int64_t src_stride, float2* out,
                                int64_t out_stride, int n, int batch, int32_t* status,
                                cudaStream_t s) {
  const GjLaSmem L(n);
  if (L.total > SMEM_LIMIT || n > 32 * GJLA_R) return cudaErrorInvalidValue;
  if (L.total > 48 * 1024)
    RCI_CUDA_TRY(cudaFuncSetAttribute(gj_lookahead_kernel,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.total));
  gj_lookahead_kernel<<<batch, GJLA_THREADS, L.total, s>>>(src, src_stride, out, out_stride, n,
                                                           status);
  rci_note_launch();
  return cudaGetLastError();
}

template <typename T, bool SMEM, int R, int TR, int TC, int NT>
cudaError_t launch_gj_reg(cplx<T>* src, int64_t src_stride, cplx<T>* out, int64_t out_stride,
                          int n, int batch, int32_t* status, cudaStream_t s,
                          const int32_t* only = nullptr) {
  const GjSmem<T> L(n, NT / 32, SMEM);
  if (L.total > SMEM_LIMIT || n > 32 * R) return cudaErrorInvalidValue;
  if (L.total > 48 * 1024)
    RCI_CUDA_TRY(cudaFuncSetAttribute(gj_regpanel_kernel<T, SMEM, R, TR, TC, NT>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.total));
  RCI_CUDA_TRY(launch_dep(gj_regpanel_kernel<T, SMEM, R, TR, TC, NT>, batch, NT, L.total, s, src, src_stride, out,
                          out_stride, n, status, only));
  rci_note_launch();
  return cudaGetLastError();
}

template <typename T, bool SMEM, int NB, int TR, int TC, int NT>
cudaError_t launch_gj_cfg(cplx<T>* src, int64_t src_stride, cplx<T>* out, int64_t out_stride,
                          int n, int batch, int32_t* status, cudaStream_t s) {
  const GjSmem<T> L(n, NB, SMEM);
  if (L.total > SMEM_LIMIT) return cudaErrorInvalidValue;
  if (L.total > 48 * 1024)
    RCI_CUDA_TRY(cudaFuncSetAttribute(gj_inverse_kernel<T, SMEM, NB, TR, TC, NT>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.total));
  gj_inverse_kernel<T, SMEM, NB, TR, TC, NT><<<batch, NT, L.total, s>>>(src, src_stride, out,
                                                                        out_stride, n, status);
  rci_note_launch();
  return cudaGetLastError();
}

// Batched inverses of n x n blocks: FP32 blocks of n <= 160 with the look-ahead kernel
// (block in shared memory, 1024 threads); other FP32 blocks up to 256 and FP64 blocks up to
// 256 with the register-panel kernel (shared memory while the block fits, else in place in
// global memory); larger blocks with gj_inverse_kernel.
template <typename T>
cudaError_t launch_gj_simt(cplx<T>* src, int64_t src_stride, cplx<T>* out, int64_t out_stride,
                           int n, int batch, int32_t* status, cudaStream_t s,
                           const int32_t* only = nullptr) {
  if (batch <= 0) return cudaSuccess;
  if (n > 1024 || (only && ((sizeof(T) == 4 && n <= 160) || n > 256))) return cudaErrorInvalidValue;
  if constexpr (sizeof(T) == 4) {
    if (n <= 160 && GjLaSmem(n).total <= SMEM_LIMIT)
      return launch_gj_lookahead(src, src_stride, out, out_stride, n, batch, status, s);
    if (n <= 160 && GjSmem<T>(n, 16, true).total <= SMEM_LIMIT)
      return launch_gj_reg<T, true, 5, 5, 5, 512>(src, src_stride, out, out_stride, n, batch,
                                                  status, s);
    if (n <= 256)
      return launch_gj_reg<T, false, 8, 5, 5, 512>(src, src_stride, out, out_stride, n, batch,
                                                   status, s, only);
    return launch_gj_cfg<T, false, 16, 5, 5, 512>(src, src_stride, out, out_stride, n, batch,
                                                  status, s);
  } else {
    if (n <= 160 && GjSmem<T>(n, 8, true).total <= SMEM_LIMIT)
      return launch_gj_reg<T, true, 5, 5, 5, 256>(src, src_stride, out, out_stride, n, batch,
                                                  status, s, only);
    if (n <= 256)
      return launch_gj_reg<T, false, 8, 5, 5, 256>(src, src_stride, out, out_stride, n, batch,
                                                   status, s, only);
    if (GjSmem<T>(n, 16, false).total <= SMEM_LIMIT)
      return launch_gj_cfg<T, false, 16, 5, 5, 256>(src, src_stride, out, out_stride, n, batch,
                                                    status, s);
    return launch_gj_cfg<T, false, 8, 5, 5, 256>(src, src_stride, out, out_stride, n, batch,
                                                 status, s);
  }
}

// Batched inverses: FP32 blocks of n <= 160 on the tensor cores (tc_gj.cu: blocked
// Gauss-Jordan with tcgen05 panel updates, block in tensor memory); everything else with the
// SIMT kernels above.
// Largest |re|, |im| over `batch` n x n blocks (stride in elements) into *maxabs (float bits,
// atomicMax), for the growth estimate of the SIMT paths (the tensor-core kernel records it
// while it reads its blocks).
template <typename T>
__global__ void block_maxabs_kernel(const cplx<T>* __restrict__ a, int64_t stride, int64_t nn,
                                    int batch, uint32_t* maxabs) {
  float m = 0.f;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nn * batch;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t z = e / nn;
    const cplx<T> v = a[z * stride + (e - z * nn)];
    m = fmaxf(m, (float)fmax(fabs(v.x), fabs(v.y)));
  }
  const uint32_t wm = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
  if ((threadIdx.x & 31) == 0) atomicMax(maxabs, wm);
}

template <typename T>
cudaError_t launch_block_maxabs(const cplx<T>* src, int64_t stride, int64_t nn, int batch, uint32_t* maxabs,
                                cudaStream_t s) {
  const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(nn * batch, 256), 4 * 152);
  block_maxabs_kernel<T><<<grid, 256, 0, s>>>(src, stride, nn, batch, maxabs);
  rci_note_launch();
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_gj(cplx<T>* src, int64_t src_stride, cplx<T>* out, int64_t out_stride, int n,
                      int batch, int32_t* status, cudaStream_t s, uint32_t* maxabs = nullptr,
                      bool tc = true) {
  if (batch <= 0) return cudaSuccess;
  if constexpr (sizeof(T) == 4) {
    if (tc && n <= 160)
      return launch_tc_gj(src, src_stride, out, out_stride, n, batch, status, s, maxabs);
  }
  if (maxabs)
    RCI_CUDA_TRY(launch_block_maxabs<T>(src, src_stride, (int64_t)n * n, batch, maxabs, s));
  return launch_gj_simt<T>(src, src_stride, out, out_stride, n, batch, status, s);
}

// Largest |re|, |im| of the operator's coefficients (diagonal and couplings)
__global__ void coeff_maxabs_kernel(const double2* __restrict__ dg, const double2* __restrict__ cx,
                                    const double2* __restrict__ cy, int64_t N, uint32_t* maxabs) {
  float m = 0.f;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N;
       e += (int64_t)gridDim.x * blockDim.x) {
    const double2 a = dg[e], b = cx[e], c = cy[e];
    const double v = fmax(fmax(fmax(fabs(a.x), fabs(a.y)), fmax(fabs(b.x), fabs(b.y))),
                          fmax(fabs(c.x), fabs(c.y)));
    m = fmaxf(m, (float)v);
  }
  const uint32_t wm = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
  if ((threadIdx.x & 31) == 0) atomicMax(maxabs, wm);
}

// ===================================================================== batched GEMM
// C[z] = alpha op(A[z]) op(B[z]) + beta C0[z]   (row-major, complex, op = N or T,
// no conjugation), z = blockIdx.z.  16 x 16 threads, each TM x TN outputs (strided
// by 16 so shared-memory reads are conflict-free), K tiles of 16.
template <typename T>
struct GemmArgs {
  int M, N, K;
  const cplx<T>* A;
  int64_t lda, sA;
  const cplx<T>* B;
  int64_t ldb, sB;
  cplx<T>* C;
  int64_t ldc, sC;
  const cplx<T>* C0;
  int64_t ldc0, sC0;
  cplx<T> alpha, beta;
};

template <typename T, int TM, int TN, bool TA, bool TB>
__global__ void __launch_bounds__(256) cgemm_kernel(GemmArgs<T> p) {
  constexpr int BM = 16 * TM, BN = 16 * TN, BK = 16;
  __shared__ cplx<T> As[BK][BM];
  __shared__ cplx<T> Bs[BK][BN];
  const int64_t z = blockIdx.z;
  const cplx<T>* A = p.A + z * p.sA;
  const cplx<T>* B = p.B + z * p.sB;
  const int i0 = blockIdx.y * BM, j0 = blockIdx.x * BN;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  cplx<T> acc[TM][TN];
#pragma unroll
  for (int r = 0; r < TM; ++r)
#pragma unroll
    for (int c = 0; c < TN; ++c) acc[r][c] = czero<T>();
  for (int k0 = 0; k0 < p.K; k0 += BK) {
#pragma unroll
    for (int e = tid; e < BM * BK; e += 256) {
      int i, kk;
      if (!TA) {
        i = e / BK;
        kk = e - i * BK;
      } else {
        kk = e / BM;
        i = e - kk * BM;
      }
      int gi = i0 + i, gk = k0 + kk;
      cplx<T> v = czero<T>();
      if (gi < p.M && gk < p.K) v = TA ? A[(int64_t)gk * p.lda + gi] : A[(int64_t)gi * p.lda + gk];
      As[kk][i] = v;
    }
#pragma unroll
    for (int e = tid; e < BK * BN; e += 256) {
      int j, kk;
      if (!TB) {
        kk = e / BN;
        j = e - kk * BN;
      } else {
        j = e / BK;
        kk = e - j * BK;
      }
      int gj = j0 + j, gk = k0 + kk;
      cplx<T> v = czero<T>();
      if (gj < p.N && gk < p.K) v = TB ? B[(int64_t)gj * p.ldb + gk] : B[(int64_t)gk * p.ldb + gj];
      Bs[kk][j] = v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      cplx<T> av[TM], bv[TN];
#pragma unroll
      for (int r = 0; r < TM; ++r) av[r] = As[kk][ty + 16 * r];
#pragma unroll
      for (int c = 0; c < TN; ++c) bv[c] = Bs[kk][tx + 16 * c];
#pragma unroll
      for (int r = 0; r < TM; ++r)
#pragma unroll
        for (int c = 0; c < TN; ++c) acc[r][c] = cfma(av[r], bv[c], acc[r][c]);
    }
    __syncthreads();
  }
  cplx<T>* C = p.C + z * p.sC;
  const cplx<T>* C0 = p.C0 ? p.C0 + z * p.sC0 : nullptr;
#pragma unroll
  for (int r = 0; r < TM; ++r) {
    int gi = i0 + ty + 16 * r;
    if (gi >= p.M) continue;
#pragma unroll
    for (int c = 0; c < TN; ++c) {
      int gj = j0 + tx + 16 * c;
      if (gj >= p.N) continue;
      cplx<T> v = p.alpha * acc[r][c];
      if (C0) v = cfma(p.beta, C0[(int64_t)gi * p.ldc0 + gj], v);
      C[(int64_t)gi * p.ldc + gj] = v;
    }
  }
}

inline int pick_tile(int d) {
  if (d % 80 == 0) return 5;
  if (d % 64 == 0) return 4;
  if (d % 48 == 0) return 3;
  if (d <= 48) return 3;
  return 4;
}

template <typename T, int TM, int TN>
cudaError_t gemm_tn(const GemmArgs<T>& a, bool ta, bool tb, int batch, cudaStream_t s) {
  dim3 grd((unsigned)ceil_div(a.N, 16 * TN), (unsigned)ceil_div(a.M, 16 * TM), (unsigned)batch);
  if (!ta && !tb) cgemm_kernel<T, TM, TN, false, false><<<grd, 256, 0, s>>>(a);
  else if (!ta && tb) cgemm_kernel<T, TM, TN, false, true><<<grd, 256, 0, s>>>(a);
  else if (ta && !tb) cgemm_kernel<T, TM, TN, true, false><<<grd, 256, 0, s>>>(a);
  else return cudaErrorInvalidValue;
  rci_note_launch();
  return cudaGetLastError();
}

template <typename T, int TM>
cudaError_t gemm_m(const GemmArgs<T>& a, bool ta, bool tb, int batch, cudaStream_t s) {
  switch (pick_tile(a.N)) {
    case 3: return gemm_tn<T, TM, 3>(a, ta, tb, batch, s);
    case 5: return gemm_tn<T, TM, 5>(a, ta, tb, batch, s);
    default: return gemm_tn<T, TM, 4>(a, ta, tb, batch, s);
  }
}

// Batched GEMM with element strides between the batch members.
template <typename T>
cudaError_t gemm(int M, int N, int K, bool ta, bool tb, cplx<T> alpha, const cplx<T>* A,
                 int64_t lda, int64_t sA, const cplx<T>* B, int64_t ldb, int64_t sB, cplx<T> beta,
                 const cplx<T>* C0, int64_t ldc0, int64_t sC0, cplx<T>* C, int64_t ldc,
                 int64_t sC, int batch, cudaStream_t s, Profiler* prof = nullptr,
                 int fam = PF_GEMM, int32_t* status = nullptr) {
  if (batch <= 0) return cudaSuccess;
  if (batch > 65535) return cudaErrorInvalidValue;
  ProfScope ps(prof, fam, s, 8.0 * M * N * K * (double)batch,
               (double)sizeof(cplx<T>) * batch * ((double)M * K + (double)K * N + (double)M * N), 1);
  GemmArgs<T> a{M, N, K, A, lda, sA, B, ldb, sB, C, ldc, sC, C0, ldc0, sC0, alpha, beta};
  // small batches (the last reduction levels) leave most SMs idle with large tiles and
  // are latency-bound: use 32 x 32 output tiles there
  const int64_t big_tiles = (int64_t)batch * ceil_div(M, 80) * ceil_div(N, 80);
  // FP32 products run on the tensor cores (3xTF32): the TMA-fed kernel at any batch where it
  // applies (its 64-row tiles keep even one product on several SMs, and a tile takes a few
  // microseconds); the register-staged kernels where enough tiles fill the GPU
  if constexpr (sizeof(T) == 4) {
    if (status && alpha.y == 0.f && beta.y == 0.f) {
      const cudaError_t e = launch_tc_cgemm_tma(M, N, K, ta, tb, alpha.x, A, lda, sA, B, ldb, sB,
                                                beta.x, C0, ldc0, sC0, C, ldc, sC, batch, status,
                                                tc_wait_limit(), s);
      if (e != cudaErrorNotSupported) return e;
    }
    const int64_t tc_tiles = (int64_t)batch * ceil_div(M, 128) * ceil_div(N, 80);
    if (status && tc_tiles >= 152)
      return launch_tc_cgemm(M, N, K, ta, tb, alpha, A, lda, sA, B, ldb, sB, beta, C0, ldc0, sC0,
                             C, ldc, sC, batch, status, s, 1);
  }
  if (big_tiles < 2 * 152) return gemm_tn<T, 2, 2>(a, ta, tb, batch, s);
  switch (pick_tile(M)) {
    case 3: return gemm_m<T, 3>(a, ta, tb, batch, s);
    case 5: return gemm_m<T, 5>(a, ta, tb, batch, s);
    default: return gemm_m<T, 4>(a, ta, tb, batch, s);
  }
}

// ===================================================================== solve kernels
// Sweeps with the tridiagonal factors for one right-hand side per thread, TRM_PF rows at a time:
// their right-hand sides and factors are loaded before the recurrence runs over them, so that a
// thread waits for memory once per TRM_PF rows.  out rows are ld apart.
constexpr int TRM_PF = 8;

template <typename T, typename Rhs>
__device__ __forceinline__ void tri_solve_rows(const TriRow<T>& f, int n, Rhs rhs, cplx<T>* out, int64_t ld) {
  cplx<T> cur = rhs(0);
  for (int j0 = 0; j0 < n - 1; j0 += TRM_PF) {
    cplx<T> nb[TRM_PF], l[TRM_PF];
    bool pv[TRM_PF];
#pragma unroll
    for (int q = 0; q < TRM_PF; ++q) {
      const int j = j0 + q < n - 1 ? j0 + q : n - 2;
      nb[q] = rhs(j + 1);
      l[q] = f.dl[j];
      pv[q] = f.piv[j] != 0;
    }
#pragma unroll
    for (int q = 0; q < TRM_PF; ++q) {
      if (j0 + q >= n - 1) break;
      out[(j0 + q) * ld] = pv[q] ? nb[q] : cur;
      cur = pv[q] ? cfms(l[q], nb[q], cur) : cfms(l[q], cur, nb[q]);
    }
  }
  out[(n - 1) * ld] = cur;
  cplx<T> g1 = czero<T>(), g2 = czero<T>();  // g_{j+1}, g_{j+2}
  for (int j0 = n - 1; j0 >= 0; j0 -= TRM_PF) {
    cplx<T> y[TRM_PF], du[TRM_PF], du2[TRM_PF], di[TRM_PF];
#pragma unroll
    for (int q = 0; q < TRM_PF; ++q) {
      const int j = j0 - q > 0 ? j0 - q : 0;
      y[q] = out[j * ld];
      du[q] = f.du[j];
      du2[q] = f.du2[j];
      di[q] = f.dinv[j];
    }
#pragma unroll
    for (int q = 0; q < TRM_PF; ++q) {
      if (j0 - q < 0) break;
      const cplx<T> g = cfms(du2[q], g2, cfms(du[q], g1, y[q])) * di[q];
      out[(j0 - q) * ld] = g;
      g2 = g1;
      g1 = g;
    }
  }
}

// Level 0 forward: t0[k] = T_{2k+1}^{-1} b[2k+1] (one thread per (k, q)).  b: nrhs columns, t0:
// ld >= nrhs columns.
template <typename T>
__global__ void __launch_bounds__(128)
fwd0_kernel(const cplx<T>* __restrict__ b, cplx<T>* __restrict__ t0, int ny, int m0, int nrhs, int ld,
            const cplx<T>* __restrict__ tdl, const cplx<T>* __restrict__ tdinv, const cplx<T>* __restrict__ tdu,
            const cplx<T>* __restrict__ tdu2, const uint8_t* __restrict__ tpiv) {
  const int64_t tt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (tt >= (int64_t)m0 * nrhs) return;
  const int k = (int)(tt / nrhs), q = (int)(tt - (int64_t)k * nrhs);
  const int64_t fb = (int64_t)k * ny;
  const TriRow<T> f{tdl + fb, tdinv + fb, tdu + fb, tdu2 + fb, tpiv + fb};
  const cplx<T>* br = b + (2 * (int64_t)k + 1) * ny * nrhs + q;
  tri_solve_rows<T>(f, ny, [&](int j) { return br[(int64_t)j * nrhs]; }, t0 + (int64_t)k * ny * ld + q, ld);
}

// Level 0 kept rows: B1[k] = b[2k] - cx[2k-1] o t0[k-1] - cx[2k] o t0[k].  b: nrhs columns, t0 and
// B1: ld (the columns from nrhs on are zero).
template <typename T>
__global__ void keep0_kernel(const cplx<T>* __restrict__ b, const cplx<T>* __restrict__ t0,
                             const double2* __restrict__ cx, cplx<T>* __restrict__ B1, int nx,
                             int ny, int n1, int nrhs, int ld) {
  const int64_t row = (int64_t)ny * ld;
  const int64_t tt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (tt >= (int64_t)n1 * row) return;
  const int64_t k = tt / row, r = tt - k * row;
  const int j = (int)(r / ld), q = (int)(r - (int64_t)j * ld);
  cplx<T> v = czero<T>();
  if (q < nrhs) {
    v = b[(2 * k * ny + j) * nrhs + q];
    if (k >= 1) v = cfms(ccast<T>(cx[(2 * k - 1) * ny + j]), t0[(k - 1) * row + r], v);
    if (2 * k + 1 < nx) v = cfms(ccast<T>(cx[(2 * k) * ny + j]), t0[k * row + r], v);
  }
  B1[tt] = v;
}

// Level 0 back substitution: x[2k] = x1[k];
// x[2k+1] = T^{-1}(b[2k+1] - cx[2k] o x1[k] - cx[2k+1] o x1[k+1]).  x1: ld columns.
template <typename T>
__global__ void __launch_bounds__(128)
bwd0_kernel(const cplx<T>* __restrict__ b, const cplx<T>* __restrict__ x1, const double2* __restrict__ cx,
            cplx<T>* __restrict__ x, int nx, int ny, int n1, int nrhs, int ld, const cplx<T>* __restrict__ tdl,
            const cplx<T>* __restrict__ tdinv, const cplx<T>* __restrict__ tdu, const cplx<T>* __restrict__ tdu2,
            const uint8_t* __restrict__ tpiv) {
  const int64_t tt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (tt >= (int64_t)n1 * nrhs) return;
  const int k = (int)(tt / nrhs), q = (int)(tt - (int64_t)k * nrhs);
  const int64_t row = (int64_t)ny * nrhs, row1 = (int64_t)ny * ld;
  const cplx<T>* xa = x1 + (int64_t)k * row1 + q;
  cplx<T>* xe = x + 2 * (int64_t)k * row + q;
#pragma unroll 8
  for (int j = 0; j < ny; ++j) xe[(int64_t)j * nrhs] = xa[(int64_t)j * ld];
  const int64_t r = 2 * (int64_t)k + 1;
  if (r >= nx) return;
  const bool has_b = r + 1 < nx;
  const cplx<T>* xb = has_b ? xa + row1 : xa;
  const cplx<T>* br = b + r * row + q;
  const double2* cl = cx + (r - 1) * ny;
  const double2* cr = cx + r * ny;
  const int64_t fb = (int64_t)k * ny;
  const TriRow<T> f{tdl + fb, tdinv + fb, tdu + fb, tdu2 + fb, tpiv + fb};
  tri_solve_rows<T>(f, ny, [&](int j) {
    cplx<T> v = cfms(ccast<T>(cl[j]), xa[(int64_t)j * ld], br[(int64_t)j * nrhs]);
    const cplx<T> c = has_b ? ccast<T>(cr[j]) : czero<T>();
    return has_b ? cfms(c, xb[(int64_t)j * ld], v) : v;
  }, x + r * row + q, nrhs);
}

// The sweeps of level 0 for few rows and right-hand sides, a block per row and at most TRG_COLS columns:
// factors and right-hand sides are staged in shared memory by the whole block, a thread per column runs the
// same recurrences there, and the results are stored together.  (A thread per row and column on global
// memory waits for it every TRM_PF rows, and few of them do so on a few SMs: with 32 rows of 224 and two
// columns its two sweeps took 105 and 169 us of a solve.)  BWD: bwd0_kernel's, else fwd0_kernel's work
// (t: t0 or x1).
constexpr int TRG_COLS = 32, TRG_THREADS = 128;

template <typename T, bool BWD>
__global__ void __launch_bounds__(TRG_THREADS)
tri_staged_kernel(const cplx<T>* __restrict__ b, cplx<T>* __restrict__ t, const double2* __restrict__ cx,
                  cplx<T>* __restrict__ x, int nx, int ny, int nrhs, int ld, int cols,
                  const cplx<T>* __restrict__ tdl, const cplx<T>* __restrict__ tdinv,
                  const cplx<T>* __restrict__ tdu, const cplx<T>* __restrict__ tdu2,
                  const uint8_t* __restrict__ tpiv) {
  extern __shared__ __align__(16) unsigned char trg_raw[];
  const int k = blockIdx.x, q0 = blockIdx.y * cols, qc = min(cols, nrhs - q0);
  const int64_t row = (int64_t)ny * nrhs, row1 = (int64_t)ny * ld;
  const int64_t r = 2 * (int64_t)k + 1;
  const cplx<T>* xa = t + k * row1 + q0;
  if (BWD) {
    cplx<T>* xe = x + 2 * k * row + q0;
    for (int e = threadIdx.x; e < ny * qc; e += TRG_THREADS) {
      const int j = e / qc, q = e - j * qc;
      xe[(int64_t)j * nrhs + q] = xa[(int64_t)j * ld + q];
    }
    if (r >= nx) return;
  }
  cplx<T>* f = reinterpret_cast<cplx<T>*>(trg_raw);  // dl, dinv, du, du2, then the columns, then piv
  cplx<T>* y = f + 4 * ny;
  uint8_t* piv = reinterpret_cast<uint8_t*>(y + (int64_t)ny * qc);
  const int64_t fb = (int64_t)k * ny;
  for (int j = threadIdx.x; j < ny; j += TRG_THREADS) {
    f[j] = tdl[fb + j];
    f[ny + j] = tdinv[fb + j];
    f[2 * ny + j] = tdu[fb + j];
    f[3 * ny + j] = tdu2[fb + j];
    piv[j] = tpiv[fb + j];
  }
  const cplx<T>* br = b + r * row + q0;
  const bool has_b = r + 1 < nx;
  for (int e = threadIdx.x; e < ny * qc; e += TRG_THREADS) {
    const int j = e / qc, q = e - j * qc;
    cplx<T> v = br[(int64_t)j * nrhs + q];
    if (BWD) {
      v = cfms(ccast<T>(cx[(r - 1) * ny + j]), xa[(int64_t)j * ld + q], v);
      if (has_b) v = cfms(ccast<T>(cx[r * ny + j]), xa[row1 + (int64_t)j * ld + q], v);
    }
    y[e] = v;
  }
  __syncthreads();
  if ((int)threadIdx.x < qc) {
    const TriRow<T> tr{f, f + ny, f + 2 * ny, f + 3 * ny, piv};
    cplx<T>* yq = y + threadIdx.x;
    tri_solve_rows<T>(tr, ny, [&](int j) { return yq[j * qc]; }, yq, qc);
  }
  __syncthreads();
  cplx<T>* out = BWD ? x + r * row + q0 : t + k * row1 + q0;
  const int64_t lo = BWD ? nrhs : ld;
  for (int e = threadIdx.x; e < ny * qc; e += TRG_THREADS) {
    const int j = e / qc, q = e - j * qc;
    out[j * lo + q] = y[e];
  }
}

// sum of a complex value over the 32 lanes of a warp (every lane gets the sum)
template <typename T>
__device__ __forceinline__ cplx<T> warp_sum(cplx<T> v) {
  for (int off = 16; off > 0; off >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
  }
  return v;
}

// ----- single right-hand side, chunked: a block per (block row k, chunk of RC rows or
// columns), so that even the last reduction levels spread over many SMs, and every lane
// issues all of its 16-byte loads before it reduces.
constexpr int RC = 32;
constexpr int CH_THREADS = 256, CH_WARPS = CH_THREADS / 32;

template <typename T> struct vec16;
template <> struct vec16<float> { using type = float4; static constexpr int per = 2; };
template <> struct vec16<double> { using type = double2; static constexpr int per = 1; };

template <typename T>
__device__ __forceinline__ cplx<T> dot_vec(const typename vec16<T>::type& v, const cplx<T>* x,
                                           int c, cplx<T> acc) {
  if constexpr (sizeof(T) == 4) {
    acc = cfma(mkc(v.x, v.y), x[c], acc);
    return cfma(mkc(v.z, v.w), x[c + 1], acc);
  } else {
    return cfma(v, x[c], acc);
  }
}

// out[r] (= sub[r] -) M[r, :] x  for the RC rows r0 .. r0+RC-1 (x in shared memory).
// Warp w handles rows r0 + w + CH_WARPS i; SMAX 16-byte vectors per lane and row.
template <typename T, int SMAX>
__device__ __forceinline__ void rows_mv(const cplx<T>* __restrict__ M, const cplx<T>* x, int ny,
                                        int r0, cplx<T>* out, const cplx<T>* sub) {
  using V = typename vec16<T>::type;
  constexpr int PER = vec16<T>::per;
  constexpr int RPW = RC / CH_WARPS;  // rows per warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nv = ny / PER;            // ny is a multiple of PER (checked by the launcher)
  V v[RPW][SMAX];
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    const int r = r0 + warp + CH_WARPS * i;
    const V* Mr = reinterpret_cast<const V*>(M + (int64_t)r * ny);
#pragma unroll
    for (int s = 0; s < SMAX; ++s) {
      const int q = lane + 32 * s;
      if (r < ny && q < nv) v[i][s] = __ldg(Mr + q);
    }
  }
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    const int r = r0 + warp + CH_WARPS * i;
    cplx<T> acc = czero<T>();
#pragma unroll
    for (int s = 0; s < SMAX; ++s) {
      const int q = lane + 32 * s;
      if (r < ny && q < nv) acc = dot_vec<T>(v[i][s], x, PER * q, acc);
    }
    acc = warp_sum<T>(acc);
    if (lane == 0 && r < ny) out[r] = sub ? sub[r] - acc : acc;
  }
}

// rows_mv split in two: the row loads (no dependence on x) and the products, so that a
// block can issue its loads before it waits for the vector it multiplies.
template <typename T, int SMAX>
struct Rows1 {
  typename vec16<T>::type v[RC / CH_WARPS][SMAX];
};

template <typename T, int SMAX>
__device__ __forceinline__ void rows_load1(Rows1<T, SMAX>& R, const cplx<T>* __restrict__ M, int ny,
                                           int r0) {
  using V = typename vec16<T>::type;
  constexpr int PER = vec16<T>::per;
  constexpr int RPW = RC / CH_WARPS;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nv = ny / PER;
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    const int r = r0 + warp + CH_WARPS * i;
    const V* Mr = reinterpret_cast<const V*>(M + (int64_t)r * ny);
#pragma unroll
    for (int s = 0; s < SMAX; ++s) {
      const int q = lane + 32 * s;
      if (r < ny && q < nv) R.v[i][s] = __ldg(Mr + q);
    }
  }
}

template <typename T, int SMAX>
__device__ __forceinline__ void rows_dot1(const Rows1<T, SMAX>& R, const cplx<T>* x, int ny, int r0,
                                          cplx<T>* out) {
  constexpr int PER = vec16<T>::per;
  constexpr int RPW = RC / CH_WARPS;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nv = ny / PER;
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    const int r = r0 + warp + CH_WARPS * i;
    cplx<T> acc = czero<T>();
#pragma unroll
    for (int s = 0; s < SMAX; ++s) {
      const int q = lane + 32 * s;
      if (r < ny && q < nv) acc = dot_vec<T>(R.v[i][s], x, PER * q, acc);
    }
    acc = warp_sum<T>(acc);
    if (lane == 0 && r < ny) out[r] = acc;
  }
}

// out[r] = sub[r] - M1[r, :] x1 - M2[r, :] x2 for the RC rows r0 .. r0+RC-1: both
// matrices' row vectors are loaded before any product, so a block streams its 2 x RC rows
// in one memory phase (the sums are formed in the order of two rows_mv calls).
template <typename T, int SMAX>
struct Rows2 {  // this thread's 16-byte vectors of the RPW rows of two matrices
  typename vec16<T>::type v1[RC / CH_WARPS][SMAX], v2[RC / CH_WARPS][SMAX];
};

// Issue the loads of rows r0 + warp + CH_WARPS i of M1 and M2 (no dependence on x).
template <typename T, int SMAX>
__device__ __forceinline__ void rows_load2(Rows2<T, SMAX>& R, const cplx<T>* __restrict__ M1,
                                           const cplx<T>* __restrict__ M2, int ny, int r0) {
  using V = typename vec16<T>::type;
  constexpr int PER = vec16<T>::per;
  constexpr int RPW = RC / CH_WARPS;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nv = ny / PER;
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    const int r = r0 + warp + CH_WARPS * i;
    const V* A = reinterpret_cast<const V*>(M1 + (int64_t)r * ny);
    const V* B = reinterpret_cast<const V*>(M2 + (int64_t)r * ny);
#pragma unroll
    for (int s = 0; s < SMAX; ++s) {
      const int q = lane + 32 * s;
      if (r < ny && q < nv) {
        R.v1[i][s] = __ldg(A + q);
        R.v2[i][s] = __ldg(B + q);
      }
    }
  }
}

// out[r] = (sub[r] - M1[r] . x1) - M2[r] . x2 for the rows loaded by rows_load2 (x1, x2 in
// shared memory).
template <typename T, int SMAX>
__device__ __forceinline__ void rows_dot2(const Rows2<T, SMAX>& R, const cplx<T>* x1,
                                          const cplx<T>* x2, int ny, int r0, cplx<T>* out,
                                          const cplx<T>* sub) {
  constexpr int PER = vec16<T>::per;
  constexpr int RPW = RC / CH_WARPS;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nv = ny / PER;
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    const int r = r0 + warp + CH_WARPS * i;
    cplx<T> a1 = czero<T>(), a2 = czero<T>();
#pragma unroll
    for (int s = 0; s < SMAX; ++s) {
      const int q = lane + 32 * s;
      if (r < ny && q < nv) {
        a1 = dot_vec<T>(R.v1[i][s], x1, PER * q, a1);
        a2 = dot_vec<T>(R.v2[i][s], x2, PER * q, a2);
      }
    }
    a1 = warp_sum<T>(a1);
    a2 = warp_sum<T>(a2);
    if (lane == 0 && r < ny) out[r] = (sub[r] - a1) - a2;
  }
}

// out[c] = sum_a M[a][c] x[a] for the RC columns c0 .. c0+RC-1 (x in shared memory);
// lanes own columns, warps stride over rows, partial sums reduced through red[CH_WARPS][RC].
template <typename T>
__device__ __forceinline__ void cols_mvT(const cplx<T>* __restrict__ M, const cplx<T>* x, int ny,
                                         int c0, cplx<T>* red, cplx<T>* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = c0 + lane;
  cplx<T> acc = czero<T>();
  constexpr int U = 5;
  for (int a0 = warp; a0 < ny; a0 += CH_WARPS * U) {
    cplx<T> m[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int a = a0 + CH_WARPS * u;
      m[u] = (a < ny && c < ny) ? __ldg(M + (int64_t)a * ny + c) : czero<T>();
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int a = a0 + CH_WARPS * u;
      if (a < ny) acc = cfma(m[u], x[a], acc);
    }
  }
  red[warp * RC + lane] = acc;
  __syncthreads();
  if (warp == 0) {
    cplx<T> s = czero<T>();
#pragma unroll
    for (int w = 0; w < CH_WARPS; ++w) s = s + red[w * RC + lane];
    if (c < ny) out[c] = s;
  }
  __syncthreads();
}

// outP[c] = sum_a X[a][c] x[a] and, if Y, outQ[c] = sum_a Y[a][c] x[a], for the RC columns
// c0 .. c0+RC-1, the loads of both matrices in one loop (the sums are formed in the order of
// two cols_mvT calls); red holds 2 x CH_WARPS x RC entries.
template <typename T>
__device__ __forceinline__ void cols_mvT2(const cplx<T>* __restrict__ X,
                                          const cplx<T>* __restrict__ Y, const cplx<T>* x, int ny,
                                          int c0, cplx<T>* red, cplx<T>* outP, cplx<T>* outQ) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = c0 + lane;
  cplx<T> ap = czero<T>(), aq = czero<T>();
  constexpr int U = 5;
  for (int a0 = warp; a0 < ny; a0 += CH_WARPS * U) {
    cplx<T> mx[U], my[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int a = a0 + CH_WARPS * u;
      const bool v = a < ny && c < ny;
      mx[u] = v ? __ldg(X + (int64_t)a * ny + c) : czero<T>();
      my[u] = (v && Y) ? __ldg(Y + (int64_t)a * ny + c) : czero<T>();
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int a = a0 + CH_WARPS * u;
      if (a < ny) {
        ap = cfma(mx[u], x[a], ap);
        aq = cfma(my[u], x[a], aq);
      }
    }
  }
  red[warp * RC + lane] = ap;
  red[(CH_WARPS + warp) * RC + lane] = aq;
  __syncthreads();
  if (warp == 0) {
    cplx<T> sp = czero<T>(), sq = czero<T>();
#pragma unroll
    for (int w = 0; w < CH_WARPS; ++w) {
      sp = sp + red[w * RC + lane];
      sq = sq + red[(CH_WARPS + w) * RC + lane];
    }
    if (c < ny) {
      outP[c] = sp;
      if (Y) outQ[c] = sq;
    }
  }
  __syncthreads();
}

// Dense level, forward: t_k = Dinv_k b_{2k+1} (rows of chunk), P_k = X_k^T b_{2k+1},
// Q_k = Y_k^T b_{2k+1} (columns of chunk).  Grid (m, ceil(ny / RC)).
template <typename T, int SMAX>
__global__ void __launch_bounds__(CH_THREADS)
fwd_chunk_kernel(const cplx<T>* __restrict__ Dinv, const cplx<T>* __restrict__ X,
                 const cplx<T>* __restrict__ Y, const cplx<T>* __restrict__ B,
                 cplx<T>* __restrict__ t, cplx<T>* __restrict__ P, cplx<T>* __restrict__ Q, int n,
                 int ny) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  cplx<T>* bs = reinterpret_cast<cplx<T>*>(sm_raw);
  cplx<T>* red = bs + ny;
  const int64_t k = blockIdx.x;
  const int c0 = blockIdx.y * RC;
  const int64_t nn = (int64_t)ny * ny;
  // the Dinv rows of the chunk are loaded before b (rows up to 192 columns in FP32)
  constexpr bool early = sizeof(T) == 4 && SMAX <= 3;
  Rows1<T, early ? SMAX : 1> R;
  if constexpr (early) rows_load1<T, SMAX>(R, Dinv + k * nn, ny, c0);
  for (int c = threadIdx.x; c < ny; c += CH_THREADS) bs[c] = B[(2 * k + 1) * ny + c];
  __syncthreads();
  if constexpr (early) rows_dot1<T, SMAX>(R, bs, ny, c0, t + k * ny);
  else rows_mv<T, SMAX>(Dinv + k * nn, bs, ny, c0, t + k * ny, nullptr);
  // X^T b and Y^T b on the chunk columns, both matrices streamed together
  cols_mvT2<T>(X + k * nn, 2 * k + 2 < n ? Y + k * nn : nullptr, bs, ny, c0, red, P + k * ny,
               Q + k * ny);
}

// Dense level, backward: x_l[2k] = x_up[k];
// x_l[2k+1] = t_k - X_k x_up[k] - Y_k x_up[k+1] (rows of chunk).  Grid (nk, ceil(ny / RC)).
template <typename T, int SMAX>
__global__ void __launch_bounds__(CH_THREADS)
bwd_chunk_kernel(const cplx<T>* __restrict__ X, const cplx<T>* __restrict__ Y,
                 const cplx<T>* __restrict__ t, const cplx<T>* __restrict__ xup,
                 cplx<T>* __restrict__ xl, int n, int m, int ny) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  cplx<T>* xa = reinterpret_cast<cplx<T>*>(sm_raw);
  cplx<T>* xb = xa + ny;
  cplx<T>* tmp = xb + ny;
  const int64_t k = blockIdx.x;
  const int c0 = blockIdx.y * RC;
  const int64_t nn = (int64_t)ny * ny;
  const bool has_b = 2 * k + 2 < n;
  // x = (t - X xa) - Y xb on the chunk rows; X and Y rows streamed together where the
  // register tiles of both fit (FP32 rows up to 192 columns), their loads issued before
  // the vectors they multiply are read, else one after the other
  // (early loads for rows up to 192 columns, where the register tiles keep two CTAs per SM)
  constexpr bool fuse = sizeof(T) == 4 && SMAX <= 6;
  constexpr bool early = fuse && SMAX <= 3;
  const bool fused = fuse && has_b && k < m;
  Rows2<T, fuse ? SMAX : 1> R;
  if constexpr (early) {
    if (fused) rows_load2<T, SMAX>(R, X + k * nn, Y + k * nn, ny, c0);
  }
  for (int c = threadIdx.x; c < ny; c += CH_THREADS) {
    xa[c] = xup[k * ny + c];
    xb[c] = has_b ? xup[(k + 1) * ny + c] : czero<T>();
  }
  for (int c = c0 + threadIdx.x; c < c0 + RC && c < ny; c += CH_THREADS)
    xl[2 * k * ny + c] = xup[k * ny + c];
  __syncthreads();
  if (k >= m) return;
  if (fused) {
    if constexpr (fuse) {
      if constexpr (!early) rows_load2<T, SMAX>(R, X + k * nn, Y + k * nn, ny, c0);
      rows_dot2<T, SMAX>(R, xa, xb, ny, c0, xl + (2 * k + 1) * ny, t + k * ny);
    }
  } else if (has_b) {
    rows_mv<T, SMAX>(X + k * nn, xa, ny, c0, tmp, t + k * ny);
    __syncthreads();
    rows_mv<T, SMAX>(Y + k * nn, xb, ny, c0, xl + (2 * k + 1) * ny, tmp);
  } else {
    rows_mv<T, SMAX>(X + k * nn, xa, ny, c0, tmp, t + k * ny);
    __syncthreads();
    for (int c = c0 + threadIdx.x; c < c0 + RC && c < ny; c += CH_THREADS)
      xl[(2 * k + 1) * ny + c] = tmp[c];
  }
}

// y_k = M_k v_k for stored inverses (level 0 forward, the last single row): the vector
// is row vrow of V (stride ny).  Grid (batch, ceil(ny / RC)).
template <typename T, int SMAX>
__global__ void __launch_bounds__(CH_THREADS)
mv_chunk_kernel(const cplx<T>* __restrict__ M, const cplx<T>* __restrict__ V, int64_t v_stride,
                int64_t v_off, cplx<T>* __restrict__ y, int ny) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  cplx<T>* vs = reinterpret_cast<cplx<T>*>(sm_raw);
  const int64_t k = blockIdx.x;
  for (int c = threadIdx.x; c < ny; c += CH_THREADS) vs[c] = V[k * v_stride + v_off + c];
  __syncthreads();
  rows_mv<T, SMAX>(M + k * (int64_t)ny * ny, vs, ny, blockIdx.y * RC, y + k * ny, nullptr);
}

// Row r of a level's right-hand side formed from the level before it (Bp, its P, Q and
// mp eliminated rows): b[r] = Bp[2r] - Qp[r-1] - Pp[r], the Q term for r >= 1 and the P term
// for r < mp, in keep_kernel's order (so the values are the ones keep_kernel would store).
template <typename T>
__device__ __forceinline__ cplx<T> kept_row(const cplx<T>* __restrict__ Bp,
                                            const cplx<T>* __restrict__ Pp,
                                            const cplx<T>* __restrict__ Qp, int mp, int64_t r,
                                            int c, int ny) {
  cplx<T> v = Bp[2 * r * ny + c];
  if (r >= 1) v = v - Qp[(r - 1) * ny + c];
  if (r < mp) v = v - Pp[r * ny + c];
  return v;
}

// Dense level l >= 2, forward, with the kept-row update of level l - 1 fused in: block
// (k, chunk) forms the odd row 2k + 1 of this level's right-hand side whole in shared memory
// and then t_k, P_k, Q_k on its chunk as fwd_chunk_kernel does; it also writes the even row
// 2k on its chunk to Bn, from which the next level forms its rows.  Grid (ceil(n / 2),
// ceil(ny / RC)): for odd n the last block row k = n / 2 has its even row only.
template <typename T, int SMAX>
__global__ void __launch_bounds__(CH_THREADS)
fwd_keep_chunk_kernel(const cplx<T>* __restrict__ Dinv, const cplx<T>* __restrict__ X,
                      const cplx<T>* __restrict__ Y, const cplx<T>* __restrict__ Bp,
                      const cplx<T>* __restrict__ Pp, const cplx<T>* __restrict__ Qp, int mp,
                      cplx<T>* __restrict__ Bn, cplx<T>* __restrict__ t, cplx<T>* __restrict__ P,
                      cplx<T>* __restrict__ Q, int n, int ny) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  cplx<T>* bs = reinterpret_cast<cplx<T>*>(sm_raw);
  cplx<T>* red = bs + ny;
  const int64_t k = blockIdx.x;
  const int c0 = blockIdx.y * RC;
  const int64_t nn = (int64_t)ny * ny;
  for (int c = c0 + threadIdx.x; c < c0 + RC && c < ny; c += CH_THREADS)
    Bn[2 * k * ny + c] = kept_row<T>(Bp, Pp, Qp, mp, 2 * k, c, ny);
  if (2 * k + 1 >= n) return;  // (uniform over the block)
  constexpr bool early = sizeof(T) == 4 && SMAX <= 3;
  Rows1<T, early ? SMAX : 1> R;
  if constexpr (early) rows_load1<T, SMAX>(R, Dinv + k * nn, ny, c0);
  for (int c = threadIdx.x; c < ny; c += CH_THREADS)
    bs[c] = kept_row<T>(Bp, Pp, Qp, mp, 2 * k + 1, c, ny);
  __syncthreads();
  if constexpr (early) rows_dot1<T, SMAX>(R, bs, ny, c0, t + k * ny);
  else rows_mv<T, SMAX>(Dinv + k * nn, bs, ny, c0, t + k * ny, nullptr);
  cols_mvT2<T>(X + k * nn, 2 * k + 2 < n ? Y + k * nn : nullptr, bs, ny, c0, red, P + k * ny,
               Q + k * ny);
}

// The single last row with the kept-row update of the level before it fused in:
// y = M b[0], b[0] = Bp[0] - Pp[0] (mp > 0).  Grid (1, ceil(ny / RC)).
template <typename T, int SMAX>
__global__ void __launch_bounds__(CH_THREADS)
mv_keep_chunk_kernel(const cplx<T>* __restrict__ M, const cplx<T>* __restrict__ Bp,
                     const cplx<T>* __restrict__ Pp, const cplx<T>* __restrict__ Qp, int mp,
                     cplx<T>* __restrict__ y, int ny) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  cplx<T>* vs = reinterpret_cast<cplx<T>*>(sm_raw);
  for (int c = threadIdx.x; c < ny; c += CH_THREADS) vs[c] = kept_row<T>(Bp, Pp, Qp, mp, 0, c, ny);
  __syncthreads();
  rows_mv<T, SMAX>(M, vs, ny, blockIdx.y * RC, y, nullptr);
}

// ----- single right-hand side, level 0 by the pivoted tridiagonal factors (5 ny values per
// eliminated row instead of the dense ny x ny inverse): one warp per eliminated row k stages
// the row's factors and right-hand side in shared memory, lane 0 runs the forward and
// backward sweeps, the warp writes the result.
//   FWD: t0[k] = T_{2k+1}^{-1} b[2k+1]
//   BWD: x[2k] = x1[k];  x[2k+1] = T_{2k+1}^{-1} (b[2k+1] - cx[2k] o x1[k] - cx[2k+1] o x1[k+1])
constexpr int TRS_WARPS = 4;

template <typename T>
__host__ __device__ size_t trs_smem_per_warp(int ny) {
  return ((size_t)5 * ny * sizeof(cplx<T>) + (size_t)ny + 15) & ~(size_t)15;
}

template <typename T, bool BWD>
__global__ void __launch_bounds__(32 * TRS_WARPS)
tri_rows_solve_kernel(const cplx<T>* __restrict__ tdl, const cplx<T>* __restrict__ tdinv,
                      const cplx<T>* __restrict__ tdu, const cplx<T>* __restrict__ tdu2,
                      const uint8_t* __restrict__ tpiv, const cplx<T>* __restrict__ b,
                      const cplx<T>* __restrict__ x1, const double2* __restrict__ cx,
                      cplx<T>* __restrict__ out, int nx, int ny, int rows) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * TRS_WARPS + w;
  if (k >= rows) return;  // whole warp
  cplx<T>* dl = reinterpret_cast<cplx<T>*>(sm_raw + (size_t)w * trs_smem_per_warp<T>(ny));
  cplx<T>* di = dl + ny;
  cplx<T>* du = di + ny;
  cplx<T>* du2 = du + ny;
  cplx<T>* v = du2 + ny;
  uint8_t* pv = reinterpret_cast<uint8_t*>(v + ny);
  const int64_t r = 2 * (int64_t)k + 1;
  const bool has = r < nx;
  if (BWD) {
    for (int j = lane; j < ny; j += 32) out[2 * (int64_t)k * ny + j] = x1[(int64_t)k * ny + j];
  }
  if (!has) return;
  const int64_t fb = (int64_t)k * ny;
  for (int j = lane; j < ny; j += 32) {
    dl[j] = tdl[fb + j];
    di[j] = tdinv[fb + j];
    du[j] = tdu[fb + j];
    du2[j] = tdu2[fb + j];
    pv[j] = tpiv[fb + j];
    cplx<T> rv = b[r * ny + j];
    if (BWD) {
      rv = cfms(ccast<T>(cx[(r - 1) * ny + j]), x1[(int64_t)k * ny + j], rv);
      if (r + 1 < nx) rv = cfms(ccast<T>(cx[r * ny + j]), x1[(int64_t)(k + 1) * ny + j], rv);
    }
    v[j] = rv;
  }
  __syncwarp();
  if (lane == 0) {
    TriRow<T> f{dl, di, du, du2, pv};
    tri_forward<T>(f, ny, [&](int j) { return v[j]; }, [&](int j, cplx<T> y) { v[j] = y; });
    tri_backward<T>(f, ny, [&](int j) { return v[j]; }, [&](int j, cplx<T> g) { v[j] = g; });
  }
  __syncwarp();
  cplx<T>* o = BWD ? out + r * ny : out + (int64_t)k * ny;
  for (int j = lane; j < ny; j += 32) o[j] = v[j];
}

}  // namespace

// ===================================================================== handle
struct BcrHandle {
  int prec;
  int nx, ny;
  std::vector<int64_t> n, m;      // rows / eliminated rows per level (index 0 = tridiagonal level)
  std::vector<int64_t> off;       // store offsets (elements) of levels >= 1
  int64_t final_off = 0;
  int Lf = 1;                     // level with a single row
  size_t esz = 0;                 // bytes per complex element
  // factor storage
  void *tdl = nullptr, *tdinv = nullptr, *tdu = nullptr, *tdu2 = nullptr;
  uint8_t* tpiv = nullptr;
  void* scratch = nullptr;        // m0 x ny x ny elements: the FP64 split path's digits and blocks
  bool simt = false;              // FP32: factor and multi-RHS products on the SIMT pipe
  void* Dw[2] = {nullptr, nullptr};
  void* Lw[2] = {nullptr, nullptr};
  void* store = nullptr;
  int32_t* status = nullptr;
  size_t factor_bytes = 0;
  Profiler* prof = nullptr;
  // solve workspace (grown on demand)
  int ws_nrhs = 0;
  void* ws = nullptr;
  size_t ws_bytes = 0;
  DevMem mem;
};

static void free_ws(BcrHandle* h) {
  h->mem.release(h->ws);
  h->ws = nullptr;
  h->ws_nrhs = 0;
  h->ws_bytes = 0;
}

void bcr_destroy(BcrHandle* h) {
  if (!h) return;
  void* ps[] = {h->tdl, h->tdinv, h->tdu, h->tdu2, h->tpiv, h->scratch, h->Dw[0], h->Dw[1],
                h->Lw[0], h->Lw[1], h->store, h->status};
  for (void* p : ps) h->mem.release(p);
  free_ws(h);
  delete h;
}

size_t bcr_bytes(const BcrHandle* h) { return h->factor_bytes + h->ws_bytes; }
void bcr_set_profiler(BcrHandle* h, Profiler* p) { h->prof = p; }
int bcr_precision(const BcrHandle* h) { return h->prec; }
void bcr_set_simt(BcrHandle* h, bool simt) { h->simt = simt && h->prec != RCI_FP64; }
bool bcr_simt(const BcrHandle* h) { return h->simt; }

// The status word handed to gemm<T>: its tensor-core paths run only with one (they record an
// expired bounded wait there), so a handle set to the SIMT pipe passes none.
static int32_t* gemm_status(const BcrHandle* h) { return h->simt ? nullptr : h->status; }

cudaError_t bcr_create(int nx, int ny, int prec, const DevMem* mem, BcrHandle** out, size_t* bytes) {
  *out = nullptr;
  if (nx < 1 || ny < 2 || ny > 1024) return cudaErrorInvalidValue;
  BcrHandle* h = new (std::nothrow) BcrHandle();
  if (!h) return cudaErrorMemoryAllocation;
  if (mem) h->mem = *mem;
  h->prec = prec;
  h->nx = nx;
  h->ny = ny;
  h->esz = prec == RCI_FP64 ? sizeof(double2) : sizeof(float2);
  const int64_t nn = (int64_t)ny * ny;
  h->n.push_back(nx);
  h->m.push_back(nx / 2);
  int64_t cur = (nx + 1) / 2;
  int64_t off = 0;
  h->off.push_back(0);
  int L = 1;
  while (cur > 1) {
    h->n.push_back(cur);
    h->m.push_back(cur / 2);
    h->off.push_back(off);
    off += 3 * (cur / 2) * nn;
    cur = (cur + 1) / 2;
    ++L;
  }
  h->n.push_back(1);
  h->m.push_back(0);
  h->off.push_back(off);
  h->Lf = L;
  h->final_off = off;
  int64_t store_elems = off + nn;
  int64_t m0 = h->m[0], n1 = (nx + 1) / 2;
  cudaError_t e = cudaSuccess;
  auto alloc = [&](void** p, size_t b) {
    if (e != cudaSuccess) return;
    e = h->mem.alloc(p, b);
    if (e == cudaSuccess) h->factor_bytes += b;
  };
  size_t m0b = (size_t)std::max<int64_t>(m0, 1) * ny;
  alloc(&h->tdl, m0b * h->esz);
  alloc(&h->tdinv, m0b * h->esz);
  alloc(&h->tdu, m0b * h->esz);
  alloc(&h->tdu2, m0b * h->esz);
  alloc((void**)&h->tpiv, m0b);
  alloc(&h->scratch, m0b * ny * h->esz);
  for (int i = 0; i < 2; ++i) {
    alloc(&h->Dw[i], (size_t)n1 * nn * h->esz);
    alloc(&h->Lw[i], (size_t)n1 * nn * h->esz);
  }
  alloc(&h->store, (size_t)store_elems * h->esz);
  alloc((void**)&h->status, 3 * sizeof(int32_t));  // status, max |A|, max |inverted block| (bits)
  if (e != cudaSuccess) {
    bcr_destroy(h);
    return e;
  }
  *out = h;
  if (bytes) *bytes = h->factor_bytes;
  return cudaSuccess;
}

cudaError_t bcr_read_status(BcrHandle* h, int32_t* st, cudaStream_t s, double* growth) {
  uint32_t w[3] = {0, 0, 0};
  RCI_CUDA_TRY(cudaMemcpyAsync(w, h->status, sizeof(w), cudaMemcpyDeviceToHost, s));
  RCI_CUDA_TRY(cudaStreamSynchronize(s));
  *st = (int32_t)w[0];
  if (growth) {
    float a, d;
    std::memcpy(&a, &w[1], 4);
    std::memcpy(&d, &w[2], 4);
    *growth = a > 0.f ? (double)d / (double)a : 0.0;
  }
  return cudaSuccess;
}

cudaError_t bcr_clear_timeout(BcrHandle* h, cudaStream_t s) {
  return cudaMemsetAsync(h->status, 0, sizeof(int32_t), s);
}

// ===================================================================== FP64 on the tensor cores
// The FP64 factorisation runs its block products through the digit split of tc_gemm64.cu and its
// block inverses as Newton iterations on an FP32 inverse, X <- X + X (I - D X), with those products:
// the FP64 pipe does neither.  At ny = 160 a product takes 1.2 us of the whole GPU where the FP64
// GEMM took 28, and an inverse of one block alone 0.4 ms where the FP64 Gauss-Jordan took 4.9: a
// new design of 500 cells 404 -> 39 ms, of 50 cells (ny = 128) 54 -> 5.5 ms.
// A block whose iteration does not contract (an FP32 inverse that resolves nothing, entries outside
// the FP32 range, a singular block) goes to the FP64 Gauss-Jordan kernel, which also reports zero
// pivots, so the factorisation accepts and refuses what it did.
//
// Scratch: the handle's (m0 blocks of ny x ny) and whatever of its working arrays and store the
// step at hand leaves unused; the blocks of a level are taken in batches that fit it.
namespace {

// a = (float) of `batch` nn-element blocks, stride elements apart
__global__ void blocks_to_f32_kernel(const double2* __restrict__ src, int64_t stride, int64_t nn,
                                     int64_t total, float2* __restrict__ out) {
  dep_begin();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int64_t z = e / nn;
  const double2 v = src[z * stride + (e - z * nn)];
  out[e] = make_float2((float)v.x, (float)v.y);
}

__global__ void blocks_to_f64_kernel(const float2* __restrict__ src, int64_t total,
                                     double2* __restrict__ out) {
  dep_begin();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < total) out[e] = make_double2((double)src[e].x, (double)src[e].y);
}

// After R = I - D X of one Newton step, per block (m = its largest |re|, |im|):
// |R^2| <= 2 n m^2 bounds the residual that this step's update X + X R leaves.  When n m^2 is well
// below rounding level the update is the last; an iteration that does not contract, or has not
// got there at the last step, marks the block for the Gauss-Jordan kernel.  `rough`: R was
// formed from the high digits only (SG_HALF), too coarse to end on.
struct NewtonFlags {
  uint32_t* maxabs;   // of R (bits of a float)
  int32_t* skip_r;    // no further residual wanted
  int32_t* skip_x;    // no further update wanted
  int32_t* failed;
  int32_t* active;    // blocks whose update of this step, and whose next residual, are wanted
};
__global__ void newton_check_kernel(NewtonFlags f, int n, int batch, int rough, int last,
                                    const int32_t* __restrict__ st32, int32_t* status) {
  dep_begin();
  const int z = blockIdx.x * blockDim.x + threadIdx.x;
  if (z == 0 && *st32 == DEV_TIMEOUT) atomicCAS(status, DEV_OK, DEV_TIMEOUT);
  if (z >= batch) return;
  if (f.skip_r[z]) {
    f.skip_x[z] = 1;
    return;
  }
  const float m = __uint_as_float(f.maxabs[z]);
  f.maxabs[z] = 0;
  const bool contracts = m * (float)n < 0.25f;
  const bool done = contracts && !rough && (float)n * m * m <= 1e-17f;
  if (!contracts || (last && !done)) f.failed[z] = f.skip_x[z] = 1;
  else atomicAdd(&f.active[0], 1);
  if (!contracts || done || last) f.skip_r[z] = 1;
  else atomicAdd(&f.active[1], 1);
}

constexpr int NEWTON_STEPS = 4;

// A split form and its exponents, for up to c operands.
struct Form {
  unsigned char* f;
  int32_t* e;
  Form() = default;
  Form(Scratch& w, int rows, int K, int planes, size_t c)
      : f(w.take<unsigned char>(c * sg_form_bytes(rows, K, planes))),
        e(w.take<int32_t>(4 * c * (size_t)sg_form_exps(rows))) {}
};

// The buffers of one batch of c blocks.  (A region's alignment is that of device allocations or of
// whole blocks: a multiple of 16 bytes, what the copies need.)
struct NewtonBuf {
  Form D, Xr, C;      // D and X as left operands; the right one in turn, X or R
  double2* R;         // first the FP32 copies of D and X
  int32_t* words;
  NewtonBuf(Scratch& w, int ny, size_t c) {
    D = Form(w, ny, ny, 3, c);
    Xr = Form(w, ny, ny, 3, c);
    C = Form(w, ny, ny, 2, c);
    R = w.take<double2>(c * ny * ny * sizeof(double2));
    words = w.take<int32_t>(4 * (4 * c + 1 + 2 * NEWTON_STEPS));
  }
};
struct LevelBuf {
  Form D, O, E, X, Y;
  LevelBuf(Scratch& w, int ny, size_t c) {
    D = Form(w, ny, ny, 3, c + 1);  // Dinv; once X and Y are formed, the columns of X
    X = D;
    O = Form(w, ny, ny, 3, c);
    E = Form(w, ny, ny, 3, c + 1);
    Y = Form(w, ny, ny, 2, c + 1);
  }
};
struct FwdBuf {
  Form D, X, Y, B;
  FwdBuf(Scratch& w, int ny, int nq, size_t c) {
    D = Form(w, ny, ny, 3, c);
    X = Form(w, ny, ny, 3, c);
    Y = Form(w, ny, ny, 3, c + 1);
    B = Form(w, nq, ny, 2, c + 1);
  }
};

}  // namespace

// out[z] = D[z]^-1 for z < m (D: stride elements apart, destroyed where the Gauss-Jordan kernel
// takes over).
static cudaError_t split_inverse(double2* D, int64_t stride, double2* out, int ny, int m, Scratch& mem,
                                 int32_t* status, cudaStream_t s) {
  const int64_t nn = (int64_t)ny * ny;
  const int cb = batch_of(mem, m, [&](int c) { NewtonBuf(mem, ny, c); });
  if (cb == 0) return cudaErrorInvalidValue;
  const long long wl = tc_wait_limit();
  for (int k0 = 0; k0 < m; k0 += cb) {
    const int c = std::min(cb, m - k0);
    mem.reset();
    const NewtonBuf w(mem, ny, c);
    if (mem.full) return cudaErrorInvalidValue;
    float2* a32 = reinterpret_cast<float2*>(w.R);
    float2* x32 = a32 + c * nn;
    double2* R = w.R;
    unsigned char *fD = w.D.f, *fXr = w.Xr.f, *fXc = w.C.f, *fR = w.C.f;
    int32_t *eD = w.D.e, *eXr = w.Xr.e, *eXc = w.C.e, *eR = w.C.e;
    int32_t* words = w.words;
    int32_t* st32 = words + 4 * c;
    double2* Dk = D + (int64_t)k0 * stride;
    double2* X = out + (int64_t)k0 * nn;
    RCI_CUDA_TRY(cudaMemsetAsync(words, 0, sizeof(int32_t) * (4 * (size_t)c + 1 + 2 * NEWTON_STEPS), s));
    const int64_t tot = (int64_t)c * nn;
    RCI_CUDA_TRY(launch_dep(blocks_to_f32_kernel, (unsigned)ceil_div(tot, 256), 256, 0, s, Dk, stride, nn, tot, a32));
    rci_note_launch();
    RCI_CUDA_TRY(cudaGetLastError());
    if (ny <= 160) RCI_CUDA_TRY(launch_tc_gj(a32, nn, x32, nn, ny, c, st32, s));
    else RCI_CUDA_TRY(launch_gj_simt<float>(a32, nn, x32, nn, ny, c, st32, s));
    RCI_CUDA_TRY(launch_dep(blocks_to_f64_kernel, (unsigned)ceil_div(tot, 256), 256, 0, s, x32, tot, X));
    rci_note_launch();
    RCI_CUDA_TRY(cudaGetLastError());
    RCI_CUDA_TRY(launch_sg_split(Dk, false, ny, stride, false, ny, ny, 3, c, fD, eD, nullptr, s));
    for (int it = 0; it < NEWTON_STEPS; ++it) {
      const NewtonFlags fl{reinterpret_cast<uint32_t*>(words), words + c, words + 2 * c, words + 3 * c,
                           st32 + 1 + 2 * it};
      RCI_CUDA_TRY(launch_sg_split(X, false, ny, nn, true, ny, ny, 2, c, fXc, eXc, fl.skip_r, s, it == 0 ? 5 : SG_SLICES));
      SgJob r{};
      r.nseg = 1;
      r.seg[0] = SgSeg{fD, eD, fXc, eXc, 3, 2, 0, 0, 0, c};
      r.neg = true;
      r.identity = true;
      r.C = R;
      r.ldc = ny;
      r.sC = nn;
      r.batch = c;
      r.maxabs = fl.maxabs;
      r.skip = fl.skip_r;
      if (it > 0) r.any = st32 + 2 * it;  // what the step before left active
      RCI_CUDA_TRY(launch_sg_gemm(ny, ny, ny, 1, &r, it == 0 ? SG_HALF : SG_FULL, status, wl, s));
      RCI_CUDA_TRY(launch_dep(newton_check_kernel, (unsigned)ceil_div(c, 128), 128, 0, s, fl, ny, c, it == 0,
                              it == NEWTON_STEPS - 1, st32, status));
      rci_note_launch();
      RCI_CUDA_TRY(cudaGetLastError());
      // (the first update corrects some 1e-5 and takes SG_HALF; the later ones correct 1e-8 or less)
      const SgDigits du = it == 0 ? SG_HALF : SG_SMALL;
      const int nd = it == 0 ? 5 : 4;
      RCI_CUDA_TRY(launch_sg_split(X, false, ny, nn, false, ny, ny, 3, c, fXr, eXr, fl.skip_x, s, nd));
      RCI_CUDA_TRY(launch_sg_split(R, false, ny, nn, true, ny, ny, 2, c, fR, eR, fl.skip_x, s, nd));
      SgJob x{};
      x.nseg = 1;
      x.seg[0] = SgSeg{fXr, eXr, fR, eR, 3, 2, 0, 0, 0, c};
      x.C0 = X;
      x.ldc0 = ny;
      x.sC0 = nn;
      x.C = X;
      x.ldc = ny;
      x.sC = nn;
      x.batch = c;
      x.skip = fl.skip_x;
      x.any = &fl.active[0];
      RCI_CUDA_TRY(launch_sg_gemm(ny, ny, ny, 1, &x, du, status, wl, s));
    }
    RCI_CUDA_TRY(launch_gj_simt<double>(Dk, stride, X, nn, ny, c, status, s, words + 3 * c));
  }
  return cudaSuccess;
}

// ---- FP32 blocks of more than 160 rows
// A block of this size fits neither tensor memory nor shared memory, and the SIMT Gauss-Jordan kernel
// works on it in L2 (7.8 us of the whole GPU a block of 224, 1.1 ms for one alone).  Instead:
//   1. inversion by halves, A = [A11 A12; A21 A22]: P = A11^-1 and T = (A22 - A21 P A12)^-1 on the
//      tensor-core Gauss-Jordan kernel, the products around them on the TMA-fed GEMM;
//   2. pivoting only within the halves costs digits, so one Newton step X + X (I - A X) follows with
//      the residual formed through the digit split (SG_SMALL: error 2^-28, where FP32 rounds at 2^-24): the
//      inverse it leaves is closer to the exact one than the SIMT kernel's.
// Blocks whose step would leave more than that kernel does (n m^2 > 2e-6 for residual entries of m: from
// 9.4e-5 on at n = 224, where ordinary blocks leave some 1e-5),
// or whose halves are singular, go to the SIMT kernel, which also reports zero pivots.
namespace {

// an h x h part of each of the blocks at src (rows lds apart) to dst (rows ldd apart)
__global__ void block_part_kernel(const float2* __restrict__ src, int64_t ss, int lds, float2* __restrict__ dst,
                                  int64_t sd, int ldd, int h, int64_t total) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int64_t hh = (int64_t)h * h, z = e / hh, r = e - z * hh;
  const int i = (int)(r / h), j = (int)(r - (int64_t)i * h);
  dst[z * sd + (int64_t)i * ldd + j] = src[z * ss + (int64_t)i * lds + j];
}

// failed[z]: the residual R = I - A X of block z is too large for one Newton step
__global__ void halves_check_kernel(const uint32_t* __restrict__ maxabs, int n, int batch, int32_t* failed,
                                    const int32_t* __restrict__ st32, int32_t* status) {
  const int z = blockIdx.x * blockDim.x + threadIdx.x;
  if (z == 0 && *st32 == DEV_TIMEOUT) atomicCAS(status, DEV_OK, DEV_TIMEOUT);
  if (z >= batch) return;
  const float m = __uint_as_float(maxabs[z]);
  failed[z] = (float)n * m * m <= 2e-6f ? 0 : 1;
}

struct HalvesBuf {
  Form D, X;
  float2 *X0, *P, *Q, *R, *S, *T, *res;  // res (n x n) takes the place of P .. T
  int32_t* words;                        // maxabs, failed, status of the halves
  int h1, h2;
  HalvesBuf(Scratch& w, int n, size_t c) {
    h1 = (int)ceil_div(n / 2, 16) * 16;
    h2 = n - h1;
    D = Form(w, n, n, 3, c);
    X = Form(w, n, n, 2, c);
    X0 = w.take<float2>(c * n * n * sizeof(float2));
    const size_t a = c * h1 * h1, b = c * h1 * h2, d = c * h2 * h2;
    P = w.take<float2>((2 * a + 2 * b + 2 * d) * sizeof(float2));  // 2 a: P and the packed A11
    res = P;
    Q = P + 2 * a;
    R = Q + b;
    S = R + b;
    T = S + d;
    words = w.take<int32_t>(4 * (2 * c + 1));
  }
};

}  // namespace

// out[z] = D[z]^-1 for z < m, FP32 blocks of 160 < ny <= SG_KMAX, even (D: stride elements apart,
// destroyed where the SIMT kernel takes over).
static cudaError_t halves_inverse(float2* D, int64_t stride, float2* out, int n, int m, Scratch& mem,
                                  int32_t* status, cudaStream_t s) {
  const int64_t nn = (int64_t)n * n;
  const int cb = batch_of(mem, m, [&](int c) { HalvesBuf(mem, n, c); });
  if (cb == 0) return cudaErrorInvalidValue;
  const long long wl = tc_wait_limit();
  // C[z] (M x N) = alpha A[z] B[z] (+ C0[z]), K terms
  auto product = [&](int M, int N, int K, const float2* A, int64_t lda, int64_t sA, const float2* B, int64_t ldb,
                     int64_t sB, float alpha, const float2* C0, int64_t ldc0, int64_t sC0, float2* C, int64_t ldc,
                     int64_t sC, int c) {
    return launch_tc_cgemm_tma(M, N, K, false, false, alpha, A, lda, sA, B, ldb, sB, C0 ? 1.f : 0.f, C0, ldc0, sC0, C,
                               ldc, sC, c, status, wl, s);
  };
  for (int k0 = 0; k0 < m; k0 += cb) {
    const int c = std::min(cb, m - k0);
    mem.reset();
    const HalvesBuf w(mem, n, c);
    if (mem.full) return cudaErrorInvalidValue;
    const int h1 = w.h1, h2 = w.h2;
    const int64_t a = (int64_t)h1 * h1, b = (int64_t)h1 * h2, d = (int64_t)h2 * h2;
    float2* A = D + (int64_t)k0 * stride;
    float2 *A12 = A + h1, *A21 = A + (int64_t)h1 * n, *A22 = A21 + h1;
    float2 *X0 = w.X0, *X12 = X0 + h1, *X21 = X0 + (int64_t)h1 * n, *X22 = X21 + h1;
    float2 *P = w.P, *A11 = P + c * a;
    uint32_t* maxabs = reinterpret_cast<uint32_t*>(w.words);
    int32_t *failed = w.words + c, *st32 = w.words + 2 * c;
    RCI_CUDA_TRY(cudaMemsetAsync(w.words, 0, sizeof(int32_t) * (2 * (size_t)c + 1), s));
    block_part_kernel<<<(unsigned)ceil_div(c * a, 256), 256, 0, s>>>(A, stride, n, A11, a, h1, h1, c * a);
    rci_note_launch();
    RCI_CUDA_TRY(cudaGetLastError());
    RCI_CUDA_TRY(launch_tc_gj(A11, a, P, a, h1, c, st32, s));
    RCI_CUDA_TRY(product(h1, h2, h1, P, h1, a, A12, n, stride, 1.f, nullptr, 0, 0, w.Q, h2, b, c));
    RCI_CUDA_TRY(product(h2, h1, h1, A21, n, stride, P, h1, a, 1.f, nullptr, 0, 0, w.R, h1, b, c));
    RCI_CUDA_TRY(product(h2, h2, h1, A21, n, stride, w.Q, h2, b, -1.f, A22, n, stride, w.S, h2, d, c));
    RCI_CUDA_TRY(launch_tc_gj(w.S, d, w.T, d, h2, c, st32, s));
    RCI_CUDA_TRY(product(h1, h2, h2, w.Q, h2, b, w.T, h2, d, -1.f, nullptr, 0, 0, X12, n, nn, c));
    RCI_CUDA_TRY(product(h2, h1, h2, w.T, h2, d, w.R, h1, b, -1.f, nullptr, 0, 0, X21, n, nn, c));
    RCI_CUDA_TRY(product(h1, h1, h2, X12, n, nn, w.R, h1, b, -1.f, P, h1, a, X0, n, nn, c));
    block_part_kernel<<<(unsigned)ceil_div(c * d, 256), 256, 0, s>>>(w.T, d, h2, X22, nn, n, h2, c * d);
    rci_note_launch();
    RCI_CUDA_TRY(cudaGetLastError());
    // one Newton step
    RCI_CUDA_TRY(launch_sg_split(A, true, n, stride, false, n, n, 3, c, w.D.f, w.D.e, nullptr, s, 4));
    RCI_CUDA_TRY(launch_sg_split(X0, true, n, nn, true, n, n, 2, c, w.X.f, w.X.e, nullptr, s, 4));
    SgJob r{};
    r.nseg = 1;
    r.seg[0] = SgSeg{w.D.f, w.D.e, w.X.f, w.X.e, 3, 2, 0, 0, 0, c};
    r.neg = true;
    r.identity = true;
    r.C32 = w.res;
    r.ldc = n;
    r.sC = nn;
    r.batch = c;
    r.maxabs = maxabs;
    RCI_CUDA_TRY(launch_sg_gemm(n, n, n, 1, &r, SG_SMALL, status, wl, s));
    halves_check_kernel<<<(unsigned)ceil_div(c, 128), 128, 0, s>>>(maxabs, n, c, failed, st32, status);
    rci_note_launch();
    RCI_CUDA_TRY(cudaGetLastError());
    float2* X = out + (int64_t)k0 * nn;
    RCI_CUDA_TRY(product(n, n, n, X0, n, nn, w.res, n, nn, 1.f, X0, n, nn, X, n, nn, c));
    RCI_CUDA_TRY(launch_gj_simt<float>(A, stride, X, nn, n, c, status, s, failed));
  }
  return cudaSuccess;
}

// The products of one FP64 reduction level (the same five as the general path), in batches of
// eliminated rows k0 .. k1 - 1:
//   X_k = Dinv_k L_{2k+1};  Y_k = Dinv_k L_{2k+2}^T
//   D'_k = D_{2k} - L_{2k} Y_{k-1} (k >= 1) - L_{2k+1}^T X_k (k < m);  L'_k = -L_{2k} X_{k-1} (k >= 1)
// Every split form serves as often as it can: the columns of L_{2k+1} as the right operand of X
// and the left one of D', the rows of L_{2k} as the right operand of Y (of the row before) and the
// left one of D' and L'.
static cudaError_t split_level(const double2* D, const double2* L, const double2* Dinv, double2* X, double2* Y,
                               double2* Dn, double2* Ln, int ny, int n, int m, int nk, Scratch& mem,
                               int32_t* status, Profiler* prof, cudaStream_t s) {
  const int64_t nn = (int64_t)ny * ny;
  const int my = (n - 1) / 2;
  const size_t f3 = sg_form_bytes(ny, ny, 3);
  const int ne = sg_form_exps(ny);
  const int cb = batch_of(mem, nk, [&](int c) { LevelBuf(mem, ny, c); });
  if (cb == 0) return cudaErrorInvalidValue;
  const long long wl = tc_wait_limit();
  for (int k0 = 0; k0 < nk; k0 += cb) {
    const int c = std::min(cb, nk - k0);           // kept rows k0 .. k0 + c - 1
    const int cm = std::min(c, m - k0);            // of which eliminated rows of the same index
    const int cy = std::max(0, std::min(c, my - k0));
    const int p0 = k0 > 0 ? 1 : 0;                 // X, Y of row k0 - 1 come first
    mem.reset();
    const LevelBuf w(mem, ny, c);
    if (mem.full) return cudaErrorInvalidValue;
    unsigned char *fD = w.D.f, *fO = w.O.f, *fE = w.E.f, *fX = w.X.f, *fY = w.Y.f;
    int32_t *eD = w.D.e, *eO = w.O.e, *eE = w.E.e, *eX = w.X.e, *eY = w.Y.e;
    // L_{2k} for k = k0 .. k0 + c while it exists (index 2k <= n - 1; L_0 is not used)
    const int nE = std::min(c + 1, nk - k0);
    const int pm = p0 + std::max(0, cm), py = p0 + cy;
    double flops = 8.0 * ny * (double)nn;
    {
      ProfScope ps(prof, PF_GEMM, s, flops * (std::max(0, cm) + cy), 3.0 * 16 * nn * (std::max(0, cm) + cy), 4);
      if (cm > 0) {
        RCI_CUDA_TRY(launch_sg_split(Dinv + k0 * nn, false, ny, nn, false, ny, ny, 3, cm, fD, eD, nullptr, s));
        RCI_CUDA_TRY(launch_sg_split(L + (2 * (int64_t)k0 + 1) * nn, false, ny, 2 * nn, true, ny, ny, 3, cm, fO,
                                     eO, nullptr, s));
      }
      // (k0 = 0: L_0 is uninitialised memory that no product reads; its form is skipped)
      const int z0 = k0 == 0 ? 1 : 0;
      if (nE > z0)
        RCI_CUDA_TRY(launch_sg_split(L + 2 * (int64_t)(k0 + z0) * nn, false, ny, 2 * nn, false, ny, ny, 3, nE - z0,
                                     fE + z0 * f3, eE + z0 * ne, nullptr, s));
      SgJob xy[2] = {};
      xy[0].nseg = 1;
      xy[0].seg[0] = SgSeg{fD, eD, fO, eO, 3, 3, 0, 0, 0, std::max(0, cm)};
      xy[0].C = X + k0 * nn;
      xy[0].ldc = ny;
      xy[0].sC = nn;
      xy[0].batch = std::max(0, cm);
      xy[1] = xy[0];
      xy[1].seg[0] = SgSeg{fD, eD, fE, eE, 3, 3, 0, 1, 0, cy};
      xy[1].C = Y + k0 * nn;
      xy[1].batch = cy;
      RCI_CUDA_TRY(launch_sg_gemm(ny, ny, ny, 2, xy, SG_FULL, status, wl, s));
    }
    ProfScope ps(prof, PF_GEMM, s, flops * (2.0 * (c - (k0 == 0)) + std::max(0, cm)), 16.0 * nn * 6 * c, 3);
    if (pm > 0)
      RCI_CUDA_TRY(launch_sg_split(X + (k0 - p0) * nn, false, ny, nn, true, ny, ny, 2, pm, fX, eX, nullptr, s));
    if (py > 0)
      RCI_CUDA_TRY(launch_sg_split(Y + (k0 - p0) * nn, false, ny, nn, true, ny, ny, 2, py, fY, eY, nullptr, s));
    SgJob sl[2] = {};
    const int lo = k0 == 0 ? 1 : 0;                // row 0 has no row before it
    sl[0].nseg = 2;
    sl[0].seg[0] = SgSeg{fE, eE, fY, eY, 3, 2, 0, p0 - 1, lo, c};
    sl[0].seg[1] = SgSeg{fO, eO, fX, eX, 3, 2, 0, p0, 0, std::max(0, cm)};
    sl[0].neg = true;
    sl[0].C0 = D + 2 * (int64_t)k0 * nn;
    sl[0].ldc0 = ny;
    sl[0].sC0 = 2 * nn;
    sl[0].C = Dn + k0 * nn;
    sl[0].ldc = ny;
    sl[0].sC = nn;
    sl[0].batch = c;
    sl[1].nseg = 1;
    sl[1].seg[0] = SgSeg{fE + lo * f3, eE + lo * ne, fX, eX, 3, 2, 0, p0 - 1 + lo, 0, c - lo};
    sl[1].neg = true;
    sl[1].C = Ln + (k0 + lo) * nn;
    sl[1].ldc = ny;
    sl[1].sC = nn;
    sl[1].batch = c - lo;
    RCI_CUDA_TRY(launch_sg_gemm(ny, ny, ny, 2, sl, SG_FULL, status, wl, s));
  }
  return cudaSuccess;
}

template <typename T>
static cudaError_t factor_t(BcrHandle* h, const double2* dg, const double2* cx, const double2* cy,
                            cudaStream_t s) {
  const int nx = h->nx, ny = h->ny;
  const int64_t nn = (int64_t)ny * ny;
  const int m0 = (int)h->m[0];
  const int n1 = (nx + 1) / 2;
  RCI_CUDA_TRY(cudaMemsetAsync(h->status, 0, 3 * sizeof(int32_t), s));
  uint32_t* maxabs = reinterpret_cast<uint32_t*>(h->status) + 1;
  {
    const int64_t N = (int64_t)nx * ny;
    const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(N, 256), 4 * 152);
    coeff_maxabs_kernel<<<grid, 256, 0, s>>>(dg, cx, cy, N, maxabs);
    rci_note_launch();
    RCI_CUDA_TRY(cudaGetLastError());
  }
  auto tdl = (cplx<T>*)h->tdl;
  auto tdinv = (cplx<T>*)h->tdinv;
  auto tdu = (cplx<T>*)h->tdu;
  auto tdu2 = (cplx<T>*)h->tdu2;
  ProfScope* l0 = new ProfScope(h->prof, PF_LEVEL0, s, 48.0 * ny * (double)ny * n1,
                                2.0 * n1 * (double)nn * sizeof(cplx<T>), 2);
  if (m0 > 0) {
    size_t tsm = TRI_WARPS * tri_smem_per_warp<T>(ny);
    if (tsm > 48 * 1024)
      RCI_CUDA_TRY(cudaFuncSetAttribute(tri_factor_kernel<T>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tsm));
    tri_factor_kernel<T><<<(unsigned)ceil_div(m0, TRI_WARPS), 32 * TRI_WARPS, tsm, s>>>(
        dg, cy, nx, ny, m0, tdl, tdinv, tdu, tdu2, h->tpiv, h->status);
    rci_note_launch();
    RCI_CUDA_TRY(cudaGetLastError());
  }
  {
    // D' and L' of the first reduced system
    constexpr bool half = sizeof(T) == 8;
    const int thr = (int)ceil_div(ny, 32) * 32;
    const size_t smem = l0_smem<T>(ny);
    if (smem > 48 * 1024)
      RCI_CUDA_TRY(cudaFuncSetAttribute(level0_schur_kernel<T, half>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    // the next level's working arrays are free during level 0 and serve as scratch
    level0_schur_kernel<T, half><<<n1, thr, smem, s>>>(dg, cx, cy, nx, ny, tdl, tdinv, tdu, tdu2,
                                                    h->tpiv, (cplx<T>*)h->Dw[0], (cplx<T>*)h->Lw[0],
                                                    (cplx<T>*)h->Dw[1], (cplx<T>*)h->Lw[1]);
    rci_note_launch();
    RCI_CUDA_TRY(cudaGetLastError());
    const int tiles = (int)ceil_div(ny, 32);
    for (int z0 = 0; half && z0 < n1; z0 += 32768) {  // (a grid's second extent ends at 65535)
      const int nz = std::min(n1 - z0, 32768);
      mirror_kernel<T><<<dim3((unsigned)(tiles * (tiles + 1) / 2), (unsigned)nz, 2), 256, 0, s>>>(
          (cplx<T>*)h->Dw[0] + z0 * nn, (cplx<T>*)h->Lw[0] + z0 * nn, ny, z0 == 0 ? 1 : 0);
      rci_note_launch();
      RCI_CUDA_TRY(cudaGetLastError());
    }
  }
  delete l0;
  const cplx<T> one = mkc(T(1), T(0)), mone = mkc(T(-1), T(0)), zero = czero<T>();
  int cur = 0;
  auto store = (cplx<T>*)h->store;
  // the scratch of an inversion (sch == false) or of the products of level l
  auto scratch_of = [&](int l, bool sch) {
    Scratch w;
    const int64_t bb = nn * (int64_t)sizeof(cplx<T>), nl = h->n[l], nk = l < h->Lf ? h->n[l + 1] : 0;
    w.add(h->scratch, std::max<int64_t>(m0, 1) * bb);
    for (void** a : {&h->Dw[0], &h->Lw[0]}) {
      w.add((char*)a[cur] + nl * bb, (n1 - nl) * bb);
      w.add((char*)a[1 - cur] + (sch ? nk * bb : 0), (n1 - (sch ? nk : 0)) * bb);
    }
    // the store of this level's products while its blocks are inverted, and of the levels to come
    const int64_t from = l >= h->Lf ? h->final_off + nn : sch ? h->off[l + 1] : h->off[l] + h->m[l] * nn;
    w.add((cplx<T>*)h->store + from, (h->final_off + nn - from) * (int64_t)sizeof(cplx<T>));
    return w;
  };
  // (taken where the scratch of every step holds at least one block: a dozen columns or more)
  bool split = sizeof(T) == 8 && ny <= SG_KMAX;
  if constexpr (sizeof(T) == 8) {
    for (int l = 1; l <= h->Lf && split; ++l) {
      Scratch wi = scratch_of(l, false);
      split = batch_of(wi, 1, [&](int c) { NewtonBuf(wi, ny, c); }) == 1;
      if (l == h->Lf || !split) break;
      Scratch ws = scratch_of(l, true);
      split = batch_of(ws, 1, [&](int c) { LevelBuf(ws, ny, c); }) == 1;
    }
  }
  // FP32 blocks above 160 rows by halves, where the scratch holds one
  auto by_halves = [&](Scratch& w) {
    return sizeof(T) == 4 && !h->simt && ny > 160 && ny <= SG_KMAX && ny % 2 == 0 &&
           batch_of(w, 1, [&](int c) { HalvesBuf(w, ny, c); }) == 1;
  };
  for (int l = 1; l < h->Lf; ++l) {
    const int n = (int)h->n[l], m = (int)h->m[l], nk = (int)h->n[l + 1];
    const int my = (n - 1) / 2;
    cplx<T>* D = (cplx<T>*)h->Dw[cur];
    cplx<T>* L = (cplx<T>*)h->Lw[cur];
    cplx<T>* Dn = (cplx<T>*)h->Dw[1 - cur];
    cplx<T>* Ln = (cplx<T>*)h->Lw[1 - cur];
    cplx<T>* Dinv = store + h->off[l];
    cplx<T>* X = Dinv + (int64_t)m * nn;
    cplx<T>* Y = X + (int64_t)m * nn;
    // D_r^{-1} for the odd rows (the working copy of D_r is destroyed)
    {
      ProfScope ps(h->prof, PF_INVERT, s, 8.0 * ny * (double)nn * m, 2.0 * m * nn * sizeof(cplx<T>), 1);
      if constexpr (sizeof(T) == 8) {
        if (split) {
          RCI_CUDA_TRY(launch_block_maxabs<T>(D + nn, 2 * nn, nn, m, maxabs + 1, s));
          Scratch w = scratch_of(l, false);
          RCI_CUDA_TRY(split_inverse(D + nn, 2 * nn, Dinv, ny, m, w, h->status, s));
        }
      }
      bool halves = false;
      if constexpr (sizeof(T) == 4) {
        Scratch w = scratch_of(l, false);
        if (by_halves(w)) {
          RCI_CUDA_TRY(launch_block_maxabs<T>(D + nn, 2 * nn, nn, m, maxabs + 1, s));
          const cudaError_t e = halves_inverse(D + nn, 2 * nn, Dinv, ny, m, w, h->status, s);
          if (e != cudaSuccess && e != cudaErrorNotSupported) return e;
          halves = e == cudaSuccess;
        }
      }
      if (!split && !halves) RCI_CUDA_TRY(launch_gj<T>(D + nn, 2 * nn, Dinv, nn, ny, m, h->status, s, maxabs + 1,
                                !h->simt));
    }
    // X_k = Dinv_k L_{2k+1};  Y_k = Dinv_k L_{2k+2}^T
    // D'_k = D_{2k} - L_{2k} Y_{k-1} (k >= 1) - L_{2k+1}^T X_k (k < m)
    // L'_k = -L_{2k} X_{k-1} (k >= 1)
    // FP32 on the tensor cores: two launches, X and Y together, then each D' as one product
    // over K = 2 ny (written once) together with L'; otherwise five batched products.
    bool fused = false;
    if constexpr (sizeof(T) == 8) {
      if (split) {
        Scratch w = scratch_of(l, true);
        RCI_CUDA_TRY(split_level(D, L, Dinv, X, Y, Dn, Ln, ny, n, m, nk, w, h->status, h->prof, s));
        fused = true;
      }
    }
    if constexpr (sizeof(T) == 4) {
      if (nk >= 2 && my >= 1) {
        const double pb = (double)sizeof(cplx<T>) * nn;
        TcJob xy[2] = {};
        xy[0].nseg = 1;
        xy[0].seg[0] = TcSegment{Dinv, ny, nn, m, false, L + nn, ny, 2 * nn, m, false, ny, 0, 0, 0, m};
        xy[0].alpha = 1.f;
        xy[0].C = X;
        xy[0].ldc = ny;
        xy[0].sC = nn;
        xy[0].batch = m;
        xy[1] = xy[0];
        xy[1].seg[0] = TcSegment{Dinv, ny, nn, my, false, L + 2 * nn, ny, 2 * nn, my, true, ny, 0, 0, 0, my};
        xy[1].C = Y;
        xy[1].batch = my;
        TcJob sl[2] = {};
        sl[0].nseg = 2;
        sl[0].seg[0] = TcSegment{L, ny, 2 * nn, nk, false, Y, ny, nn, my, false, ny, 0, -1, 1, nk};
        sl[0].seg[1] = TcSegment{L + nn, ny, 2 * nn, m, true, X, ny, nn, m, false, ny, 0, 0, 0, m};
        sl[0].alpha = -1.f;
        sl[0].beta = 1.f;
        sl[0].C0 = D;
        sl[0].ldc0 = ny;
        sl[0].sC0 = 2 * nn;
        sl[0].C = Dn;
        sl[0].ldc = ny;
        sl[0].sC = nn;
        sl[0].batch = nk;
        sl[1].nseg = 1;
        sl[1].seg[0] = TcSegment{L + 2 * nn, ny, 2 * nn, nk - 1, false, X, ny, nn, m, false, ny, 0, 0, 0, nk - 1};
        sl[1].alpha = -1.f;
        sl[1].C = Ln + nn;
        sl[1].ldc = ny;
        sl[1].sC = nn;
        sl[1].batch = nk - 1;
        cudaError_t e;
        {
          ProfScope ps(h->prof, PF_GEMM, s, 8.0 * ny * (double)nn * (m + my), pb * 3.0 * (m + my), 1);
          e = h->simt ? cudaErrorNotSupported
                      : launch_tc_cgemm_tma_jobs(ny, ny, 2, xy, h->status, tc_wait_limit(), s);
        }
        if (e == cudaSuccess) {
          ProfScope ps(h->prof, PF_GEMM, s, 8.0 * ny * (double)nn * (2 * (nk - 1) + m),
                       pb * (2.0 * (nk - 1 + m) + 2.0 * nk + 3.0 * (nk - 1)), 1);
          RCI_CUDA_TRY(launch_tc_cgemm_tma_jobs(ny, ny, 2, sl, h->status, tc_wait_limit(), s));
          fused = true;
        } else if (e != cudaErrorNotSupported) {
          return e;
        }
      }
    }
    if (!fused) {
      RCI_CUDA_TRY(gemm<T>(ny, ny, ny, false, false, one, Dinv, ny, nn, L + nn, ny, 2 * nn, zero,
                           nullptr, 0, 0, X, ny, nn, m, s, h->prof, PF_GEMM, gemm_status(h)));
      RCI_CUDA_TRY(gemm<T>(ny, ny, ny, false, true, one, Dinv, ny, nn, L + 2 * nn, ny, 2 * nn, zero,
                           nullptr, 0, 0, Y, ny, nn, my, s, h->prof, PF_GEMM, gemm_status(h)));
      RCI_CUDA_TRY(cudaMemcpyAsync(Dn, D, nn * sizeof(cplx<T>), cudaMemcpyDeviceToDevice, s));
      RCI_CUDA_TRY(gemm<T>(ny, ny, ny, false, false, mone, L + 2 * nn, ny, 2 * nn, Y, ny, nn, one,
                           D + 2 * nn, ny, 2 * nn, Dn + nn, ny, nn, nk - 1, s, h->prof, PF_GEMM,
                           gemm_status(h)));
      RCI_CUDA_TRY(gemm<T>(ny, ny, ny, true, false, mone, L + nn, ny, 2 * nn, X, ny, nn, one, Dn,
                           ny, nn, Dn, ny, nn, m, s, h->prof, PF_GEMM, gemm_status(h)));
      RCI_CUDA_TRY(gemm<T>(ny, ny, ny, false, false, mone, L + 2 * nn, ny, 2 * nn, X, ny, nn, zero,
                           nullptr, 0, 0, Ln + nn, ny, nn, nk - 1, s, h->prof, PF_GEMM, gemm_status(h)));
    }
    cur = 1 - cur;
  }
  // last single row
  {
    ProfScope ps(h->prof, PF_INVERT, s, 8.0 * ny * (double)nn, 2.0 * nn * sizeof(cplx<T>), 1);
    if constexpr (sizeof(T) == 8) {
      if (split) {
        RCI_CUDA_TRY(launch_block_maxabs<T>((cplx<T>*)h->Dw[cur], nn, nn, 1, maxabs + 1, s));
        Scratch w = scratch_of(h->Lf, false);
        return split_inverse((cplx<T>*)h->Dw[cur], nn, store + h->final_off, ny, 1, w, h->status, s);
      }
    }
    if constexpr (sizeof(T) == 4) {
      Scratch w = scratch_of(h->Lf, false);
      if (by_halves(w)) {
        RCI_CUDA_TRY(launch_block_maxabs<T>((cplx<T>*)h->Dw[cur], nn, nn, 1, maxabs + 1, s));
        const cudaError_t e = halves_inverse((cplx<T>*)h->Dw[cur], nn, store + h->final_off, ny, 1, w, h->status, s);
        if (e != cudaErrorNotSupported) return e;
      }
    }
    RCI_CUDA_TRY(launch_gj<T>((cplx<T>*)h->Dw[cur], 0, store + h->final_off, 0, ny, 1, h->status, s,
                              maxabs + 1, !h->simt));
  }
  return cudaSuccess;
}

cudaError_t bcr_factor(BcrHandle* h, const double2* dg, const double2* cx, const double2* cy,
                       cudaStream_t s) {
  return h->prec == RCI_FP64 ? factor_t<double>(h, dg, cx, cy, s)
                             : factor_t<float>(h, dg, cx, cy, s);
}

// columns of the workspace rows for nrhs right-hand sides (even in FP32: the TMA-fed products take
// 16-byte aligned rows)
static int ws_cols(const BcrHandle* h, int nrhs) { return h->prec == RCI_FP64 ? nrhs : (nrhs + 1) & ~1; }

// workspace layout (elements of cplx<T>); one right-hand side:
//   t0 [m0 row] | B_l [n_l row] (l = 1..Lf) | t_l [m_l row] (l = 1..Lf-1) | P, Q of the odd levels,
//   of the even levels | xf [row]
// several: t0 [m0 row] | B_1 [n_1 row] | t_l [m_l row] (l = 1..Lf-1) | xf [row]
static int64_t ws_elems(const BcrHandle* h, int nrhs) {
  const int64_t row = (int64_t)h->ny * (nrhs == 1 ? 1 : ws_cols(h, nrhs));
  int64_t t = 0, B = 0;
  for (int l = 1; l <= h->Lf; ++l) B += h->n[l];
  for (int l = 1; l < h->Lf; ++l) t += h->m[l];
  if (nrhs > 1) return std::max((h->m[0] + h->n[1] + t + 1) * row, ws_elems(h, 1));
  const int64_t m1 = h->Lf > 1 ? h->m[1] : 0, m2 = h->Lf > 2 ? h->m[2] : 0;
  return (h->m[0] + B + t + 2 * m1 + 2 * m2 + 1) * row;
}

cudaError_t bcr_reserve_ws(BcrHandle* h, int nrhs) {
  if (h->ws_nrhs >= nrhs) return cudaSuccess;
  free_ws(h);
  size_t bytes = (size_t)ws_elems(h, nrhs) * h->esz;
  RCI_CUDA_TRY(h->mem.alloc(&h->ws, bytes));
  h->ws_bytes = bytes;
  h->ws_nrhs = nrhs;
  return cudaSuccess;
}

// ===================================================================== several right-hand sides
// The rows of every level live in one array B1 (level l: rows 2^(l-1) apart), so that a level's
// kept rows are updated in place, the solution of a level is found where the level below reads
// it, and no copies or separate sums remain:
//   forward   t_k = Dinv_k b_{2k+1};  b_{2e} -= Y_{e-1}^T b_{2e-1} + X_e^T b_{2e+1}
//   backward  x_{2k+1} = t_k - X_k x_{2k} - Y_k x_{2k+2}
// Each line is one launch: FP32 on the TMA-fed tensor-core kernel (a product over two K segments),
// FP64 on the digit split of tc_gemm64.cu; the SIMT pipe and sizes the split does not take run
// the products one by one.
namespace {

// One level of the solve: dst_z = c0_z - A0_z[op] src_{z+z0} - A1_z[op] src_{z+z1} over the z that
// have them; rows of src `ss`, of dst `sd`, of c0 `sc` elements apart.
template <typename T>
struct MultiTerm {
  const cplx<T>* A;   // null: the term is not there
  int nA;             // members
  bool ta;
  int zA, zB, zlo, zhi;
};

}  // namespace

template <typename T>
static cudaError_t multi_update(BcrHandle* h, int ny, int nq, const MultiTerm<T> (&tm)[2], const cplx<T>* src,
                                int64_t ss, int nsrc, const cplx<T>* c0, int64_t sc, cplx<T>* dst, int64_t sd,
                                int batch, cudaStream_t s) {
  const int64_t nn = (int64_t)ny * ny;
  const cplx<T> one = mkc(T(1), T(0)), mone = mkc(T(-1), T(0));
  if (batch <= 0) return cudaSuccess;
  if constexpr (sizeof(T) == 4) {
    if (!h->simt) {
      TcJob j{};
      for (const MultiTerm<T>& t : tm)
        if (t.A && t.zhi > t.zlo)
          j.seg[j.nseg++] = TcSegment{t.A, ny, nn, t.nA, t.ta, src, nq, ss, nsrc, false, ny, t.zA, t.zB, t.zlo, t.zhi};
      if (j.nseg > 0) {
        j.alpha = -1.f;
        j.beta = 1.f;
        j.C0 = c0;
        j.ldc0 = nq;
        j.sC0 = sc;
        j.C = dst;
        j.ldc = nq;
        j.sC = sd;
        j.batch = batch;
        const cudaError_t e = launch_tc_cgemm_tma_jobs(ny, nq, 1, &j, h->status, tc_wait_limit(), s);
        if (e != cudaErrorNotSupported) return e;
      }
    }
  }
  // one product after the other: the first takes c0 (it covers every row where c0 is not dst)
  bool first = true;
  for (const MultiTerm<T>& t : tm) {
    if (!t.A || t.zhi <= t.zlo) continue;
    const cplx<T>* c = first ? c0 + t.zlo * sc : dst + t.zlo * sd;
    RCI_CUDA_TRY(gemm<T>(ny, nq, ny, t.ta, false, mone, t.A + (t.zlo + t.zA) * nn, ny, nn,
                         src + (t.zlo + t.zB) * ss, nq, ss, one, c, nq, first ? sc : sd, dst + t.zlo * sd, nq, sd,
                         t.zhi - t.zlo, s, nullptr, PF_SOLVE, gemm_status(h)));
    first = false;
  }
  return cudaSuccess;
}

// The split solve's scratch: the handle's and, after the factorisation, its working arrays.
static Scratch solve_scratch(const BcrHandle* h) {
  const int64_t bb = (int64_t)h->ny * h->ny * (int64_t)sizeof(double2), n1 = (h->nx + 1) / 2;
  Scratch w;
  w.add(h->scratch, std::max<int64_t>(h->m[0], 1) * bb);
  for (void* a : {h->Dw[0], h->Dw[1], h->Lw[0], h->Lw[1]}) w.add(a, n1 * bb);
  return w;
}

// One forward level in FP64: rows n of B (st elements apart), m eliminated.
static cudaError_t split_fwd(BcrHandle* h, Scratch& mem, const double2* Dinv, const double2* X, const double2* Y,
                             double2* B, int64_t st, double2* t, int n, int m, int nk, int nq, cudaStream_t s) {
  const int ny = h->ny, my = (n - 1) / 2;
  const int64_t nn = (int64_t)ny * ny, row = (int64_t)ny * nq;
  const int cb = batch_of(mem, nk, [&](int c) { FwdBuf(mem, ny, nq, c); });
  if (cb == 0) return cudaErrorInvalidValue;
  for (int k0 = 0; k0 < nk; k0 += cb) {
    const int c = std::min(cb, nk - k0), cm = std::min(c, m - k0), p0 = k0 > 0 ? 1 : 0;
    const int ny1 = std::max(0, std::min(k0 + c - 1, my) - (k0 - p0));  // Y of rows k0 - p0 .. k0 + c - 2
    const int nb1 = p0 + cm;                                            // odd rows from index k0 - p0 on
    mem.reset();
    const FwdBuf w(mem, ny, nq, c);
    if (mem.full) return cudaErrorInvalidValue;
    unsigned char *fD = w.D.f, *fX = w.X.f, *fY = w.Y.f, *fB = w.B.f;
    int32_t *eD = w.D.e, *eX = w.X.e, *eY = w.Y.e, *eB = w.B.e;
    RCI_CUDA_TRY(launch_sg_split(Dinv + k0 * nn, false, ny, nn, false, ny, ny, 3, cm, fD, eD, nullptr, s));
    RCI_CUDA_TRY(launch_sg_split(X + k0 * nn, false, ny, nn, true, ny, ny, 3, cm, fX, eX, nullptr, s));
    RCI_CUDA_TRY(launch_sg_split(Y + (k0 - p0) * nn, false, ny, nn, true, ny, ny, 3, ny1, fY, eY, nullptr, s));
    RCI_CUDA_TRY(launch_sg_split(B + (2 * (int64_t)(k0 - p0) + 1) * st, false, nq, 2 * st, true, nq, ny, 2, nb1, fB,
                                 eB, nullptr, s));
    SgJob j[2] = {};
    j[0].nseg = 1;
    j[0].seg[0] = SgSeg{fD, eD, fB, eB, 3, 2, 0, p0, 0, cm};
    j[0].C = t + k0 * row;
    j[0].ldc = nq;
    j[0].sC = row;
    j[0].batch = cm;
    j[1].nseg = 2;
    j[1].seg[0] = SgSeg{fY, eY, fB, eB, 3, 2, p0 - 1, p0 - 1, 1 - p0, c};
    j[1].seg[1] = SgSeg{fX, eX, fB, eB, 3, 2, 0, p0, 0, cm};
    j[1].neg = true;
    j[1].C = B + 2 * (int64_t)k0 * st;
    j[1].ldc = nq;
    j[1].sC = 2 * st;
    j[1].C0 = j[1].C;
    j[1].ldc0 = nq;
    j[1].sC0 = 2 * st;
    j[1].batch = c;
    RCI_CUDA_TRY(launch_sg_gemm(ny, nq, ny, 2, j, SG_FULL, h->status, tc_wait_limit(), s));
  }
  return cudaSuccess;
}

// One backward level in FP64.
static cudaError_t split_bwd(BcrHandle* h, Scratch& mem, const double2* X, const double2* Y, double2* B, int64_t st,
                             const double2* t, int n, int m, int nq, cudaStream_t s) {
  const int ny = h->ny, my = (n - 1) / 2;
  const int64_t nn = (int64_t)ny * ny, row = (int64_t)ny * nq;
  const int nk = (n + 1) / 2;
  const int cb = batch_of(mem, m, [&](int c) { FwdBuf(mem, ny, nq, c); });
  if (cb == 0) return cudaErrorInvalidValue;
  for (int k0 = 0; k0 < m; k0 += cb) {
    const int c = std::min(cb, m - k0), cy = std::max(0, std::min(c, my - k0)), nb1 = std::min(c + 1, nk - k0);
    mem.reset();
    const FwdBuf w(mem, ny, nq, c);
    if (mem.full) return cudaErrorInvalidValue;
    unsigned char *fX = w.X.f, *fY = w.Y.f, *fB = w.B.f;
    int32_t *eX = w.X.e, *eY = w.Y.e, *eB = w.B.e;
    RCI_CUDA_TRY(launch_sg_split(X + k0 * nn, false, ny, nn, false, ny, ny, 3, c, fX, eX, nullptr, s));
    RCI_CUDA_TRY(launch_sg_split(Y + k0 * nn, false, ny, nn, false, ny, ny, 3, cy, fY, eY, nullptr, s));
    RCI_CUDA_TRY(launch_sg_split(B + 2 * (int64_t)k0 * st, false, nq, 2 * st, true, nq, ny, 2, nb1, fB, eB, nullptr, s));
    SgJob j{};
    j.nseg = 2;
    j.seg[0] = SgSeg{fX, eX, fB, eB, 3, 2, 0, 0, 0, c};
    j.seg[1] = SgSeg{fY, eY, fB, eB, 3, 2, 0, 1, 0, cy};
    j.neg = true;
    j.C0 = t + k0 * row;
    j.ldc0 = nq;
    j.sC0 = row;
    j.C = B + (2 * (int64_t)k0 + 1) * st;
    j.ldc = nq;
    j.sC = 2 * st;
    j.batch = c;
    RCI_CUDA_TRY(launch_sg_gemm(ny, nq, ny, 1, &j, SG_FULL, h->status, tc_wait_limit(), s));
  }
  return cudaSuccess;
}

template <typename T>
static cudaError_t solve_multi(BcrHandle* h, const double2* cx, const cplx<T>* b, cplx<T>* x, int nrhs,
                               cudaStream_t s) {
  const int nx = h->nx, ny = h->ny, nq = ws_cols(h, nrhs);
  const int64_t nn = (int64_t)ny * ny, row = (int64_t)ny * nq;
  const int m0 = (int)h->m[0], n1 = (nx + 1) / 2;
  RCI_CUDA_TRY(bcr_reserve_ws(h, nrhs));
  cplx<T>* p = (cplx<T>*)h->ws;
  cplx<T>* t0 = p;
  p += m0 * row;
  cplx<T>* B1 = p;
  p += n1 * row;
  std::vector<cplx<T>*> tl(h->Lf + 1, nullptr);
  for (int l = 1; l < h->Lf; ++l) {
    tl[l] = p;
    p += h->m[l] * row;
  }
  cplx<T>* xf = p;
  auto store = (const cplx<T>*)h->store;
  const cplx<T> one = mkc(T(1), T(0)), zero = czero<T>();
  double sbytes = 2.0 * m0 * 5.0 * ny * sizeof(cplx<T>), sflops = 2.0 * 30.0 * m0 * (double)ny * nrhs;
  for (int l = 1; l < h->Lf; ++l) {
    sbytes += 5.0 * h->m[l] * (double)nn * sizeof(cplx<T>);
    sflops += 5.0 * 8.0 * h->m[l] * (double)nn * nrhs;
  }
  sbytes += (double)nn * sizeof(cplx<T>) + 2.0 * nx * (double)ny * nrhs * sizeof(cplx<T>);
  const int dense = h->Lf - 1;
  ProfScope ps(h->prof, PF_SOLVE, s, sflops, sbytes, (m0 > 0 ? 1 : 0) + 1 + 2 * dense + 1 + dense + 1);
  bool split = false;
  Scratch mem;
  if constexpr (sizeof(T) == 8) {
    mem = solve_scratch(h);
    FwdBuf(mem, ny, nq, 1);
    split = ny <= SG_KMAX && !mem.full;
  }

  // ---- level 0 forward by tridiagonal sweeps, then its kept rows
  // FP32: staged while rows and columns do not fill the GPU.  Measured at 3 to 500 cells of 48 to 224 rows
  // with 2 to 128 columns, a whole solve gains up to 1.37-fold by it, 1.03 at 32768 of them and nothing at
  // 49000 (250 cells of 224 rows, 48 columns).
  const bool staged = sizeof(T) == 4 && (int64_t)m0 * nrhs <= 32768;
  const int parts = (int)ceil_div(nrhs, TRG_COLS), cols = (int)ceil_div(nrhs, parts);
  const size_t trg = sizeof(cplx<T>) * ny * (4 + (size_t)cols) + ny;
  if constexpr (sizeof(T) == 4) {
    if (staged && trg > 48 * 1024) {
      RCI_CUDA_TRY(cudaFuncSetAttribute(tri_staged_kernel<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)trg));
      RCI_CUDA_TRY(cudaFuncSetAttribute(tri_staged_kernel<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)trg));
    }
  }
  auto sweep_staged = [&](auto kernel, unsigned rows, cplx<T>* t) {
    kernel<<<dim3(rows, (unsigned)parts), TRG_THREADS, trg, s>>>(
        b, t, cx, x, nx, ny, nrhs, nq, cols, (const cplx<T>*)h->tdl, (const cplx<T>*)h->tdinv,
        (const cplx<T>*)h->tdu, (const cplx<T>*)h->tdu2, h->tpiv);
  };
  if (m0 > 0) {
    if (staged) {
      if constexpr (sizeof(T) == 4) sweep_staged(tri_staged_kernel<T, false>, (unsigned)m0, t0);
    } else {
      fwd0_kernel<T><<<(unsigned)ceil_div((int64_t)m0 * nrhs, 128), 128, 0, s>>>(
          b, t0, ny, m0, nrhs, nq, (const cplx<T>*)h->tdl, (const cplx<T>*)h->tdinv, (const cplx<T>*)h->tdu,
          (const cplx<T>*)h->tdu2, h->tpiv);
    }
    rci_note_launch();
    RCI_CUDA_TRY(cudaGetLastError());
  }
  keep0_kernel<T><<<(unsigned)ceil_div(n1 * row, 256), 256, 0, s>>>(b, t0, cx, B1, nx, ny, n1, nrhs, nq);
  rci_note_launch();
  RCI_CUDA_TRY(cudaGetLastError());
  // ---- dense levels forward
  for (int l = 1; l < h->Lf; ++l) {
    const int n = (int)h->n[l], m = (int)h->m[l], nk = (int)h->n[l + 1], my = (n - 1) / 2;
    const cplx<T>* Dinv = store + h->off[l];
    const cplx<T>* X = Dinv + (int64_t)m * nn;
    const cplx<T>* Y = X + (int64_t)m * nn;
    const int64_t st = row << (l - 1);
    if constexpr (sizeof(T) == 8) {
      if (split) {
        RCI_CUDA_TRY(split_fwd(h, mem, Dinv, X, Y, B1, st, tl[l], n, m, nk, nq, s));
        continue;
      }
    }
    RCI_CUDA_TRY(gemm<T>(ny, nq, ny, false, false, one, Dinv, ny, nn, B1 + st, nq, 2 * st, zero, nullptr, 0, 0,
                         tl[l], nq, row, m, s, nullptr, PF_SOLVE, gemm_status(h)));
    const MultiTerm<T> tm[2] = {{Y, my, true, -1, -1, 1, my + 1}, {X, m, true, 0, 0, 0, m}};
    RCI_CUDA_TRY(multi_update<T>(h, ny, nq, tm, B1 + st, 2 * st, m, B1, 2 * st, B1, 2 * st, nk, s));
  }
  // ---- single remaining row
  {
    const cplx<T>* Dinv = store + h->final_off;
    bool done = false;
    if constexpr (sizeof(T) == 8) {
      if (split) {
        mem.reset();
        const FwdBuf w(mem, ny, nq, 1);
        if (mem.full) return cudaErrorInvalidValue;
        unsigned char *fD = w.D.f, *fB = w.B.f;
        int32_t *eD = w.D.e, *eB = w.B.e;
        RCI_CUDA_TRY(launch_sg_split(Dinv, false, ny, nn, false, ny, ny, 3, 1, fD, eD, nullptr, s));
        RCI_CUDA_TRY(launch_sg_split(B1, false, nq, row, true, nq, ny, 2, 1, fB, eB, nullptr, s));
        SgJob j{};
        j.nseg = 1;
        j.seg[0] = SgSeg{fD, eD, fB, eB, 3, 2, 0, 0, 0, 1};
        j.C = B1;  // (the operand is its split form)
        j.ldc = nq;
        j.sC = row;
        j.batch = 1;
        RCI_CUDA_TRY(launch_sg_gemm(ny, nq, ny, 1, &j, SG_FULL, h->status, tc_wait_limit(), s));
        done = true;
      }
    }
    if (!done) {
      RCI_CUDA_TRY(gemm<T>(ny, nq, ny, false, false, one, Dinv, ny, 0, B1, nq, 0, zero, nullptr, 0, 0, xf, nq, 0, 1, s,
                           nullptr, PF_SOLVE, gemm_status(h)));
      RCI_CUDA_TRY(cudaMemcpyAsync(B1, xf, row * sizeof(cplx<T>), cudaMemcpyDeviceToDevice, s));
    }
  }
  // ---- dense levels backward
  for (int l = h->Lf - 1; l >= 1; --l) {
    const int n = (int)h->n[l], m = (int)h->m[l], nk = (int)h->n[l + 1], my = (n - 1) / 2;
    const cplx<T>* X = store + h->off[l] + (int64_t)m * nn;
    const cplx<T>* Y = X + (int64_t)m * nn;
    const int64_t st = row << (l - 1);
    if constexpr (sizeof(T) == 8) {
      if (split) {
        RCI_CUDA_TRY(split_bwd(h, mem, X, Y, B1, st, tl[l], n, m, nq, s));
        continue;
      }
    }
    const MultiTerm<T> tm[2] = {{X, m, false, 0, 0, 0, m}, {Y, my, false, 0, 1, 0, my}};
    RCI_CUDA_TRY(multi_update<T>(h, ny, nq, tm, B1, 2 * st, nk, tl[l], row, B1 + st, 2 * st, m, s));
  }
  // ---- level 0 backward by tridiagonal sweeps (and the kept rows copied)
  if (staged) {
    if constexpr (sizeof(T) == 4) sweep_staged(tri_staged_kernel<T, true>, (unsigned)n1, B1);
  } else {
    bwd0_kernel<T><<<(unsigned)ceil_div((int64_t)n1 * nrhs, 128), 128, 0, s>>>(
        b, B1, cx, x, nx, ny, n1, nrhs, nq, (const cplx<T>*)h->tdl, (const cplx<T>*)h->tdinv, (const cplx<T>*)h->tdu,
        (const cplx<T>*)h->tdu2, h->tpiv);
  }
  rci_note_launch();
  return cudaGetLastError();
}

template <typename T>
static cudaError_t solve_one(BcrHandle* h, const double2* cx, const cplx<T>* b, cplx<T>* x, cudaStream_t s) {
  const int nx = h->nx, ny = h->ny;
  const int64_t nn = (int64_t)ny * ny;
  const int64_t row = ny;
  const int m0 = (int)h->m[0], n1 = (nx + 1) / 2;
  RCI_CUDA_TRY(bcr_reserve_ws(h, 1));
  // carve the workspace
  cplx<T>* p = (cplx<T>*)h->ws;
  cplx<T>* t0 = p;
  p += h->m[0] * row;
  std::vector<cplx<T>*> B(h->Lf + 1, nullptr), tl(h->Lf + 1, nullptr);
  for (int l = 1; l <= h->Lf; ++l) {
    B[l] = p;
    p += h->n[l] * row;
  }
  for (int l = 1; l < h->Lf; ++l) {
    tl[l] = p;
    p += h->m[l] * row;
  }
  int64_t m1 = h->Lf > 1 ? h->m[1] : 0, m2 = h->Lf > 2 ? h->m[2] : 0;
  cplx<T>* P = p;
  p += m1 * row;
  cplx<T>* Q = p;
  p += m1 * row;
  // a second pair for the even levels: one right-hand side forms a level's rows from the P
  // and Q of the level before while it writes its own
  cplx<T>* P2 = p;
  p += m2 * row;
  cplx<T>* Q2 = p;
  p += m2 * row;
  cplx<T>* xf = p;

  auto store = (const cplx<T>*)h->store;

  // level 0: the tridiagonal factors twice; levels >= 1: Dinv, X, Y forward and X, Y backward
  double sbytes = 2.0 * m0 * 5.0 * ny * sizeof(cplx<T>), sflops = 2.0 * 30.0 * m0 * (double)ny;
  for (int l = 1; l < h->Lf; ++l) {
    sbytes += 5.0 * h->m[l] * (double)nn * sizeof(cplx<T>);
    sflops += 5.0 * 8.0 * h->m[l] * (double)nn;
  }
  sbytes += (double)nn * sizeof(cplx<T>) + 2.0 * nx * (double)ny * sizeof(cplx<T>);
  // kernels launched: level-0 pair, per dense level forward and backward, the last row
  const int dense = h->Lf - 1, l0 = m0 > 0 ? 1 : 0;
  ProfScope ps(h->prof, PF_SOLVE, s, sflops, sbytes, l0 + 1 + dense + 1 + dense + 1);

  if (ny % vec16<T>::per != 0 || ny > 256 * vec16<T>::per)
    return cudaErrorInvalidValue;  // (grid creation keeps ny within these limits)
  const int smax = (int)ceil_div(ny, 32 * vec16<T>::per);
  const unsigned nch = (unsigned)ceil_div(ny, RC);
  const size_t red_smem = (size_t)2 * CH_WARPS * RC * sizeof(cplx<T>);
#define RCI_SMAX_DISPATCH(KERNEL, GRID, SMEM, ...)                                   \
  do {                                                                               \
    switch (smax) {                                                                  \
      case 1: KERNEL<T, 1><<<GRID, CH_THREADS, SMEM, s>>>(__VA_ARGS__); break;       \
      case 2: KERNEL<T, 2><<<GRID, CH_THREADS, SMEM, s>>>(__VA_ARGS__); break;       \
      case 3: KERNEL<T, 3><<<GRID, CH_THREADS, SMEM, s>>>(__VA_ARGS__); break;       \
      case 4: KERNEL<T, 4><<<GRID, CH_THREADS, SMEM, s>>>(__VA_ARGS__); break;       \
      case 5: KERNEL<T, 5><<<GRID, CH_THREADS, SMEM, s>>>(__VA_ARGS__); break;       \
      case 6: KERNEL<T, 6><<<GRID, CH_THREADS, SMEM, s>>>(__VA_ARGS__); break;       \
      case 7: KERNEL<T, 7><<<GRID, CH_THREADS, SMEM, s>>>(__VA_ARGS__); break;       \
      default: KERNEL<T, 8><<<GRID, CH_THREADS, SMEM, s>>>(__VA_ARGS__); break;      \
    }                                                                                \
    rci_note_launch();                                                               \
    RCI_CUDA_TRY(cudaGetLastError());                                                \
  } while (0)
  // the chunked level-0 backward pass reads b while other blocks write x: no aliasing
  const cplx<T>* bsrc = b;
  if ((const void*)b == (const void*)x) return cudaErrorInvalidValue;
  // ---- level 0 forward: t0[k] = T_{2k+1}^{-1} b[2k+1] by tridiagonal sweeps
  const size_t trs_smem = TRS_WARPS * trs_smem_per_warp<T>(ny);
  auto trs_attr = [&](auto kern) -> cudaError_t {
    return trs_smem > 48 * 1024 ? cudaFuncSetAttribute(kern,
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)trs_smem)
                                : cudaSuccess;
  };
  // Many FP64 rows: one thread per row.  The FP64 pipe takes as long for a warp's one busy lane as for
  // all of them, so with a warp per row 2020 rows of 160 take 340 us a sweep; with a thread per row
  // 235 and 255.  Few rows are bound by one row's chain of operations, which is shorter on a warp's
  // staged copies (220 rows of 128: 84 us against 170 and 200).  The line lies where a ninth warp comes
  // to an SM: whole solves of 64 to 224 rows take 3 to 4 % less with warps at 1200 columns, 2 to 4 % less
  // with threads at 1400.
  const bool thread_per_row = sizeof(T) == 8 && m0 > 8 * 152;
  if (m0 > 0) {
    if (thread_per_row) {
      fwd0_kernel<T><<<(unsigned)ceil_div(m0, 32), 32, 0, s>>>(
          bsrc, t0, ny, m0, 1, 1, (const cplx<T>*)h->tdl, (const cplx<T>*)h->tdinv, (const cplx<T>*)h->tdu,
          (const cplx<T>*)h->tdu2, h->tpiv);
    } else {
      RCI_CUDA_TRY(trs_attr(tri_rows_solve_kernel<T, false>));
      tri_rows_solve_kernel<T, false><<<(unsigned)ceil_div(m0, TRS_WARPS), 32 * TRS_WARPS, trs_smem, s>>>(
          (const cplx<T>*)h->tdl, (const cplx<T>*)h->tdinv, (const cplx<T>*)h->tdu,
          (const cplx<T>*)h->tdu2, h->tpiv, bsrc, nullptr, cx, t0, nx, ny, m0);
    }
    rci_note_launch();
    RCI_CUDA_TRY(cudaGetLastError());
  }
  {
    int64_t nt = (int64_t)n1 * row;
    keep0_kernel<T><<<(unsigned)ceil_div(nt, 256), 256, 0, s>>>(bsrc, t0, cx, B[1], nx, ny, n1, 1, 1);
    rci_note_launch();
    RCI_CUDA_TRY(cudaGetLastError());
  }
  // ---- dense levels forward: level 1 from the kept rows of level 0; every later level forms
  // its rows from the level before (the kept-row update fused into its forward kernel), the
  // P and Q of odd levels in (P, Q), of even levels in (P2, Q2)
  auto Pl = [&](int l) { return (l & 1) ? P : P2; };
  auto Ql = [&](int l) { return (l & 1) ? Q : Q2; };
  for (int l = 1; l < h->Lf; ++l) {
    const int n = (int)h->n[l], m = (int)h->m[l];
    const cplx<T>* Dinv = store + h->off[l];
    const cplx<T>* X = Dinv + (int64_t)m * nn;
    const cplx<T>* Y = X + (int64_t)m * nn;
    if (l == 1) {
      RCI_SMAX_DISPATCH(fwd_chunk_kernel, dim3(m, nch), ny * sizeof(cplx<T>) + red_smem, Dinv,
                        X, Y, B[1], tl[1], Pl(1), Ql(1), n, ny);
    } else {
      RCI_SMAX_DISPATCH(fwd_keep_chunk_kernel, dim3((unsigned)h->n[l + 1], nch),
                        ny * sizeof(cplx<T>) + red_smem, Dinv, X, Y, B[l - 1], Pl(l - 1),
                        Ql(l - 1), (int)h->m[l - 1], B[l], tl[l], Pl(l), Ql(l), n, ny);
    }
  }
  // ---- single remaining row (from the level before it when there is one, written straight
  // to B[Lf], which nothing reads as input then)
  if (h->Lf >= 2) {
    const int lp = h->Lf - 1;
    RCI_SMAX_DISPATCH(mv_keep_chunk_kernel, dim3(1, nch), ny * sizeof(cplx<T>),
                      store + h->final_off, B[lp], Pl(lp), Ql(lp), (int)h->m[lp], B[h->Lf], ny);
  } else {
    RCI_SMAX_DISPATCH(mv_chunk_kernel, dim3(1, nch), ny * sizeof(cplx<T>), store + h->final_off,
                      B[h->Lf], (int64_t)0, (int64_t)0, xf, ny);
    RCI_CUDA_TRY(cudaMemcpyAsync(B[h->Lf], xf, row * sizeof(cplx<T>), cudaMemcpyDeviceToDevice, s));
  }
  // ---- dense levels backward (the solution of level l overwrites B[l])
  for (int l = h->Lf - 1; l >= 1; --l) {
    const int n = (int)h->n[l], m = (int)h->m[l], nk = (int)h->n[l + 1];
    const cplx<T>* Dinv = store + h->off[l];
    const cplx<T>* X = Dinv + (int64_t)m * nn;
    const cplx<T>* Y = X + (int64_t)m * nn;
    RCI_SMAX_DISPATCH(bwd_chunk_kernel, dim3(nk, nch), 3 * ny * sizeof(cplx<T>), X, Y, tl[l],
                      B[l + 1], B[l], n, m, ny);
  }
  // ---- level 0 backward by tridiagonal sweeps (and the kept rows copied)
  if (thread_per_row) {
    bwd0_kernel<T><<<(unsigned)ceil_div(n1, 32), 32, 0, s>>>(
        bsrc, B[1], cx, x, nx, ny, n1, 1, 1, (const cplx<T>*)h->tdl, (const cplx<T>*)h->tdinv,
        (const cplx<T>*)h->tdu, (const cplx<T>*)h->tdu2, h->tpiv);
  } else {
    RCI_CUDA_TRY(trs_attr(tri_rows_solve_kernel<T, true>));
    tri_rows_solve_kernel<T, true><<<(unsigned)ceil_div(n1, TRS_WARPS), 32 * TRS_WARPS, trs_smem, s>>>(
        (const cplx<T>*)h->tdl, (const cplx<T>*)h->tdinv, (const cplx<T>*)h->tdu,
        (const cplx<T>*)h->tdu2, h->tpiv, bsrc, B[1], cx, x, nx, ny, n1);
  }
  rci_note_launch();
  RCI_CUDA_TRY(cudaGetLastError());
#undef RCI_SMAX_DISPATCH
  return cudaSuccess;
}

cudaError_t bcr_solve(BcrHandle* h, const double2* cx, const void* b, void* x, int nrhs,
                      cudaStream_t s) {
  if (nrhs < 1) return cudaErrorInvalidValue;
  if (h->prec == RCI_FP64)
    return nrhs == 1 ? solve_one<double>(h, cx, (const double2*)b, (double2*)x, s)
                     : solve_multi<double>(h, cx, (const double2*)b, (double2*)x, nrhs, s);
  return nrhs == 1 ? solve_one<float>(h, cx, (const float2*)b, (float2*)x, s)
                   : solve_multi<float>(h, cx, (const float2*)b, (float2*)x, nrhs, s);
}

cudaError_t bcr_block_inverse(const void* src, void* out, int n, int batch, int prec, int kernel,
                              int32_t* status, cudaStream_t s) {
  const int64_t nn = (int64_t)n * n;
  if (kernel == 3) {
    const bool f64 = prec == RCI_FP64;
    if (n > SG_KMAX || (!f64 && (n <= 160 || n % 2))) return cudaErrorInvalidValue;
    Scratch need, mem;
    need.add(nullptr, (int64_t)1 << 60);  // (only counted)
    if (f64) NewtonBuf(need, n, batch);
    else HalvesBuf(need, n, batch);
    void* w = nullptr;
    RCI_CUDA_TRY(cudaMalloc(&w, need.r[0].used));
    mem.add(w, (int64_t)need.r[0].used);
    cudaError_t e = f64 ? split_inverse((double2*)src, nn, (double2*)out, n, batch, mem, status, s)
                        : halves_inverse((float2*)src, nn, (float2*)out, n, batch, mem, status, s);
    if (e == cudaErrorNotSupported) e = cudaErrorInvalidValue;
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(w);
    return e;
  }
  if (prec == RCI_FP64) {
    if (kernel == 2) return cudaErrorInvalidValue;
    return launch_gj<double>((double2*)src, nn, (double2*)out, nn, n, batch, status, s);
  }
  if (kernel == 1) return launch_gj_simt<float>((float2*)src, nn, (float2*)out, nn, n, batch, status, s);
  if (kernel == 2) return launch_tc_gj((const float2*)src, nn, (float2*)out, nn, n, batch, status, s);
  return launch_gj<float>((float2*)src, nn, (float2*)out, nn, n, batch, status, s);
}

cudaError_t bcr_gemm(int M, int N, int K, bool ta, bool tb, double alpha, const void* A,
                     int64_t lda, int64_t sA, const void* B, int64_t ldb, int64_t sB, double beta,
                     const void* C0, int64_t ldc0, int64_t sC0, void* C, int64_t ldc, int64_t sC,
                     int batch, int prec, int kernel, int32_t* status, cudaStream_t s) {
  if (prec == RCI_FP64) {
    if (kernel == 1 || kernel == 2) return cudaErrorInvalidValue;
    if (kernel == 4) {
      if (K > SG_KMAX || (alpha != 1.0 && alpha != -1.0) || (C0 && beta != 1.0)) return cudaErrorInvalidValue;
      const size_t fa = batch * sg_form_bytes(M, K, 3), fb = batch * sg_form_bytes(N, K, 2);
      const size_t ea = sizeof(int32_t) * batch * sg_form_exps(M), eb = sizeof(int32_t) * batch * sg_form_exps(N);
      unsigned char* w = nullptr;
      RCI_CUDA_TRY(cudaMalloc(&w, fa + fb + ea + eb));
      unsigned char* wb = w + fa;
      int32_t *xa = reinterpret_cast<int32_t*>(wb + fb), *xb = reinterpret_cast<int32_t*>(wb + fb + ea);
      SgJob j{};
      j.nseg = 1;
      j.seg[0] = SgSeg{w, xa, wb, xb, 3, 2, 0, 0, 0, batch};
      j.neg = alpha < 0;
      j.C0 = (const double2*)C0;
      j.ldc0 = ldc0;
      j.sC0 = sC0;
      j.C = (double2*)C;
      j.ldc = ldc;
      j.sC = sC;
      j.batch = batch;
      cudaError_t e = launch_sg_split(A, false, lda, sA, ta, M, K, 3, batch, w, xa, nullptr, s);
      if (e == cudaSuccess) e = launch_sg_split(B, false, ldb, sB, !tb, N, K, 2, batch, wb, xb, nullptr, s);
      if (e == cudaSuccess) e = launch_sg_gemm(M, N, K, 1, &j, SG_FULL, status, tc_wait_limit(), s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      cudaFree(w);
      return e;
    }
    const cplx<double> al{alpha, 0.0}, be{beta, 0.0};
    return gemm<double>(M, N, K, ta, tb, al, (const double2*)A, lda, sA, (const double2*)B, ldb,
                        sB, be, (const double2*)C0, ldc0, sC0, (double2*)C, ldc, sC, batch, s);
  }
  const float2 al = make_float2((float)alpha, 0.f), be = make_float2((float)beta, 0.f);
  const float2 *a = (const float2*)A, *b = (const float2*)B, *c0 = (const float2*)C0;
  float2* c = (float2*)C;
  switch (kernel) {
    case 1:
      return launch_tc_cgemm(M, N, K, ta, tb, al, a, lda, sA, b, ldb, sB, be, c0, ldc0, sC0, c, ldc,
                             sC, batch, status, s, 1);
    case 2: {
      if (N > 160) return cudaErrorInvalidValue;  // (the entry point's stated limit)
      const cudaError_t e = launch_tc_cgemm_tma(M, N, K, ta, tb, (float)alpha, a, lda, sA, b, ldb, sB,
                                                (float)beta, c0, ldc0, sC0, c, ldc, sC, batch,
                                                status, tc_wait_limit(), s);
      return e == cudaErrorNotSupported ? cudaErrorInvalidValue : e;
    }
    case 3:  // SIMT: no status word, so the dispatch keeps off the tensor cores
      return gemm<float>(M, N, K, ta, tb, al, a, lda, sA, b, ldb, sB, be, c0, ldc0, sC0, c, ldc, sC,
                         batch, s);
    default:
      return gemm<float>(M, N, K, ta, tb, al, a, lda, sA, b, ldb, sB, be, c0, ldc0, sC0, c, ldc, sC,
                         batch, s, nullptr, PF_GEMM, status);
  }
}
