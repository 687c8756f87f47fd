// Small dense FP64 kernels of the Rayleigh-Ritz step (Section 2.1, Algorithm 1): the Cholesky factor
// of the B-Gram matrix with its inverse, and the symmetric eigensolver of the projected matrix.
//
// On this GPU FP64 arithmetic is scarce (about 2 DFMA per clock per SM) and the N x N problems
// (N = 60 ... 2400) are too small to fill the chip, so these steps are bound by the length of
// their sequential dependency chains.  The kernels keep every chain on the device and pay few
// exchanges between CTAs:
//   * chol_inv_blocked_kernel: Cholesky G = L L^T and L^-1 together, in 32 x 32 tiles on a cooperative
//     grid, two grid barriers per 32 columns (chol_inv_smem_kernel and chol_inv_kernel, a barrier per
//     column, stand in where it could not be resident);
//   * tridiag_xch_kernel: Householder reduction to tridiagonal form Q^T M Q = T for orders up to 1024, one
//     exchange per column, in one thread-block cluster through distributed shared memory (orders up to
//     320) or on a cooperative grid through L2; above, or where its columns do not fit in shared memory,
//     tridiag_smem_kernel and tridiag_kernel (two barriers per column: after the symmetric matrix-vector
//     product, after the rank-2 update);
//   * tri_eig_kernel: an eigenvalue of T and its vector per warp (orders up to 1408): Sturm multisection in
//     FP32, then FP64 with secant steps, the vector from a twisted factorisation; above, bisect_kernel
//     (multisection in FP64, 32 trial points per step) and inverse iteration for every vector;
//   * inviter_kernel: the vectors of clusters of numerically equal eigenvalues (gap <= 1e-9 ||T||) by
//     inverse iteration (tridiagonal LU with partial pivoting) with Gram-Schmidt inside the cluster;
//   * one Newton-Schulz step Z <- Z (3 I - Z^T Z) / 2 (two products) for the O(eps ||T|| / gap) residue
//     between the others, which leaves each residual at O(eps ||T||);
//   * backtransform_reg_kernel (orders up to 1024; above, backtransform_kernel): V = Q Z, four reflectors
//     per round.
// Multi-CTA kernels run as one thread-block cluster when the matrix is small, or as a cooperative grid
// when more SMs pay for the dearer exchange.  Data written by another CTA is read with ld.global.cg (L2),
// never through a possibly stale L1 line.
#include <cooperative_groups.h>

#include <cfloat>

#include "common.cuh"
#include "oz_digits.cuh"
#include "oz_gemm.cuh"
#include "prof.cuh"
#include "tc_ptx.cuh"

namespace cg = cooperative_groups;

namespace rchfsi {
namespace {

constexpr int EIG_THREADS = 512;

template <bool CLUSTER>
__device__ __forceinline__ void all_sync() {
  if constexpr (CLUSTER) {
    cg::this_cluster().sync();
  } else {
    cg::this_grid().sync();
  }
}

// Sum over the CTA; every thread receives the result.  `red` holds 33 doubles.
__device__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  if (w == 0) {
    double t = (l < (int)(blockDim.x >> 5)) ? red[l] : 0.0;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (l == 0) red[32] = t;
  }
  __syncthreads();
  return red[32];
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// What an FP64 instruction costs here (clock64): every SM sub-partition issues one warp-wide FP64
// instruction per 64 clocks, whatever its active lanes and however independent it is of the one
// before (16 dependent or independent DFMAs of a warp: 1000 clocks).  The kernels below therefore
// count FP64 instructions per sub-partition: full lanes, no redundant scalar work in FP64, sums
// across lanes and seeds in the integer and FP32 units.

// Sum over the warp of one double per lane, every lane receiving it, in integer arithmetic: the
// lanes' significands are aligned to the largest exponent (9 guard bits below its last place), cut
// into 26-bit limbs and added with redux.sync.  The result is within 1/8 unit in the last place of
// the largest addend plus one rounding, closer than a tree of FP64 adds, and costs one FP64
// instruction (a conversion) instead of five.  Non-finite addends, and such that a sum of 32 may leave the
// range, take the FP64 tree (NaN and Inf propagate); a result below the normal range is 0.
constexpr uint32_t kFxTop = 0x7f8;  // the largest exponent field the integer sum takes is one less
__device__ __forceinline__ double fx_scaled(long long t, uint32_t top) {  // t 2^(top - 1075 - 9 + 5)
  const double d = __ll2double_rn(t);
  const int he = __double2hiint(d), ef = ((he >> 20) & 0x7ff) + (int)top - 1079;
  return t != 0 && ef > 0 ? __hiloint2double(he + (((int)top - 1079) << 20), __double2loint(d)) : 0.0;
}
__device__ __forceinline__ double warp_sum_fx(double v) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const uint32_t e0 = (hi >> 20) & 0x7ffu;
  const uint32_t ex = max(e0, 1u);
  const uint32_t top = __reduce_max_sync(0xffffffffu, ex);
  if (top >= kFxTop) return warp_sum(v);
  const uint32_t sh = min(top - ex, 63u);
  const uint32_t mh = (hi & 0xfffffu) | (e0 ? 0x100000u : 0u);
  const unsigned long long mant = ((((unsigned long long)mh << 32) | lo) << 9) >> sh;
  const long long f = (int32_t)hi < 0 ? -(long long)mant : (long long)mant;
  // f = h 2^52 + m 2^26 + l with 0 <= m, l < 2^26: 32 limbs of 26 bits add up below 2^31
  const uint32_t l = (uint32_t)f & 0x3ffffffu, m = (uint32_t)(f >> 26) & 0x3ffffffu;
  const int h = (int)(f >> 52);
  const uint32_t sl = __reduce_add_sync(0xffffffffu, l), sm = __reduce_add_sync(0xffffffffu, m);
  const int sg = __reduce_add_sync(0xffffffffu, h);
  return fx_scaled(((long long)sg << 47) + ((long long)sm << 21) + (long long)(sl >> 5), top);
}

__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// 1 / sqrt(a) for a normal a > 0: FP32 seed y (22 bits), then one step of the third-order Householder
// iteration y (1 + e / 2 + 3 e^2 / 8), e = 1 - a y^2 (error e^3): 5 FP64 instructions.
__device__ __forceinline__ double rsqrt_h3(double a) {
  const int hi = __double2hiint(a), lo = __double2loint(a);
  const int eb = ((hi >> 20) & 0x7ff) - 1023, hf = eb >> 1;  // a = m 4^hf, m in [1, 4)
  const float m = __int_as_float(((eb - 2 * hf + 127) << 23) | ((hi & 0xfffff) << 3) | (int)((uint32_t)lo >> 29));
  const int yb = __float_as_int(rsqrtf(m));
  const double y = __hiloint2double((((yb >> 23) - 127 + 1023 - hf) << 20) | ((yb >> 3) & 0xfffff), yb << 29);
  const double e = fma(-a, y * y, 1.0);
  return fma(e * y, fma(0.375, e, 0.5), y);
}

// 1 / a for a normal a > 0: FP32 seed r (22 bits), then r (1 + e + e^2), e = 1 - a r: 3 FP64 instructions.
__device__ __forceinline__ double rcp_h3(double a) {
  const int hi = __double2hiint(a), lo = __double2loint(a);
  const int eb = ((hi >> 20) & 0x7ff) - 1023;
  const float m = __int_as_float((127 << 23) | ((hi & 0xfffff) << 3) | (int)((uint32_t)lo >> 29));
  const int yb = __float_as_int(__fdividef(1.0f, m));
  const double r = __hiloint2double((((yb >> 23) - 127 + 1023 - eb) << 20) | ((yb >> 3) & 0xfffff), yb << 29);
  const double e = fma(-a, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// ------------------------------------------------------------------ Cholesky and L^-1
// A (n x n, column-major, symmetric; its lower triangle is destroyed), L and Linv (outputs,
// lower triangular with zero upper part).  info = j + 1 when pivot j is not positive / finite.
// Column k of the trailing matrix is owned by CTA k mod P.
template <bool CLUSTER>
__global__ void __launch_bounds__(EIG_THREADS) chol_inv_kernel(int n, double* A, double* L, double* Linv,
                                                               int* info) {
  extern __shared__ double sm[];
  double* col = sm;      // n: scaled pivot column of the current step
  double* col2 = sm + n; // n: second buffer for the inverse phase
  const int P = gridDim.x, r = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
  bool bad = false;
  for (int j = 0; j < n; ++j) {
    const double ajj = __ldcg(A + (int64_t)j * n + j);
    if (!(ajj > 0.0) || !isfinite(ajj)) {
      // every CTA reads the same value, so all leave the loop at the same step
      if (r == 0 && tid == 0) *info = j + 1;
      bad = true;
      break;
    }
    const double piv = sqrt(ajj), inv = 1.0 / piv;
    for (int i = j + 1 + tid; i < n; i += blockDim.x) col[i] = __ldcg(A + (int64_t)j * n + i) * inv;
    __syncthreads();
    if (j % P == r) {
      for (int i = tid; i < n; i += blockDim.x) L[(int64_t)j * n + i] = i < j ? 0.0 : (i == j ? piv : col[i]);
    }
    // trailing update of the owned columns k > j (lower part): A(i,k) -= L(i,j) L(k,j)
    const int k0 = j + 1 + ((r - (j + 1)) % P + P) % P;  // first owned column > j
    for (int k = k0 + warp * P; k < n; k += nw * P) {
      const double lk = col[k];
      double* ak = A + (int64_t)k * n;
      for (int i = k + lane; i < n; i += 32) ak[i] -= col[i] * lk;
    }
    all_sync<CLUSTER>();
  }
  if (bad) return;
  if (r == 0 && tid == 0) *info = 0;
  // L^-1: column c solves L x = e_c; the warp owning c does every step of that column
  for (int c = r + warp * P; c < n; c += nw * P)
    for (int i = lane; i < n; i += 32) Linv[(int64_t)c * n + i] = (i == c) ? 1.0 : 0.0;
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    double* lc = (k & 1) ? col2 : col;
    for (int i = k + tid; i < n; i += blockDim.x) lc[i] = __ldcg(L + (int64_t)k * n + i);
    __syncthreads();
    const double inv = 1.0 / lc[k];
    for (int c = r + warp * P; c <= k && c < n; c += nw * P) {
      double* x = Linv + (int64_t)c * n;
      const double xk = x[k] * inv;
      __syncwarp();
      if (lane == 0) x[k] = xk;
      for (int i = k + 1 + lane; i < n; i += 32) x[i] -= lc[i] * xk;
      __syncwarp();
    }
    // the other buffer is refilled next step, after every warp has left this one (2 steps apart)
  }
}

// Same factorisation with the owned columns resident in shared memory (nq = ceil(n / P) columns per
// CTA), the pivot column exchanged through a double-buffered L2 slot (xch, 2 n doubles: the owner of
// column j + 1 publishes it during step j while the others may still read column j), one barrier
// per column.  L^-1 then runs as in chol_inv_kernel, with the next column of L prefetched into
// registers (rows tid + 256 t, t < 16, so n <= 4096).
template <bool CLUSTER>
__global__ void __launch_bounds__(256) chol_inv_smem_kernel(int n, const double* __restrict__ A, double* L,
                                                            double* Linv, double* xch, double* dinv, int* info) {
  extern __shared__ double sm[];
  constexpr int MAXT = 16;
  const int P = gridDim.x, r = blockIdx.x;
  const int nq = (n - r + P - 1) / P;
  double* cols = sm;                  // nq x n
  double* col = cols + (size_t)nq * n;  // n (scaled pivot column), later the first L^-1 buffer
  double* col2 = col + n;             // n
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5, bd = blockDim.x;
  for (int q = 0; q < nq; ++q)
    for (int i = tid; i < n; i += bd) cols[(size_t)q * n + i] = A[(size_t)(r + q * P) * n + i];
  __syncthreads();
  if (r == 0)
    for (int i = tid; i < n; i += bd) __stcg(xch + i, cols[i]);
  all_sync<CLUSTER>();
  bool bad = false;
  for (int j = 0; j < n; ++j) {
    const double* xj = xch + (size_t)(j & 1) * n;
    const double ajj = __ldcg(xj + j);
    if (!(ajj > 0.0) || !isfinite(ajj)) {
      if (r == 0 && tid == 0) *info = j + 1;
      bad = true;
      break;
    }
    const double inv = rsqrt(ajj), piv = ajj * inv;
    for (int i = j + 1 + tid; i < n; i += bd) col[i] = __ldcg(xj + i) * inv;
    __syncthreads();
    if (j % P == r) {
      for (int i = tid; i < n; i += bd) L[(size_t)j * n + i] = i < j ? 0.0 : (i == j ? piv : col[i]);
      if (tid == 0) __stcg(dinv + j, inv);
    }
    const int qa = (j + 1 - r + P - 1) / P > 0 ? (j + 1 - r + P - 1) / P : 0;
    for (int q = qa + warp; q < nq; q += nw) {
      const int k = r + q * P;
      const double lk = col[k];
      double* ak = cols + (size_t)q * n;
      for (int i = k + lane; i < n; i += 32) ak[i] -= col[i] * lk;
    }
    __syncthreads();
    if (j + 1 < n && (j + 1) % P == r) {
      const double* ak = cols + (size_t)((j + 1 - r) / P) * n;
      double* xn = xch + (size_t)((j + 1) & 1) * n;
      for (int i = j + 1 + tid; i < n; i += bd) __stcg(xn + i, ak[i]);
    }
    all_sync<CLUSTER>();
  }
  if (bad) return;
  if (r == 0 && tid == 0) *info = 0;
  for (int c = r + warp * P; c < n; c += nw * P)
    for (int i = lane; i < n; i += 32) Linv[(size_t)c * n + i] = (i == c) ? 1.0 : 0.0;
  double cur[MAXT], nxt[MAXT];
  double dcur = __ldcg(dinv), dnxt = 0.0;
#pragma unroll
  for (int t = 0; t < MAXT; ++t) {
    const int i = tid + bd * t;
    cur[t] = i < n ? __ldcg(L + i) : 0.0;
  }
  for (int k = 0; k < n; ++k) {
    double* lc = (k & 1) ? col2 : col;
#pragma unroll
    for (int t = 0; t < MAXT; ++t) {
      const int i = tid + bd * t;
      if (i >= k && i < n) lc[i] = cur[t];
    }
    if (k + 1 < n) {
#pragma unroll
      for (int t = 0; t < MAXT; ++t) {
        const int i = tid + bd * t;
        nxt[t] = (i >= k + 1 && i < n) ? __ldcg(L + (size_t)(k + 1) * n + i) : 0.0;
      }
      dnxt = __ldcg(dinv + k + 1);
    }
    __syncthreads();
    const double inv = dcur;
    for (int c = r + warp * P; c <= k && c < n; c += nw * P) {
      double* x = Linv + (size_t)c * n;
      const double xk = x[k] * inv;
      __syncwarp();
      if (lane == 0) x[k] = xk;
      for (int i = k + 1 + lane; i < n; i += 32) x[i] -= lc[i] * xk;
      __syncwarp();
    }
#pragma unroll
    for (int t = 0; t < MAXT; ++t) cur[t] = nxt[t];
    dcur = dnxt;
  }
}

// ------------------------------------------------------------------ blocked Cholesky and L^-1
// A = L L^T (A symmetric positive definite, n x n column-major, lower triangle read) and L^-1, on a
// cooperative grid, in 32 x 32 tiles.  Per block column K, with B = I in Linv at the start:
//   1. every CTA factors the diagonal tile and inverts its factor (DI_K = L_KK^-1) for itself: the
//      same bits everywhere, and no barrier before they are used;
//   2. panel L_IK = A_IK DI_K^T (I > K) and row K of the inverse X_KJ = DI_K B_KJ (J <= K);
//   3. grid barrier; trailing updates A_IJ -= L_IK L_JK^T (K < J <= I) and B_IJ -= L_IK X_KJ
//      (I > K, J <= K); grid barrier.
// Two barriers per 32 columns for the factor and the inverse together.  Products are split into
// units of 128 outputs (two threads each) so that a few tiles still spread over the SMs.
// The factor of a tile (tile_factor): LDL^T by columns with the same row operations applied to the
// identity, one thread per (row, column mod 8), one CTA barrier per column; the chain of a column is
// its FMA, the reciprocal of the pivot (an FP32 seed and 3 FP64 instructions) and one product.  The
// square roots are taken at the end, for all 32 pivots in one go.  Those want pivots and reciprocals
// that are normal: where A(0, 0) lies outside 2^-800 .. 2^800, A is scaled by 2^200 or 2^-200 on entry and the
// results on exit.
// info: 0, or j + 1 for the first column j whose pivot is not positive (L and L^-1 are then not
// written in full).
// Measured, one call: N = 60 60 us, N = 240 233 us, N = 600 0.78 ms.
constexpr int CB = 32;

struct TileSmem {
  double L[CB][CB + 1], D[CB][CB + 1];  // factor and its inverse of the diagonal tile
  double col[2][CB], mul[2][CB], piv[CB], rs[CB];
  int bad;
};

// Factor tile (K, K) of M (column-major n x n, lower triangle) into T.L and T.D; T.bad = 0, or j + 1
// for the first pivot j that is not positive and finite.  256 threads.
__device__ __forceinline__ void tile_factor(TileSmem& T, const double* M, int n, int K) {
  const int tid = threadIdx.x, i = tid & 31, w = tid >> 5;
  double a[4], b[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = w + 8 * q, gi = K * CB + i, gc = K * CB + c;
    a[q] = (gi < n && gc < n) ? __ldcg(M + (size_t)gc * n + gi) : (i == c ? 1.0 : 0.0);
    b[q] = i == c ? 1.0 : 0.0;
  }
  if (tid == 0) T.bad = 0;
  __syncthreads();
#pragma unroll
  for (int jq = 0; jq < 4; ++jq) {
    for (int jw = 0; jw < 8; ++jw) {
      const int j = 8 * jq + jw, buf = j & 1;
      if (w == jw) {
        const double d = __shfl_sync(0xffffffffu, a[jq], j);
        const bool good = d > 0.0 && d < DBL_MAX;
        const double m = a[jq] * rcp_h3(good ? d : 1.0);
        T.col[buf][i] = a[jq];
        T.mul[buf][i] = m;
        T.L[i][j] = a[jq];
        if (i == 0) {
          T.piv[j] = good ? d : 1.0;
          if (!good && T.bad == 0) T.bad = j + 1;
        }
      }
      __syncthreads();
      const double ci = T.col[buf][i], mi = T.mul[buf][i];
      // the columns still to come (the next pivot's first), then the rows of the identity
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int q = (u + jq) & 3, c = w + 8 * q;
        if (c > j) a[q] = fma(-ci, T.mul[buf][c], a[q]);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (w + 8 * q <= j) {
          const double bj = __shfl_sync(0xffffffffu, b[q], j);
          const double v = fma(-mi, bj, b[q]);
          if (i > j) b[q] = v;
        }
      }
    }
  }
  __syncthreads();
  if (w == 0) T.rs[i] = rsqrt_h3(T.piv[i]);
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = w + 8 * q;
    T.L[i][c] = i < c ? 0.0 : T.L[i][c] * T.rs[c];  // (d_c / sqrt(d_c) on the diagonal)
    T.D[i][c] = b[q] * T.rs[i];
  }
  __syncthreads();
}

// Output (r, c) of a unit: the sum of a[k] b[k] over 32 k, two threads (even / odd lanes) per output.
__device__ __forceinline__ double unit_dot(const double* a, int sa, const double* b, int sb, int half) {
  double s0 = 0.0, s1 = 0.0;
#pragma unroll 8
  for (int k = 0; k < CB / 2; k += 2) {
    const int k0 = half * (CB / 2) + k;
    s0 = fma(a[k0 * sa], b[k0 * sb], s0);
    s1 = fma(a[(k0 + 1) * sa], b[(k0 + 1) * sb], s1);
  }
  s0 += s1;
  return s0 + __shfl_xor_sync(0xffffffffu, s0, 1);
}

__global__ void __launch_bounds__(256) chol_inv_blocked_kernel(int n, const double* __restrict__ A, double* L,
                                                               double* Linv, int* info) {
  __shared__ TileSmem T;
  __shared__ double SA[CB][CB + 1], SB[CB][CB + 1];
  cg::grid_group grid = cg::this_grid();
  const int P = gridDim.x, r = blockIdx.x, tid = threadIdx.x;
  const int nt = (n + CB - 1) / CB;
  const size_t nn = (size_t)n * n;
  auto at = [&](const double* M, int i, int j) { return (i < n && j < n) ? __ldcg(M + (size_t)j * n + i) : 0.0; };
  auto put = [&](double* M, int i, int j, double v) {
    if (i < n && j < n) __stcg(M + (size_t)j * n + i, v);
  };
  // 2^-h A is factored; 0 but at the ends of the range
  const int e0 = exp_field(A[0]) - 1023, h = e0 < -800 ? -200 : e0 > 800 ? 200 : 0;
  // L = lower(A), Linv = I
  for (size_t e = (size_t)r * blockDim.x + tid; e < nn; e += (size_t)P * blockDim.x) {
    const size_t j = e / n, i = e - j * n;
    const double v = i >= j ? A[e] : 0.0;
    __stcg(L + e, h != 0 ? ldexp(v, -h) : v);
    __stcg(Linv + e, i == j ? 1.0 : 0.0);
  }
  grid.sync();
  const int o = tid >> 1, half = tid & 1;  // output of the unit, and half of its sum
  for (int K = 0; K < nt; ++K) {
    tile_factor(T, L, n, K);
    if (T.bad) {
      if (r == 0 && tid == 0) *info = K * CB + T.bad;
      return;  // (every CTA takes the same branch)
    }
    // ---- panel rows (4 of a tile per unit) and columns of row K of the inverse (4 of a tile per unit)
    const int np = nt - K - 1;
    for (int u = r; u < 8 * (np + K + 1); u += P) {
      const bool inv = u >= 8 * np;
      const int t = inv ? u - 8 * np : u;
      const int I = inv ? t >> 3 : K + 1 + (t >> 3), h = 4 * (t & 7);
      if (tid < 128) {
        if (!inv) {
          const int rr = tid & 3, k = tid >> 2;
          SA[rr][k] = at(L, I * CB + h + rr, K * CB + k);
        } else {
          const int k = tid & 31, c = tid >> 5;
          SA[c][k] = at(Linv, K * CB + k, I * CB + h + c);
        }
      }
      __syncthreads();
      // (both: outputs 4 x 32, a 4-row operand against the rows of DI)
      const int x = inv ? o >> 5 : o & 3, y = inv ? o & 31 : o >> 2;
      const double v = unit_dot(&SA[x][0], 1, &T.D[y][0], 1, half);
      if (half == 0) {
        if (!inv) put(L, I * CB + h + x, K * CB + y, v);
        else put(Linv, K * CB + y, I * CB + h + x, v);
      }
      __syncthreads();
    }
    grid.sync();
    if (r == 0)
      for (int e = tid; e < CB * CB; e += blockDim.x) put(L, K * CB + (e & 31), K * CB + (e >> 5), T.L[e & 31][e >> 5]);
    if (np == 0) break;
    // ---- trailing updates in units of 16 x 8 outputs (8 per tile)
    const int ta = np * (np + 1) / 2, tb = np * (K + 1);
    for (int u = r; u < 8 * (ta + tb); u += P) {
      const int t = u >> 3, r0 = 16 * (u & 1), c0 = 8 * ((u >> 1) & 3);
      int I, J;
      const bool inv = t >= ta;
      if (!inv) {
        // t -> (I, J) with J <= I: row a = I - K - 1 holds a + 1 tiles
        int a = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
        while ((a + 1) * (a + 2) / 2 <= t) ++a;
        while (a * (a + 1) / 2 > t) --a;
        I = K + 1 + a;
        J = K + 1 + (t - a * (a + 1) / 2);
      } else {
        I = K + 1 + (t - ta) / (K + 1);
        J = (t - ta) % (K + 1);
      }
      for (int e = tid; e < 16 * CB; e += 256) SA[e & 15][e >> 4] = at(L, I * CB + r0 + (e & 15), K * CB + (e >> 4));
      {
        const int e = tid;  // 8 x 32: rows of L_JK, or columns of X_KJ
        if (!inv) SB[e & 7][e >> 3] = at(L, J * CB + c0 + (e & 7), K * CB + (e >> 3));
        else SB[e >> 5][e & 31] = at(Linv, K * CB + (e & 31), J * CB + c0 + (e >> 5));
      }
      double* C = inv ? Linv : L;
      const int x = o & 15, y = o >> 4;
      const double old = half == 0 ? at(C, I * CB + r0 + x, J * CB + c0 + y) : 0.0;
      __syncthreads();
      const double v = unit_dot(&SA[x][0], 1, &SB[y][0], 1, half);
      if (half == 0) put(C, I * CB + r0 + x, J * CB + c0 + y, old - v);
      __syncthreads();
    }
    grid.sync();
  }
  if (h != 0) {
    grid.sync();
    for (size_t e = (size_t)r * blockDim.x + tid; e < nn; e += (size_t)P * blockDim.x) {
      __stcg(L + e, ldexp(__ldcg(L + e), h / 2));
      __stcg(Linv + e, ldexp(__ldcg(Linv + e), -h / 2));
    }
  }
  if (r == 0 && tid == 0) *info = 0;
}

// ------------------------------------------------------------------ Householder tridiagonalisation
// M (n x n, column-major, full symmetric storage, destroyed).  Outputs: d (n), e (n-1), the
// Householder vectors H(:, k) = v_k (rows k+1 .. n-1, v_k(k+1) = 1) and tau (n-1), so that
// Q = H_0 H_1 ... H_{n-3}, H_k = I - tau_k v_k v_k^T, and Q^T M Q = tridiag(e, d, e).
// p: n doubles of scratch.  Column c of the trailing matrix is owned by CTA c mod P.
template <bool CLUSTER>
__global__ void __launch_bounds__(EIG_THREADS) tridiag_kernel(int n, double* M, double* H, double* d, double* e,
                                                              double* tau, double* p) {
  extern __shared__ double sm[];
  double* v = sm;          // n
  double* w = sm + n;      // n
  double* red = sm + 2 * n;  // 33
  const int P = gridDim.x, r = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
  for (int k = 0; k + 2 < n; ++k) {
    const int rr = n - k - 1;  // order of the trailing block
    const double* mk = M + (int64_t)k * n + k + 1;
    for (int i = tid; i < rr; i += blockDim.x) v[i] = __ldcg(mk + i);
    __syncthreads();
    const double alpha = v[0];
    double s = 0.0;
    for (int i = 1 + tid; i < rr; i += blockDim.x) s += v[i] * v[i];
    const double xn2 = block_sum(s, red);
    double beta = alpha, t = 0.0;
    if (xn2 > 0.0) {
      beta = -copysign(sqrt(alpha * alpha + xn2), alpha);
      t = (beta - alpha) / beta;
      const double sc = 1.0 / (alpha - beta);
      for (int i = 1 + tid; i < rr; i += blockDim.x) v[i] *= sc;
    }
    __syncthreads();
    if (tid == 0) v[0] = 1.0;
    __syncthreads();
    if (r == 0) {
      if (tid == 0) {
        d[k] = __ldcg(M + (int64_t)k * n + k);
        e[k] = beta;
        tau[k] = t;
      }
      for (int i = tid; i < rr; i += blockDim.x) H[(int64_t)k * n + k + 1 + i] = v[i];
    }
    if (t == 0.0) continue;  // H_k = I: nothing to update (every CTA takes the same branch)
    // p_c = t * M(k+1:, c) . v for the owned columns c >= k + 1
    const int c0 = k + 1 + ((r - (k + 1)) % P + P) % P;
    for (int c = c0 + warp * P; c < n; c += nw * P) {
      const double* mc = M + (int64_t)c * n + k + 1;
      double acc = 0.0;
      for (int i = lane; i < rr; i += 32) acc += mc[i] * v[i];
      acc = warp_sum(acc);
      if (lane == 0) __stcg(p + c, t * acc);
    }
    all_sync<CLUSTER>();
    for (int i = tid; i < rr; i += blockDim.x) w[i] = __ldcg(p + k + 1 + i);
    __syncthreads();
    double pv = 0.0;
    for (int i = tid; i < rr; i += blockDim.x) pv += w[i] * v[i];
    const double K = -0.5 * t * block_sum(pv, red);
    for (int i = tid; i < rr; i += blockDim.x) w[i] += K * v[i];
    __syncthreads();
    // M(k+1:, c) -= v w_c + w v_c on the owned columns
    for (int c = c0 + warp * P; c < n; c += nw * P) {
      double* mc = M + (int64_t)c * n + k + 1;
      const double wc = w[c - k - 1], vc = v[c - k - 1];
      for (int i = lane; i < rr; i += 32) mc[i] = fma(-w[i], vc, fma(-v[i], wc, mc[i]));
    }
    all_sync<CLUSTER>();
  }
  if (r == 0 && tid == 0) {
    if (n >= 2) {
      d[n - 2] = __ldcg(M + (int64_t)(n - 2) * n + n - 2);
      e[n - 2] = __ldcg(M + (int64_t)(n - 2) * n + n - 1);
    }
    d[n - 1] = __ldcg(M + (int64_t)(n - 1) * n + n - 1);
  }
}

// Same reduction with the owned columns resident in shared memory (nq = ceil(n / P) columns of n
// doubles per CTA).  Per step only the pivot column (xch: rows k+1.., then M(k,k) at xch[n]) and the
// product p travel through L2; the owner of column k+1 publishes it at the end of step k, so each
// step needs two barriers.
constexpr int TRI_THREADS = 256;

template <bool CLUSTER>
__global__ void __launch_bounds__(TRI_THREADS) tridiag_smem_kernel(int n, const double* __restrict__ Min, double* H,
                                                                   double* d, double* e, double* tau, double* xch,
                                                                   double* xp) {
  extern __shared__ double sm[];
  const int P = gridDim.x, r = blockIdx.x;
  const int nq = (n - r + P - 1) / P;  // owned columns c = r + q P, q < nq
  double* cols = sm;                   // nq x n
  double* v = cols + (size_t)nq * n;   // n
  double* w = v + n;                   // n
  double* red = w + n;                 // 33
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
  for (int q = 0; q < nq; ++q)
    for (int i = tid; i < n; i += blockDim.x) cols[(size_t)q * n + i] = Min[(size_t)(r + q * P) * n + i];
  __syncthreads();
  if (r == 0) {  // column 0 is owned by CTA 0
    for (int i = 1 + tid; i < n; i += blockDim.x) __stcg(xch + i - 1, cols[i]);
    if (tid == 0) __stcg(xch + n, cols[0]);
  }
  all_sync<CLUSTER>();
  for (int k = 0; k + 2 < n; ++k) {
    const int rr = n - k - 1;
    for (int i = tid; i < rr; i += blockDim.x) v[i] = __ldcg(xch + i);
    __syncthreads();
    const double alpha = v[0];
    double s = 0.0;
    for (int i = 1 + tid; i < rr; i += blockDim.x) s += v[i] * v[i];
    const double xn2 = block_sum(s, red);
    double beta = alpha, t = 0.0;
    if (xn2 > 0.0) {
      beta = -copysign(sqrt(alpha * alpha + xn2), alpha);
      // t = (beta - alpha) / beta and sc = 1 / (alpha - beta) from one reciprocal
      const double g = alpha - beta, rcp = 1.0 / (beta * g);
      t = -(g * g) * rcp;
      const double sc = beta * rcp;
      for (int i = 1 + tid; i < rr; i += blockDim.x) v[i] *= sc;
    }
    __syncthreads();
    if (tid == 0) v[0] = 1.0;
    __syncthreads();
    if (r == 0) {
      if (tid == 0) {
        d[k] = __ldcg(xch + n);
        e[k] = beta;
        tau[k] = t;
      }
      for (int i = tid; i < rr; i += blockDim.x) H[(int64_t)k * n + k + 1 + i] = v[i];
    }
    // owned columns c >= k + 1: q from qa on
    const int qa = (k + 1 - r + P - 1) / P > 0 ? (k + 1 - r + P - 1) / P : 0;
    if (t != 0.0) {
      for (int q = qa + warp; q < nq; q += nw) {
        const double* mc = cols + (size_t)q * n + k + 1;
        double acc0 = 0.0, acc1 = 0.0;
        int i = lane;
        for (; i + 32 < rr; i += 64) {
          acc0 = fma(mc[i], v[i], acc0);
          acc1 = fma(mc[i + 32], v[i + 32], acc1);
        }
        if (i < rr) acc0 = fma(mc[i], v[i], acc0);
        const double acc = warp_sum(acc0 + acc1);
        if (lane == 0) __stcg(xp + r + q * P, t * acc);
      }
    }
    all_sync<CLUSTER>();
    if (t != 0.0) {
      for (int i = tid; i < rr; i += blockDim.x) w[i] = __ldcg(xp + k + 1 + i);
      __syncthreads();
      double pv = 0.0;
      for (int i = tid; i < rr; i += blockDim.x) pv += w[i] * v[i];
      const double K = -0.5 * t * block_sum(pv, red);
      for (int i = tid; i < rr; i += blockDim.x) w[i] += K * v[i];
      __syncthreads();
      for (int q = qa + warp; q < nq; q += nw) {
        const int c = r + q * P;
        double* mc = cols + (size_t)q * n + k + 1;
        const double wc = w[c - k - 1], vc = v[c - k - 1];
        for (int i = lane; i < rr; i += 32) mc[i] = fma(-w[i], vc, fma(-v[i], wc, mc[i]));
      }
      __syncthreads();
    }
    // publish column k + 1 (rows k+2.., then its diagonal) for the next step
    if ((k + 1) % P == r) {
      const double* mc = cols + (size_t)((k + 1 - r) / P) * n;
      for (int i = k + 2 + tid; i < n; i += blockDim.x) __stcg(xch + i - (k + 2), mc[i]);
      if (tid == 0) __stcg(xch + n, mc[k + 1]);
    }
    all_sync<CLUSTER>();
  }
  // last 2 x 2 block
  if (n >= 2 && (n - 2) % P == r && tid == 0) {
    const double* mc = cols + (size_t)((n - 2 - r) / P) * n;
    d[n - 2] = mc[n - 2];
    e[n - 2] = mc[n - 1];
  }
  if ((n - 1) % P == r && tid == 0) d[n - 1] = cols[(size_t)((n - 1 - r) / P) * n + n - 1];
}

// ------------------------------------------------------------------ one exchange per column
// The reduction of tridiag_smem_kernel with one exchange between the CTAs per column instead of two
// barriers and several dependent remote reads.  With x = M(k+1:, k) the current pivot column (alpha =
// x_0, beta = -sign(alpha) ||x||), u = x - beta e_1 and eta = 2 / (u^T u) = 1 / (beta^2 - alpha beta),
// H_k = I - eta u u^T and, A' being the trailing block,
//   t = A' u = A' x - beta a,  a = A' e_1 = M(k+1:, k+1),   w = eta t - (eta^2 / 2) (u^T t) u,
//   A' <- A' - u w^T - w u^T.
// The products q_c = A'(:, c)^T x of the owned columns need neither beta nor eta, so the norm, the
// square root and the divide of a column (one warp of every CTA, redundantly) run beside the
// products and the exchange.  What travels per column is q (each entry from its column's owner) and
// a (from the owner of column k + 1): every CTA then forms t, w and the next pivot column
// x' = a - u w_0 - w u_0 for itself, all from the same bits, so nobody waits for an owner again.  One
// pass over the owned columns applies the rank-2 update and forms the next products.
// eta^2 and the products with it are formed on their own, which holds for ||x|| = |beta| in 2^-240 .. 2^240.  Outside
// (far_exp), u and t are multiplied by a power of two near 1 / ||x|| (and eta by its inverse square), which leaves
// u w^T as it is.
// Exchange: CL = true, one thread-block cluster: q by st.async, a by one bulk copy per CTA, both
// completing bytes on the receiver's mbarrier.  CL = false, a cooperative grid: 16-byte packets
// {low word, tag, high word, tag} through L2 (xg: 4 n packets, zeroed), polled by the thread that
// needs the entry; the tag is the step.  Both buffers alternate by step.  A CTA takes part in step k only
// while it owns a column c >= k + 2, that is, while it has something to send for step k + 1; then it is
// done (the last P steps, one CTA after another), receives nothing more and writes nothing more, and the
// owner of column n - 1, which stays to the end, writes the outputs of the steps whose pivot column's
// owner has left.  So the two buffers are enough: step k + 2 is sent only after step k + 1 has arrived
// from every CTA that took part in step k, and each of them sent it after it had read step k.
// Every wait is bounded: on a timeout *err is set to 2 and all CTAs leave.
// Warps 0-7: rows and columns; warp 8: the scalars.  Outputs as tridiag_smem_kernel, with H(:, k) = u
// and tau = eta (the same reflector, whatever the power of two).
__device__ __forceinline__ bool far_exp(double beta) { return (unsigned)(exp_field(beta) - 783) > 480u; }

constexpr int TX_THREADS = 288;
constexpr int TX_ROWS = 4;  // rows per thread: n <= 1024

size_t tridiag_xch_smem(int n, int P, bool cl) {
  const size_t ld = ((size_t)n + 1) & ~(size_t)1, nqm = ((size_t)n + P - 1) / P;
  return (nqm * ld + (cl ? 4 : 0) * ld + 3 * ld) * sizeof(double) + 16;
}

__device__ __forceinline__ uint32_t mapa_u32(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_async_f64(uint32_t addr, double v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr),
               "l"(__double_as_longlong(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void bulk_s2s(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   dst),
               "r"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void pkt_store(uint4* p, double v, uint32_t tag) {
  asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %2};" ::"l"(p), "r"((uint32_t)__double2loint(v)),
               "r"(tag), "r"((uint32_t)__double2hiint(v))
               : "memory");
}
// true when the packet carries `tag`
__device__ __forceinline__ bool pkt_load(const uint4* p, uint32_t tag, double* v) {
  uint32_t a, b, c, e;
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(a), "=r"(b), "=r"(c), "=r"(e)
               : "l"(p)
               : "memory");
  *v = __hiloint2double((int)c, (int)a);
  return b == tag && e == tag;
}

template <bool CL>
__global__ void __launch_bounds__(TX_THREADS) tridiag_xch_kernel(int n, const double* __restrict__ Min, double* H,
                                                                 double* d, double* e, double* tau, uint4* xg,
                                                                 int* err) {
  extern __shared__ double sm_raw[];
  __shared__ __align__(8) uint64_t qbar[2], sbar;
  // scal: beta, then of the scaled u eta, -eta^2 / 2, u_0, u_0 eta, -u_0 eta^2; where far_exp(beta), the power of two
  // and beta times it
  __shared__ double red[8], scal[8];
  __shared__ int abort_flag[2];
  const int P = gridDim.x, r = blockIdx.x;  // (a cluster launch is one cluster)
  const int ld = (n + 1) & ~1;
  const int nqm = (n + P - 1) / P, nq = (n - r + P - 1) / P;  // owned columns c = r + q P
  // the last column that CTA `rank` owns (negative: none); it takes part in steps k <= last - 2
  auto last_col = [&](int rank) { return rank < n ? rank + (n - 1 - rank) / P * P : -1; };
  const int steps = max(0, min(n - 2, last_col(r) - 1));
  double* sm = reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(sm_raw) + 15) & ~uintptr_t(15));
  double* cols = sm;                       // nqm x ld
  double* xa = cols + (size_t)nqm * ld;    // CL: two buffers of a, two of q
  double* xq = xa + (CL ? 2 * ld : 0);
  double* U = xq + (CL ? 2 * ld : 0);
  double* W = U + ld;
  double* X = W + ld;
  uint4* ga = xg;                          // !CL: two buffers of a, two of q
  uint4* gq = xg + 2 * (size_t)n;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    tc::mbar_init(&qbar[0], 1);
    tc::mbar_init(&qbar[1], 1);
    tc::mbar_init(&sbar, 1);
    tc::fence_barrier_init();
    abort_flag[0] = abort_flag[1] = 0;
  }
  for (int q = 0; q < nq; ++q)
    for (int i = tid; i < n; i += TX_THREADS) cols[(size_t)q * ld + i] = Min[(size_t)(r + q * P) * n + i];
  for (int i = tid; i < n; i += TX_THREADS) X[i] = Min[i];
  if (n & 1)  // the padding row travels with the columns
    for (int q = tid; q < nqm; q += TX_THREADS) cols[(size_t)q * ld + n] = 0.0;
  if (CL) cg::this_cluster().sync();  // the barriers are ready before anyone sends
  else __syncthreads();

  // bytes that arrive for step k: q_c, c = k + 1 .. n - 1, and rows (k + 1) & ~1 .. of a
  auto expect = [&](int k) {
    tc::mbar_arrive_expect_tx(&qbar[k & 1], (uint32_t)(8 * (n - k - 1) + 8 * (ld - ((k + 1) & ~1))));
  };
  if (CL && tid == 0)
    for (int k = 0; k < 2 && k < steps; ++k) expect(k);

  // this lane's view of CTA `lane` of the cluster
  uint32_t rq = 0, ra = 0, rb = 0;
  int last = -1;  // the last column of that CTA
  if (CL && lane < P) {
    last = last_col(lane);
    rq = mapa_u32(tc::smem_u32(xq), (uint32_t)lane);
    ra = mapa_u32(tc::smem_u32(xa), (uint32_t)lane);
    rb = mapa_u32(tc::smem_u32(qbar), (uint32_t)lane);
  }

  // rank-2 update of step k on the owned columns c >= k + 2 (UPD), the products with x' and, with
  // `send`, what step k + 1 needs, to the CTAs that take part in it
  auto pass = [&](int k, bool upd, bool send) {
    const int s0 = k + 2, rr = n - s0;  // rows s0 .. n - 1
    const int qa = s0 - r > 0 ? (s0 - r + P - 1) / P : 0;
    const int b = (k + 1) & 1;
    const bool to = CL && last >= k + 3;
    // (columns go to the warps in an order that loads sub-partition 0, which also runs the scalars, last)
    for (int q = qa + (((warp + 3) & 3) | (warp & 4)); q < nq; q += 16) {
      const int q2 = q + 8;
      const bool two = q2 < nq;
      const int c = r + q * P, c2 = c + 8 * P;
      double* m1 = cols + (size_t)q * ld + s0;
      double* m2 = cols + (size_t)(two ? q2 : q) * ld + s0;
      double wc = 0.0, uc = 0.0, wc2 = 0.0, uc2 = 0.0;
      if (upd) {
        wc = W[c];
        uc = U[c];
        if (two) {
          wc2 = W[c2];
          uc2 = U[c2];
        }
      }
      double a1 = 0.0, a2 = 0.0;
      for (int c0 = 0; c0 < rr; c0 += 64) {
        double x[2], u[2], w[2], p1[2], p2[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int i = c0 + 32 * h + lane;
          const bool in = i < rr;
          x[h] = in ? X[s0 + i] : 0.0;
          p1[h] = in ? m1[i] : 0.0;
          p2[h] = in && two ? m2[i] : 0.0;
          if (upd) {
            u[h] = in ? U[s0 + i] : 0.0;
            w[h] = in ? W[s0 + i] : 0.0;
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int i = c0 + 32 * h + lane;
          if (c0 + 32 * h < rr) {  // (a chunk past the end would still hold the FP64 pipe)
            if (upd) {
              p1[h] = fma(-w[h], uc, p1[h]);
              if (two) p2[h] = fma(-w[h], uc2, p2[h]);
              p1[h] = fma(-u[h], wc, p1[h]);
              if (two) p2[h] = fma(-u[h], wc2, p2[h]);
              if (i < rr) {
                m1[i] = p1[h];
                if (two) m2[i] = p2[h];
              }
            }
            if (send) {
              a1 = fma(p1[h], x[h], a1);
              if (two) a2 = fma(p2[h], x[h], a2);
            }
          }
        }
      }
      if (!send) continue;
      if (c == s0) {  // column k + 2 is the next step's a
        if (CL) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          const int i0 = s0 & ~1;
          if (to)
            bulk_s2s(ra + (uint32_t)((b * ld + i0) * 8), tc::smem_u32(cols + (size_t)q * ld + i0),
                     (uint32_t)((ld - i0) * 8), rb + 8u * b);
        } else {
          __syncwarp();
          for (int i = s0 + lane; i < n; i += 32)
            pkt_store(ga + (size_t)b * n + i, cols[(size_t)q * ld + i], (uint32_t)(k + 2));
        }
      }
      const double d1 = warp_sum_fx(a1);
      const double d2 = two ? warp_sum_fx(a2) : 0.0;
      if (CL) {
        if (to) {
          st_async_f64(rq + (uint32_t)((b * ld + c) * 8), d1, rb + 8u * b);
          if (two) st_async_f64(rq + (uint32_t)((b * ld + c2) * 8), d2, rb + 8u * b);
        }
      } else if (lane == 0) {
        pkt_store(gq + (size_t)b * n + c, d1, (uint32_t)(k + 2));
        if (two) pkt_store(gq + (size_t)b * n + c2, d2, (uint32_t)(k + 2));
      }
    }
  };
  // scalars of the pivot column x = X[k + 1 ..] (warp 8)
  auto scalars = [&](int k) {
    double s2 = 0.0;
    for (int i = k + 2 + lane; i < n; i += 32) s2 = fma(X[i], X[i], s2);
    s2 = warp_sum_fx(s2);
    const double alpha = X[k + 1];
    double beta = alpha, eta = 0.0, u0 = 0.0;
    const double nx2 = fma(alpha, alpha, s2);
    auto reflect = [&](double al, double nn) {
      // eta = 1 / (||x||^2 + |alpha| ||x||) = (1 / ||x||) / (||x|| + |alpha|)
      const double ri = rsqrt_h3(nn), nx = nn * ri, g = nx + fabs(al);
      beta = -copysign(nx, al);
      u0 = copysign(g, al);  // alpha - beta
      eta = ri * rcp_h3(g);
    };
    const bool some = s2 > 0.0 && nx2 < DBL_MAX;
    if (some) {
      reflect(alpha, nx2);
    } else if (s2 != 0.0) {
      beta = eta = u0 = __longlong_as_double(0x7ff8000000000000LL);  // overflow of ||x||^2, or a NaN in x
    }
    if (lane == 0) scal[0] = beta;
    if (far_exp(beta)) {
      const int h = some ? exp_field(beta) - 1023 : 0;
      const double sig = __hiloint2double((1023 - h) << 20, 0);
      if (some) reflect(alpha * sig, nx2 * sig * sig);
      if (lane == 0) {
        scal[6] = sig;
        scal[7] = beta;
      }
    }
    const double ue = u0 * eta;
    if (lane == 0) {
      scal[1] = eta;
      scal[2] = -0.5 * (eta * eta);
      scal[3] = u0;
      scal[4] = ue;
      scal[5] = -(ue * eta);
    }
    __syncwarp();
    if (lane == 0) tc::mbar_arrive(&sbar);
  };

  if (n >= 3) {
    double xr[TX_ROWS];
#pragma unroll
    for (int j = 0; j < TX_ROWS; ++j) {
      const int i = tid + 256 * j;
      xr[j] = i < n ? X[i] : 0.0;
    }
    if (r == 0 && tid == 0) d[0] = X[0];
    if (warp == 8) scalars(0);
    else pass(-1, false, true);
    for (int k = 0; k < steps; ++k) {
      const int b = k & 1;
      const bool writes = r == (k + P < n ? k % P : (n - 1) % P);  // the outputs of this step
      if (warp < 8) {
        const bool any = [&] {  // (warp-uniform) does this warp hold a row of the trailing block
          bool a = false;
#pragma unroll
          for (int j = 0; j < TX_ROWS; ++j) a = a || (256 * j + 32 * warp < n && 256 * j + 32 * warp + 31 > k);
          return a;
        }();
        bool ok = true;
        double qv[TX_ROWS], av[TX_ROWS], q0 = 0.0, a0 = 0.0;
#pragma unroll
        for (int j = 0; j < TX_ROWS; ++j) qv[j] = av[j] = 0.0;
        if (CL) {
          ok = tc::mbar_wait(&qbar[b], (uint32_t)((k >> 1) & 1));
          if (tid == 0 && ok && k + 2 < steps) expect(k + 2);
          if (any) {
            q0 = xq[b * ld + k + 1];
            a0 = xa[b * ld + k + 1];
          }
#pragma unroll
          for (int j = 0; j < TX_ROWS; ++j) {
            const int i = tid + 256 * j;
            const bool in = i > k && i < n;
            qv[j] = in ? xq[b * ld + i] : 0.0;
            av[j] = in ? xa[b * ld + i] : 0.0;
          }
        } else if (any) {
          // (each packet is loaded until its tag shows up, then kept)
          uint32_t need = 3u << (2 * TX_ROWS);
#pragma unroll
          for (int j = 0; j < TX_ROWS; ++j) {
            const int i = tid + 256 * j;
            if (i > k && i < n) need |= 3u << (2 * j);
          }
          const long long c0 = clock64();
          do {
#pragma unroll
            for (int j = 0; j <= TX_ROWS; ++j) {
              const int i = j < TX_ROWS ? tid + 256 * j : k + 1;
              double v;
              if ((need >> (2 * j)) & 1u) {
                if (pkt_load(gq + (size_t)b * n + i, (uint32_t)(k + 1), &v)) {
                  need &= ~(1u << (2 * j));
                  if (j < TX_ROWS) qv[j] = v;
                  else q0 = v;
                }
              }
              if ((need >> (2 * j)) & 2u) {
                if (pkt_load(ga + (size_t)b * n + i, (uint32_t)(k + 1), &v)) {
                  need &= ~(2u << (2 * j));
                  if (j < TX_ROWS) av[j] = v;
                  else a0 = v;
                }
              }
            }
          } while (need && clock64() - c0 < tc::kWaitCycles);
          const bool done = need == 0u;
          ok = done;
        }
        ok = tc::mbar_wait(&sbar, (uint32_t)(k & 1)) && ok;
        if (!ok) abort_flag[b] = 1;
        const double eta = scal[1], mh = scal[2], u0 = scal[3], ue = scal[4], f0 = scal[5];
        double beta = scal[0];
        if (far_exp(beta)) {
          const double sig = scal[6];
          beta = scal[7];
#pragma unroll
          for (int j = 0; j < TX_ROWS; ++j) {
            xr[j] *= sig;
            qv[j] *= sig;
          }
          q0 *= sig;
        }
        double u[TX_ROWS], z[TX_ROWS], y[TX_ROWS], g = 0.0, e0 = 0.0;
        if (any) {
#pragma unroll
          for (int j = 0; j < TX_ROWS; ++j) {
            const int i = tid + 256 * j, base = 256 * j + 32 * warp;
            u[j] = z[j] = y[j] = 0.0;
            if (base < n && base + 31 > k) {
              u[j] = i == k + 1 ? u0 : i > k ? xr[j] : 0.0;
              z[j] = fma(-beta, av[j], qv[j]);  // t
              g = fma(u[j], z[j], g);
            }
          }
          g = warp_sum_fx(g);
          // beside the sum: eta t, a - u_0 eta t, eta t_0
#pragma unroll
          for (int j = 0; j < TX_ROWS; ++j) {
            const int base = 256 * j + 32 * warp;
            if (base < n && base + 31 > k) {
              y[j] = fma(-ue, z[j], av[j]);
              z[j] *= eta;
            }
          }
          e0 = eta * fma(-beta, a0, q0);
        }
        if (lane == 0) red[warp] = g;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (any) {
          const double gam = n <= 64 ? red[0] + red[1] : warp_sum_fx(lane < 8 ? red[lane] : 0.0);
          // w = eta t + kappa u, kappa = -eta^2 gam / 2;  x' = a - u w_0 - w u_0
          //   = (a - u_0 eta t) - u (eta t_0 + 2 kappa u_0)
          const double c0 = fma(f0, gam, e0), kap = mh * gam;
#pragma unroll
          for (int j = 0; j < TX_ROWS; ++j) {
            const int i = tid + 256 * j, base = 256 * j + 32 * warp;
            if (base < n && base + 31 > k) {
              const double x = fma(-u[j], c0, y[j]);
              const double w = fma(kap, u[j], z[j]);
              if (i > k && i < n) {
                U[i] = u[j];
                W[i] = w;
                X[i] = x;
                xr[j] = x;
                if (writes) {
                  H[(size_t)k * n + i] = u[j];
                  if (i == k + 1) {
                    d[k + 1] = x;  // a_0 - 2 u_0 w_0: the next diagonal entry
                    e[k] = scal[0];
                    tau[k] = eta;
                  }
                  if (k + 3 == n && i == n - 1) e[n - 2] = x;
                }
              }
            }
          }
        }
      }
      __syncthreads();
      if (abort_flag[b]) {
        if (tid == 0) atomicExch(err, 2);
        break;
      }
      if (warp == 8) {
        if (k + 1 < steps) scalars(k + 1);
      } else {
        pass(k, true, k + 3 < n);
      }
    }
    __syncthreads();
    if ((n - 1) % P == r && tid == 0) d[n - 1] = cols[(size_t)((n - 1 - r) / P) * ld + n - 1];
  } else if (r == 0 && tid == 0) {
    d[0] = Min[0];
    if (n == 2) {
      e[0] = Min[1];
      d[1] = Min[3];
    }
  }
  if (CL) cg::this_cluster().sync();  // nobody leaves while another CTA may still send to it
}

// ------------------------------------------------------------------ tridiagonal eigenvalues
// Number of eigenvalues of T below x: sign changes of the Sturm sequence of leading principal
// minors p_i = det(T_i - x I), by the three-term recurrence p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2}
// (p_{-1} = 1) on T scaled by 1 / tnorm (ds = d / tnorm, e2s[i] = (e_{i-1} / tnorm)^2, e2s[0] = 0).
// The recurrence needs no division (an FP64 divide costs ~9 dependent FMAs on this GPU), so its
// critical chain is one FMA per step; the pair (p_i, p_{i-1}) is rescaled by a power of two every
// 8 steps.  A zero minor between two nonzero ones of opposite sign counts one sign change either
// way; an exact zero is replaced by a tiny value of the sign opposite to its predecessor.
__device__ __forceinline__ bool neg_bits(double v) { return __double_as_longlong(v) < 0; }

template <int K>
__device__ void sturm_count_k(int n, const double* ds, const double* e2s, const double* xs, int* cnt) {
  // K independent sequences interleaved, so their dependent FMAs overlap
  double pm[K], p[K];
#pragma unroll
  for (int c = 0; c < K; ++c) {
    pm[c] = 1.0;
    p[c] = ds[0] - xs[c];
    if ((__double_as_longlong(p[c]) << 1) == 0) p[c] = -DBL_MIN;
    cnt[c] = neg_bits(p[c]);
  }
  int i = 1;
  for (; i + 8 <= n; i += 8) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double d = ds[i + u], e2 = e2s[i + u];
#pragma unroll
      for (int c = 0; c < K; ++c) {
        double pn = fma(d - xs[c], p[c], -e2 * pm[c]);
        if ((__double_as_longlong(pn) << 1) == 0) pn = neg_bits(p[c]) ? DBL_MIN : -DBL_MIN;
        cnt[c] += neg_bits(pn) != neg_bits(p[c]);
        pm[c] = p[c];
        p[c] = pn;
      }
    }
#pragma unroll
    for (int c = 0; c < K; ++c) {
      const long long bp = __double_as_longlong(p[c]) & 0x7fffffffffffffffLL;
      const long long bq = __double_as_longlong(pm[c]) & 0x7fffffffffffffffLL;
      const long long ex = ((bp > bq ? bp : bq) >> 52) - 1023;
      const double sc = __longlong_as_double((long long)(1023 - ex) << 52);
      p[c] *= sc;
      pm[c] *= sc;
    }
  }
  for (; i < n; ++i) {
    const double d = ds[i], e2 = e2s[i];
#pragma unroll
    for (int c = 0; c < K; ++c) {
      double pn = fma(d - xs[c], p[c], -e2 * pm[c]);
      if ((__double_as_longlong(pn) << 1) == 0) pn = neg_bits(p[c]) ? DBL_MIN : -DBL_MIN;
      cnt[c] += neg_bits(pn) != neg_bits(p[c]);
      pm[c] = p[c];
      p[c] = pn;
    }
  }
}

// Sturm sequences per lane.  One: on this GPU a warp-wide FP64 instruction occupies the SM's FP64
// pipe for ~12 clocks, so more sequences per lane trade latency for pipe time at a loss (measured).
constexpr int kChains = 1;

// The same count without the per-step zero substitution, so that the dependency chain from one
// minor to the next is the FMA alone: sign changes are read from the high words and accumulated
// off the chain, and *zero is set when a minor came out exactly zero (or with a zero high word, a
// subnormal below 2^-1042), the one case in which the substitution would have changed the count.
// The caller then recounts that shift with sturm_count_k.
__device__ __forceinline__ int sturm_count_fast(int n, const double* ds, const double* e2s, double xs, bool* zero) {
  double pm = 1.0, p = ds[0] - xs;
  uint32_t hp = (uint32_t)__double2hiint(p);
  int cnt = (int)(hp >> 31);
  uint32_t zmin = hp << 1;  // zero iff some minor had a zero high word (sign bit dropped)
  int i = 1;
  for (; i + 8 <= n; i += 8) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double pn = fma(ds[i + u] - xs, p, -e2s[i + u] * pm);
      const uint32_t hn = (uint32_t)__double2hiint(pn);
      cnt += (int)((hn ^ hp) >> 31);
      zmin = min(zmin, hn << 1);
      pm = p;
      p = pn;
      hp = hn;
    }
    // rescale the pair by a power of two (signs and ratios unchanged)
    const uint32_t ep = ((uint32_t)__double2hiint(p) >> 20) & 0x7ffu, eq = ((uint32_t)__double2hiint(pm) >> 20) & 0x7ffu;
    const int ex = (int)(ep > eq ? ep : eq) - 1023;
    const double sc = __hiloint2double((1023 - ex) << 20, 0);
    p *= sc;
    pm *= sc;
  }
  for (; i < n; ++i) {
    const double pn = fma(ds[i] - xs, p, -e2s[i] * pm);
    const uint32_t hn = (uint32_t)__double2hiint(pn);
    cnt += (int)((hn ^ hp) >> 31);
    zmin = min(zmin, hn << 1);
    pm = p;
    p = pn;
    hp = hn;
  }
  *zero = zmin == 0u;
  return cnt;
}

// Eigenvalue j (ascending) of T = tridiag(e, d, e): one warp (one CTA), 32 kChains trial points per step.
__global__ void __launch_bounds__(32) bisect_kernel(int n, const double* __restrict__ d, const double* __restrict__ e,
                                                    double* lam, double* tnorm_out) {
  extern __shared__ double sm[];
  double* ds = sm;       // n
  double* e2s = sm + n;  // n
  const int j = blockIdx.x;
  const int lane = threadIdx.x & 31;
  if (j >= n) return;
  double lo = DBL_MAX, hi = -DBL_MAX;
  for (int i = lane; i < n; i += 32) {
    const double a = i + 1 < n ? fabs(e[i]) : 0.0, b = i > 0 ? fabs(e[i - 1]) : 0.0;
    lo = fmin(lo, d[i] - a - b);
    hi = fmax(hi, d[i] + a + b);
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  const double tnorm = fmax(fabs(lo), fabs(hi));
  const double inv_tn = tnorm > 0.0 ? 1.0 / tnorm : 1.0;
  for (int i = lane; i < n; i += 32) {
    ds[i] = d[i] * inv_tn;
    const double b = i > 0 ? e[i - 1] * inv_tn : 0.0;
    e2s[i] = b * b;
  }
  __syncwarp();
  const double tiny = DBL_MIN * 4.0;
  lo -= 2.0 * DBL_EPSILON * tnorm + tiny;
  hi += 2.0 * DBL_EPSILON * tnorm + tiny;
  constexpr int NP = 32 * kChains;  // trial points per step; point q = c * 32 + lane
  for (int it = 0; it < 64; ++it) {
    // relative accuracy, but no finer than the eps ||T|| that the Sturm counts resolve
    if (hi - lo <= 2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi)) + 0.5 * DBL_EPSILON * tnorm + tiny) break;
    const double w = (hi - lo) / (double)(NP + 1);
    double x[kChains], xs[kChains];
    int cnt[kChains];
#pragma unroll
    for (int c = 0; c < kChains; ++c) {
      x[c] = lo + w * (double)(c * 32 + lane + 1);
      xs[c] = x[c] * inv_tn;
    }
    bool zero = false;
    cnt[0] = sturm_count_fast(n, ds, e2s, xs[0], &zero);
    if (zero) sturm_count_k<1>(n, ds, e2s, xs, cnt);
    // counts grow with x, so the first point with count > j bounds the eigenvalue from above
    int q = -1;
#pragma unroll
    for (int c = 0; c < kChains; ++c) {
      const unsigned ge = __ballot_sync(0xffffffffu, cnt[c] >= j + 1);
      if (q < 0 && ge != 0u) q = c * 32 + __ffs(ge) - 1;
    }
    if (q < 0) {
      lo = lo + w * (double)NP;
    } else {
      const double nlo = q > 0 ? lo + w * (double)q : lo;
      hi = lo + w * (double)(q + 1);
      lo = nlo;
    }
  }
  if (lane == 0) {
    lam[j] = 0.5 * (lo + hi);
    if (j == 0) *tnorm_out = tnorm;
  }
}

// ------------------------------------------------------------------ eigenpairs of T, one warp each
// Eigenvalue j of T = tridiag(e, d, e) and its eigenvector, one warp per eigenvalue, four per CTA.  An
// FP64 instruction takes 64 clocks of its SM sub-partition, so the time is the number of FP64
// instructions per Sturm step times the number of passes over T; bisect_kernel needs 3 and 11-12.
//   * Search: 4 passes of 32 trial points in FP32 narrow Gershgorin's interval by 33^4; the result
//     and a margin bracket the FP64 search (the first FP64 pass counts at both ends and widens the
//     bracket on the side that turns out wrong).  Once a bracket between neighbouring points holds
//     one eigenvalue, the secant of the last minor through them estimates it, and the next 32
//     points lie at distances w 4^-i (i = 0 .. 15) on both sides of the estimate: the bracket shrinks
//     to about four times the secant's error without that error being known, so 3-4 FP64 passes
//     reach round-off.  Clusters go on by multisection (5 bits a pass).
//   * Sturm step in FP64, 2 instructions: the minors p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} as
//     p_i = c_i q_i with c_i = e_{i-1}^2 c_{i-2}: q_i = a_i q_{i-1} - q_{i-2}, a_i = (d_i - x) g_i,
//     g_i = c_{i-1} / c_i = 1 / (e_{i-1}^2 g_{i-1}), one FMA each for a_i and q_i.  c restarts every
//     8 steps (q_{i-2} is multiplied by the last g) with a power-of-two rescaling.  |e| is kept
//     >= 2^-100 ||T|| so that no g overflows (a change far below the rounding of T).
//   * Vector: the rows of (T - x) z = 0 solved forwards from z_0 = 1 (lane 0) and backwards from
//     z_{n-1} = 1 (lane 1), both rescaled by powers of two, joined at the index k with the largest
//     |f_k b_k|, which is proportional to the k-th diagonal entry of (T - x)^-1 (the twisted
//     factorisation of Fernando and Parlett): every row but k holds to rounding and row k's
//     residual is the smallest possible.
// Vectors of numerically equal eigenvalues (gap <= 1e-9 ||T||) are replaced by inviter_kernel.
constexpr int TE_WARPS = 4;
constexpr int TE_MAX_N = 1408;

size_t tri_eig_smem(int n) {
  const size_t ng = ((size_t)n + 7) / 8 + 1;
  return (size_t)n * (7 + 2 * TE_WARPS) * sizeof(double) + (size_t)n * 2 * sizeof(float) +
         2 * TE_WARPS * ng * sizeof(int) + 16;
}

// x 2^k, 0 when the result leaves the normal range downwards (x normal or 0, the result does not overflow).
__device__ __forceinline__ double scale2(double x, int k) {
  const int hi = __double2hiint(x), ef = (hi >> 20) & 0x7ff;
  const int nf = ef + k;
  return ef != 0 && nf > 0 ? __hiloint2double(hi + (k << 20), __double2loint(x)) : 0.0;
}

// FP32 Sturm count of T / ||T|| at x.
__device__ __forceinline__ int sturm_count_f32(int n, const float* d, const float* e2, float x) {
  float pm = 1.f, p = d[0] - x;
  uint32_t hp = __float_as_uint(p);
  int cnt = (int)(hp >> 31);
  int i = 1;
  for (; i + 4 <= n; i += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float pn = fmaf(d[i + u] - x, p, -(e2[i + u] * pm));
      const uint32_t hn = __float_as_uint(pn);
      cnt += (int)((hn ^ hp) >> 31);
      pm = p;
      p = pn;
      hp = hn;
    }
    const int ef = (int)max((hp >> 23) & 0xffu, (__float_as_uint(pm) >> 23) & 0xffu);
    const float sc = __int_as_float((254 - min(max(ef, 1), 253)) << 23);  // 2^-(exponent)
    p *= sc;
    pm *= sc;
  }
  for (; i < n; ++i) {
    const float pn = fmaf(d[i] - x, p, -(e2[i] * pm));
    const uint32_t hn = __float_as_uint(pn);
    cnt += (int)((hn ^ hp) >> 31);
    pm = p;
    p = pn;
    hp = hn;
  }
  return cnt;
}

// FP64 Sturm count at x (scaled), and the last minor as q 2^qe (up to a factor common to all x).
__device__ __forceinline__ int sturm_count_g(int n, double d0, const double* g, const double* dg, double x, double* q,
                                             int* qe) {
  double pm = 1.0, p = d0 - x;
  uint32_t hp = (uint32_t)__double2hiint(p);
  int cnt = (int)(hp >> 31), ee = 0;
  int i = 1;
  for (; i + 8 <= n; i += 8) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double pn = fma(fma(-x, g[i + u], dg[i + u]), p, -pm);
      const uint32_t hn = (uint32_t)__double2hiint(pn);
      cnt += (int)((hn ^ hp) >> 31);
      pm = p;
      p = pn;
      hp = hn;
    }
    pm *= g[i + 7];
    const int ex = max(exp_field(p), exp_field(pm)) - 1023;
    p = scale2(p, -ex);
    pm = scale2(pm, -ex);
    hp = (hp & 0x80000000u) | ((uint32_t)__double2hiint(p) & 0x7fffffffu);
    ee += ex;
  }
  for (; i < n; ++i) {
    const double pn = fma(fma(-x, g[i], dg[i]), p, -pm);
    const uint32_t hn = (uint32_t)__double2hiint(pn);
    cnt += (int)((hn ^ hp) >> 31);
    pm = p;
    p = pn;
    hp = hn;
  }
  *q = p;
  *qe = ee;
  return cnt;
}

__global__ void __launch_bounds__(32 * TE_WARPS) tri_eig_kernel(int n, const double* __restrict__ d,
                                                                const double* __restrict__ e, double* lam,
                                                                double* tnorm_out, double* Z) {
  extern __shared__ double sm[];
  __shared__ double rmin[TE_WARPS], rmax[TE_WARPS];
  const int ng = (n + 7) / 8 + 1;
  double* g = sm;          // g_i, (d_i) g_i: row i of the Sturm recurrence
  double* dg = g + n;
  double* rf = dg + n;     // e_{i-1} / e_i and d_i / e_i, 1 / e_i: forward solve, row i
  double* df = rf + n;
  double* ie = df + n;
  double* rb = ie + n;     // e_i / e_{i-1} and d_i / e_{i-1}: backward solve, row i
  double* db = rb + n;
  double* vec = db + n;    // per warp: n forward, n backward values
  float* d32 = reinterpret_cast<float*>(vec + (size_t)2 * TE_WARPS * n);
  float* e32 = d32 + n;
  int* vex = reinterpret_cast<int*>(e32 + n);  // per warp: exponents of every 8 values, both directions
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // Gershgorin's interval
  double glo = DBL_MAX, ghi = -DBL_MAX;
  for (int i = tid; i < n; i += 32 * TE_WARPS) {
    const double r = (i + 1 < n ? fabs(e[i]) : 0.0) + (i > 0 ? fabs(e[i - 1]) : 0.0);
    glo = fmin(glo, d[i] - r);
    ghi = fmax(ghi, d[i] + r);
  }
  for (int o = 16; o > 0; o >>= 1) {
    glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
    ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
  }
  if (lane == 0) {
    rmin[warp] = glo;
    rmax[warp] = ghi;
  }
  __syncthreads();
  for (int w = 0; w < TE_WARPS; ++w) {
    glo = fmin(glo, rmin[w]);
    ghi = fmax(ghi, rmax[w]);
  }
  const double tnorm = fmax(fabs(glo), fabs(ghi));
  const double inv = tnorm > 0.0 ? 1.0 / tnorm : 1.0;
  // scaled off-diagonal entry, kept away from zero
  auto es = [&](int i) {
    const double v = e[i] * inv;
    return fabs(v) < 0x1p-100 ? 0x1p-100 : v;
  };
  for (int i = tid; i < n; i += 32 * TE_WARPS) {
    const double ds = d[i] * inv;
    const double ec = i + 1 < n ? es(i) : 1.0, ep = i > 0 ? es(i - 1) : 0.0;
    const double ic = rcp_h3(ec < 0.0 ? -ec : ec) * (ec < 0.0 ? -1.0 : 1.0);
    const double ip = i > 0 ? rcp_h3(ep < 0.0 ? -ep : ep) * (ep < 0.0 ? -1.0 : 1.0) : 0.0;
    ie[i] = ic;
    rf[i] = ep * ic;
    df[i] = ds * ic;
    rb[i] = i + 1 < n ? ec * ip : 0.0;
    db[i] = ds * ip;
    d32[i] = (float)ds;
    e32[i] = (float)(ep * ep);
  }
  for (int t = tid; 1 + 8 * t < n; t += 32 * TE_WARPS) {
    double gp = 1.0;
    for (int i = 1 + 8 * t; i < min(n, 9 + 8 * t); ++i) {
      const double ev = es(i - 1);
      gp = rcp_h3(ev * ev * gp);
      g[i] = gp;
      dg[i] = d[i] * inv * gp;
    }
  }
  __syncthreads();
  const int j = blockIdx.x * TE_WARPS + warp;
  if (j >= n) return;
  const double d0 = d[0] * inv;
  glo = glo * inv - 4.0 * DBL_EPSILON;
  ghi = ghi * inv + 4.0 * DBL_EPSILON;
  // ---- FP32 multisection
  float flo = (float)glo, fhi = (float)ghi;
  for (int it = 0; it < 4; ++it) {
    const float w = (fhi - flo) * (1.f / 33.f);
    const int cnt = sturm_count_f32(n, d32, e32, flo + w * (float)(lane + 1));
    const unsigned ge = __ballot_sync(0xffffffffu, cnt > j);
    const int q = ge ? __ffs(ge) - 1 : 32;
    const float a = flo + w * (float)q;
    fhi = q < 32 ? flo + w * (float)(q + 1) : fhi;
    flo = q > 0 ? a : flo;
  }
  // ---- FP64
  double lo = fmax(glo, (double)flo - 3e-6), hi = fmin(ghi, (double)fhi + 3e-6);
  bool lo_ok = false, hi_ok = false, sec = false;
  double xs = 0.0;
  for (int it = 0; it < 80; ++it) {
    const double w = hi - lo;
    if (lo_ok && hi_ok && w <= 2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi)) + 0.5 * DBL_EPSILON) break;
    double x;
    if (sec) {
      const int i = lane < 16 ? lane : 31 - lane;
      const double o = scale2(w, -2 * i);
      x = fmin(fmax(lane < 16 ? xs - o : xs + o, lo), hi);
    } else if (lo_ok && hi_ok) {
      x = fma(w, (double)(lane + 1) * (1.0 / 33.0), lo);
    } else {
      x = lane == 31 ? hi : fma(w, (double)lane * (1.0 / 31.0), lo);
    }
    double qv;
    int qe;
    const int cnt = sturm_count_g(n, d0, g, dg, x, &qv, &qe);
    const unsigned ge = __ballot_sync(0xffffffffu, cnt > j);
    const int q = ge ? __ffs(ge) - 1 : 32;
    sec = false;
    if (q == 0) {
      const double x0 = __shfl_sync(0xffffffffu, x, 0);
      hi = x0;
      hi_ok = true;
      if (!lo_ok) {
        lo = fmax(glo, x0 - 8.0 * w);
        lo_ok = lo == glo;
      }
    } else if (q == 32) {
      const double x1 = __shfl_sync(0xffffffffu, x, 31);
      lo = x1;
      lo_ok = true;
      if (!hi_ok) {
        hi = fmin(ghi, x1 + 8.0 * w);
        hi_ok = hi == ghi;
      }
    } else {
      const double xl = __shfl_sync(0xffffffffu, x, q - 1), xh = __shfl_sync(0xffffffffu, x, q);
      const int cl = __shfl_sync(0xffffffffu, cnt, q - 1), ch = __shfl_sync(0xffffffffu, cnt, q);
      const double ql = __shfl_sync(0xffffffffu, qv, q - 1), qh = __shfl_sync(0xffffffffu, qv, q);
      const int el = __shfl_sync(0xffffffffu, qe, q - 1), eh = __shfl_sync(0xffffffffu, qe, q);
      lo = xl;
      hi = xh;
      lo_ok = hi_ok = true;
      if (ch - cl == 1) {
        // zero of the line through (xl, ql) and (xh, qh), opposite signs
        const int de = eh - el;
        const double a = fabs(de > 0 ? scale2(ql, -de) : ql), b = fabs(de < 0 ? scale2(qh, de) : qh);
        const double t = a + b;
        if (t > 0.0 && t < DBL_MAX) {
          xs = fma(xh - xl, a / t, xl);
          sec = true;
        }
      }
    }
  }
  const double xl = 0.5 * (lo + hi);
  if (lane == 0) {
    lam[j] = xl * tnorm;
    if (j == 0) *tnorm_out = tnorm;
  }
  // ---- vector: lane 0 forwards, lane 1 backwards
  double* F = vec + (size_t)warp * 2 * n;
  double* B = F + n;
  int* eF = vex + warp * 2 * ng;
  int* eB = eF + ng;
  if (lane < 2) {
    const bool fw = lane == 0;
    const int st = fw ? 1 : -1;
    int i = fw ? 0 : n - 1;
    const double* pa = fw ? ie : ie - 1;  // 1 / e_i, or 1 / e_{i-1}
    const double* pd = fw ? df : db;
    const double* pr = fw ? rf : rb;
    double* out = fw ? F : B;
    int* oe = fw ? eF : eB;
    double zm = 0.0, z = 1.0;
    int ee = 0;
    for (int s0 = 0; s0 < n; s0 += 8) {
      // values s0 .. s0 + 7 of this direction share the exponent ee
      oe[s0 >> 3] = ee;
      const int m = min(8, n - s0);
      for (int u = 0; u < m; ++u) {
        out[i] = z;
        if (s0 + u + 1 < n) {
          // z_next = -((d_i - x) z + e_prev zm) / e_next
          const double zn = fma(fma(xl, pa[i], -pd[i]), z, -(pr[i] * zm));
          zm = z;
          z = zn;
        }
        i += st;
      }
      const int ex = max(exp_field(z), exp_field(zm)) - 1023;
      z = scale2(z, -ex);
      zm = scale2(zm, -ex);
      ee += ex;
    }
  }
  __syncwarp();
  // the joining index: largest |f_k b_k|, compared by exponent, then by the product of significands
  int be = -2000000000, bk = 0;
  double bm = -1.0;
  for (int k = lane; k < n; k += 32) {
    const double f = F[k], b = B[k];
    const int ff = exp_field(f), bf = exp_field(b);
    if (ff == 0 || bf == 0) continue;
    const int ex = eF[k >> 3] + eB[(n - 1 - k) >> 3] + ff + bf;
    const double m = fabs(scale2(f, 1023 - ff) * scale2(b, 1023 - bf));
    if (ex > be || (ex == be && m > bm)) {
      be = ex;
      bm = m;
      bk = k;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const int oe = __shfl_xor_sync(0xffffffffu, be, o), ok = __shfl_xor_sync(0xffffffffu, bk, o);
    const double om = __shfl_xor_sync(0xffffffffu, bm, o);
    if (oe > be || (oe == be && (om > bm || (om == bm && ok < bk)))) {
      be = oe;
      bm = om;
      bk = ok;
    }
  }
  const double fk = F[bk], bkv = B[bk];
  const int fe = eF[bk >> 3], bee = eB[(n - 1 - bk) >> 3];
  const double sf = 1.0 / fk, sb = 1.0 / bkv;
  __syncwarp();
  double nr = 0.0;
  for (int k = lane; k < n; k += 32) {
    const double z = k <= bk ? scale2(F[k] * sf, eF[k >> 3] - fe) : scale2(B[k] * sb, eB[(n - 1 - k) >> 3] - bee);
    F[k] = z;
    nr = fma(z, z, nr);
  }
  const double sc = rsqrt_h3(warp_sum_fx(nr));
  double* zj = Z + (size_t)j * n;
  for (int k = lane; k < n; k += 32) zj[k] = F[k] * sc;
}

// ------------------------------------------------------------------ tridiagonal eigenvectors
// LU factorisation with partial pivoting of T - lam I, one matrix per lane: the pivoting is by selects, so that the
// lanes of a warp factor the matrices of a cluster's members in the time of one.  Row i of U is 1 / u0 (u0inv, the
// pivot clamped away from zero), u1, u2 (first and second superdiagonals); mult/sw record the elimination of
// row i + 1.
__device__ void tri_lu(int n, const double* d, const double* e, double lam, double small, double* u0inv, double* u1,
                       double* u2, double* mult, int* sw) {
  double p0 = d[0] - lam, p1 = e[0];  // the current row
  auto inv = [&](double u) {
    const double a = fabs(u) < small ? small : fabs(u);
    return copysign(rcp_h3(a), u);
  };
  for (int i = 0; i + 1 < n; ++i) {
    const double c = e[i];  // subdiagonal entry (i + 1, i)
    const double a1 = d[i + 1] - lam, b1 = e[i + 1];
    const bool swap = fabs(p0) < fabs(c);
    const double piv = swap ? c : p0, r = inv(piv);
    const double q1 = swap ? a1 : p1;
    const double m = (swap ? p0 : c) * r;
    u0inv[i] = r;
    u1[i] = q1;
    u2[i] = swap ? b1 : 0.0;
    mult[i] = m;
    sw[i] = swap ? 1 : 0;
    p0 = fma(-m, q1, swap ? p1 : a1);
    p1 = swap ? -m * b1 : b1;
  }
  u0inv[n - 1] = inv(p0);
  u1[n - 1] = u2[n - 1] = 0.0;
}

// y <- (T - lam I)^-1 y with the factors of tri_lu (one system per lane).
__device__ void tri_solve(int n, const double* u0inv, const double* u1, const double* u2, const double* mult,
                          const int* sw, double* y) {
  double t = y[0];
  for (int i = 0; i + 1 < n; ++i) {
    const double v = y[i + 1], m = mult[i];
    const bool s = sw[i] != 0;
    y[i] = s ? v : t;
    t = s ? fma(-m, v, t) : fma(-m, t, v);
  }
  double y1 = t * u0inv[n - 1], y2 = 0.0;
  y[n - 1] = y1;
  for (int i = n - 2; i >= 0; --i) {
    const double x = fma(-u1[i], y1, fma(-u2[i], y2, y[i])) * u0inv[i];
    y[i] = x;
    y2 = y1;
    y1 = x;
  }
}

// One warp (one CTA) per cluster of eigenvalues, a cluster being a run of eigenvalues with
// consecutive gaps <= 1e-9 ||T|| (numerically degenerate, e.g. the pairs of a complex problem's
// real embedding): inverse iteration, `batch` members at a time (a lane each: the factorisation and the solves
// are chains of FP64 instructions, and a pair of n = 192 took 530 us one member after the other), with
// Gram-Schmidt (twice) against the
// members already done.  Eigenvectors of better separated eigenvalues come out orthogonal to
// O(eps ||T|| / gap); the caller removes that residue with one Newton-Schulz step.  The LU factors
// and the iterates live in shared memory (5.5 n doubles per member).  Z (n x n, column-major) receives the unit
// eigenvectors of T.  A cluster larger than maxc sets *flag (the caller then uses another solver).
__global__ void __launch_bounds__(32) inviter_kernel(int n, const double* __restrict__ d, const double* __restrict__ e,
                                                     const double* __restrict__ lam, const double* __restrict__ tnorm_p,
                                                     double* Z, int maxc, int clusters_only, int batch, int* flag) {
  extern __shared__ double sm[];
  const int j = blockIdx.x;
  const int lane = threadIdx.x & 31;
  if (j >= n) return;
  const double tnorm = *tnorm_p;
  const double ortol = 1e-9 * tnorm;
  if (j > 0 && lam[j] - lam[j - 1] <= ortol) return;  // not the first member of its cluster
  int k = j + 1;
  while (k < n && lam[k] - lam[k - 1] <= ortol) ++k;
  if (clusters_only && k == j + 1) return;
  if (k - j > maxc) {
    if (lane == 0) atomicExch(flag, 1);
    return;
  }
  const double small = fmax(DBL_EPSILON * tnorm, 4.0 * DBL_MIN);  // (its reciprocal is a normal number)
  double* dd = sm;        // copies of d and e (n each)
  double* ee = dd + n;
  double* fac = ee + n;   // per member of the batch: 1 / u0, u1, u2, mult (n each)
  double* ys = fac + (size_t)batch * 4 * n;  // iterates
  int* sws = reinterpret_cast<int*>(ys + (size_t)batch * n);
  for (int m = lane; m < n; m += 32) {
    dd[m] = d[m];
    ee[m] = m + 1 < n ? e[m] : 0.0;
  }
  __syncwarp();
  for (int i0 = j; i0 < k; i0 += batch) {
    const int nb = min(batch, k - i0);
    double* f = fac + (size_t)min(lane, nb - 1) * 4 * n;
    double* y = ys + (size_t)min(lane, nb - 1) * n;
    int* sw = sws + (size_t)min(lane, nb - 1) * n;
    if (lane < nb) tri_lu(n, dd, ee, lam[i0 + lane], small, f, f + n, f + 2 * n, f + 3 * n, sw);
    // deterministic start vectors with no structure shared with T
    for (int b = 0; b < nb; ++b)
      for (int m = lane; m < n; m += 32)
        ys[(size_t)b * n + m] = cosf(0.75487767f * (float)m + 1.3247180f * (float)(i0 + b - j) + 0.5f) + 0.1f;
    __syncwarp();
    // the shift is accurate to a few ulps, so two solves already give the eigenvector to round-off
    for (int it = 0; it < 2; ++it) {
      if (lane < nb) tri_solve(n, f, f + n, f + 2 * n, f + 3 * n, sw, y);
      __syncwarp();
      for (int b = 0; b < nb; ++b) {
        double* yb = ys + (size_t)b * n;
        // (unit length first: the solve has blown the vector up)
        for (int rep = 0; rep < 3; ++rep) {
          double nr = 0.0;
          for (int m = lane; m < n; m += 32) nr = fma(yb[m], yb[m], nr);
          nr = warp_sum(nr);
          const double sc = 1.0 / sqrt(nr);
          for (int m = lane; m < n; m += 32) yb[m] *= sc;
          __syncwarp();
          if (rep == 2) break;
          for (int l = j; l < i0 + b; ++l) {
            const double* zl = l < i0 ? Z + (size_t)l * n : ys + (size_t)(l - i0) * n;
            double dt = 0.0;
            for (int m = lane; m < n; m += 32) dt = fma(zl[m], yb[m], dt);
            dt = warp_sum(dt);
            for (int m = lane; m < n; m += 32) yb[m] = fma(-dt, zl[m], yb[m]);
            __syncwarp();
          }
        }
      }
    }
    for (int b = 0; b < nb; ++b) {
      double* zi = Z + (size_t)(i0 + b) * n;
      for (int m = lane; m < n; m += 32) zi[m] = ys[(size_t)b * n + m];
    }
    __syncwarp();
  }
}

size_t inviter_smem(int n, int batch) { return (2 * (size_t)n + (size_t)batch * 5 * n + ((size_t)batch * n + 1) / 2) * sizeof(double); }

// Four warp sums at once: lane l receives the sum of v[l & 3], one conversion for all four.
__device__ __forceinline__ double warp_sum4_fx(const double (&v)[4], int lane) {
  long long t = 0;
  uint32_t top = 0;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const uint32_t hi = (uint32_t)__double2hiint(v[a]), lo = (uint32_t)__double2loint(v[a]);
    const uint32_t e0 = (hi >> 20) & 0x7ffu, ex = max(e0, 1u);
    const uint32_t tp = __reduce_max_sync(0xffffffffu, ex), sh = min(tp - ex, 63u);
    const uint32_t mh = (hi & 0xfffffu) | (e0 ? 0x100000u : 0u);
    const unsigned long long mant = ((((unsigned long long)mh << 32) | lo) << 9) >> sh;
    const long long f = (int32_t)hi < 0 ? -(long long)mant : (long long)mant;
    const uint32_t sl = __reduce_add_sync(0xffffffffu, (uint32_t)f & 0x3ffffffu);
    const uint32_t sm = __reduce_add_sync(0xffffffffu, (uint32_t)(f >> 26) & 0x3ffffffu);
    const int sg = __reduce_add_sync(0xffffffffu, (int)(f >> 52));
    if ((lane & 3) == a) {
      t = ((long long)sg << 47) + ((long long)sm << 21) + (long long)(sl >> 5);
      top = tp;
    }
  }
  // (a non-finite addend, or one above 2^1016, which reflectors of norm up to 2^241 and unit vectors do not make)
  if (top >= kFxTop) return __longlong_as_double(0x7ff8000000000000LL);
  return fx_scaled(t, top);
}

// The reflectors of the back-transform in groups of four, k0 = n - 3 - 4 g first: with p_a = v_a . z for the
// untouched z, the four steps are z -= sum_a s_a v_a, s = T p (T lower triangular, T_aa = tau_a,
// T_ab = -tau_a sum_{b <= c < a} (v_a . v_c) T_cb).  One warp per group writes T (16 doubles).
__global__ void __launch_bounds__(32) reflector_groups_kernel(int n, const double* __restrict__ H,
                                                              const double* __restrict__ tau, double* __restrict__ T) {
  const int lane = threadIdx.x, k0 = n - 3 - 4 * (int)blockIdx.x;
  double g[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};  // (1,0) (2,0) (2,1) (3,0) (3,1) (3,2)
  for (int i = max(k0 - 2, 0) + lane; i < n; i += 32) {
    double v[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) v[a] = (k0 - a >= 0 && i > k0 - a) ? H[(size_t)(k0 - a) * n + i] : 0.0;
    g[0] = fma(v[1], v[0], g[0]);
    g[1] = fma(v[2], v[0], g[1]);
    g[2] = fma(v[2], v[1], g[2]);
    g[3] = fma(v[3], v[0], g[3]);
    g[4] = fma(v[3], v[1], g[4]);
    g[5] = fma(v[3], v[2], g[5]);
  }
#pragma unroll
  for (int q = 0; q < 6; ++q) g[q] = warp_sum_fx(g[q]);
  if (lane == 0) {
    double t[4][4] = {}, ta[4];
    for (int a = 0; a < 4; ++a) ta[a] = k0 - a >= 0 ? tau[k0 - a] : 0.0;
    const double ga[4][4] = {{0, 0, 0, 0}, {g[0], 0, 0, 0}, {g[1], g[2], 0, 0}, {g[3], g[4], g[5], 0}};
    for (int a = 0; a < 4; ++a) {
      t[a][a] = ta[a];
      for (int b = 0; b < a; ++b) {
        double x = 0.0;
        for (int c = b; c < a; ++c) x = fma(ga[a][c], t[c][b], x);
        t[a][b] = -ta[a] * x;
      }
    }
    for (int a = 0; a < 4; ++a)
      for (int b = 0; b < 4; ++b) T[16 * (size_t)blockIdx.x + 4 * a + b] = t[a][b];
  }
}

// V = Q Z = H_0 H_1 ... H_{n-3} Z (in place on V), S warps per column, the column in registers (rows
// lane + 32 t, t = r S + part, r < RR), four reflectors per round (see above).  Bound: FP64 instructions, 64
// clocks each per sub-partition.  One warp per column used two of the four sub-partitions of 120 SMs at
// n = 240, and paid a warp sum (about 700 clocks with its waits) per reflector: 240 us there, 26 us at n = 60,
// 2.41 ms at n = 600.  S is the largest with which n S warps fit on the 608 sub-partitions.
template <int RR, int S>
__global__ void __launch_bounds__(128) backtransform_reg_kernel(int n, const double* __restrict__ H,
                                                                const double* __restrict__ T, double* V) {
  constexpr bool kKeep = RR <= 5;  // the reflectors' chunks stay in registers between the two uses
  __shared__ double part_sum[2][4][4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cb = warp / S, part = warp % S;
  const int col = blockIdx.x * (4 / S) + cb;
  if (col >= n) return;
  double* zc = V + (size_t)col * n;
  double z[RR], h[kKeep ? 4 : 1][kKeep ? RR : 1], hn[kKeep ? 4 : 1][kKeep ? RR : 1];
#pragma unroll
  for (int r = 0; r < RR; ++r) {
    const int i = lane + 32 * (r * S + part);
    z[r] = i < n ? zc[i] : 0.0;
  }
  auto at = [&](int k, int r) {
    const int i = lane + 32 * (r * S + part);
    return (k >= 0 && i > k && i < n) ? __ldg(H + (size_t)k * n + i) : 0.0;
  };
  const int groups = (n - 2 + 3) / 4;
  if (kKeep && groups > 0) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int r = 0; r < RR; ++r) hn[a][r] = at(n - 3 - a, r);
  }
  for (int g = 0; g < groups; ++g) {
    const int k0 = n - 3 - 4 * g;
    const double2* tp = reinterpret_cast<const double2*>(T + 16 * (size_t)g + 4 * (lane & 3));  // row of T
    const double2 t01 = __ldg(tp), t23 = __ldg(tp + 1);
    double p[4] = {0.0, 0.0, 0.0, 0.0};
    // (rows up to k are not touched: chunks without any other are skipped, an FP64 instruction costs the
    // same with zeros; likewise the chunks past n)
    if (kKeep) {
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int r = 0; r < RR; ++r) {
          h[a][r] = hn[a][r];
          hn[a][r] = at(k0 - 4 - a, r);
        }
    }
#pragma unroll
    for (int r = 0; r < RR; ++r) {
      const int t = r * S + part;
      if (32 * t + 31 > k0 - 3 && 32 * t < n) {
#pragma unroll
        for (int a = 0; a < 4; ++a) p[a] = fma(kKeep ? h[a][r] : at(k0 - a, r), z[r], p[a]);
      }
    }
    double mine = warp_sum4_fx(p, lane);  // of reflector lane & 3
    if (S > 1) {
      double* ps = &part_sum[g & 1][0][0];
      if (lane < 4) ps[4 * warp + lane] = mine;
      asm volatile("bar.sync %0, %1;" ::"r"(1 + cb), "r"(32 * S) : "memory");
      mine = ps[4 * cb * S + (lane & 3)];
#pragma unroll
      for (int q = 1; q < S; ++q) mine += ps[4 * (cb * S + q) + (lane & 3)];
    }
    // s = T p: lane a & 3 holds row a
    double sa = 0.0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const double pb = __shfl_sync(0xffffffffu, mine, b);
      sa = fma(b == 0 ? t01.x : b == 1 ? t01.y : b == 2 ? t23.x : t23.y, pb, sa);
    }
    double s[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) s[a] = -__shfl_sync(0xffffffffu, sa, a);
#pragma unroll
    for (int r = 0; r < RR; ++r) {
      const int t = r * S + part;
      if (32 * t + 31 > k0 - 3 && 32 * t < n) {
#pragma unroll
        for (int a = 0; a < 4; ++a) z[r] = fma(s[a], kKeep ? h[a][r] : at(k0 - a, r), z[r]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < RR; ++r) {
    const int i = lane + 32 * (r * S + part);
    if (i < n) zc[i] = z[r];
  }
}

// V = Q Z = H_0 H_1 ... H_{n-3} Z, one warp per column (in place on V).
__global__ void __launch_bounds__(64) backtransform_kernel(int n, const double* __restrict__ H,
                                                           const double* __restrict__ tau, double* V) {
  const int col = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (col >= n) return;
  double* z = V + (size_t)col * n;
  for (int k = n - 3; k >= 0; --k) {
    const double t = tau[k];
    if (t == 0.0) continue;
    const double* h = H + (size_t)k * n;
    double s = 0.0;
    for (int i = k + 1 + lane; i < n; i += 32) s += h[i] * z[i];
    s = warp_sum(s) * t;
    for (int i = k + 1 + lane; i < n; i += 32) z[i] -= s * h[i];
    __syncwarp();
  }
}

// C = val * I (n x n, column-major)
// S = 1.5 I - 0.5 S (n x n): the Newton-Schulz factor from the Gram matrix Z^T Z.
__global__ void ns_shift_kernel(int n, double* S) {
  const int64_t tot = (int64_t)n * n;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = t / n, i = t - j * n;
    S[t] = fma(-0.5, S[t], i == j ? 1.5 : 0.0);
  }
}

__global__ void diag_fill_kernel(int n, double* C, double val) {
  const int64_t tot = (int64_t)n * n;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x)
    C[t] = (t / n == t % n) ? val : 0.0;
}

}  // namespace

// ------------------------------------------------------------------ launchers
namespace {

constexpr int CLUSTER_MAX_N = 1024;     // global-memory variants: above this the cooperative grid is used
constexpr int INV_MAX_CLUSTER = 256;    // inverse iteration handles clusters up to this size
constexpr size_t SMEM_CAP = 220 * 1024; // dynamic shared memory of the resident variants

size_t multi_smem(int n) { return (2 * (size_t)n + 33) * sizeof(double); }

// Shared memory of a resident kernel (owned columns + two n-vectors + reduction slots) for P CTAs.
size_t resident_smem(int n, int P) {
  const size_t nq = ((size_t)n + P - 1) / P;
  return (nq * n + 2 * (size_t)n + 40) * sizeof(double);
}

cudaLaunchConfig_t cluster_cfg(int cs, int threads, size_t smem, cudaStream_t s, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cs);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

// Largest cluster size (16, else 8, else 0) with which `kernel` can be resident.
int cluster_size_for(const void* kernel, int threads, size_t smem) {
  RC_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_CAP));
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    cudaGetLastError();
  for (int cs : {16, 8}) {
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = cluster_cfg(cs, threads, smem, nullptr, at);
    int num = 0;
    if (cudaOccupancyMaxActiveClusters(&num, kernel, &cfg) == cudaSuccess && num >= 1) return cs;
    cudaGetLastError();
  }
  return 0;
}

// Launch a multi-CTA kernel pair (cluster / cooperative grid variants) with 2 n + 33 doubles of
// shared memory.
template <typename... Args>
void launch_multi(cudaStream_t s, void (*kc)(Args...), void (*kg)(Args...), int n, int num_sms, Args... args) {
  const size_t smem = multi_smem(n);
  if (n <= CLUSTER_MAX_N) {
    // one query per kernel (per instantiation), at the largest shared-memory size of this path
    static const int csz = cluster_size_for(reinterpret_cast<const void*>(kc), EIG_THREADS,
                                            multi_smem(CLUSTER_MAX_N));
    if (csz > 0) {
      cudaLaunchAttribute at[1];
      cudaLaunchConfig_t cfg = cluster_cfg(csz, EIG_THREADS, smem, s, at);
      RC_CUDA(cudaLaunchKernelEx(&cfg, kc, args...));
      RC_LAUNCH();
      return;
    }
  }
  RC_CUDA(cudaFuncSetAttribute(reinterpret_cast<const void*>(kg), cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)SMEM_CAP));
  int per_sm = 0;
  RC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kg, EIG_THREADS, smem));
  RC_CHECK(per_sm >= 1, RCHFSI_ERR_UNSUPPORTED, "eigensolver kernel does not fit on an SM");
  const int ctas = std::max(1, std::min(num_sms, std::max(8, n / 16)));
  void* argv[] = {(void*)&args...};
  RC_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kg), dim3(ctas), dim3(EIG_THREADS), argv, smem,
                                      s));
  RC_LAUNCH();
}

// Launch a shared-memory-resident kernel pair (256 threads): one cluster when its CTAs can hold the
// owned columns, else a cooperative grid of one CTA per SM; false when neither fits.
template <typename... Args>
bool launch_resident(cudaStream_t s, void (*kc)(Args...), void (*kg)(Args...), int n, int num_sms, Args... args) {
  static const int csz = cluster_size_for(reinterpret_cast<const void*>(kc), TRI_THREADS, SMEM_CAP);
  if (csz > 0 && resident_smem(n, csz) <= SMEM_CAP) {
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = cluster_cfg(csz, TRI_THREADS, resident_smem(n, csz), s, at);
    RC_CUDA(cudaLaunchKernelEx(&cfg, kc, args...));
    RC_LAUNCH();
    return true;
  }
  const int P = num_sms;
  const size_t smem = resident_smem(n, P);
  if (smem > SMEM_CAP) return false;
  RC_CUDA(cudaFuncSetAttribute(reinterpret_cast<const void*>(kg), cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)SMEM_CAP));
  int per_sm = 0;
  RC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kg, TRI_THREADS, smem));
  if (per_sm < 1) return false;
  void* argv[] = {(void*)&args...};
  RC_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kg), dim3(P), dim3(TRI_THREADS), argv, smem, s));
  RC_LAUNCH();
  return true;
}

// tridiag_xch_kernel: one cluster up to this order, above it a cooperative grid (a grid's exchange
// through L2 costs ~1 us more per column, but spreads the FP64 work over more SMs).  Measured (us),
// cluster of 16 / grid of 96: n = 240 1036 / 1237, 300 1607 / 1704, 384 2573 / 2338, 480 4016 / 3220.
constexpr int kTriClusterMaxN = 320;

// The workspace tridiag_xch_kernel needs on a grid, in doubles (4 n packets of 16 bytes).
size_t tridiag_xch_ws(int n) { return 8 * (size_t)n + 2; }

// False when the matrix does not fit (n > 1024, or no shared memory for the owned columns).
bool launch_tridiag_xch(cudaStream_t s, int n, int num_sms, const double* M, double* H, double* d, double* e,
                        double* tau, double* xg, int* err) {
  if (n > 256 * TX_ROWS) return false;
  if (n <= kTriClusterMaxN) {
    static const int csz = cluster_size_for(reinterpret_cast<const void*>(tridiag_xch_kernel<true>), TX_THREADS,
                                            tridiag_xch_smem(kTriClusterMaxN, 16, true));
    // 8 CTAs reach the floor of the exchange for small orders (n = 60: 158 us, 4: 166, 16: 164)
    const int P = std::min(csz, n <= 96 ? 8 : 16);
    const size_t smem = P > 0 ? tridiag_xch_smem(n, P, true) : 0;
    if (P > 0 && smem <= SMEM_CAP) {
      cudaLaunchAttribute at[1];
      cudaLaunchConfig_t cfg = cluster_cfg(P, TX_THREADS, smem, s, at);
      RC_CUDA(cudaLaunchKernelEx(&cfg, tridiag_xch_kernel<true>, n, M, H, d, e, tau, (uint4*)nullptr, err));
      RC_LAUNCH();
      return true;
    }
  }
  const int P = std::min(num_sms, n <= 512 ? 96 : 128);
  const size_t smem = tridiag_xch_smem(n, P, false);
  if (smem > SMEM_CAP) return false;
  set_smem_limit(reinterpret_cast<const void*>(tridiag_xch_kernel<false>), (int)SMEM_CAP);
  int per_sm = 0;
  RC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, tridiag_xch_kernel<false>, TX_THREADS, smem));
  if (per_sm < 1) return false;
  uint4* pk = reinterpret_cast<uint4*>((reinterpret_cast<uintptr_t>(xg) + 15) & ~uintptr_t(15));
  RC_CUDA(cudaMemsetAsync(pk, 0, 64 * (size_t)n, s));  // no packet carries a tag yet
  void* argv[] = {(void*)&n, (void*)&M, (void*)&H, (void*)&d, (void*)&e, (void*)&tau, (void*)&pk, (void*)&err};
  RC_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(tridiag_xch_kernel<false>), dim3(P),
                                      dim3(TX_THREADS), argv, smem, s));
  RC_LAUNCH();
  return true;
}

template <int RR, int S>
void launch_backtransform(cudaStream_t s, int n, const double* H, const double* T, double* V) {
  backtransform_reg_kernel<RR, S><<<cdiv(n, 4 / S), 128, 0, s>>>(n, H, T, V);
  RC_LAUNCH();
}

}  // namespace

int cholesky_inverse_f64(cudaStream_t s, int n, double* A, double* L, double* Linv, int* d_info, int num_sms,
                         DevBuf<double>& scratch) {
  RC_CHECK(n >= 1 && n <= 6144, RCHFSI_ERR_UNSUPPORTED, "cholesky_inverse: order out of [1, 6144]");
  {
    const int nt = (n + CB - 1) / CB;
    int per_sm = 0;
    RC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, chol_inv_blocked_kernel, 256, 0));
    if (per_sm >= 1) {
      // no more CTAs than the largest phase has units (a barrier costs more with more CTAs)
      const int P = std::max(1, std::min(num_sms, 2 * nt * (nt + 1)));
      const double* Ac = A;
      void* argv[] = {(void*)&n, (void*)&Ac, (void*)&L, (void*)&Linv, (void*)&d_info};
      RC_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(chol_inv_blocked_kernel), dim3(P), dim3(256),
                                          argv, 0, s));
      RC_LAUNCH();
      return 0;
    }
  }
  double* xch = scratch.ensure(3 * (size_t)n);
  double* dinv = xch + 2 * (size_t)n;
  if (n <= 4096 && launch_resident(s, chol_inv_smem_kernel<true>, chol_inv_smem_kernel<false>, n, num_sms, n,
                                   (const double*)A, L, Linv, xch, dinv, d_info))
    return 0;
  launch_multi(s, chol_inv_kernel<true>, chol_inv_kernel<false>, n, num_sms, n, A, L, Linv, d_info);
  return 0;
}

bool sym_eig_f64(cudaStream_t s, int n, double* M, double* V, double* evals, DevBuf<double>& ws, int* d_flag,
                 int num_sms, const OzScratch* oz) {
  if (n < 1 || n > 3072) return false;
  // workspace: T (16 per group of four reflectors), H, S, V2 (n^2 each), d, e, tau, p (n each), xch (n + 8), tnorm,
  // exchange packets
  const size_t nn = (size_t)n * n, tn = ((size_t)(n + 3) / 4 * 16 + 31) / 32 * 32;
  double* T = ws.ensure(tn + 3 * nn + 6 * (size_t)n + 16 + tridiag_xch_ws(n));
  double* H = T + tn;
  double* S = H + nn;
  double* V2 = S + nn;
  double* d = V2 + nn;
  double* e = d + n;
  double* tau = e + n;
  double* p = tau + n;
  double* xch = p + n;
  double* tnorm = xch + n + 8;
  double* pkts = tnorm + 8;
  RC_CUDA(cudaMemsetAsync(d_flag, 0, sizeof(int), s));
  if (n == 1) {
    RC_CUDA(cudaMemcpyAsync(evals, M, sizeof(double), cudaMemcpyDeviceToDevice, s));
    const double one = 1.0;
    RC_CUDA(cudaMemcpyAsync(V, &one, sizeof(double), cudaMemcpyHostToDevice, s));
    RC_CUDA(cudaStreamSynchronize(s));
    return true;
  }
  RC_CUDA(cudaMemsetAsync(e, 0, sizeof(double) * 2 * n, s));  // and tau behind it
  // 1. Q^T M Q = T
  if (!launch_tridiag_xch(s, n, num_sms, M, H, d, e, tau, pkts, d_flag) &&
      !launch_resident(s, tridiag_smem_kernel<true>, tridiag_smem_kernel<false>, n, num_sms, n, (const double*)M, H,
                       d, e, tau, xch, p))
    launch_multi(s, tridiag_kernel<true>, tridiag_kernel<false>, n, num_sms, n, M, H, d, e, tau, p);
  // 2. eigenvalues and eigenvectors of T (into V2), 3. the vectors of clusters
  const bool pairs = n <= TE_MAX_N;
  if (pairs) {
    set_smem_limit(reinterpret_cast<const void*>(tri_eig_kernel), (int)SMEM_CAP);
    tri_eig_kernel<<<cdiv(n, TE_WARPS), 32 * TE_WARPS, tri_eig_smem(n), s>>>(n, d, e, evals, tnorm, V2);
  } else {
    bisect_kernel<<<n, 32, 2 * (size_t)n * sizeof(double), s>>>(n, d, e, evals, tnorm);
  }
  RC_LAUNCH();
  set_smem_limit(reinterpret_cast<const void*>(inviter_kernel), (int)SMEM_CAP);
  int batch = 4;
  while (batch > 1 && inviter_smem(n, batch) > 48 * 1024) --batch;
  inviter_kernel<<<n, 32, inviter_smem(n, batch), s>>>(n, d, e, evals, tnorm, V2, INV_MAX_CLUSTER, pairs ? 1 : 0, batch,
                                                       d_flag);
  RC_LAUNCH();
  // 4. one Newton-Schulz step towards the orthogonal factor: Z <- Z (3 I - Z^T Z) / 2
  if (oz && n <= kSmallGemmMaxN) {
    // S = 1.5 I - 0.5 Z^T Z, V = Z S
    gemm_small_f64(s, n, V2, n, 1, V2, 1, n, -0.5, 1.5, S, RCHFSI_KERNEL_EIG);
    gemm_small_f64(s, n, V2, 1, n, S, 1, n, 1.0, 0.0, V, RCHFSI_KERNEL_EIG);
  } else if (oz) {
    // FP64-accurate products from BF16 slices: G = Z^T Z (symmetric), S = 1.5 I - 0.5 G, V = Z S
    oz_slice(s, n, n, V2, n, 1, *oz->a);  // row i = column i of Z
    oz_gemm(s, oz->num_sms, *oz->a, *oz->a, S, n, *oz->ws, oz->err, true);
    ns_shift_kernel<<<cdiv((int64_t)n * n, 256) < 1216 ? cdiv((int64_t)n * n, 256) : 1216, 256, 0, s>>>(n, S);
    RC_LAUNCH();
    oz_slice(s, n, n, V2, 1, n, *oz->b);  // row i of Z
    oz_slice(s, n, n, S, n, 1, *oz->a);   // column j of S as row j
    oz_gemm(s, oz->num_sms, *oz->b, *oz->a, V, n, *oz->ws, oz->err);
  } else {
  diag_fill_kernel<<<cdiv((int64_t)n * n, 256) < 1216 ? cdiv((int64_t)n * n, 256) : 1216, 256, 0, s>>>(n, S, 1.5);
  RC_LAUNCH();
  EpiArgs g;
  g.kind = EPI_STORE;
  g.C = S;
  g.ldc = n;
  g.alpha = -0.5;
  g.beta = 1.0;
  g.prof_cls = RCHFSI_KERNEL_EIG;
  gemm_f64(s, n, n, n, V2, n, true, V2, n, true, g);
  EpiArgs z;
  z.kind = EPI_STORE;
  z.C = V;
  z.ldc = n;
  z.prof_cls = RCHFSI_KERNEL_EIG;
  gemm_f64(s, n, n, n, V2, n, false, S, n, true, z);
  }
  // 5. V = Q Z
  if (n > 1024) {
    backtransform_kernel<<<cdiv(n, 2), 64, 0, s>>>(n, H, tau, V);
    RC_LAUNCH();
    return true;
  }
  if (n > 2) {
    reflector_groups_kernel<<<(n - 2 + 3) / 4, 32, 0, s>>>(n, H, tau, T);
    RC_LAUNCH();
  }
  if (n <= 64) launch_backtransform<1, 2>(s, n, H, T, V);
  else if (n <= 128) launch_backtransform<1, 4>(s, n, H, T, V);
  else if (n <= 152) launch_backtransform<2, 4>(s, n, H, T, V);
  else if (n <= 320) launch_backtransform<5, 2>(s, n, H, T, V);
  else if (n <= 640) launch_backtransform<20, 1>(s, n, H, T, V);
  else launch_backtransform<32, 1>(s, n, H, T, V);
  return true;
}

}  // namespace rchfsi
