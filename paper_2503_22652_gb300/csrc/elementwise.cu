// Memory-bound helper kernels: layout changes, casts, column norms, the reconstruction of
// Algorithm 3 (Y_p = D^-1 R_Y + X Lambda_Y), the product-free part of the recurrence update, and
// the small reductions used by the Lanczos estimate.  Grid-stride loops sized to the SM count.
#include <algorithm>

#include "common.cuh"

namespace rchfsi {
namespace {

__device__ __forceinline__ unsigned grid_threads() { return gridDim.x * blockDim.x; }

inline unsigned ew_blocks(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  if (b < 1) b = 1;
  return (unsigned)b;
}

__global__ void transpose_kernel(int64_t rows, int64_t cols, const double* __restrict__ in, int64_t ldin,
                                 double* __restrict__ out, int64_t ldout) {
  __shared__ double t[32][33];
  const int64_t r0 = (int64_t)blockIdx.y * 32, c0 = (int64_t)blockIdx.x * 32;
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    int64_t r = r0 + k, c = c0 + threadIdx.x;
    if (r < rows && c < cols) t[k][threadIdx.x] = in[r * ldin + c];
  }
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    int64_t c = c0 + k, r = r0 + threadIdx.x;
    if (r < rows && c < cols) out[c * ldout + r] = t[threadIdx.x][k];
  }
}

// FP64 <-> FP32 conversions by integer arithmetic for normal values (others: the conversion instruction).
// A conversion from or to a double holds the FP64 pipe like a multiply (about two per clock per SM), which
// bounded the passes that open and close the FE filter: 262144 x 600, 1105 and 1187 us against 0.37 and
// 0.47 ms of HBM traffic.
// (the conversions proper stay behind a call: inlined, they are executed for every value and selected away)
__device__ __noinline__ float f32_cvt(double x) { return (float)x; }
__device__ __noinline__ double f64_cvt(float x) { return (double)x; }
__device__ __forceinline__ float f32_rn(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned long long r = u + 0x0fffffffULL + ((u >> 29) & 1ULL);  // round to nearest even at bit 29
  const uint32_t e = (uint32_t)(r >> 52) & 0x7ffu;
  if (e - 897u > 253u) return f32_cvt(x);  // zero, subnormal, overflow, non-finite
  const uint32_t v = (uint32_t)((r & 0x7fffffffffffffffULL) >> 29) - (896u << 23);
  return __uint_as_float(v | ((uint32_t)(u >> 32) & 0x80000000u));
}
__device__ __forceinline__ double f64_of(float x) {
  const uint32_t b = __float_as_uint(x), e = (b >> 23) & 0xffu;
  if (e - 1u > 253u) return f64_cvt(x);
  return __longlong_as_double((long long)(((unsigned long long)(b & 0x80000000u) << 32) |
                                          (((unsigned long long)(b & 0x7fffffffu) << 29) + (896ULL << 52))));
}

// One column per lane, one warp per block: a chain of 3 FP64 instructions (64 clocks each) per step.
__global__ void __launch_bounds__(32) filter_tables_kernel(const __grid_constant__ FilterTables t) {
  const int j = blockIdx.x * 32 + threadIdx.x;
  if (j < t.N) {
    const double lm = t.lam[j] - t.cc;
    double lx = 1.0, ly = t.s1e * lm;
    t.tab[j] = 1.0;
    t.tab[(int64_t)t.N + j] = ly;
    for (int k = 0; k < t.steps; ++k) {
      if (t.lamf) t.lamf[(int64_t)k * t.N + j] = f32_rn(ly);
      const double nx = fma(t.a[k] * lm, ly, t.c[k] * lx);
      lx = ly;
      ly = nx;
      t.tab[(int64_t)(k + 2) * t.N + j] = ly;
    }
  }
  const int stride = gridDim.x * 32;
  if (t.coef)
    for (int k = j; k < t.steps; k += stride) {
      t.coef[3 * k] = f32_rn(t.a[k]);
      t.coef[3 * k + 1] = f32_rn(t.b[k]);
      t.coef[3 * k + 2] = f32_rn(t.c[k]);
    }
  for (int i = j; i < t.ncounters; i += stride) t.counters[i] = 0;
}

// o1(i, j) = (float)(W(i, j) s1), o2(i, j) = (float)(W(i, j) s2): W column-major (leading dimension
// m), o1 and o2 row-major m x n.  32 x 32 shared-memory tiles, rows on blockIdx.x.
__global__ void __launch_bounds__(256) cols_to_rows_f32x2_kernel(int64_t m, int64_t n, const double* __restrict__ W,
                                                                 double s1, double s2, float* __restrict__ o1,
                                                                 float* __restrict__ o2) {
  __shared__ double t[32][33];
  const int64_t i0 = (int64_t)blockIdx.x * 32, j0 = (int64_t)blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
  for (int c = ty; c < 32; c += 8) {
    const int64_t i = i0 + tx, j = j0 + c;
    t[c][tx] = (i < m && j < n) ? W[j * m + i] : 0.0;
  }
  __syncthreads();
  for (int r = ty; r < 32; r += 8) {
    const int64_t i = i0 + r, j = j0 + tx;
    if (i < m && j < n) {
      const double w = t[tx][r];
      const float f2 = f32_rn(s2 == 1.0 ? w : w * s2);
      o1[i * n + j] = s1 == s2 ? f2 : f32_rn(w * s1);
      o2[i * n + j] = f2;
    }
  }
}

// The same for a row-major W: elementwise, pairs where the arrays allow it.
template <bool PAIRS>
__global__ void __launch_bounds__(256) rows_f32x2_kernel(int64_t total, const double* __restrict__ W, double s1,
                                                         double s2, float* __restrict__ o1, float* __restrict__ o2) {
  const int64_t cnt = PAIRS ? total / 2 : total;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < cnt; e += grid_threads()) {
    if (PAIRS) {
      const double2 w = reinterpret_cast<const double2*>(W)[e];
      const float2 f2 = s2 == 1.0 ? make_float2(f32_rn(w.x), f32_rn(w.y)) : make_float2(f32_rn(w.x * s2), f32_rn(w.y * s2));
      reinterpret_cast<float2*>(o1)[e] = s1 == s2 ? f2 : make_float2(f32_rn(w.x * s1), f32_rn(w.y * s1));
      reinterpret_cast<float2*>(o2)[e] = f2;
    } else {
      const double w = W[e];
      const float f2 = f32_rn(s2 == 1.0 ? w : w * s2);
      o1[e] = s1 == s2 ? f2 : f32_rn(w * s1);
      o2[e] = f2;
    }
  }
}

// Y(i, j) = dinv[i] rs R(i, j) + X(i, j) lam[j] (dinv optional): R row-major float (leading
// dimension n); X and Y column-major (leading dimension m).  32 x 32 shared-memory tiles.
__global__ void __launch_bounds__(256) rows_to_cols_recon_kernel(int64_t m, int64_t n, const float* __restrict__ R,
                                                                 double rs, const double* __restrict__ dinv,
                                                                 const double* X, const double* __restrict__ lam,
                                                                 double* Y) {
  __shared__ float t[32][33];
  const int64_t i0 = (int64_t)blockIdx.x * 32, j0 = (int64_t)blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
  for (int r = ty; r < 32; r += 8) {
    const int64_t i = i0 + r, j = j0 + tx;
    t[r][tx] = (i < m && j < n) ? R[i * n + j] : 0.f;
  }
  __syncthreads();
  const int64_t i = i0 + tx;
  if (i >= m) return;
  const double d = dinv ? dinv[i] * rs : rs;
#pragma unroll
  for (int c = ty; c < 32; c += 8) {
    const int64_t j = j0 + c;
    if (j < n) Y[j * m + i] = fma(X[j * m + i], lam[j], d * f64_of(t[tx][c]));
  }
}

// The same with X and Y row-major (leading dimension n): a warp per row, four pairs (PAIRS) or values of the
// row in flight per lane.
template <bool PAIRS>
__global__ void __launch_bounds__(256) rows_recon_kernel(int64_t m, int64_t n, const float* __restrict__ R, double rs,
                                                         const double* __restrict__ dinv, const double* X,
                                                         const double* __restrict__ lam, double* Y) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x / 32);
  const int64_t cnt = PAIRS ? n / 2 : n;
  for (int64_t i = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; i < m; i += nw) {
    const double d = dinv ? dinv[i] * rs : rs;
    for (int64_t j0 = lane; j0 < cnt; j0 += 128) {
      if (PAIRS) {
        const float2* r2 = reinterpret_cast<const float2*>(R + i * n);
        const double2* x2 = reinterpret_cast<const double2*>(X + i * n);
        float2 r[4];
        double2 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j0 + 32 * u < cnt) {
            r[u] = r2[j0 + 32 * u];
            x[u] = x2[j0 + 32 * u];
          }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j0 + 32 * u < cnt) {
            const double2 l = reinterpret_cast<const double2*>(lam)[j0 + 32 * u];
            reinterpret_cast<double2*>(Y + i * n)[j0 + 32 * u] =
                make_double2(fma(x[u].x, l.x, d * f64_of(r[u].x)), fma(x[u].y, l.y, d * f64_of(r[u].y)));
          }
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int64_t j = j0 + 32 * u;
          if (j < cnt) Y[i * n + j] = fma(X[i * n + j], lam[j], d * f64_of(R[i * n + j]));
        }
      }
    }
  }
}

// Four rows in flight per thread, one column per blockIdx.y step (no division per element).
__global__ void __launch_bounds__(256) scale_cols_kernel(int64_t m, int64_t n, double* X, int64_t ld,
                                                         const double* scale) {
  for (int64_t j = blockIdx.y; j < n; j += gridDim.y) {
    const double f = scale[j];
    double* col = X + j * ld;
    for (int64_t i = blockIdx.x * (int64_t)1024 + threadIdx.x; i < m; i += (int64_t)gridDim.x * 1024) {
      double v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = i + 256 * u < m ? col[i + 256 * u] : 0.0;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i + 256 * u < m) col[i + 256 * u] = v[u] * f;
    }
  }
}

// One CTA per column: out[j] = 1 / ||X(:,j)||_2 (column-major); bad[0] / bad[1]: the smallest column whose
// norm is not finite / is zero (preset above every column).
__global__ void __launch_bounds__(1024) col_norms_inv_kernel(int64_t m, const double* __restrict__ X, int64_t ld,
                                                             double* out, int* bad) {
  __shared__ double red[32];
  const int64_t j = blockIdx.x;
  const double* col = X + j * ld;
  double s = 0.0, t = 0.0;
  int64_t i = threadIdx.x;
  for (; i + 3 * (int64_t)blockDim.x < m; i += 4 * (int64_t)blockDim.x) {
    const double a = col[i], b = col[i + blockDim.x], c = col[i + 2 * blockDim.x], d = col[i + 3 * blockDim.x];
    s = fma(a, a, s);
    t = fma(b, b, t);
    s = fma(c, c, s);
    t = fma(d, d, t);
  }
  for (; i < m; i += blockDim.x) s = fma(col[i], col[i], s);
  s += t;
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) {
      const double nrm = sqrt(s);
      if (!isfinite(nrm)) atomicMin(bad, (int)j);
      else if (nrm == 0.0) atomicMin(bad + 1, (int)j);
      out[j] = 1.0 / nrm;
    }
  }
}

__global__ void scale_rows_kernel(int64_t m, int64_t n, const double* in, double* out, const double* d, int cols) {
  const int64_t total = m * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += grid_threads()) {
    const int64_t i = e / n, j = e - i * n;
    out[e] = in[e] * (cols ? d[j] : d[i]);
  }
}

// Round an FP32 value to TF32 (10 explicit mantissa bits), round-to-nearest, ties away from zero
// (the cvt.rna.tf32.f32 rounding).
__device__ __forceinline__ float to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

__global__ void cast_f64_f32_kernel(int64_t n, const double* in, float* out, double scale, int tf32) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += grid_threads()) {
    float v = (float)(in[e] * scale);
    out[e] = tf32 ? to_tf32(v) : v;
  }
}

__global__ void cast_f64_bf16_kernel(int64_t n, const double* in, __nv_bfloat16* out, double scale) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += grid_threads())
    out[e] = __float2bfloat16_rn((float)(in[e] * scale));
}

__global__ void cast_f32_f64_kernel(int64_t n, const float* in, double* out, double scale) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += grid_threads())
    out[e] = scale * (double)in[e];
}

__global__ void scaled_copy_kernel(int64_t n, const double* in, double* out, double scale) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += grid_threads())
    out[e] = in[e] * scale;
}

template <typename R>
__device__ __forceinline__ double ld_r(const R* p, int64_t o) { return (double)p[o]; }
template <>
__device__ __forceinline__ double ld_r<__nv_bfloat16>(const __nv_bfloat16* p, int64_t o) {
  return (double)__bfloat162float(p[o]);
}

__device__ __forceinline__ void st_r(float* p, double v) { *p = f32_rn(v); }
__device__ __forceinline__ void st_r(__nv_bfloat16* p, double v) { *p = __float2bfloat16_rn(f32_rn(v)); }

// Row-major W (m x n) -> column-major o1 = s1 W, o2 = W (optional) of pitch ld.  One launch in place of a
// transpose and two casts; 32 x 32 tiles.
template <typename R>
__global__ void __launch_bounds__(256) rows_to_cols_lowp_kernel(int64_t m, int64_t n, const double* __restrict__ W,
                                                                double s1, R* __restrict__ o1, R* __restrict__ o2,
                                                                int64_t ld) {
  __shared__ double t[32][33];
  const int64_t i0 = (int64_t)blockIdx.x * 32, j0 = (int64_t)blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
  for (int r = ty; r < 32; r += 8) {
    const int64_t i = i0 + r, j = j0 + tx;
    t[r][tx] = (i < m && j < n) ? W[i * n + j] : 0.0;
  }
  __syncthreads();
#pragma unroll
  for (int c = ty; c < 32; c += 8) {
    const int64_t i = i0 + tx, j = j0 + c;
    if (i < m && j < n) {
      const double w = t[tx][c];
      st_r(o1 + j * ld + i, w * s1);
      if (o2) st_r(o2 + j * ld + i, w);
    }
  }
}

// Y = D^-1 R + X diag(lam) with R column-major of pitch ldr, X and Y row-major: one launch in place of the
// reconstruction and two transposes.
template <typename R>
__global__ void __launch_bounds__(256) cols_to_rows_recon_kernel(int64_t m, int64_t n, const R* __restrict__ Rr,
                                                                 int64_t ldr, const double* __restrict__ dinv,
                                                                 const double* X, const double* __restrict__ lam,
                                                                 double* Y) {
  __shared__ double t[32][33];
  const int64_t i0 = (int64_t)blockIdx.x * 32, j0 = (int64_t)blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const double d = dinv && i0 + tx < m ? dinv[i0 + tx] : 1.0;
#pragma unroll
  for (int c = ty; c < 32; c += 8) {
    const int64_t i = i0 + tx, j = j0 + c;
    t[c][tx] = (i < m && j < n) ? ld_r(Rr, j * ldr + i) * d : 0.0;
  }
  __syncthreads();
#pragma unroll
  for (int r = ty; r < 32; r += 8) {
    const int64_t i = i0 + r, j = j0 + tx;
    if (i < m && j < n) Y[i * n + j] = fma(X[i * n + j], lam[j], t[tx][r]);
  }
}

// Y = D^-1 R + X diag(lam), all column-major m x n with leading dimension m.
template <typename R>
__global__ void reconstruct_kernel(int64_t m, int64_t n, const R* __restrict__ Rr, int64_t ldr,
                                   const double* __restrict__ dinv, const double* __restrict__ X,
                                   const double* __restrict__ lam, double* __restrict__ Y) {
  const int64_t total = m * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += grid_threads()) {
    const int64_t j = e / m, i = e - j * m;
    double r = ld_r(Rr, j * ldr + i);
    if (dinv) r *= dinv[i];
    Y[e] = fma(X[e], lam[j], r);
  }
}

// Rx = b*Ry + c*Rx + a*W*lam[j]  (float storage, column-major)
__global__ void recur_axpby_kernel(int64_t m, int64_t n, const float* __restrict__ Ry, float* __restrict__ Rx,
                                   const float* __restrict__ W, const double* __restrict__ lam, float a, float b,
                                   float c) {
  const int64_t total = m * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += grid_threads()) {
    const int64_t j = e / m;
    float v = b * Ry[e] + c * Rx[e];
    if (W) v += a * W[e] * (float)lam[j];
    Rx[e] = v;
  }
}

__global__ void resid_norms_kernel(int64_t m, const double* __restrict__ W, const double* __restrict__ X,
                                   double* out_abs, double* out_x) {
  __shared__ double red[2][32];
  const int64_t j = blockIdx.x;
  double s = 0.0, t = 0.0;
  const double *cw = W + j * m, *cx = X ? X + j * m : nullptr;  // X: optional
  int64_t i = threadIdx.x;
  for (; i + 3 * (int64_t)blockDim.x < m; i += 4 * (int64_t)blockDim.x) {
    double w[4], x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      w[u] = cw[i + u * blockDim.x];
      x[u] = X ? cx[i + u * blockDim.x] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      s = fma(w[u], w[u], s);
      if (X) t = fma(x[u], x[u], t);
    }
  }
  for (; i < m; i += blockDim.x) {
    s = fma(cw[i], cw[i], s);
    if (X) t = fma(cx[i], cx[i], t);
  }
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = s;
    red[1][threadIdx.x >> 5] = t;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const bool ok = threadIdx.x < (blockDim.x >> 5);
    s = ok ? red[0][threadIdx.x] : 0.0;
    t = ok ? red[1][threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, o);
      t += __shfl_xor_sync(0xffffffffu, t, o);
    }
    if (threadIdx.x == 0) {
      out_abs[j] = sqrt(s);
      if (X) out_x[j] = sqrt(t);
    }
  }
}

// Single-CTA dot product: *out = x . y
__global__ void dot_kernel(int64_t n, const double* __restrict__ x, const double* __restrict__ y, double* out) {
  __shared__ double red[32];
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s = fma(x[i], y[i], s);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) *out = s;
  }
}

}  // namespace

void transpose_f64(cudaStream_t s, int64_t rows, int64_t cols, const double* in, int64_t ldin, double* out,
                   int64_t ldout) {
  if (rows <= 0 || cols <= 0) return;
  RC_CHECK(cdiv(rows, 32) <= 65535u, RCHFSI_ERR_INVALID_ARG, "transpose: too many rows for the grid");
  dim3 grid(cdiv(cols, 32), cdiv(rows, 32));
  transpose_kernel<<<grid, dim3(32, 8), 0, s>>>(rows, cols, in, ldin, out, ldout);
  RC_LAUNCH();
}

void scale_cols_f64(cudaStream_t s, int64_t m, int64_t n, double* X, int64_t ld, const double* scale) {
  if (m <= 0 || n <= 0) return;
  const dim3 grid(std::min<unsigned>(cdiv(m, 1024), 1024u), (unsigned)std::min<int64_t>(n, 65535));
  scale_cols_kernel<<<grid, 256, 0, s>>>(m, n, X, ld, scale);
  RC_LAUNCH();
}

void col_norms_inv_f64(cudaStream_t s, int64_t m, int64_t n, const double* X, int64_t ld, double* out, int* bad) {
  if (n <= 0) return;
  RC_CUDA(cudaMemsetAsync(bad, 0x7f, 2 * sizeof(int), s));
  // few columns: wide CTAs (m = 13,824, 48 columns: 13.6 us with 256 threads); many: several per SM
  col_norms_inv_kernel<<<(unsigned)n, n < 300 ? 1024 : 256, 0, s>>>(m, X, ld, out, bad);
  RC_LAUNCH();
}

void scale_rows_f64(cudaStream_t s, int64_t m, int64_t n, const double* in, double* out, const double* d,
                    bool cols) {
  scale_rows_kernel<<<ew_blocks(m * n), 256, 0, s>>>(m, n, in, out, d, cols ? 1 : 0);
  RC_LAUNCH();
}

void cols_to_rows_f32x2(cudaStream_t s, int64_t m, int64_t n, const double* W, double s1, double s2, float* o1,
                        float* o2) {
  if (m <= 0 || n <= 0) return;
  RC_CHECK(cdiv(n, 32) <= 65535u, RCHFSI_ERR_INVALID_ARG, "cols_to_rows: too many columns for the grid");
  cols_to_rows_f32x2_kernel<<<dim3(cdiv(m, 32), cdiv(n, 32)), 256, 0, s>>>(m, n, W, s1, s2, o1, o2);
  RC_LAUNCH();
}

template <typename R>
static void rows_to_cols_lowp(cudaStream_t s, int64_t m, int64_t n, const double* W, double s1, R* o1, R* o2,
                              int64_t ld) {
  if (m <= 0 || n <= 0) return;
  RC_CHECK(cdiv(n, 32) <= 65535u, RCHFSI_ERR_INVALID_ARG, "rows_to_cols: too many columns for the grid");
  rows_to_cols_lowp_kernel<R><<<dim3(cdiv(m, 32), cdiv(n, 32)), 256, 0, s>>>(m, n, W, s1, o1, o2, ld);
  RC_LAUNCH();
}
template <typename R>
static void cols_to_rows_recon(cudaStream_t s, int64_t m, int64_t n, const R* r, int64_t ldr, const double* dinv,
                               const double* X, const double* lam, double* Y) {
  if (m <= 0 || n <= 0) return;
  RC_CHECK(cdiv(n, 32) <= 65535u, RCHFSI_ERR_INVALID_ARG, "cols_to_rows: too many columns for the grid");
  cols_to_rows_recon_kernel<R><<<dim3(cdiv(m, 32), cdiv(n, 32)), 256, 0, s>>>(m, n, r, ldr, dinv, X, lam, Y);
  RC_LAUNCH();
}
void rows_to_cols_lowp_f32(cudaStream_t s, int64_t m, int64_t n, const double* W, double s1, float* o1, float* o2,
                           int64_t ld) {
  rows_to_cols_lowp<float>(s, m, n, W, s1, o1, o2, ld);
}
void rows_to_cols_lowp_bf16(cudaStream_t s, int64_t m, int64_t n, const double* W, double s1, __nv_bfloat16* o1,
                            __nv_bfloat16* o2, int64_t ld) {
  rows_to_cols_lowp<__nv_bfloat16>(s, m, n, W, s1, o1, o2, ld);
}
void cols_to_rows_recon_f32(cudaStream_t s, int64_t m, int64_t n, const float* R, int64_t ldr, const double* dinv,
                            const double* X, const double* lam, double* Y) {
  cols_to_rows_recon<float>(s, m, n, R, ldr, dinv, X, lam, Y);
}
void cols_to_rows_recon_bf16(cudaStream_t s, int64_t m, int64_t n, const __nv_bfloat16* R, int64_t ldr,
                             const double* dinv, const double* X, const double* lam, double* Y) {
  cols_to_rows_recon<__nv_bfloat16>(s, m, n, R, ldr, dinv, X, lam, Y);
}

void filter_tables(cudaStream_t s, const FilterTables& t) {
  filter_tables_kernel<<<cdiv(t.N, 32), 32, 0, s>>>(t);
  RC_LAUNCH();
}

static bool pairs_ok(int64_t n, const void* a, const void* b) {
  return n % 2 == 0 && ((uintptr_t)a & 15) == 0 && ((uintptr_t)b & 15) == 0;
}

void rows_f32x2(cudaStream_t s, int64_t m, int64_t n, const double* W, double s1, double s2, float* o1, float* o2) {
  if (m <= 0 || n <= 0) return;
  if (pairs_ok(n, W, W)) rows_f32x2_kernel<true><<<ew_blocks(m * n / 2), 256, 0, s>>>(m * n, W, s1, s2, o1, o2);
  else rows_f32x2_kernel<false><<<ew_blocks(m * n), 256, 0, s>>>(m * n, W, s1, s2, o1, o2);
  RC_LAUNCH();
}

void rows_recon(cudaStream_t s, int64_t m, int64_t n, const float* R, double rs, const double* dinv, const double* X,
                const double* lam, double* Y) {
  if (m <= 0 || n <= 0) return;
  const unsigned blocks = (unsigned)std::min<int64_t>((m + 7) / 8, 152 * 32);
  if (pairs_ok(n, X, Y) && pairs_ok(n, lam, R))
    rows_recon_kernel<true><<<blocks, 256, 0, s>>>(m, n, R, rs, dinv, X, lam, Y);
  else rows_recon_kernel<false><<<blocks, 256, 0, s>>>(m, n, R, rs, dinv, X, lam, Y);
  RC_LAUNCH();
}

void rows_to_cols_recon(cudaStream_t s, int64_t m, int64_t n, const float* R, double rs, const double* dinv,
                        const double* X, const double* lam, double* Y) {
  if (m <= 0 || n <= 0) return;
  RC_CHECK(cdiv(n, 32) <= 65535u, RCHFSI_ERR_INVALID_ARG, "rows_to_cols: too many columns for the grid");
  rows_to_cols_recon_kernel<<<dim3(cdiv(m, 32), cdiv(n, 32)), 256, 0, s>>>(m, n, R, rs, dinv, X, lam, Y);
  RC_LAUNCH();
}

void cast_f64_to_f32(cudaStream_t s, int64_t n, const double* in, float* out, double scale, int round_tf32) {
  cast_f64_f32_kernel<<<ew_blocks(n), 256, 0, s>>>(n, in, out, scale, round_tf32);
  RC_LAUNCH();
}

void cast_f64_to_bf16(cudaStream_t s, int64_t n, const double* in, __nv_bfloat16* out, double scale) {
  cast_f64_bf16_kernel<<<ew_blocks(n), 256, 0, s>>>(n, in, out, scale);
  RC_LAUNCH();
}

void cast_f32_to_f64(cudaStream_t s, int64_t n, const float* in, double* out, double scale) {
  cast_f32_f64_kernel<<<ew_blocks(n), 256, 0, s>>>(n, in, out, scale);
  RC_LAUNCH();
}

namespace {
// A += factor * tr(A) * I (one block: the trace, then the diagonal update)
__global__ void shift_diag_trace_kernel(int n, double* A, int lda, double factor) {
  __shared__ double part[256];
  double t = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) t += A[(int64_t)i * lda + i];
  part[threadIdx.x] = t;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  const double shift = factor * part[0];
  for (int i = threadIdx.x; i < n; i += blockDim.x) A[(int64_t)i * lda + i] += shift;
}
}  // namespace

void shift_diag_by_trace_f64(cudaStream_t s, int n, double* A, int lda, double factor) {
  shift_diag_trace_kernel<<<1, 256, 0, s>>>(n, A, lda, factor);
  RC_LAUNCH();
}

void fill_zero(cudaStream_t s, void* p, size_t bytes) { RC_CUDA(cudaMemsetAsync(p, 0, bytes, s)); }

void scaled_copy_f64(cudaStream_t s, int64_t n, const double* in, double* out, double scale) {
  scaled_copy_kernel<<<ew_blocks(n), 256, 0, s>>>(n, in, out, scale);
  RC_LAUNCH();
}

void reconstruct_f64(cudaStream_t s, int64_t m, int64_t n, const double* R, int64_t ldr, const double* dinv,
                     const double* X, const double* lam, double* Y) {
  reconstruct_kernel<double><<<ew_blocks(m * n), 256, 0, s>>>(m, n, R, ldr, dinv, X, lam, Y);
  RC_LAUNCH();
}

void reconstruct_f32(cudaStream_t s, int64_t m, int64_t n, const float* R, int64_t ldr, const double* dinv,
                     const double* X, const double* lam, double* Y) {
  reconstruct_kernel<float><<<ew_blocks(m * n), 256, 0, s>>>(m, n, R, ldr, dinv, X, lam, Y);
  RC_LAUNCH();
}

void reconstruct_bf16(cudaStream_t s, int64_t m, int64_t n, const __nv_bfloat16* R, int64_t ldr,
                      const double* dinv, const double* X, const double* lam, double* Y) {
  reconstruct_kernel<__nv_bfloat16><<<ew_blocks(m * n), 256, 0, s>>>(m, n, R, ldr, dinv, X, lam, Y);
  RC_LAUNCH();
}

namespace {
__global__ void cast2d_f32_kernel(int64_t rows, int64_t cols, const double* in, int64_t ldin, float* out,
                                  int64_t ldout, double scale, int tf32) {
  const int64_t total = rows * cols;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += grid_threads()) {
    const int64_t r = e / cols, c = e - r * cols;
    const float v = (float)(in[r * ldin + c] * scale);
    out[r * ldout + c] = tf32 ? to_tf32(v) : v;
  }
}
__global__ void cast2d_bf16_kernel(int64_t rows, int64_t cols, const double* in, int64_t ldin, __nv_bfloat16* out,
                                   int64_t ldout, double scale) {
  const int64_t total = rows * cols;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += grid_threads()) {
    const int64_t r = e / cols, c = e - r * cols;
    out[r * ldout + c] = __float2bfloat16_rn((float)(in[r * ldin + c] * scale));
  }
}
}  // namespace

void cast2d_f64_to_f32(cudaStream_t s, int64_t rows, int64_t cols, const double* in, int64_t ldin, float* out,
                       int64_t ldout, double scale, int round_tf32) {
  cast2d_f32_kernel<<<ew_blocks(rows * cols), 256, 0, s>>>(rows, cols, in, ldin, out, ldout, scale, round_tf32);
  RC_LAUNCH();
}

void cast2d_f64_to_bf16(cudaStream_t s, int64_t rows, int64_t cols, const double* in, int64_t ldin,
                        __nv_bfloat16* out, int64_t ldout, double scale) {
  cast2d_bf16_kernel<<<ew_blocks(rows * cols), 256, 0, s>>>(rows, cols, in, ldin, out, ldout, scale);
  RC_LAUNCH();
}

void recur_axpby_f32(cudaStream_t s, int64_t m, int64_t n, const float* Ry, float* Rx, const float* W,
                     const double* lam, double a, double b, double c) {
  recur_axpby_kernel<<<ew_blocks(m * n), 256, 0, s>>>(m, n, Ry, Rx, W, lam, (float)a, (float)b, (float)c);
  RC_LAUNCH();
}

void resid_rel_norms(cudaStream_t s, int64_t m, int64_t n, const double* W, const double* X, double* out_abs,
                     double* out_xnorm) {
  if (n <= 0) return;
  // (203 columns of 64000 with 256 threads and one row in flight: 90 us against 31 us of HBM traffic)
  resid_norms_kernel<<<(unsigned)n, m >= 4096 ? 1024 : 256, 0, s>>>(m, W, X, out_abs, out_xnorm);
  RC_LAUNCH();
}

void dot_f64(cudaStream_t s, int64_t n, const double* x, const double* y, double* out) {
  dot_kernel<<<1, 1024, 0, s>>>(n, x, y, out);
  RC_LAUNCH();
}

}  // namespace rchfsi
