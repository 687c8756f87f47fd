// Exact base-256 digits of FP64 values for the BF16-slice products (oz_gemm.cu, fe_oz.cu).
#pragma once
#include <cstdint>

namespace rchfsi {

// FP64 arithmetic is scarce on this GPU, so the slicing works on the bits: the binary exponent E
// with |x| in [2^(E-1), 2^E) (E = -100000 for 0), and the digits of x 2^(56 - e) in base 256 by
// integer shifts.
__device__ __forceinline__ int exp_of(double x) {
  const long long b = __double_as_longlong(x) & 0x7fffffffffffffffLL;
  if (b == 0) return -100000;
  const int eb = (int)(b >> 52);
  if (eb != 0) return eb - 1022;
  // subnormal: 2^-1074 times the 52-bit fraction
  return -1074 + (64 - __clzll(b));
}

// round(x 2^(56 - e)) as a signed 64-bit integer (half away from zero), for |x| < 2^e (so |result| <= 2^56).
// x = mant 2^ex with ex + 56 - e <= 4 (but for a row of subnormals only), so the significand goes four places
// up and then right by r >= 0; r > 58 gives 0.
__device__ __forceinline__ long long fixed56(double x, int e) {
  const long long bits = __double_as_longlong(x);
  const int eb = (int)(bits >> 52) & 0x7ff;
  unsigned long long mant = (unsigned long long)bits & 0x000fffffffffffffULL;
  if (eb != 0) mant |= 0x0010000000000000ULL;
  const int r = min(4 - ((eb != 0 ? eb : 1) - 1075 + 56 - e), 63);
  const long long f = r >= 0 ? (long long)(((mant << 4) + ((1ULL << r) >> 1)) >> r) : (long long)(mant << (4 - r));
  return bits < 0 ? -f : f;
}

// The 7 digits of f = round(x 2^(56 - e)): f = sum_s t_s 2^(48 - 8 s), |t_0| <= 256 and -128 <= t_s <= 127,
// each as an exact FP32 value.  Adding 128 to every lower digit turns them into the bytes of one integer;
// a byte placed under the exponent of 2^23 is an FP32 value 2^23 + byte, so a digit costs one byte permute
// and one FP32 add.  (A shift, a rounding and an integer-to-float conversion per digit bound the slicing
// passes by the integer pipe: 262144 x 600 by columns into row-major planes 1252 us against 0.51 ms of HBM.)
__device__ __forceinline__ void digits7(long long f, float* t) {
  const unsigned long long u = (unsigned long long)f + 0x0000808080808080ULL;
  const uint32_t lo = (uint32_t)u, hi = (uint32_t)(u >> 32);
  t[0] = __uint_as_float(0x4B400000u + (uint32_t)((int)hi >> 16)) - 12582912.0f;
  t[1] = __uint_as_float(__byte_perm(hi, 0x4B000000u, 0x7441)) - 8388736.0f;
  t[2] = __uint_as_float(__byte_perm(hi, 0x4B000000u, 0x7440)) - 8388736.0f;
  t[3] = __uint_as_float(__byte_perm(lo, 0x4B000000u, 0x7443)) - 8388736.0f;
  t[4] = __uint_as_float(__byte_perm(lo, 0x4B000000u, 0x7442)) - 8388736.0f;
  t[5] = __uint_as_float(__byte_perm(lo, 0x4B000000u, 0x7441)) - 8388736.0f;
  t[6] = __uint_as_float(__byte_perm(lo, 0x4B000000u, 0x7440)) - 8388736.0f;
}

// Two FP32 values that BF16 holds exactly as a packed pair (a in the low half).
__device__ __forceinline__ uint32_t bf16_pair(float a, float b) {
  return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}

// v 2^e as an FP64 value, rounded to nearest even: one conversion on the FP64 pipe, the scaling by
// exponent arithmetic.
__device__ __forceinline__ double fixed_to_f64(long long v, int e) {
  if (v == 0) return 0.0;
  const double d = (double)v;
  const long long be = (long long)((__double_as_longlong(d) >> 52) & 0x7ff) + e;
  if (be <= 0 || be >= 2047) return ldexp(d, e);  // out of the normal range: rare
  return __longlong_as_double(__double_as_longlong(d) + ((long long)e << 52));
}

// The same in integer arithmetic, for passes that need the FP64 pipe for something else.
__device__ __forceinline__ double fixed_to_f64_int(long long v, int e) {
  if (v == 0) return 0.0;
  const unsigned long long sgn = v < 0 ? (1ull << 63) : 0ull;
  unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int lz = __clzll((long long)a);
  a <<= lz;                          // leading one at bit 63
  unsigned long long mant = a >> 11;  // 53 significant bits
  const unsigned long long rem = a & 0x7ffull;
  if (rem > 0x400ull || (rem == 0x400ull && (mant & 1ull))) ++mant;
  const int be = 1086 - lz + e;  // v 2^e = 1.f 2^(63 - lz + e); a carry of the rounding runs into the exponent
  if (be <= 0 || be >= 2046) return ldexp((double)v, e);  // out of the normal range: rare
  return __longlong_as_double((long long)(sgn | (((unsigned long long)be << 52) + (mant - (1ull << 52)))));
}

}  // namespace rchfsi
