// FP64 helpers that spend few FP64 instructions (two a clock and SM on GB300):
// comparisons as integers, and the reciprocal and roots by Halley's third-order
// iteration from the FP32 unit's approximation (relative error e0 < 2^-21; the
// step leaves a relative error of order e0^3 < 2^-63 beside its own roundings).
// Published method: E. Halley (1694); cubic forms of Newton-Raphson reciprocal
// and reciprocal square root as in J.-M. Muller, Elementary Functions, ch. 9.
// Arguments outside the positive normal range take the CUDA functions.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace dgswe {

__device__ __forceinline__ bool pos_normal(double x) {
  return (unsigned)__double2hiint(x) - 0x00100000u < 0x7fe00000u;
}
// max(x, y) for y > 0: a positive double orders as its bits, a negative one below
__device__ __forceinline__ double max_pos(double x, double y) {
  return __longlong_as_double(max(__double_as_longlong(x), __double_as_longlong(y)));
}
// bits whose signed order is that of the values
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ (long long)((unsigned long long)(b >> 63) >> 1);
}
__device__ __forceinline__ double min_f64(double x, double y) { return order_key(x) < order_key(y) ? x : y; }
__device__ __forceinline__ double max_f64(double x, double y) { return order_key(x) < order_key(y) ? y : x; }

// x = m 2^k with m in [1, 2) (EVEN: k even, m in [1, 4)): m rounded down to a float.
template <bool EVEN>
__device__ __forceinline__ float split_exp(double x, int& k) {
  const int hi = __double2hiint(x);
  k = (hi >> 20) - 1023;
  if (EVEN) k &= ~1;
  const int mh = hi - ((k + 1023 - 127) << 20);  // exponent biased by 127
  return __uint_as_float(__funnelshift_l((unsigned)__double2loint(x), (unsigned)mh, 3));
}
// the float f in (2^-2, 2) times 2^k, as a double
__device__ __forceinline__ double join_exp(float f, int k) {
  const unsigned b = __float_as_uint(f);
  return __hiloint2double((int)(b >> 3) + ((k + 1023 - 127) << 20), (int)(b << 29));
}

__device__ __forceinline__ double rcp_pos(double x) {
  if (!pos_normal(x)) return 1.0 / x;
  int k;
  const float m = split_exp<false>(x, k);
  if (k > 1000) return 1.0 / x;  // the start would be subnormal
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(m));
  const double y = join_exp(r, -k);
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
// 1 / sqrt(x) and sqrt(x)
__device__ __forceinline__ double rsqrt_pos(double x) {
  if (!pos_normal(x)) return rsqrt(x);
  int k;
  const float m = split_exp<true>(x, k);
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(m));
  const double y = join_exp(r, -(k >> 1));
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double sqrt_pos(double x) {
  if (!pos_normal(x)) return sqrt(x);
  int k;
  const float m = split_exp<true>(x, k);
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(m));
  const double y = join_exp(r, -(k >> 1));
  const double s = x * y;
  const double e = fma(-s, y, 1.0);
  return fma(s * e, fma(0.375, e, 0.5), s);
}

}  // namespace dgswe
