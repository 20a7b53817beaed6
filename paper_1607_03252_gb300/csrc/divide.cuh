// FP64 quotients and reciprocals for the operator set-up, which is bound by the FP64 pipe: GB300 runs
// FP64 at 1/64 of the FP32 rate, so every operation counts. Newton's iteration from an FP32
// reciprocal with a final residual correction (P. W. Markstein, IBM J. Res. Dev. 34, 1990): y0 = the
// hardware's FP32 reciprocal of the truncated d (relative error below 2^-22), y = y0 + y0 (1 - d y0)
// (2^-44), q = n y, q + (n - d q) y: before its last rounding the quotient is within 2^-88 of n / d,
// so it is the correctly rounded one except next to a tie. Five operations (a reciprocal four); the
// conversions run on the integer pipe. Operands whose magnitude leaves 2^-100 .. 2^100 take the
// language's division.
#pragma once
#include <cuda_runtime.h>

namespace mlmc {

#if defined(__CUDA_ARCH__)
// biased exponent of |d| within 100 of 1
__device__ __forceinline__ bool div_in_range(double d) {
  return (((unsigned)__double2hiint(d) >> 20) & 0x7ffu) - 923u <= 200u;
}
// FP32 reciprocal of d in range, as an FP64 value
__device__ __forceinline__ double div_start(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const float f = __uint_as_float((hi & 0x80000000u) | (((hi & 0x7fffffffu) - (896u << 20)) << 3) | (lo >> 29));
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
  const unsigned b = __float_as_uint(y);
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}
__device__ __forceinline__ double divide(double n, double d) {
  if (!(div_in_range(n) && div_in_range(d))) return __ddiv_rn(n, d);
  const double y0 = div_start(d), y = fma(y0, fma(-d, y0, 1.0), y0), q = n * y;
  return fma(fma(-d, q, n), y, q);
}
__device__ __forceinline__ double reciprocal(double d) {
  if (!div_in_range(d)) return 1.0 / d;
  const double y0 = div_start(d), y = fma(y0, fma(-d, y0, 1.0), y0);
  return fma(y, fma(-d, y, 1.0), y);
}
// 2 a b / (a + b): seven operations (the doubling of a b in its exponent)
__device__ __forceinline__ double harmonic(double a, double b) {
  const double m = __dmul_rn(a, b), s = __dadd_rn(a, b);
  if (!(div_in_range(m) && div_in_range(s))) return __ddiv_rn(__dmul_rn(2.0 * a, b), s);
  return divide(__hiloint2double(__double2hiint(m) + (1 << 20), __double2loint(m)), s);
}
#else
inline double divide(double n, double d) { return n / d; }
inline double reciprocal(double d) { return 1.0 / d; }
inline double harmonic(double a, double b) { return (2.0 * a * b) / (a + b); }
#endif
__host__ __device__ __forceinline__ float reciprocal(float d) { return 1.0f / d; }

}  // namespace mlmc
