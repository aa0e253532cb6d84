// FP64 operations by the cheapest pipe. On this part an FP64 operation costs a warp 64 clocks of its sub-partition
// (19 of the SM), a division nine times that, and a conversion between the floating types as much as an operation, while
// integer operations cost 2 clocks of the SM a warp.
#pragma once
#include <cuda_runtime.h>

namespace nlmg {

// 1 / x from the hardware's approximation (about 20 bits) and one third-order step, r (1 + e + e^2) with e = 1 - x r
// (the truncated geometric series: the remaining error e^3 is below 2^-60); x away from the ends of the exponent range.
__device__ __forceinline__ double rcp_core(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
// 2^-960 <= |x| <= 2^960: the core's range (a zero, an infinity or a NaN is outside)
__device__ __forceinline__ bool rcp_in_range(double x) {
  const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
  return ex - 63u < 1921u;
}
__device__ __forceinline__ double fast_rcp(double x) { return rcp_in_range(x) ? rcp_core(x) : 1.0 / x; }
// a / b: the reciprocal's quotient with its residual added back by a fused multiply-add (Markstein's correction; about half
// a division's chain of operations). Both operands in 2^-480 .. 2^480, so that the quotient is far from the ends of the
// range as well (an overflowing one would have an infinite residual), else the division.
__device__ __forceinline__ bool div_in_range(double x) {
  const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
  return ex - 543u < 961u;
}
__device__ __forceinline__ double fast_div(double a, double b) {
  if (!div_in_range(b) || !div_in_range(a)) return a / b;
  const double r = rcp_core(b), q = a * r;
  return fma(fma(-b, q, a), r, q);
}

// Exact double of a float, by its bits (a conversion instruction takes as long as an FP64 addition).
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f), ex = (b >> 23) & 0xffu;
  if (ex == 0u || ex == 255u) return (double)f;
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}
// Nearest float of a double (ties to even), by its bits where the result is a normal number.
__device__ __forceinline__ float narrow(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned ex = (unsigned)(b >> 52) & 0x7ffu;
  if (ex - 897u >= 253u) return (float)v;
  unsigned long long m = (b & 0x7fffffffffffffffull) - (896ull << 52);
  m += 0xfffffffull + ((m >> 29) & 1ull);
  return __uint_as_float((unsigned)(m >> 29) | ((unsigned)(b >> 32) & 0x80000000u));
}

}  // namespace nlmg
