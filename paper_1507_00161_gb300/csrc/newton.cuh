// FP64 division, reciprocal and square root for latency, with the results of the library's, shared by
// the Jacobi kernels.  One FP64 instruction of a warp takes 64 clocks here whatever follows it, so a
// dependent operation less is what counts (measured: division 564 -> 364 clocks, root 598 -> 430).
#pragma once
#include <cuda_runtime.h>

namespace dmrg {

// Quotient, reciprocal and square root, rounded to nearest, by Newton's iteration with a final
// correction from the exact remainder (P. Markstein, IBM J. Res. Dev. 34 (1990) 111): from a 2^-23
// seed one step gives a reciprocal good to 2^-46 and, with the remainder, a result good to ~2^-90
// before its one rounding.  Operands in 2^-400 .. 2^400.
__device__ __forceinline__ int exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ bool mid_range(double x) {
  const int e = exponent(x);
  return e > 623 && e < 1423;
}
__device__ __forceinline__ bool is_zero(double x) {
  return ((__double2hiint(x) & 0x7fffffff) | __double2loint(x)) == 0;
}
__device__ __forceinline__ double times_pow2(double x, int e) {   // x and the result normal
  return __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x));
}
__device__ __forceinline__ double flip_if(double x, bool neg) {
  return __hiloint2double(__double2hiint(x) ^ (neg ? int(0x80000000) : 0), __double2loint(x));
}
__device__ __forceinline__ double quick_rcp_step(double b) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
  return fma(fma(-b, y, 1.0), y, y);
}
__device__ __forceinline__ double quick_div(double a, double b) {
  const double y = quick_rcp_step(b), q = a * y;
  return fma(fma(-b, q, a), y, q);
}
__device__ __forceinline__ double quick_rcp(double b) {
  const double y = quick_rcp_step(b);
  return fma(fma(-b, y, 1.0), y, y);
}
__device__ __forceinline__ double quick_sqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double g = x * y, h = times_pow2(y, -1);
  const double e = fma(-g, h, 0.5);
  g = fma(g, e, g);
  h = fma(h, e, h);
  return fma(fma(-g, g, x), h, g);
}

}  // namespace dmrg
