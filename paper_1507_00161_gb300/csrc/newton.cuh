// FP64 division, reciprocal and square root for latency, shared by the Jacobi kernels (the Ritz problem
// and the SVD).  One FP64 instruction of a warp takes 64 clocks here whatever follows it, so a
// dependent operation less is what counts (measured: division 564 -> 364 clocks, root 598 -> 430).
#pragma once
#include <cuda_runtime.h>

namespace dmrg {

// Quotient, reciprocal and square root by Newton's iteration with a final correction from the
// remainder, formed by a fused multiply-add (P. Markstein, IBM J. Res. Dev. 34 (1990) 111).  The seed
// instructions read the upper 32 bits of their operand and give the upper 32 bits of a result, so a
// seed is good to 2^-19 (two cuts at a 20-bit mantissa); one step gives 2^-38, and the correction a
// value good to 2^-75 before its one rounding.  That rounds to nearest unless the exact value lies
// within 2^-75 of the middle between two numbers (at most one operand in 2^21); there the result may
// be the other neighbour, one unit in the last place from the library's.  Operands in 2^-399 .. 2^400.
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
