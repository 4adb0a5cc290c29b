// f64_ops.cuh -- FP64 arithmetic in the form the FP64 unit takes fastest.
//
// The unit needs 16 clocks per warp for a DFMA whose three operands are vector registers and 19
// for a DADD, a DMUL or a DFMA with a constant or uniform operand (measured: 2.00 and 1.68
// lanes per clock and SM, from four warps per SM on).  So the FP64-bound kernels do every
// operation as a three-register DFMA: a + b = a 1 + b and a b = a b + (-0), both exact, with 1
// and -0 held in registers, and constants read from a table in shared memory at each use,
// through an address that depends on the thread (a provably uniform one would end in a uniform
// register).  Characteristic FP64 Euler, 2048^2 stage: 21.2 ms with plain operators, 18.8 ms so.
#pragma once
#include <cuda_runtime.h>

#include "rcp64.h"

namespace hw {

struct Ops {
  double one, nz;
  unsigned tab;  // shared address of the table
  template <int I>
  __device__ __forceinline__ double k() const {
    double v;  // volatile: a constant is loaded where it is used, not kept in registers
    asm volatile("ld.shared.f64 %0, [%1+%2];" : "=d"(v) : "r"(tab), "n"(8 * I));
    return v;
  }
  __device__ __forceinline__ double add(double a, double b) const { return fma(a, one, b); }
  __device__ __forceinline__ double sub(double a, double b) const { return fma(-b, one, a); }
  __device__ __forceinline__ double mul(double a, double b) const { return fma(a, b, nz); }
};

// The operations on the table `tab` (entries One and MinusZero hold 1 and -0), which a barrier has
// made visible to the thread.  k is the stage number, at most 3: k >> 2 is 0 for every thread,
// which the compiler cannot prove.
template <int One, int MinusZero>
__device__ __forceinline__ Ops make_ops(const double* tab, int k) {
  // the reads below are volatile and follow this statement, which no memory access crosses: none
  // moves above the barrier after the table's filling
  asm volatile("" : : : "memory");
  Ops o;
  o.tab = (unsigned)__cvta_generic_to_shared(tab) + (unsigned)((k >> 2) * (int)threadIdx.x);
  o.one = o.k<One>();
  o.nz = o.k<MinusZero>();
  return o;
}

// 1/x of a normal double with exponent field in [1, 2044], from the hardware's reciprocal of about
// 20 bits (its residual e = 1 - x y is below 2^-19.9, measured over all the leading words it looks
// at), by the first terms of the geometric series 1/(1 - e) = 1 + e + e^2 + ..  On integers (rcp64.h),
// within 0.51 ulp, where many warps share the FP64 unit: about 30 integer instructions instead of
// three FP64 operations, 1/40 of a 2D Euler cell's time (2048^2 step 56.5 -> 55.1 ms, 768^2
// component-wise 5.50 -> 5.30 ms).
__device__ __forceinline__ double rcp_in_range(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return rcp64_refine(x, y);
}
// The same in three FMAs, within 0.51 ulp, for the 1D kernels' lone warps and the FP32-bulk kernels.
__device__ __forceinline__ double rcp_in_range(const Ops& o, double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, o.one);  // y / (1 - e) = y (1 + e + e^2 + ..)
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ bool rcp_applies(double x) {
  const int eb = (__double2hiint(x) >> 20) & 0x7ff;
  return eb >= 1 && eb <= 2044;
}
__device__ __forceinline__ double rcp_any(double x) {
  return rcp_applies(x) ? rcp_in_range(x) : 1.0 / x;
}
__device__ __forceinline__ double rcp_any(const Ops& o, double x) {
  return rcp_applies(x) ? rcp_in_range(o, x) : 1.0 / x;
}

// 1/sqrt(x): the hardware's 20-bit value y refined by the first three terms of the binomial series
// of (1 - e)^(-1/2) = 1 + e/2 + 3 e^2/8 + .., e = 1 - x y^2 (the next, 5 e^3/16, is below 2^-58);
// the library's where x is near the ends of the range or not positive.  Within 1 ulp (measured
// 0.99; the rounding of x y shows in e).  half and c38: 1/2 and 3/8.
__device__ __forceinline__ bool root_applies(double x) {
  const int eb = __double2hiint(x) >> 20;
  return eb >= 64 && eb <= 1983;
}
__device__ __forceinline__ double rsqrt_any(const Ops& o, double x, double half, double c38) {
  if (!root_applies(x)) return rsqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-o.mul(x, y), y, o.one);
  return fma(o.mul(y, e), fma(c38, e, half), y);
}

// sqrt(x): g = x y refined by the same series, then by one step of Newton's iteration with the
// exact residual, s + (x - s^2) y/2 (y/2 by its exponent field): within 0.501 ulp (the library's bits
// in 2^20 values of the whole range), for the wave speeds that set alpha and dt.  One FP64
// operation more than x rsqrt_any(x), which would be within 2 ulp.
__device__ __forceinline__ double sqrt_any(const Ops& o, double x, double half, double c38) {
  if (!root_applies(x)) return sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double g = o.mul(x, y), e = fma(-g, y, o.one);
  const double s = fma(o.mul(g, e), fma(c38, e, half), g);
  const double yh = __hiloint2double(__double2hiint(y) - 0x100000, __double2loint(y));
  return fma(fma(-s, s, x), yh, s);
}

}  // namespace hw
