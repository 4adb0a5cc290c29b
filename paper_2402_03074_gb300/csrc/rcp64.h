// rcp64.h -- a double's reciprocal completed on integers, in plain C++ that also compiles for the host
// (tests/test_rcp64_host.py).  An SM takes one FP64 instruction of a warp in 16 clocks but two
// 32-bit integer instructions in one, beside those of the other warps.
#pragma once
#include <cstring>
#if defined(__CUDACC__)
#define HW_RCP64 __host__ __device__ __forceinline__
#else
#define HW_RCP64 inline
#endif

namespace hw {

HW_RCP64 unsigned long long bits_of(double x) {
#if defined(__CUDA_ARCH__)
  return (unsigned long long)__double_as_longlong(x);
#else
  unsigned long long b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}
HW_RCP64 double from_bits(unsigned long long b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)b);
#else
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}

// 1/x of a normal double with exponent field in [1, 2044] from y, its reciprocal to about 20 bits
// (the low word of y is zero, |1 - x y| < 2^-19, and y is in the binade of 1/x or, for x next to a
// power of two, at its lower end): y (1 + e + e^2), e = 1 - x y, the first terms of the geometric
// series of 1/(1 - e), on the mantissas.  Within 0.58 ulp: a rounding, e^3 < 2^-57 (1/16 ulp) and
// the truncation of e (1/128 ulp).
HW_RCP64 double rcp64_refine(double x, double y) {
  const unsigned long long bx = bits_of(x);
  const unsigned hy = (unsigned)(bits_of(y) >> 32);
  const unsigned long long M = (bx & 0xfffffffffffffull) | 0x10000000000000ull;
  unsigned Y = (hy & 0xfffffu) | 0x100000u;  // 21 bits
  unsigned top = (hy & 0xfff00000u) - 0x100000u;
  // M Y is next to 2^73, but next to 2^72 where x is just above a power of two and y was not
  // rounded below one
  if ((M & 0x1ffff000000000ull) == 0x10000000000000ull && !(Y & 0x80000u)) {
    Y <<= 1;
    top -= 0x100000u;
  }
  const long long e = -(long long)(M * Y);  // 2^73 e: the product's upper bits are known
  const int eh = (int)(e >> 24);
  const long long e2 = e + (((long long)eh * eh) >> 25);     // 2^73 (e + e^2)
  const long long corr = ((long long)Y * (e2 >> 13)) >> 25;  // 2^35 Y (e + e^2)
  const unsigned long long Z = ((unsigned long long)Y << 35) + (unsigned long long)corr;  // 56 bits
  return from_bits(((Z + 4) >> 3) + ((unsigned long long)top << 32));
}

}  // namespace hw
