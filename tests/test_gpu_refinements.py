"""The refined reciprocals and roots of csrc/f64_ops.cuh on the device, from the hardware's own
starting values, in units in the last place.

The hardware looks at the leading word alone, so all 2^20 leading mantissa words (roots: of both
exponent parities), each with the least, the largest and a random trailing word, cover every
starting value; the rest of the range (exponent ends, both sides of the cut-offs of the library
fallback, subnormals, zeros, infinities, NaN, both signs) is compared with CUDA's operations bit by
bit within one ulp.

Tolerances, with starting residuals e below 2^-19 (checked first): reciprocal in FMAs half an ulp
and e^3 < 2^-57 (1/16 ulp): 0.57; on integers also 1/128: 0.58; inverse root half an ulp, the
rounding of x y (half an ulp) and 5 e^3/16 (0.02): 1.03; root half an ulp, its correction's error
being some 2^-20 of an ulp: 0.501."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include "f64_ops.cuh"
using namespace hw;
__device__ Ops ops(double* tab) {
  if (threadIdx.x == 0) { tab[0] = 1.0; tab[1] = -0.0; }
  __syncthreads();
  return make_ops<0, 1>(tab, 1);
}
__device__ double ulp(double z) {  // z > 0, normal
  return __longlong_as_double(__double_as_longlong(z) + 1) - z;
}
__device__ void raise(double* m, double v) {
  if (!(v >= 0.0)) v = 1e9;
  atomicMax((unsigned long long*)m, (unsigned long long)__double_as_longlong(v));
}
// worst[0..1]: residuals of the starting values; [2] reciprocal on integers, [3] in FMAs, [4] inverse
// root, [5] root
__global__ void dense(double* worst) {
  __shared__ double tab[2];
  const Ops o = ops(tab);
  const unsigned n = blockIdx.x * blockDim.x + threadIdx.x;  // 2^20 threads
  for (int low = 0; low < 3; ++low)
    for (int ex = 1023; ex <= 1024; ++ex) {
      const unsigned lo = low == 0 ? 0u : (low == 1 ? 0xffffffffu : n * 2654435761u + 12345u);
      const double x = __hiloint2double((int)((unsigned)ex << 20 | n), (int)lo);
      double y;
      asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
      raise(&worst[0], fabs(fma(-x, y, 1.0)));
      const double a = rcp_any(x), b = rcp_any(o, x);
      raise(&worst[2], fabs(fma(-x, a, 1.0) / x) / ulp(a));
      raise(&worst[3], fabs(fma(-x, b, 1.0) / x) / ulp(b));
      asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
      const double q = y * y;  // 41 bits: exact
      raise(&worst[1], fabs(fma(-x, q, 1.0)));
      const double r = rsqrt_any(o, x, 0.5, 0.375), s = sqrt_any(o, x, 0.5, 0.375);
      const double p = x * r, pe = fma(x, r, -p);           // x r = p + pe
      const double res = fma(-p, r, 1.0) - pe * r;          // 1 - x r^2
      raise(&worst[4], fabs(0.5 * res * r) / ulp(r));
      raise(&worst[5], fabs(fma(-s, s, x) / (2.0 * s)) / ulp(s));
    }
}
__device__ long long distance(double a, double b) {
  if (isnan(a) && isnan(b)) return 0;
  const long long u = __double_as_longlong(a), v = __double_as_longlong(b);
  if ((u < 0) != (v < 0)) return 1ll << 60;
  return u > v ? u - v : v - u;
}
__global__ void whole(const double* x, int n, unsigned long long* far) {
  __shared__ double tab[2];
  const Ops o = ops(tab);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i];
  atomicMax(&far[0], (unsigned long long)distance(rcp_any(v), 1.0 / v));
  atomicMax(&far[1], (unsigned long long)distance(rcp_any(o, v), 1.0 / v));
  atomicMax(&far[2], (unsigned long long)distance(rsqrt_any(o, v, 0.5, 0.375), rsqrt(v)));
  atomicMax(&far[3], (unsigned long long)distance(sqrt_any(o, v, 0.5, 0.375), sqrt(v)));
}
int main() {
  const int n = 1 << 20;
  double *worst, *x;
  unsigned long long* far;
  if (cudaMallocManaged(&worst, 6 * 8) || cudaMallocManaged(&x, n * 8) ||
      cudaMallocManaged(&far, 4 * 8))
    return 2;
  memset(worst, 0, 48);
  memset(far, 0, 32);
  unsigned long long s = 88172645463325252ULL;
  const int edge[] = {0, 1, 2, 62, 63, 64, 65, 66, 1981, 1982, 1983, 1984, 1985, 2043, 2044, 2045, 2046, 2047};
  for (int i = 0; i < n; ++i) {
    s ^= s << 13; s ^= s >> 7; s ^= s << 17;
    unsigned long long b = s;
    if (i % 4 == 0) b = (b & 0x800fffffffffffffull) | (unsigned long long)edge[(i / 4) % 18] << 52;
    if (i % 8 == 1) b = (b & 0xfff00000000000ffull);                    // mantissas next to 1
    if (i % 8 == 2) b = b | 0x000ffffffffff000ull;                      // and next to 2
    if (i % 1024 == 3) b &= 0x8000000000000000ull;                      // zeros
    if (i % 1024 == 7) b = (b & 0x8000000000000000ull) | 0x7ff0000000000000ull;  // infinities
    memcpy(&x[i], &b, 8);
  }
  dense<<<(1 << 20) / 256, 256>>>(worst);
  whole<<<n / 256, 256>>>(x, n, far);
  if (cudaDeviceSynchronize() != cudaSuccess) return 3;
  for (int i = 0; i < 6; ++i) printf("%.17g ", worst[i]);
  for (int i = 0; i < 4; ++i) printf("%llu ", far[i]);
  return 0;
}
"""


def test_refinements_against_the_operations_they_stand_for(tmp_path):
    src, exe = tmp_path / "r.cu", tmp_path / "r"
    src.write_text(SRC)
    subprocess.run(["nvcc", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-I",
                    os.path.join(ROOT, "paper_2402_03074_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    v = r.stdout.split()
    seed_rcp, seed_rsqrt, rcp_int, rcp_fma, inv_root, root = map(float, v[:6])
    assert seed_rcp < 2.0 ** -19 and seed_rsqrt < 2.0 ** -19, (seed_rcp, seed_rsqrt)
    assert rcp_int <= 0.58 and rcp_fma <= 0.57, (rcp_int, rcp_fma)
    assert inv_root <= 1.03 and root <= 0.501, (inv_root, root)
    assert [int(t) <= bound for t, bound in zip(v[6:], (1, 1, 2, 1))] == [True] * 4, v[6:]
