"""The no-allocation entry point on the host side: a C++ program whose own operator new counts every
heap allocation made by the library (the program's definition takes the place of the library's)
calls hweno_stage_batch_static after a first call has set the device up; the count stays zero in
both precisions and for one solve as for the largest batch."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CLIENT = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include "hweno.h"
static bool counting = false;
static long allocations = 0;
void* operator new(std::size_t n) {
  if (counting) ++allocations;
  void* p = std::malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

int main() {
  for (int precision = 0; precision < 2; ++precision) {
    const int N = HWENO_STATIC_BATCH_MAX;
    hweno_problem p[N];
    double *in[N], *vh[N], *out[N], *a[N], *b[N], *dt[N];
    uint32_t* st[N];
    for (int s = 0; s < N; ++s) {
      std::memset(&p[s], 0, sizeof p[s]);
      p[s].dim = 2; p[s].equation = HWENO_BURGERS;
      p[s].nx = 20 + s; p[s].ny = 40 + s;
      p[s].x1 = p[s].nx; p[s].y1 = p[s].ny; p[s].gamma = 1.4;
      p[s].cfl = 0.6; p[s].precision = precision ? HWENO_MIXED32 : HWENO_FP64;
      p[s].gamma_lo = 1.0 / 400.0; p[s].eps = 1e-10;
      const size_t plane = sizeof(double) * p[s].nx * p[s].ny;
      if (cudaMalloc((void**)&in[s], 3 * plane) || cudaMalloc((void**)&vh[s], 2 * plane) ||
          cudaMalloc((void**)&out[s], 3 * plane) || cudaMalloc((void**)&a[s], 16) ||
          cudaMalloc((void**)&b[s], 16) || cudaMalloc((void**)&dt[s], 8) ||
          cudaMalloc((void**)&st[s], 4))
        return 2;
      cudaMemset(in[s], 0, 3 * plane);
      cudaMemset(vh[s], 0, 2 * plane);
      cudaMemset(a[s], 0, 16);
      cudaMemset(b[s], 0, 16);
      cudaMemset(dt[s], 0, 8);
      cudaMemset(st[s], 0, 4);
    }
    for (int n : {1, N}) {
      for (int rep = 0; rep < 2; ++rep) {
        allocations = 0;
        counting = rep == 1;
        for (int k = 1; k <= 3; ++k)
          if (hweno_stage_batch_static(n, p, k, in, in, vh, out, a, b, dt, st, nullptr) != HWENO_OK)
            return 3;
        counting = false;
      }
      std::printf("%ld\n", allocations);
    }
    if (cudaDeviceSynchronize() != cudaSuccess) return 4;
  }
  return 0;
}
"""


def test_static_batch_makes_no_heap_allocation(tmp_path):
    from paper_2402_03074_gb300 import build as B
    lib = B.build()
    src, exe = tmp_path / "client.cpp", tmp_path / "client"
    src.write_text(CLIENT)
    subprocess.run(["nvcc", "-std=c++17", "-O1", "-I",
                    os.path.join(ROOT, "include"), str(src), "-o", str(exe), lib, "-Xlinker",
                    "-rpath," + os.path.dirname(lib)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    assert [int(x) for x in r.stdout.split()] == [0, 0, 0, 0]
