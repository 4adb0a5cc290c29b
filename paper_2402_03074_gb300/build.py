"""Build libhweno.so in-tree: nvcc for sm_103a, one translation unit per process, linked
into a shared library with the C ABI of include/hweno.h."""
from __future__ import annotations

import concurrent.futures as cf
import fcntl
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libhweno.so")
SOURCES = ["stage2d.cu", "stage2d_w96.cu", "stage2d_w64.cu", "stage2d_w192.cu", "stage2d_w32.cu",
           "stage1d.cu",
           "batch.cu", "static_batch.cu", "engine.cu", "server.cu", "tune.cu", "peaks.cu"]
HEADERS = ["hweno_device.cuh", "f64_ops.cuh", "rcp64.h", "launch.h", "server.h", "batch.h", "geometry.h",
           "stage1d_item.cuh", "stage1d_lanes64.cuh",
           "stage2d_item.cuh", "recon64.cuh", "stage2d_char64.cuh",
           "stage2d_comp64.cuh", "stage2d_tile64.cuh", "stage2d_impl.cuh"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-std=c++17", "-O3", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall",
              "-I" + os.path.join(ROOT, "include")]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile what is out of date.  Processes that build at the same time (one per rank of a
    multi-GPU launch) take turns on a lock file; the later ones find everything current."""
    os.makedirs(BUILD, exist_ok=True)
    with open(os.path.join(BUILD, ".lock"), "w") as lk:
        fcntl.flock(lk, fcntl.LOCK_EX)
        try:
            return _build(force, verbose)
        finally:
            fcntl.flock(lk, fcntl.LOCK_UN)


def _build(force: bool, verbose: bool) -> str:
    hdrs = [os.path.join(CSRC, h) for h in HEADERS] + [os.path.join(ROOT, "include", "hweno.h")]
    jobs = []
    objs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(BUILD, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + hdrs):
            jobs.append([_nvcc(), *ARCH, *NVCC_FLAGS, "-c", s, "-o", o])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        if verbose:
            sys.stdout.write(r.stdout + r.stderr)

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        for f in [ex.submit(run, j) for j in jobs]:
            f.result()
    if force or jobs or _stale(LIB, objs):
        tmp = LIB + f".tmp{os.getpid()}"
        run([_nvcc(), *ARCH, "-shared", "-o", tmp, *objs])
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
