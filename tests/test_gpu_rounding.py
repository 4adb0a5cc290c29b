"""Rounding of the FP64 stages: their rms error against the scheme in long double (the oracle's source
compiled with long double in the place of double: 80 or 128 bits), per class, on smooth waves and on
Riemann data; run with -s to print the figures.

Tolerance: a stage combines the state with three roundings of its scale at most (rms 2^-53 together),
and adds dt/h times differences of fluxes with some eight roundings each, dt/h at most 0.6 over the
speed they scale with: below 2 x 2^-53 of the component's largest average, averages and first
moments each."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

import oracle as O
from paper_2402_03074_gb300 import inputs as I
from gpu_helpers import gpu_stage, problems

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

ENTRY = r"""
int wide_stage(int dim, int eq, int nx, int ny, F64 x1, F64 y1, const int* bc, int ch, int k, const F64* Uin,
               const F64* Un, const F64* Vh, F64 a0, F64 a1, F64 dt, F64* hi, F64* lo) {
  orc_problem P;
  memset(&P, 0, sizeof P);
  P.dim = dim; P.eq = eq; P.nx = nx; P.ny = ny; P.x1 = x1; P.y1 = y1; P.ax = 1; P.ay = -(F64)0.7; P.gam = (F64)1.4;
  for (int i = 0; i < 4; ++i) P.bc[i] = bc[i];
  P.characteristic = ch; P.gamma_lo = (F64)1 / 400; P.eps = (F64)1e-10; P.cfl = (F64)0.6;
  const size_t N = (size_t)nx * ny * orc_ncomp(&P) * orc_nmom(&P);
  const size_t V = (size_t)nx * ny * orc_ncomp(&P) * (orc_nmom(&P) - 1);
  WIDE *a = malloc(sizeof(WIDE) * N), *b = malloc(sizeof(WIDE) * N), *c = malloc(sizeof(WIDE) * V),
       *o = malloc(sizeof(WIDE) * N);
  for (size_t i = 0; i < N; ++i) { a[i] = Uin[i]; b[i] = Un[i]; }
  for (size_t i = 0; i < V; ++i) c[i] = Vh[i];
  WIDE al[2] = {a0, a1};
  const int rc = orc_stage(&P, k, a, b, c, al, dt, o);
  for (size_t i = 0; i < N; ++i) { hi[i] = (F64)o[i]; lo[i] = (F64)(o[i] - (WIDE)hi[i]); }
  free(a); free(b); free(c); free(o);
  return rc;
}
"""


@pytest.fixture(scope="module")
def wide(tmp_path_factory):
    d = tmp_path_factory.mktemp("wide")

    def widen(name):
        s = open(os.path.join(ROOT, "oracle", name)).read()
        s = re.sub(r"(?<![\w.])(\d+\.\d*(?:[eE][+-]?\d+)?)(?![\w.])", r"\1L", s)
        s = re.sub(r"\bdouble\b", "WIDE", s)
        return re.sub(r"\b(fabs|sqrt|fmax|fmin|pow)\(", r"\1l(", s)
    head = "#ifndef WIDE\ntypedef double F64;\n#define WIDE long double\n#endif\n"
    (d / "hweno_oracle.h").write_text(head + widen("hweno_oracle.h"))
    (d / "wide.c").write_text(head + widen("hweno_oracle.c") + ENTRY)
    so = d / "wide.so"
    subprocess.run(["gcc", "-O2", "-std=gnu11", "-fopenmp", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    str(d), "-o", str(so), str(d / "wide.c"), "-lm"], check=True)
    L = ctypes.CDLL(str(so))

    def stage(op, k, Uin, Un, Vh, a, dt):
        f64 = ctypes.c_double
        arr = lambda x: x.ctypes.data_as(ctypes.POINTER(f64))
        hi, lo = np.empty_like(Uin), np.empty_like(Uin)
        Uin, Un, Vh = (np.ascontiguousarray(x) for x in (Uin, Un, Vh))
        bc = (ctypes.c_int * 4)(*op.bc)
        rc = L.wide_stage(op.dim, op.eq, op.nx, op.ny, f64(op.x1), f64(op.y1), bc, op.characteristic, k,
                          arr(Uin), arr(Un), arr(Vh), f64(a[0]), f64(a[1]), f64(dt), arr(hi), arr(lo))
        assert rc == 0
        return hi, lo
    return stage


def _initial(dim, eq, data, seed):
    if eq != "euler":
        U = (I.burgers_sine_1d(128) if dim == 1 else I.burgers_sine_2d(24)).U0.copy()
        U[:, 0] += 0.37 * (seed + 1)
        return U, 0
    if data == "riemann":
        w = I.shock_tube_1d(seed, n=128, t_end=1.0) if dim == 1 else I.quadrant_vortex_2d(seed, 24)
        return w.U0, 1
    return (I.euler_density_wave_1d(128) if dim == 1 else I.euler_density_wave_2d(24, k=0.5)).U0, 0


@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("eq,ch,data", [("adv", 0, "wave"), ("burg", 0, "wave"), ("euler", 0, "wave"),
                                        ("euler", 1, "wave"), ("euler", 0, "riemann"), ("euler", 1, "riemann")])
def test_rms_error_against_long_double(wide, dim, eq, ch, data):
    err = np.zeros(2)
    seeds = (0, 1, 2, 3) if dim == 1 else (0, 1)
    for seed in seeds:
        U, bc = _initial(dim, eq, data, seed)
        ny, nx = U.shape[2:]
        op, hp = problems(dim, eq, nx, ny, bc=bc, characteristic=ch, L=2.0)
        S = np.abs(U[:, 0]).max(axis=(1, 2)).reshape(-1, 1, 1)
        a = np.zeros(2)
        a[:] = O.alpha(op, U)
        dt = 0.6 * 2.0 / nx / a[:dim].sum()
        state, Vh = U, np.zeros((U.shape[0], dim, ny, nx))
        for k in (1, 2, 3):
            out, vh, aout, status = gpu_stage(hp, k, state, U, Vh, a, dt)
            assert status == 0
            hi, lo = wide(op, k, state, U, Vh, a, dt)
            e = (out - hi) - lo
            err += [np.mean((e[:, 0] / S) ** 2), np.mean((e[:, 1:] / S[:, None]) ** 2)]
            state, Vh, a = out, vh, aout
    err = np.sqrt(err / (3 * len(seeds)))
    print(f"\n{dim}D {eq} characteristic={ch} {data}: averages {err[0]:.2e}, first moments {err[1]:.2e}")
    assert (err <= 2.0 * 2.0 ** -53).all(), err
