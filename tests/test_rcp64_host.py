"""The reciprocal completed on integers (csrc/rcp64.h, the code the kernels run), compiled with g++,
against exact rational arithmetic, from starting values of both sides of the rounding to 20 bits.

Tolerance: one rounding (2^-53), e^3 < 2^-57 from a start with |e| < 2^-19, and three truncations of
at most 2^-55: below 1.9 2^-53."""
import math
import os
import random
import shutil
import subprocess
from fractions import Fraction as F

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2402_03074_gb300", "csrc")
DRIVER = r"""
#include <cstdio>
#include "rcp64.h"
int main() {
  double x, y;
  while (std::scanf("%la %la", &x, &y) == 2) std::printf("%a\n", hw::rcp64_refine(x, y));
  return 0;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("rcp64")
    src, exe = d / "driver.cc", d / "driver"
    src.write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o",
                    str(exe)], check=True)

    def call(lines):
        r = subprocess.run([str(exe)], input="\n".join(lines) + "\n", capture_output=True,
                           text=True, check=True)
        return [float.fromhex(ln) for ln in r.stdout.split()]
    return call


# mantissas of x: the ends of [1, 2), where the reciprocal crosses a power of two, and between
ENDS = [1.0, 1.0 + 2.0 ** -52, 1.0 + 2.0 ** -21, 1.0 + 2.0 ** -20, 2.0 - 2.0 ** -52, 2.0 - 2.0 ** -21]


@pytest.mark.parametrize("where", ["ends", "near one", "near two", "between"])
def test_reciprocal(run, where):
    rng = random.Random(where)
    high = lambda v: math.ldexp(math.floor(math.ldexp(math.frexp(v)[0], 21)), math.frexp(v)[1] - 21)
    pairs = []
    for _ in range(4000):
        m = {"ends": rng.choice(ENDS), "near one": 1 + rng.random() * 2.0 ** -19,
             "near two": 2 - rng.uniform(0.01, 1) * 2.0 ** -19, "between": rng.uniform(1, 1.99)}[where]
        x = math.ldexp(rng.choice([-1, 1]) * m, rng.choice([-1022, 1021, rng.randint(-1022, 1021)]))
        y = high(high(1.0 / x) * (1.0 + rng.choice([0.0, 2.0 ** -20])))
        pairs.append((x, y))
    got = run([f"{float.hex(x)} {float.hex(y)}" for x, y in pairs])
    assert len(got) == len(pairs)
    for (x, _), z in zip(pairs, got):
        assert abs(F(z) * F(x) - 1) <= F(19, 10) * F(1, 2 ** 53)
