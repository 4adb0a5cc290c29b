"""The integer reciprocal (csrc/rcp64.h), compiled with g++, over the whole of its stated precondition:
starting values with a residual up to 2^-19 on either side, against exact rational arithmetic, in
units in the last place of the result.

Tolerance: half an ulp for the rounding, e^3 < 2^-57 (at most 1/16 ulp) and the truncation of e
(1/128 ulp): below 0.58 ulp."""
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


@pytest.mark.parametrize("where", ["near one", "near two", "between"])
def test_reciprocal_up_to_the_stated_residual(tmp_path, where):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "driver.cc", tmp_path / "driver"
    src.write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o",
                    str(exe)], check=True)
    rng = random.Random(where)
    pairs = []
    while len(pairs) < 6000:
        m = {"near one": 1 + rng.random() * 2.0 ** -17, "near two": 2 - rng.random() * 2.0 ** -17,
             "between": rng.uniform(1, 2)}[where]
        x = math.ldexp(rng.choice([-1, 1]) * m, rng.choice([-1022, 1021, rng.randint(-1022, 1021)]))
        y = (1.0 / x) * (1.0 + rng.uniform(-1, 1) * 2.0 ** -19)
        fr, ex = math.frexp(y)
        y = math.ldexp(round(math.ldexp(fr, 21)), ex - 21)   # a low word of zero
        if abs(1 - F(x) * F(y)) < F(1, 2 ** 19) and (m < 1.5 or abs(y) >= math.ldexp(1, -math.frexp(x)[1])):
            pairs.append((x, y))
    r = subprocess.run([str(exe)], input="".join(f"{float.hex(x)} {float.hex(y)}\n" for x, y in pairs),
                       capture_output=True, text=True, check=True)
    got = [float.fromhex(ln) for ln in r.stdout.split()]
    assert len(got) == len(pairs)
    worst = max(abs(F(z) - 1 / F(x)) / F(math.ulp(z)) for (x, _), z in zip(pairs, got))
    assert worst <= F(58, 100), float(worst)
