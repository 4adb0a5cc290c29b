"""Host logic of the FP64 tiles' launch geometry (csrc/geometry.h), compiled with g++: the
default tile covers the grid, and its modelled time is the least over the alternatives; the
batched rows are the cheapest."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2402_03074_gb300", "csrc")
DRIVER = r"""
#include <cstdio>
#include <vector>
#include "geometry.h"
int main() {
  char op;
  while (std::scanf(" %c", &op) == 1) {
    if (op == 'D') {
      int nx, ny, sms;
      if (std::scanf("%d %d %d", &nx, &ny, &sms) != 3) return 2;
      const int bx[3] = {32, 64, 96}, slots[3] = {sms, sms, sms};
      const hw::Tile64 t = hw::default_tile64(nx, ny, sms, bx, slots, 3);
      const hw::Geom2D g = hw::geom2d(nx, ny, t.bx, sms, t.rows, 0, false);
      std::printf("%d %d %d %d %d %d %d %d\n", t.bx, t.rows, g.bands, g.wout, g.chunks, g.rows, g.seg, g.blocks);
    } else if (op == 'B') {
      int n, bx, slots, per;
      if (std::scanf("%d %d %d %d", &n, &bx, &slots, &per) != 4) return 2;
      std::vector<int> b(n), w(n), y(n);
      for (int s = 0; s < n; ++s)
        if (std::scanf("%d %d %d", &b[s], &w[s], &y[s]) != 3) return 2;
      std::printf("%d\n", hw::batch_rows64(b.data(), w.data(), y.data(), n, bx, slots, per));
    } else {
      return 3;
    }
  }
  return 0;
}
"""
BY = {32: 8, 64: 4, 96: 2}


@pytest.fixture(scope="module")
def geo(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("tile64")
    src, exe = d / "driver.cc", d / "driver"
    src.write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o",
                    str(exe)], check=True)

    def run(lines):
        r = subprocess.run([str(exe)], input="\n".join(lines) + "\n", capture_output=True,
                           text=True, check=True)
        return [list(map(int, ln.split())) for ln in r.stdout.strip().splitlines()]
    return run


def _time(warps, by, rows, per, step=4.6):
    full, rest = divmod(rows + 2, by)
    w = warps * per
    last = 0.5 * step if rest == 1 else (max(step, w * rest) if rest else 0.0)
    t = full * max(step, w * by) + last - 1.08 * w
    return max(t, step * (full + (1.0 if rest > 1 else 0.5 * rest)))


def test_default_tile_covers_the_grid(geo):
    rng = np.random.default_rng(5)
    grids = [(2, 2), (30, 1000), (1000, 2), (40, 40), (240, 240), (2048, 2048), (5000, 3)]
    grids += [tuple(int(v) for v in np.exp(rng.uniform(0.7, 8.3, 2)).astype(int)) for _ in range(200)]
    out = geo([f"D {nx} {ny} 152" for nx, ny in grids])
    for (nx, ny), (bx, rows, bands, wout, chunks, crows, seg, blocks) in zip(grids, out):
        assert bx in BY and 1 <= wout <= bx - 2
        assert bands * wout >= nx and (bands - 1) * wout < nx
        if seg:
            assert rows == -seg and blocks * seg >= bands * ny and (blocks - 1) * seg < bands * ny
        else:
            assert chunks * crows >= ny and (chunks - 1) * crows < ny and blocks == bands * chunks
    by_grid = dict(zip(grids, out))
    assert by_grid[(240, 240)][:6] == [32, 13, 8, 30, 19, 13]
    assert by_grid[(2048, 2048)][0] == 96 and by_grid[(2048, 2048)][6] == 297
    assert by_grid[(40, 40)][0] == 32


def test_batched_rows_are_the_cheapest(geo):
    rng = np.random.default_rng(9)
    sets = []
    for _ in range(30):
        n = int(rng.integers(1, 9))
        per = int(rng.integers(1, 3))
        sets.append((n, 64, 152 * per, per, [(int(rng.integers(1, 18)), int(rng.integers(1, 3)),
                                   int(rng.integers(2, 400))) for _ in range(n)]))
    got = geo(["B %d %d %d %d %s" % (n, bx, sl, per, " ".join(f"{b} {w} {y}" for b, w, y in g))
               for n, bx, sl, per, g in sets])
    for (n, bx, slots, per, g), (r,) in zip(sets, got):
        def cost(q):
            items = sum(b * math.ceil(y / q) for b, _, y in g)
            return math.ceil(items / slots) * max(_time(w, BY[bx], min(q, y), per) for _, w, y in g)
        best = min(cost(q) for q in range(1, max(y for _, _, y in g) + 1))
        assert cost(r) == pytest.approx(best, rel=1e-12)
