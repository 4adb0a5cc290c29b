"""The tile rule (csrc/geometry.h) with FP32-bulk tiles and several blocks per SM, compiled with g++:
the chosen tile covers the grid, and no other width or chunk height it may choose from has a smaller
modelled time by more than the rule's margin of 0.5 %."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2402_03074_gb300", "csrc")
DRIVER = r"""
#include <cstdio>
#include "geometry.h"
int main() {
  int nx, ny, sms, per, mixed;
  while (std::scanf("%d %d %d %d %d", &nx, &ny, &sms, &per, &mixed) == 5) {
    const int bx[3] = {32, 64, 96}, slots[3] = {sms * per, sms * per, sms * per};
    const hw::Tile64 t = hw::default_tile64(nx, ny, sms, bx, slots, 3, mixed != 0);
    const hw::Geom2D g = hw::geom2d(nx, ny, t.bx, sms * per, t.rows, 0, false);
    std::printf("%d %d %d %d %d %d %d %d\n", t.bx, t.rows, g.bands, g.wout, g.chunks, g.rows, g.seg, g.blocks);
  }
  return 0;
}
"""
BY = {0: {32: 8, 64: 4, 96: 2}, 1: {32: 6, 64: 3, 96: 2}}
STEP = {0: 4.6, 1: 7.0}


def _sweep(warps, by, rows, blocks, step):
    full, rest = divmod(rows + 2, by)
    w = warps * blocks
    last = 0.5 * step if rest == 1 else (max(step, w * rest) if rest else 0.0)
    t = full * max(step, w * by) + last - 1.08 * w
    return max(t, step * (full + (1.0 if rest > 1 else 0.5 * rest)))


def _launch(bx, rows, pieces, blocks, warps, sms, per, mixed):
    """Modelled time of `blocks` blocks of `rows` rows in `pieces` pieces."""
    waves, rest = divmod(blocks, sms * per)
    by, step = BY[mixed][bx], STEP[mixed]
    t = waves * _sweep(warps, by, rows, per, step)
    if rest:
        t += _sweep(warps, by, rows, -(-rest // sms), step)
    return t + (waves + (rest > 0)) * 2.5 + (pieces - 1) * (2.5 + 0.92 * warps * per)


@pytest.mark.parametrize("mixed,per", [(1, 2), (1, 3), (0, 2), (1, 1)])
def test_chosen_tile_covers_and_costs_least(tmp_path, mixed, per):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "driver.cc", tmp_path / "driver"
    src.write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o",
                    str(exe)], check=True)
    rng = np.random.default_rng(10 * mixed + per)
    grids = [(2, 2), (30, 1000), (1000, 2), (40, 40), (2048, 2048), (5000, 3)]
    grids += [tuple(int(v) for v in np.exp(rng.uniform(0.7, 8.0, 2))) for _ in range(150)]
    grids = [(max(2, a), max(2, b)) for a, b in grids]
    sms = 152
    r = subprocess.run([str(exe)], input="".join(f"{a} {b} {sms} {per} {mixed}\n" for a, b in grids),
                       capture_output=True, text=True, check=True)
    out = [list(map(int, ln.split())) for ln in r.stdout.strip().splitlines()]
    assert len(out) == len(grids)
    for (nx, ny), (bx, rows, bands, wout, chunks, crows, seg, blocks) in zip(grids, out):
        assert bx in BY[mixed] and 1 <= wout <= bx - 2
        assert bands * wout >= nx and (bands - 1) * wout < nx
        warps = (wout + 2 + 31) // 32
        if seg:
            assert rows == -seg and blocks * seg >= bands * ny and (blocks - 1) * seg < bands * ny
            mine = _launch(bx, seg, -(-(seg - 1 + ny) // ny), blocks, warps, sms, per, mixed)
        else:
            assert chunks * crows >= ny and (chunks - 1) * crows < ny and blocks == bands * chunks
            mine = _launch(bx, crows, 1, blocks, warps, sms, per, mixed)
        for b in BY[mixed]:
            nb = -(-nx // (b - 2))
            w = -(-nx // nb)
            nb = -(-nx // w)
            wp = (w + 2 + 31) // 32
            for h in range(1, min(16, ny) + 1):
                other = _launch(b, h, 1, nb * -(-ny // h), wp, sms, per, mixed)
                assert mine <= other * 1.0051 + 1e-9, (nx, ny, bx, rows, b, h)
