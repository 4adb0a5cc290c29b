"""The 2D tiles in FP32-bulk arithmetic at their edges, for every equation and weight, against the
FP64 oracle at the bound of that path (1e-5 of the component's scale, derived in
test_gpu_parity.py::test_mixed_precision_stage), and in both precisions the same bits in every width
(32 to 192 columns) and chunk height: the decomposition changes no cell's arithmetic.  States vary
little about a mean (see test_gpu_char64.py)."""
import numpy as np
import pytest

import oracle as O
from paper_2402_03074_gb300 import _binding as H
from gpu_helpers import gpu_stage, problems, rel_err
from test_gpu_tile64 import EQ, _state

pytestmark = pytest.mark.gpu
CLASSES = [("adv", 0), ("burg", 0), ("euler", 0), ("euler", 1)]
TOL = {H.HWENO_FP64: 1e-12, H.HWENO_MIXED32: 1e-5}


def _check(eq, ch, nx, ny, bc, k, weights=0, precision=H.HWENO_MIXED32):
    op, hp = problems(2, eq, nx, ny, bc=bc, characteristic=ch, weights=weights, precision=precision)
    U = _state(eq, nx, ny, 3 * nx + ny)
    Un = U if k == 1 else _state(eq, nx, ny, nx + ny)
    Vh = np.random.default_rng(nx).uniform(-0.05, 0.05, (U.shape[0], 2, ny, nx))
    a = O.alpha(op, U)
    dt = 0.2 / 64.0 / a.sum()
    ref, vref, st = O.stage(op, k, U, Un, Vh if k > 1 else None, a, dt)
    assert st == 0
    got, vgot, aout, status = gpu_stage(hp, k, U, Un, Vh, a, dt)
    assert status == 0
    assert rel_err(got, ref, U) <= TOL[precision]
    if k == 1:
        assert np.abs(vgot - vref).max() <= TOL[precision] * np.abs(U).max()
    return got


@pytest.mark.parametrize("eq,ch", CLASSES)
@pytest.mark.parametrize("nx,ny,bc,k,weights", [
    (2, 2, 0, 1, 0), (29, 4, 1, 2, 1), (30, 5, 0, 1, 2), (31, 6, (2, 1, 1, 2), 3, 0), (60, 7, 2, 1, 1),
    (62, 11, 0, 2, 2), (95, 13, (1, 2, 0, 0), 3, 0), (100, 1000, 1, 1, 0), (700, 9, (1, 1, 2, 2), 1, 0)])
def test_default_tile_fp32_bulk(eq, ch, nx, ny, bc, k, weights):
    _check(eq, ch, nx, ny, bc, k, weights)


@pytest.mark.parametrize("precision", [H.HWENO_FP64, H.HWENO_MIXED32])
@pytest.mark.parametrize("eq,ch", CLASSES)
def test_same_bits_in_every_width_and_chunk_height(tmp_path, eq, ch, precision):
    import torch
    name = torch.cuda.get_device_name(0).replace(" ", "_")
    nx, ny = 131, 11
    path = str(tmp_path / "t.txt")

    def entry(rows, bands, width):
        with open(path, "w") as f:
            f.write(f"{name} {EQ[eq]} {ch} {int(precision == H.HWENO_MIXED32)} {nx} {ny} {rows} {bands} "
                    f"{width} 0\n")
        assert H.hweno_tuning_load(path) == 1

    entry(0, 0, 0)
    ref = _check(eq, ch, nx, ny, 2, 2, precision=precision)
    try:
        for width in (32, 64, 96, 128, 192):
            for rows in (-1, 1, 2, 3, 8, -5, -23):
                entry(rows, -1, width)
                np.testing.assert_array_equal(
                    _check(eq, ch, nx, ny, 2, 2, precision=precision), ref)
    finally:
        entry(0, 0, 0)
