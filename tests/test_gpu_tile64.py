"""The FP64 2D tiles (bx columns x several rows of threads) at their edges, for every equation,
against the oracle at the FP64 parity bar (1e-12 of the component's scale): grids one column
around a band and one row around the tile's rows, in the tile the launch chooses and in every
width a tuning table can ask for.  States vary little about a mean (see test_gpu_char64.py)."""
import numpy as np
import pytest

import oracle as O
from paper_2402_03074_gb300 import _binding as H
from gpu_helpers import gpu_stage, problems, rel_err

pytestmark = pytest.mark.gpu
EQ = {"adv": 0, "burg": 1, "euler": 2}


def _state(eq, nx, ny, seed):
    rng = np.random.default_rng(seed)
    nc = 4 if eq == "euler" else 1
    U = np.zeros((nc, 3, ny, nx))
    U[:, 0] = rng.uniform(0.8, 1.2, (nc, ny, nx))
    if eq == "euler":
        U[1:3, 0] -= 1.0
        U[3, 0] += 1.7
    U[:, 1:] = rng.uniform(-0.01, 0.01, (nc, 2, ny, nx))
    return U


def _check(eq, ch, nx, ny, bc, k):
    op, hp = problems(2, eq, nx, ny, bc=bc, characteristic=ch)
    U = _state(eq, nx, ny, 3 * nx + ny)
    Un = U if k == 1 else _state(eq, nx, ny, nx + ny)
    Vh = np.random.default_rng(nx).uniform(-0.05, 0.05, (U.shape[0], 2, ny, nx))
    a = O.alpha(op, U)
    dt = 0.2 / 64.0 / a.sum()
    ref, vref, st = O.stage(op, k, U, Un, Vh if k > 1 else None, a, dt)
    assert st == 0
    got, vgot, aout, status = gpu_stage(hp, k, U, Un, Vh, a, dt)
    assert status == 0
    assert rel_err(got, ref, U) <= 1e-12
    if k == 1:
        assert np.abs(vgot - vref).max() <= 1e-12 * np.abs(U).max()
    return got


@pytest.mark.parametrize("eq,ch", [("adv", 0), ("burg", 0), ("euler", 0), ("euler", 1)])
@pytest.mark.parametrize("nx,ny,bc,k", [
    (2, 2, 0, 1), (29, 5, 1, 2), (30, 6, 0, 1), (31, 7, (2, 1, 1, 2), 3), (60, 8, 2, 1), (61, 13, 0, 2),
    (100, 1000, 1, 1), (700, 9, (1, 1, 2, 2), 1)])
def test_default_tile(eq, ch, nx, ny, bc, k):
    _check(eq, ch, nx, ny, bc, k)


@pytest.mark.parametrize("eq,ch", [("adv", 0), ("burg", 0), ("euler", 0), ("euler", 1)])
def test_every_width_and_chunk_height(tmp_path, eq, ch):
    """Chunks of 1, 2, 3 and 8 rows and segments, in every width: the same bits (the decomposition
    changes no cell's arithmetic), at 1e-12 of the oracle."""
    import torch
    name = torch.cuda.get_device_name(0).replace(" ", "_")
    nx, ny = 131, 11
    path = str(tmp_path / "t.txt")

    def entry(rows, width):
        with open(path, "w") as f:
            f.write(f"{name} {EQ[eq]} {ch} 0 {nx} {ny} {rows} 0 {width} 0\n")
        assert H.hweno_tuning_load(path) == 1

    ref = _check(eq, ch, nx, ny, 2, 1)
    try:
        for width in (64, 96, 128, 192):
            for rows in (1, 2, 3, 8, -5, -23):
                entry(rows, width)
                np.testing.assert_array_equal(_check(eq, ch, nx, ny, 2, 1), ref)
    finally:
        entry(0, 0)


def test_an_overflowed_sound_speed_stays_infinite():
    """gamma (gamma - 1) e / rho beyond the double range at finite, admissible averages (a uniform
    state at rest, linear weights, dt = 0): the output's wave speeds are infinite, not lost."""
    _, hp = problems(2, "euler", 9, 7, characteristic=0, weights=2)
    U = np.zeros((4, 3, 7, 9))
    U[0, 0], U[3, 0] = 1e-10, 1e300
    out, _, speeds, status = gpu_stage(hp, 1, U, U, np.zeros((4, 2, 7, 9)), (1.0, 1.0), 0.0)
    assert status == 0 and np.array_equal(out[:, 0], U[:, 0])
    assert np.isposinf(speeds).all()
