"""The FP64 1D layouts -- four lanes per cell (short grids) and one thread per cell -- at the edges
of their blocks, against the oracle at the FP64 parity bar (1e-12 of the component's scale), and
against each other: they do the same operations, so their results are the same bits.  States
vary little about a mean (see test_gpu_char64.py)."""
import numpy as np
import pytest

import oracle as O
from paper_2402_03074_gb300 import _binding as H
from gpu_helpers import gpu_stage, problems, rel_err

pytestmark = pytest.mark.gpu
EQ = {"adv": 0, "burg": 1, "euler": 2}
CLASSES = [("adv", 0), ("burg", 0), ("euler", 0), ("euler", 1)]


def _state(eq, nx, seed):
    rng = np.random.default_rng(seed)
    nc = 3 if eq == "euler" else 1
    U = np.zeros((nc, 2, 1, nx))
    U[:, 0] = rng.uniform(0.8, 1.2, (nc, 1, nx))
    if eq == "euler":
        U[1, 0] -= 1.0
        U[2, 0] += 1.7
    U[:, 1] = rng.uniform(-0.01, 0.01, (nc, 1, nx))
    return U


def _check(eq, ch, nx, bc, k, weights=0):
    op, hp = problems(1, eq, nx, bc=bc, characteristic=ch, weights=weights)
    U = _state(eq, nx, nx + k)
    Un = U if k == 1 else _state(eq, nx, nx + 17)
    Vh = np.random.default_rng(nx).uniform(-0.05, 0.05, (U.shape[0], 1, 1, nx))
    a = O.alpha(op, U)
    dt = 0.2 / 64.0 / a[0]
    ref, vref, st = O.stage(op, k, U, Un, Vh if k > 1 else None, a, dt)
    assert st == 0
    got, vgot, aout, status = gpu_stage(hp, k, U, Un, Vh, a, dt)
    assert status == 0
    assert rel_err(got, ref, U) <= 1e-12
    if k == 1:
        assert np.abs(vgot - vref).max() <= 1e-12 * np.abs(U).max()
    assert np.allclose(aout[0], O.alpha(op, ref)[0], rtol=1e-13)
    return got


@pytest.mark.parametrize("eq,ch", CLASSES)
@pytest.mark.parametrize("nx,bc,k,weights", [
    (2, 0, 1, 0), (3, 2, 2, 0), (29, 1, 3, 0), (30, 0, 1, 1), (31, 2, 1, 0), (60, 1, 2, 2), (61, 0, 3, 0),
    (480, 2, 1, 0), (481, 0, 2, 0), (4560, 1, 1, 0), (4561, 0, 1, 0), (5001, 2, 3, 0)])
def test_default_layout(eq, ch, nx, bc, k, weights):
    _check(eq, ch, nx, bc, k, weights)


@pytest.mark.parametrize("eq,ch", CLASSES)
def test_layouts_give_the_same_bits(tmp_path, eq, ch):
    import torch
    name = torch.cuda.get_device_name(0).replace(" ", "_")
    nx = 97
    path = str(tmp_path / "t.txt")

    def entry(width, lanes):
        with open(path, "w") as f:
            f.write(f"{name} {EQ[eq]} {ch} 0 {nx} 1 0 0 {width} {lanes}\n")
        assert H.hweno_tuning_load(path) == 1

    try:
        for bc in (0, 1, 2):
            ref = _check(eq, ch, nx, bc, 2)
            for width, lanes in ((32, 1), (128, 1), (32, 4), (64, 4), (128, 4)):
                entry(width, lanes)
                np.testing.assert_array_equal(_check(eq, ch, nx, bc, 2), ref)
            entry(0, 0)
    finally:
        entry(0, 0)
