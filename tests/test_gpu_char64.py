"""The characteristic FP64 2D Euler stage at the edges of its bands and chunks, against the
oracle: every stage, mixed boundary conditions, grids of one band and of ragged bands, through
the single-solve and the batched launches.  Tolerance: the FP64 parity bar of the other stage
tests (1e-12 of the component's scale per cell and moment).  The states vary by a third about a
mean, so that no reconstructed point comes near vacuum: there a flux m^2/rho amplifies rounding
without bound, and the oracle itself is further than 1e-12 from the scheme evaluated in 80-bit
arithmetic."""
import numpy as np
import pytest

import oracle as O
from paper_2402_03074_gb300 import _binding as H
from gpu_helpers import gpu_stage, problems, rel_err

pytestmark = pytest.mark.gpu


def _state(nx, ny, seed):
    rng = np.random.default_rng(seed)
    U = np.zeros((4, 3, ny, nx))
    U[0, 0] = rng.uniform(0.8, 1.2, (ny, nx))
    U[1, 0] = rng.uniform(-0.6, 0.6, (ny, nx))
    U[2, 0] = rng.uniform(-0.6, 0.6, (ny, nx))
    U[3, 0] = rng.uniform(2.5, 3.0, (ny, nx))
    U[:, 1:] = rng.uniform(-0.01, 0.01, (4, 2, ny, nx))
    return U


def _case(nx, ny, bc, k, weights):
    op, hp = problems(2, "euler", nx, ny, bc=bc, weights=weights)
    U = _state(nx, ny, nx * 7 + ny)
    Un = U if k == 1 else _state(nx, ny, nx + ny)
    Vh = np.random.default_rng(nx).uniform(-0.05, 0.05, (4, 2, ny, nx))
    a = O.alpha(op, U)
    dt = 0.2 / 64.0 / a.sum()
    ref, vref, st = O.stage(op, k, U, Un, Vh if k > 1 else None, a, dt)
    assert st == 0
    return hp, U, Un, Vh, a, dt, ref, vref


@pytest.mark.parametrize("nx,ny,bc,k,weights", [
    (2, 2, 0, 1, 0), (3, 2, (1, 1, 2, 2), 2, 0), (2, 5, 2, 3, 1), (61, 3, 0, 1, 0), (63, 4, 1, 2, 0),
    (93, 3, (2, 1, 1, 2), 1, 0), (94, 2, 0, 2, 0), (95, 5, 2, 1, 0), (96, 3, 1, 3, 2),
    (187, 4, 0, 1, 0), (188, 3, 2, 2, 0), (189, 2, (1, 2, 0, 0), 3, 0), (33, 311, (0, 0, 2, 1), 1, 0),
])
def test_stage_at_tile_edges(nx, ny, bc, k, weights):
    hp, U, Un, Vh, a, dt, ref, vref = _case(nx, ny, bc, k, weights)
    got, vgot, aout, status = gpu_stage(hp, k, U, Un, Vh, a, dt)
    assert status == 0
    assert rel_err(got, ref, U) <= 1e-12
    if k == 1:
        assert np.abs(vgot - vref).max() <= 1e-12 * np.abs(U).max()


@pytest.mark.parametrize("sizes", [[(2, 2), (95, 3)], [(126, 4), (127, 2), (63, 65)]])
def test_batched_stage_at_tile_edges(sizes):
    import torch
    cases = [_case(nx, ny, (1, 2, 2, 1), 1, 0) for nx, ny in sizes]
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    U = [dev(c[1]) for c in cases]
    V = [dev(c[3]) for c in cases]
    out = [torch.full_like(u, float("nan")) for u in U]
    ain = [dev(c[4]) for c in cases]
    aout = [torch.zeros(2, dtype=torch.float64, device="cuda") for _ in cases]
    dt = [dev(np.array([c[5]])) for c in cases]
    st = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in cases]
    H.hweno_stage_batch_static([c[0] for c in cases], 1, U, U, V, out, ain, aout, dt, st,
                               torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    for c, o, s in zip(cases, out, st):
        assert int(s.item()) == 0
        assert rel_err(o.cpu().numpy(), c[6], c[1]) <= 1e-12
