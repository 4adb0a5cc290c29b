"""Performance cases: what a program asks of this library, from a 200-cell line to a 2048^2 grid.

A case is a dict of plain values and a way of calling the library:

  "stages"   one SSP-RK3 step on the caller's own device buffers: the wave speeds of the state,
             then the three fused stages (hweno_alpha_device, hweno_stage_device);
  "batch"    the same for several 2D solves at once through the entry point that allocates
             nothing (hweno_stage_batch_static);
  "advance"  a solve held by an engine: state in, time steps, state out (hweno_set_state,
             hweno_advance, hweno_get_state);
  "serve"    requests of different grids and precisions submitted to the serving loop and
             collected when they are done (hweno_submit, hweno_serve, hweno_poll).

prepare() makes the inputs (seeded initial data projected onto the moments by 5-point Gauss
quadrature), run() is one pass, exact() the same pass in plain torch in 64 bits, written from
the scheme's formulas.
"""
import math
import random

import numpy as np
import torch

from paper_2402_03074_gb300 import _binding as H

EQUATIONS = {"advection": H.HWENO_ADVECTION, "burgers": H.HWENO_BURGERS, "euler": H.HWENO_EULER}
BOUNDARIES = {"periodic": H.HWENO_BC_PERIODIC, "transmissive": H.HWENO_BC_TRANSMISSIVE,
              "reflective": H.HWENO_BC_REFLECTIVE}
PRECISIONS = {"fp64": H.HWENO_FP64, "mixed32": H.HWENO_MIXED32}
WEIGHTS = {"scale_invariant": H.HWENO_W_SCALE_INVARIANT, "original": H.HWENO_W_ORIGINAL,
           "linear": H.HWENO_W_LINEAR}
GAMMA = 1.4
CFL = 0.6
GAMMA_LO = 1.0 / 400.0
EPS = 1e-10
AX, AY = 1.0, -0.7  # advection speeds


def _case(call, dim, equation, nx, ny=1, **more):
    c = {"call": call, "dim": dim, "equation": equation, "nx": nx, "ny": ny, "data": "wave",
         "bc_x": "periodic", "bc_y": "periodic", "precision": "fp64", "characteristic": True,
         "weights": "scale_invariant", "steps": 1}
    c.update(more)
    return c


def listed():
    open_box = {"data": "quadrants", "bc_x": "transmissive", "bc_y": "transmissive"}
    return [
        # the headline grid: a 2D Riemann problem with a vortex, one time step in FP64
        _case("stages", 2, "euler", 2048, 2048, name="euler2d_2048_fp64", **open_box),
        # the same grid in the FP32-bulk arithmetic
        _case("stages", 2, "euler", 2048, 2048, name="euler2d_2048_mixed32", precision="mixed32",
              **open_box),
        # a ragged channel with walls: neither side a multiple of a tile
        _case("stages", 2, "euler", 517, 389, name="euler2d_ragged_channel", data="quadrants",
              bc_x="transmissive", bc_y="reflective"),
        # component-wise reconstruction: the cheaper option for Euler flows
        _case("stages", 2, "euler", 768, 768, name="euler2d_768_componentwise",
              characteristic=False, **open_box),
        # the paper's finest 2D Euler accuracy grid, a few steps of a solve held by an engine
        _case("advance", 2, "euler", 240, 240, name="euler2d_240_advance", steps=12),
        # its coarsest grid: a step is a handful of short launches
        _case("advance", 2, "euler", 40, 40, name="euler2d_40_advance", steps=24),
        # 2D Burgers on the paper's finest grid
        _case("advance", 2, "burgers", 240, 240, name="burgers2d_240_advance", steps=48),
        # 1D advection, 200 cells, to T = 2 (one period)
        _case("advance", 1, "advection", 200, name="advection1d_200", steps=334),
        # the paper's finest 1D Euler accuracy grid
        _case("advance", 1, "euler", 240, name="euler1d_240", steps=400),
        # a 4000-cell shock tube
        _case("advance", 1, "euler", 4000, name="euler1d_tube_4000", steps=128, data="quadrants",
              bc_x="transmissive"),
        # a batch of mid-size 2D solves advanced by a caller that cannot allocate
        _case("batch", 2, "euler", 200, 184, name="euler2d_batch", count=8, **open_box),
        # a served mix of grids and of both precisions
        _case("serve", 2, "euler", 128, 128, name="euler2d_served", count=6, steps=16, **open_box),
    ]


def draw(rng: random.Random):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def options(dim, eq):
        data = rng.choice(["wave", "quadrants"]) if eq == "euler" else "wave"
        more = {"data": data, "precision": rng.choice(["fp64", "fp64", "mixed32"]),
                "weights": rng.choice(["scale_invariant"] * 4 + ["original"])}
        if data == "quadrants":
            more["bc_x"] = rng.choice(["transmissive", "reflective"])
            more["bc_y"] = rng.choice(["transmissive", "reflective"]) if dim == 2 else "periodic"
        if eq == "euler":
            more["characteristic"] = rng.random() < 0.8
        return more

    call = rng.choice(["stages"] * 5 + ["advance"] * 7 + ["batch", "serve"])
    if call == "stages":
        eq = rng.choice(["euler"] * 5 + ["burgers", "advection"])
        nx = size(32, 2048)
        ny = min(2048, max(24, int(nx * math.exp(rng.uniform(-0.5, 0.5)))))
        return _case(call, 2, eq, nx, ny, **options(2, eq))
    if call == "advance":
        if rng.random() < 0.55:
            eq = rng.choice(["euler", "euler", "burgers", "advection"])
            return _case(call, 1, eq, size(32, 8000), steps=size(16, 256), **options(1, eq))
        eq = rng.choice(["euler", "euler", "euler", "burgers"])
        nx = size(32, 400)
        ny = max(24, int(nx * math.exp(rng.uniform(-0.4, 0.4))))
        return _case(call, 2, eq, nx, ny, steps=size(4, 16), **options(2, eq))
    more = options(2, "euler")
    n = size(48, 256)
    if call == "batch":
        return _case(call, 2, "euler", n, max(24, n - rng.randint(0, 40)),
                     count=rng.randint(2, 12), **more)
    more["precision"] = "fp64"  # a served mix holds both precisions in any case
    return _case(call, 2, "euler", n, n, count=rng.randint(2, 6), steps=rng.randint(4, 16), **more)


# ---- the grids of a case ------------------------------------------------------------------
def _grids(case):
    """(nx, ny, precision) of every solve: one, or `count` of growing size in which a served mix
    takes every third in the FP32-bulk arithmetic."""
    if case["call"] not in ("batch", "serve"):
        return [(case["nx"], case["ny"], case["precision"])]
    out = []
    for s in range(case["count"]):
        grow = 1.0 + 0.35 * s if case["call"] == "serve" else 1.0 + 0.06 * s
        mixed = case["call"] == "serve" and s % 3 == 1
        out.append((int(case["nx"] * grow), int(case["ny"] * grow),
                    "mixed32" if mixed else case["precision"]))
    return out


def _problem(case, nx, ny, precision, t_end=0.0):
    length = 2.0 if case["data"] == "wave" else 1.0
    bx, by = BOUNDARIES[case["bc_x"]], BOUNDARIES[case["bc_y"]]
    return H.make_problem(dim=case["dim"], equation=EQUATIONS[case["equation"]], nx=nx, ny=ny,
                          x0=0.0, x1=length, y0=0.0,
                          y1=length * ny / nx if case["dim"] == 2 else 1.0, ax=AX, ay=AY,
                          gamma=GAMMA, bc=(bx, bx, by, by), cfl=CFL, t_end=t_end,
                          precision=PRECISIONS[precision],
                          characteristic=int(case["characteristic"]),
                          weights=WEIGHTS[case["weights"]], gamma_lo=GAMMA_LO, eps=EPS)


# flops of one cell and stage (multiplications, additions, divisions and roots of the scheme's
# formulas, repeated ones counted once; the mean over the three stages)
STAGE_FLOPS = {(2, "euler", True): 10102.0, (2, "euler", False): 5037.0,
               (2, "burgers", False): 1192.0, (2, "advection", False): 1150.0,
               (1, "euler", True): 895.0, (1, "euler", False): 648.0,
               (1, "burgers", False): 206.0, (1, "advection", False): 198.0}


def work(case):
    """The scheme's flops, and the bytes of its three stages: each reads its input (and, after
    the first, the base averages and first-moment modifications) and writes its output (the
    first also the modifications)."""
    ch = case["characteristic"] and case["equation"] == "euler"
    flops = STAGE_FLOPS[case["dim"], case["equation"], ch]
    nc = (2 + case["dim"]) if case["equation"] == "euler" else 1
    nm = 1 + case["dim"]
    per_step = 8.0 * (6 * nc * nm + nc * (nm - 1) + 2 * nc * nm)
    cells = sum(nx * ny for nx, ny, _ in _grids(case))
    n = cells * case["steps"]
    return {"bytes": per_step * n, "flops": 3.0 * flops * n}


# ---- initial data -------------------------------------------------------------------------
_NODES, _NODE_W = (torch.from_numpy(a) for a in np.polynomial.legendre.leggauss(5))
_NODES, _NODE_W = _NODES / 2.0, _NODE_W / 2.0


def _device():
    return torch.device("cuda:0" if torch.cuda.is_available() else "cpu")


def _moments(fn, dim, nx, ny, length):
    """Cell averages and first moments of fn (points -> list of components): U[nc, nm, ny, nx]."""
    dev = _device()
    h = length / nx
    X = (torch.arange(nx, dtype=torch.float64, device=dev) + 0.5) * h
    Y = (torch.arange(ny, dtype=torch.float64, device=dev) + 0.5) * h
    out = None
    for a in range(5):
        for b in range(5 if dim == 2 else 1):
            x = (X + _NODES[a].item() * h)[None, :]
            y = (Y + _NODES[b].item() * h)[:, None] if dim == 2 else torch.zeros_like(Y)[:, None]
            w = _NODE_W[a].item() * (_NODE_W[b].item() if dim == 2 else 1.0)
            vals = fn(*torch.broadcast_tensors(x, y))
            if out is None:
                out = torch.zeros((len(vals), 1 + dim, ny, nx), dtype=torch.float64, device=dev)
            for c, v in enumerate(vals):
                out[c, 0] += w * v
                out[c, 1] += (w * _NODES[a].item()) * v
                if dim == 2:
                    out[c, 2] += (w * _NODES[b].item()) * v
    return out


def _conserved(dim, rho, u, v, p):
    e = p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)
    return [rho, rho * u, e] if dim == 1 else [rho, rho * u, rho * v, e]


def _initial(case, nx, ny, seed):
    """Seeded initial moments: a smooth periodic wave, or constant states meeting at the middle
    of the domain with a smooth structure on top (in 2D a vortex, in 1D an entropy wave)."""
    rng = np.random.default_rng(seed)
    dim, eq = case["dim"], case["equation"]
    length = 2.0 if case["data"] == "wave" else 1.0
    pick = lambda lo, hi, n=None: rng.uniform(lo, hi, size=n)
    if case["data"] == "wave":
        # one period along x; along y the nearest whole number of periods to the domain's height
        ky = max(1, round(ny / nx)) * nx / ny if dim == 2 else 0.0
        amp, ph, mean = pick(0.15, 0.25), pick(0.0, 2.0 * math.pi), pick(0.9, 1.1)
        if eq != "euler":
            return _moments(lambda x, y: [0.5 * mean + 4.0 * amp *
                                          torch.sin(math.pi * (x + ky * y) + ph)],
                            dim, nx, ny, length)
        u, v, p = pick(0.8, 1.2), pick(0.8, 1.2), pick(0.9, 1.1)

        def wave(x, y):
            rho = mean + amp * torch.sin(math.pi * (x + ky * y) + ph)
            one = torch.ones_like(rho)
            return _conserved(dim, rho, u * one, (v if dim == 2 else 0.0) * one, p * one)

        return _moments(wave, dim, nx, ny, length)
    nq = 4 if dim == 2 else 2
    rho, p = pick(0.2, 2.0, nq), pick(0.2, 2.0, nq)
    u, v = pick(-0.75, 0.75, nq), pick(-0.75, 0.75, nq)
    xc, yc, k = pick(0.3, 0.7), pick(0.3, 0.7), pick(30.0, 80.0)
    dev = _device()
    rho, p, u, v = (torch.tensor(a, dtype=torch.float64, device=dev) for a in (rho, p, u, v))
    half = length * ny / nx / 2.0

    def states(x, y):
        if dim == 1:
            q = (x >= 0.5).to(torch.int64)
            r = rho[q] * torch.where(q == 1, 1.0 + 0.2 * torch.sin(k * x), torch.ones_like(x))
            return _conserved(1, r, u[q], torch.zeros_like(x), p[q])
        q = (x >= 0.5).to(torch.int64) + 2 * (y >= half).to(torch.int64)
        dx, dy = (x - xc) / 0.05, (y - 2.0 * half * yc) / 0.05
        g = torch.exp(0.5 * (1.0 - dx * dx - dy * dy))
        s = 5.0 / (2.0 * math.pi)
        temp = 1.0 - (GAMMA - 1.0) * 25.0 / (8.0 * GAMMA * math.pi ** 2) * g * g
        return _conserved(2, rho[q] * temp ** 2.5, u[q] - s * g * dy, v[q] + s * g * dx,
                          p[q] * temp ** 3.5)

    return _moments(states, dim, nx, ny, length)


def _speeds(case, U):
    """max |f'| and max |g'| over the cell averages."""
    u = U[:, 0]
    if case["equation"] == "advection":
        return [abs(AX), abs(AY) if case["dim"] == 2 else 0.0]
    if case["equation"] == "burgers":
        a = float(u.abs().max())
        return [a, a if case["dim"] == 2 else 0.0]
    rho, m, E = u[0], u[1:-1], u[-1]
    vel = m / rho
    c = torch.sqrt(GAMMA * (GAMMA - 1.0) * (E - 0.5 * (m * vel).sum(0)) / rho)
    return [float((vel[d].abs() + c).max()) if d < case["dim"] else 0.0 for d in range(2)]


def _cfl_step(case, nx, a):
    h = (2.0 if case["data"] == "wave" else 1.0) / nx
    return CFL / (a[0] / h + (a[1] / h if case["dim"] == 2 else 0.0))


# ---- prepare and run -----------------------------------------------------------------------
_engine = None


def _the_engine():
    global _engine
    if _engine is None:
        _engine = H.hweno_create()
    return _engine


class _Solve:
    """A solve open on the engine, closed with its owner."""

    def __init__(self, problem, U):
        self.id = H.hweno_open(_the_engine(), problem, U)

    def __del__(self):
        H.hweno_close(_engine, self.id)


def _host(U):
    """A state in pinned host memory."""
    t = torch.empty(U.shape, dtype=U.dtype, pin_memory=U.is_cuda)
    t.copy_(U)
    return t.numpy()


def prepare(case, seed):
    call = case["call"]
    grids = _grids(case)
    states = [_initial(case, nx, ny, seed + 1000 * s) for s, (nx, ny, _) in enumerate(grids)]
    S = {"call": call, "case": case}
    if call in ("stages", "batch"):
        S["solves"] = []
        for (nx, ny, prec), U in zip(grids, states):
            nc, nm = U.shape[:2]
            dt = _cfl_step(case, nx, _speeds(case, U))
            S["solves"].append({
                "problem": _problem(case, nx, ny, prec), "U": U, "U1": torch.empty_like(U),
                "U2": torch.empty_like(U), "out": torch.empty_like(U),
                "Vh": torch.zeros((nc, nm - 1, ny, nx), dtype=U.dtype, device=U.device),
                "speeds": torch.zeros((4, 2), dtype=U.dtype, device=U.device),
                "dt": torch.tensor([dt], dtype=U.dtype, device=U.device),
                "status": torch.zeros(1, dtype=torch.int32, device=U.device)})
        return S
    S["hosts"] = [_host(U) for U in states]
    if call == "advance":
        (nx, ny, prec), = grids
        S["solve"] = _Solve(_problem(case, nx, ny, prec), S["hosts"][0])
        S["result"] = _host(states[0])
        return S
    S["results"] = [_host(U) for U in states]
    S["problems"] = [_problem(case, nx, ny, prec, _end_time(case, nx, U))
                     for (nx, ny, prec), U in zip(grids, states)]
    return S


def _end_time(case, nx, U):
    """The end time of a served request: about `steps` steps."""
    return (case["steps"] - 0.5) * _cfl_step(case, nx, _speeds(case, U))


def run(S):
    if S["call"] in ("stages", "batch"):
        stream = torch.cuda.current_stream().cuda_stream
        for s in S["solves"]:
            s["speeds"].zero_()
            s["status"].zero_()
            H.hweno_alpha_device(s["problem"], s["U"], s["speeds"][0], stream)
        for k, (src, dst) in enumerate((("U", "U1"), ("U1", "U2"), ("U2", "out")), 1):
            if S["call"] == "stages":
                s, = S["solves"]
                H.hweno_stage_device(s["problem"], k, s[src], s["U"], s["Vh"], s[dst],
                                     s["speeds"][k - 1], s["speeds"][k], s["dt"], s["status"],
                                     stream)
            else:
                q = S["solves"]
                H.hweno_stage_batch_static(
                    [s["problem"] for s in q], k, [s[src] for s in q], [s["U"] for s in q],
                    [s["Vh"] for s in q], [s[dst] for s in q], [s["speeds"][k - 1] for s in q],
                    [s["speeds"][k] for s in q], [s["dt"] for s in q], [s["status"] for s in q],
                    stream)
        return [{"U": s["out"], "Vh": s["Vh"], "speeds": s["speeds"], "status": s["status"]}
                for s in S["solves"]]
    eng = _the_engine()
    if S["call"] == "advance":
        sid = S["solve"].id
        H.hweno_set_state(eng, sid, S["hosts"][0], 0.0)
        steps = H.hweno_advance(eng, sid, 1e9, S["case"]["steps"])
        U, t = H.hweno_get_state(eng, sid, S["result"])
        return [{"U": U, "t": t, "steps": steps}]
    tickets = [H.hweno_submit(eng, p, u) for p, u in zip(S["problems"], S["hosts"])]
    while H.hweno_serve(eng, 8) > 0:
        pass
    out = []
    for ticket, result in zip(tickets, S["results"]):
        _, info = H.hweno_poll(eng, ticket, result)
        out.append({"U": result, "t": info.t, "steps": int(info.steps)})
    return out


# ---- the same in plain torch, 64 bits --------------------------------------------------------
_S15 = math.sqrt(15.0) / 10.0
_GAUSS = ((-_S15, 5.0 / 18.0), (0.0, 4.0 / 9.0), (_S15, 5.0 / 18.0))
_POWERS = ((0, 0), (1, 0), (0, 1), (2, 0), (1, 1), (0, 2), (3, 0), (2, 1), (1, 2), (0, 3),
           (4, 0), (3, 1), (2, 2), (1, 3), (0, 4))


def _ghosts(n, bc, dev):
    """Stored index of the cells -2 .. n+1 and whether each is a mirror image."""
    idx, flip = [], []
    for i in range(-2, n + 2):
        f = False
        while i < 0 or i >= n:
            if bc == "periodic":
                i += n if i < 0 else -n
            elif bc == "transmissive":
                i = 0 if i < 0 else n - 1
            else:
                i, f = (-1 - i if i < 0 else 2 * n - 1 - i), not f
        idx.append(i)
        flip.append(f)
    return torch.tensor(idx, device=dev), torch.tensor(flip, device=dev)


def _padded(case, U):
    """The state with two ghost cells on every side of each of its directions."""
    nc = U.shape[0]
    for axis in range(case["dim"]):  # 0: x (last axis), 1: y
        n = U.shape[3 - axis]
        idx, flip = _ghosts(n, case["bc_x"] if axis == 0 else case["bc_y"], U.device)
        U = U.index_select(3 - axis, idx)
        shape = [1, 1, 1, 1]
        shape[3 - axis] = n + 4
        neg = flip.reshape(shape)
        sign = torch.ones(U.shape[:2] + (1, 1), dtype=U.dtype, device=U.device)
        sign[:, 1 + axis] *= -1.0  # the first moment normal to the wall
        if nc > 1:
            sign[1 + axis] *= -1.0  # the momentum normal to the wall
        U = torch.where(neg, U * sign, U)
    return U


def _omegas(case, betas, u_ave):
    """Nonlinear weights, returned as the factors a0 of p_0 and b_m of p_m."""
    n = len(betas)
    lin = [1.0 - (n - 1) * GAMMA_LO] + [GAMMA_LO] * (n - 1)
    if case["weights"] == "linear":
        return torch.ones_like(u_ave), [torch.zeros_like(u_ave)] * (n - 1)
    if case["weights"] == "original":
        u_ave = torch.ones_like(u_ave)
    tau = (sum((betas[0] - b).abs() for b in betas[1:]) / (n - 1)) ** 2
    w = [g * (1.0 + tau / (b * u_ave + EPS)) for g, b in zip(lin, betas)]
    total = sum(w)
    a0 = w[0] / total / lin[0]
    return a0, [x / total - a0 * g for x, g in zip(w[1:], lin[1:])]


def _poly_1d(case, u, v):
    """Combined quartic of every cell: u averages and v first moments of the 3 stencil cells."""
    um, u0, up = u
    vm, vp = v[0], v[2]
    c = [-43.0 / 384.0 * um + 235.0 / 192.0 * u0 - 43.0 / 384.0 * up - 27.0 / 64.0 * vm + 27.0 / 64.0 * vp,
         -63.0 / 76.0 * um + 63.0 / 76.0 * up - 75.0 / 19.0 * vm - 75.0 / 19.0 * vp,
         23.0 / 16.0 * um - 23.0 / 8.0 * u0 + 23.0 / 16.0 * up + 45.0 / 8.0 * vm - 45.0 / 8.0 * vp,
         5.0 / 19.0 * um - 5.0 / 19.0 * up + 60.0 / 19.0 * vm + 60.0 / 19.0 * vp,
         -5.0 / 8.0 * um + 5.0 / 4.0 * u0 - 5.0 / 8.0 * up - 15.0 / 4.0 * vm + 15.0 / 4.0 * vp]
    slope = [u0 - um, up - u0]
    betas = [(c[1] + 0.25 * c[3]) ** 2 + 13.0 / 3.0 * (c[2] + 63.0 / 130.0 * c[4]) ** 2 +
             781.0 / 20.0 * c[3] ** 2 + 1421461.0 / 2275.0 * c[4] ** 2, slope[0] ** 2, slope[1] ** 2]
    a0, b = _omegas(case, betas, ((um.abs() + u0.abs() + up.abs()) / 3.0) ** 2)
    return [a0 * c[0] + (b[0] + b[1]) * u0, a0 * c[1] + b[0] * slope[0] + b[1] * slope[1],
            a0 * c[2], a0 * c[3], a0 * c[4]]


def _poly_2d(case, u, v, w):
    """Combined quartic of every cell from the 9 averages and the x and y first moments."""
    u1, u2, u3, u4, u5, u6, u7, u8, u9 = u
    v2, v4, v6, v8 = v[1], v[3], v[5], v[7]
    w2, w4, w6, w8 = w[1], w[3], w[5], w[7]
    corners, cross = u1 + u3 + u7 + u9, u2 + u4 + u6 + u8
    twist = u1 - u3 - u7 + u9
    c = [corners / 576.0 - 133.0 / 1152.0 * cross + 419.0 / 288.0 * u5 +
         27.0 / 64.0 * (v6 - v4 + w8 - w2),
         (u1 - u3 + u7 - u9) / 48.0 - 397.0 / 456.0 * (u4 - u6) - 75.0 / 19.0 * (v4 + v6),
         (u1 + u3 - u7 - u9) / 48.0 - 397.0 / 456.0 * (u2 - u8) - 75.0 / 19.0 * (w2 + w8),
         -corners / 48.0 + (u2 + u8) / 24.0 + 71.0 / 48.0 * (u4 + u6) - 71.0 / 24.0 * u5 +
         45.0 / 8.0 * (v4 - v6),
         -7.0 / 22.0 * twist + 75.0 / 11.0 * (v8 - v2 + w6 - w4),
         -corners / 48.0 + 71.0 / 48.0 * (u2 + u8) + (u4 + u6) / 24.0 - 71.0 / 24.0 * u5 +
         45.0 / 8.0 * (w2 - w8),
         5.0 / 19.0 * (u4 - u6) + 60.0 / 19.0 * (v4 + v6),
         -(u1 + u3 - u7 - u9) / 4.0 + (u2 - u8) / 2.0,
         -(u1 - u3 + u7 - u9) / 4.0 + (u4 - u6) / 2.0,
         5.0 / 19.0 * (u2 - u8) + 60.0 / 19.0 * (w2 + w8),
         -5.0 / 8.0 * (u4 + u6) + 5.0 / 4.0 * u5 + 15.0 / 4.0 * (v6 - v4),
         5.0 / 22.0 * twist + 60.0 / 11.0 * (v2 - v8),
         corners / 4.0 - cross / 2.0 + u5,
         5.0 / 22.0 * twist + 60.0 / 11.0 * (w4 - w6),
         -5.0 / 8.0 * (u2 + u8) + 5.0 / 4.0 * u5 + 15.0 / 4.0 * (w8 - w2)]
    sq = lambda t: t * t
    b0 = (0.5 * (sq(c[1] + 0.5 * c[6]) + sq(c[1] + c[8] / 6.0) + sq(c[2] + c[7] / 6.0) +
                 sq(c[2] + 0.5 * c[9])) +
          13.0 / 6.0 * (sq(c[3] + 63.0 / 65.0 * c[10]) + sq(c[3] + c[12] / 6.0) +
                        sq(c[5] + c[12] / 6.0) + sq(c[5] + 63.0 / 65.0 * c[14])) +
          7.0 / 12.0 * (sq(c[4] + 17.0 / 35.0 * c[11]) + sq(c[4] + 17.0 / 35.0 * c[13])) +
          3119.0 / 80.0 * sq(c[6] + 5.0 / 9357.0 * c[8]) +
          3379.0 / 720.0 * sq(c[7] + 15.0 / 3379.0 * c[9]) +
          2634769.0 / 561420.0 * sq(c[8]) + 2634769.0 / 67580.0 * sq(c[9]) +
          5676583.0 / 9100.0 * sq(c[10] + 3185.0 / 11353166.0 * c[12]) +
          709573.0 / 16800.0 * sq(c[11] + 1155.0 / 709573.0 * c[13]) +
          230094013357.0 / 12261419280.0 * sq(c[12] + 2145748374.0 / 230094013357.0 * c[14]) +
          31468281769.0 / 745051650.0 * sq(c[13]) +
          25118160529227568.0 / 40266452337475.0 * sq(c[14]))
    l, r, d, t = u5 - u4, u6 - u5, u5 - u2, u8 - u5
    betas = [b0, sq(l) + sq(d), sq(r) + sq(d), sq(l) + sq(t), sq(r) + sq(t)]
    a0, b = _omegas(case, betas, sq((u2.abs() + u4.abs() + u5.abs() + u6.abs() + u8.abs()) / 5.0))
    C = [a0 * x for x in c]
    C[0] = C[0] + sum(b) * u5
    C[1] = C[1] + (b[0] + b[2]) * l + (b[1] + b[3]) * r
    C[2] = C[2] + (b[0] + b[1]) * d + (b[2] + b[3]) * t
    return C


def _at(C, x, y):
    return sum(c * (x ** p * y ** q) for c, (p, q) in zip(C, _POWERS) if x ** p * y ** q != 0.0)


def _flux(case, d, u):
    if case["equation"] == "advection":
        return (AX, AY)[d] * u
    if case["equation"] == "burgers":
        return 0.5 * u * u
    m, E = u[1:-1], u[-1]
    vel = m / u[0]
    p = (GAMMA - 1.0) * (E - 0.5 * (m * vel).sum(0))
    f = u * vel[d]
    f[1 + d] += p
    f[-1] += p * vel[d]
    return f


def _eigen(case, d, u):
    """L and R of the flux Jacobian in direction d at the states u, as [field][component] and
    [component][field] lists of tensors or plain numbers."""
    rho, E = u[0], u[-1]
    vel = [m / rho for m in u[1:-1]]
    q = 0.5 * sum(x * x for x in vel)
    p = (GAMMA - 1.0) * (E - rho * q)
    c = torch.sqrt(GAMMA * p / rho)
    Hs = (E + p) / rho
    n = vel[d]
    b1 = (GAMMA - 1.0) / (c * c)
    b2 = b1 * q
    if case["dim"] == 1:
        L = [[0.5 * (b2 + n / c), -0.5 * (b1 * n + 1.0 / c), 0.5 * b1], [1.0 - b2, b1 * n, -b1],
             [0.5 * (b2 - n / c), -0.5 * (b1 * n - 1.0 / c), 0.5 * b1]]
        R = [[1.0, 1.0, 1.0], [n - c, n, n + c], [Hs - n * c, q, Hs + n * c]]
        return L, R
    t = vel[1 - d]
    L = [[0.5 * (b2 + n / c), -0.5 * (b1 * n + 1.0 / c), -0.5 * b1 * t, 0.5 * b1],
         [1.0 - b2, b1 * n, b1 * t, -b1], [-t, 0.0, 1.0, 0.0],
         [0.5 * (b2 - n / c), -0.5 * (b1 * n - 1.0 / c), -0.5 * b1 * t, 0.5 * b1]]
    R = [[1.0, 1.0, 0.0, 1.0], [n - c, n, 0.0, n + c], [t, t, 1.0, t],
         [Hs - n * c, q, t, Hs + n * c]]
    if d == 1:  # the momentum components change places
        L = [[r[0], r[2], r[1], r[3]] for r in L]
        R = [R[0], R[2], R[1], R[3]]
    return L, R


def _apply(M, u):
    return torch.stack([sum(a * x for a, x in zip(row, u)) for row in M])


def _reconstruct(case, d, cells, points):
    """Values at `points` and the first-moment modification of direction d, from the moments of
    the 3 or 9 stencil cells (each [nc, nm, ...])."""
    mid = len(cells) // 2
    back = None
    if case["equation"] == "euler" and case["characteristic"]:
        L, back = _eigen(case, d, cells[mid][:, 0])
        cells = [torch.stack([_apply(L, s[:, m]) for m in range(s.shape[1])], 1) for s in cells]
    if case["dim"] == 1:
        C = _poly_1d(case, [s[:, 0] for s in cells], [s[:, 1] for s in cells])
        vals = [sum(c * x ** n for n, c in enumerate(C)) for x, _ in points]
        vals.append(C[1] / 12.0 + C[3] / 80.0)
    else:
        C = _poly_2d(case, [s[:, 0] for s in cells], [s[:, 1] for s in cells],
                     [s[:, 2] for s in cells])
        vals = [_at(C, x, y) for x, y in points]
        vals.append(C[1] / 12.0 + C[6] / 80.0 + C[8] / 144.0 if d == 0 else
                    C[2] / 12.0 + C[9] / 80.0 + C[7] / 144.0)
    if back is not None:
        vals = [_apply(back, v) for v in vals]
    return vals[:-1], vals[-1]


def _combine(k, dt, own, base, rhs):
    adv = own + dt * rhs
    return adv if k == 1 else (0.75 * base + 0.25 * adv if k == 2 else base / 3.0 + 2.0 / 3.0 * adv)


def _stage_1d(case, k, P, Un, Vh, a, dt, h):
    n = P.shape[3] - 4
    cells = [P[:, :, 0, i:i + n + 2] for i in range(3)]
    s5 = math.sqrt(5.0) / 10.0
    pts, vh = _reconstruct(case, 0, cells, [(-0.5, 0), (-s5, 0), (s5, 0), (0.5, 0)])
    f = [_flux(case, 0, u) for u in pts]
    face = 0.5 * (f[3][:, :-1] + f[0][:, 1:] - a[0] * (pts[0][:, 1:] - pts[3][:, :-1]))
    lo, hi = face[:, :-1], face[:, 1:]
    vol = ((f[0] + f[3]) / 12.0 + 5.0 / 12.0 * (f[1] + f[2]))[:, 1:-1]
    rhs = torch.stack([-(hi - lo) / h, (vol - 0.5 * (lo + hi)) / h], 1)
    own = torch.stack([P[:, 0, 0, 2:-2], vh[:, 1:-1]], 1)
    if k == 1:
        Vh[:, 0, 0] = vh[:, 1:-1]
    base = torch.stack([Un[:, 0, 0], Vh[:, 0, 0]], 1)
    return _combine(k, dt, own, base, rhs)[:, :, None]


def _stage_2d(case, k, P, Un, Vh, a, dt, h, rows=160):
    ny, nx = P.shape[2] - 4, P.shape[3] - 4
    out = torch.empty_like(Un)
    inner = [(x, y) for x, _ in _GAUSS for y, _ in _GAUSS]
    wts = [p * q for _, p in _GAUSS for _, q in _GAUSS]
    w = [q for _, q in _GAUSS]
    wx = [p * q for p, q in _GAUSS]
    gs = lambda wt, fs: sum(q * f for q, f in zip(wt, fs))
    for j0 in range(0, ny, rows):
        j1 = min(ny, j0 + rows)
        win = P[:, :, j0:j1 + 4]
        cells = [win[:, :, j:j + j1 - j0 + 2, i:i + nx + 2] for j in range(3) for i in range(3)]
        # x: traces on the left and right edges, the volume sum of f, v-hat
        edges = [(-0.5, y) for y, _ in _GAUSS] + [(0.5, y) for y, _ in _GAUSS]
        pts, vh = _reconstruct(case, 0, cells, edges + inner)
        vol_f = gs(wts, [_flux(case, 0, u) for u in pts[6:]])[:, 1:-1, 1:-1]
        F = []
        for g in range(3):
            uL, uR = pts[3 + g][:, 1:-1, :-1], pts[g][:, 1:-1, 1:]
            F.append(0.5 * (_flux(case, 0, uL) + _flux(case, 0, uR) - a[0] * (uR - uL)))
        # y: traces on the bottom and top edges, the volume sum of g, w-hat
        edges = [(x, -0.5) for x, _ in _GAUSS] + [(x, 0.5) for x, _ in _GAUSS]
        pts, wh = _reconstruct(case, 1, cells, edges + inner)
        vol_g = gs(wts, [_flux(case, 1, u) for u in pts[6:]])[:, 1:-1, 1:-1]
        G = []
        for g in range(3):
            uB, uT = pts[3 + g][:, :-1, 1:-1], pts[g][:, 1:, 1:-1]
            G.append(0.5 * (_flux(case, 1, uB) + _flux(case, 1, uT) - a[1] * (uT - uB)))
        fl, fr = [f[:, :, :-1] for f in F], [f[:, :, 1:] for f in F]
        gb, gt = [g[:, :-1] for g in G], [g[:, 1:] for g in G]
        rhs = torch.stack([
            -(gs(w, fr) - gs(w, fl)) / h - (gs(w, gt) - gs(w, gb)) / h,
            (vol_f - 0.5 * (gs(w, fl) + gs(w, fr))) / h - (gs(wx, gt) - gs(wx, gb)) / h,
            -(gs(wx, fr) - gs(wx, fl)) / h + (vol_g - 0.5 * (gs(w, gb) + gs(w, gt))) / h], 1)
        vh, wh = vh[:, 1:-1, 1:-1], wh[:, 1:-1, 1:-1]
        own = torch.stack([win[:, 0, 2:-2, 2:-2], vh, wh], 1)
        if k == 1:
            Vh[:, 0, j0:j1] = vh
            Vh[:, 1, j0:j1] = wh
        base = torch.stack([Un[:, 0, j0:j1], Vh[:, 0, j0:j1], Vh[:, 1, j0:j1]], 1)
        out[:, :, j0:j1] = _combine(k, dt, own, base, rhs)
    return out


def _step(case, U, Vh, dt, speeds):
    """One SSP-RK3 step; `speeds` receives those of the input and of the three stages."""
    h = (2.0 if case["data"] == "wave" else 1.0) / U.shape[3]
    stage = _stage_1d if case["dim"] == 1 else _stage_2d
    V = U
    for k in (1, 2, 3):
        V = stage(case, k, _padded(case, V), U, Vh, speeds[-1], dt, h)
        speeds.append(_speeds(case, V))
    return V


def exact(case, seed):
    out = []
    for s, (nx, ny, _) in enumerate(_grids(case)):
        U = _initial(case, nx, ny, seed + 1000 * s)
        Vh = torch.zeros((U.shape[0], U.shape[1] - 1, ny, nx), dtype=U.dtype, device=U.device)
        a = _speeds(case, U)
        if case["call"] in ("stages", "batch"):
            speeds = [a]
            V = _step(case, U, Vh, _cfl_step(case, nx, a), speeds)
            out.append({"U": V, "Vh": Vh, "speeds": torch.tensor(speeds, dtype=torch.float64),
                        "status": None})
            continue
        end = _end_time(case, nx, U) if case["call"] == "serve" else 1e9
        limit = case["steps"] if case["call"] == "advance" else 1 << 30
        t, n = 0.0, 0
        while t < end and n < limit:
            dt = _cfl_step(case, nx, a)
            dt, t = (dt, t + dt) if t + dt < end else (end - t, end)
            speeds = [a]
            U = _step(case, U, Vh, dt, speeds)
            a, n = speeds[-1], n + 1
        out.append({"U": U, "t": t, "steps": n})
    return out
