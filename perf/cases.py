"""Performance cases of the immersed boundary framework and their 64-bit values.

Every case goes through the public Python entry points (ibm.Grid, ibm.Batch,
ibm.cd_nu_objective, ibm.ibm_rhs_dt_noalloc) the way a user's program does:

  run        set_state, step(k), forces, get_state of one grid: 2D or 3D,
             FP32 or FP64, static or moving body, direct launches or graphs
  batch      the same over a batch of uneven 2D grids
  gradient   J = a C_d + b Nu of a k-step run and its gradient: FP64 grids for
             shape (marker positions) and wall temperatures, FP32 grids for
             wall temperatures
  body       a new body on an existing grid: set_markers and its weights
  operators  rhs, interpolate, spread, surface_pressure on a user's fields
  rhs        L(U) and the step size without a handle (ibm_rhs_dt_noalloc)

Marker values of FP32 grids are kept in the grid's own precision.  exact() restates the method in plain torch FP64 operations.
"""
import math
import random

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2301_09349_gb300 import cases as C
from paper_2301_09349_gb300 import ibm

DEV = "cuda"


def listed():
    return [
        # the smallest call: one explicit evaluation of a coarse 3D grid, for
        # a host code that drives its own time loop
        dict(name="rhs_48", kind="rhs", dim=3, nx=48, ny=48, nz=48, fp=4, div=8, mach=0.3, re=300.0),
        # the paper's heated cylinder (Sec. 3) on its small FP64 grid, steps
        # replayed from graphs: latency of a step
        dict(name="cylinder_fp64_128x64", kind="run", dim=2, nx=128, ny=64, nz=1, fp=8, div=8,
             mach=0.1, re=40.0, tw=1.1, steps=20, graphs=10, moving=0, reading=0, stage_forcing=0),
        # the oscillating cylinder (Sec. 5) at its configured size: bins,
        # forced cells and weights rebuilt every step
        dict(name="moving_cylinder_1024x512", kind="run", dim=2, nx=1024, ny=512, nz=1, fp=4, div=32,
             mach=0.2, re=100.0, tw=1.2, steps=20, graphs=10, moving=1, reading=0, stage_forcing=0),
        # the heated sphere (Sec. 4) at full size: the flagship workload
        dict(name="sphere_256", kind="run", dim=3, nx=256, ny=256, nz=256, fp=4, div=32,
             mach=0.3, re=300.0, tw=1.5, steps=10, graphs=0, moving=0, reading=0, stage_forcing=0),
        # a sphere on a grid of odd sizes, cold wall, heat source on the total
        # energy (the other reading of the method)
        dict(name="sphere_ragged_131x97x113", kind="run", dim=3, nx=131, ny=97, nz=113, fp=4, div=16,
             mach=0.5, re=100.0, tw=0.8, steps=10, graphs=0, moving=0, reading=1, stage_forcing=0),
        # a double-precision sphere, as used to check the single-precision runs
        dict(name="sphere_fp64_64", kind="run", dim=3, nx=64, ny=64, nz=64, fp=8, div=8,
             mach=0.3, re=300.0, tw=1.5, steps=5, graphs=0, moving=0, reading=0, stage_forcing=0),
        # a sphere oscillating across the stream: a 3D body whose weights are
        # solved again every step
        dict(name="moving_sphere_96", kind="run", dim=3, nx=96, ny=96, nz=96, fp=4, div=12,
             mach=0.3, re=100.0, tw=1.2, steps=10, graphs=0, moving=1, reading=0, stage_forcing=0),
        # a design-space sweep of 64 uneven 2D cases in one batch
        dict(name="batch_64", kind="batch", ncases=64, nmax=512, layout=4, fp=4, steps=25),
        # one gradient of drag and heat transfer for wall-temperature design,
        # at the adjoint sphere's size (Mach 0.5, Re 100)
        dict(name="gradient_sphere_128", kind="gradient", dim=3, nx=128, ny=128, nz=128, fp=4, div=16,
             mach=0.5, re=100.0, tw=1.5, steps=10, every=5),
        # the same of a 2D cylinder in double precision, for its shape too
        dict(name="gradient_cylinder_fp64_128x64", kind="gradient", dim=2, nx=128, ny=64, nz=1, fp=8,
             div=8, mach=0.3, re=40.0, tw=1.3, steps=20, every=10),
        # a new body placed on the full-size grid (one design of many)
        dict(name="body_256", kind="body", dim=3, nx=256, ny=256, nz=256, fp=4, div=32, mach=0.3,
             re=300.0, tw=1.5),
        # post-processing operators on the fields of a mid-size grid
        dict(name="operators_128", kind="operators", dim=3, nx=128, ny=128, nz=128, fp=4, div=16,
             mach=0.3, re=300.0, tw=1.5),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sizes(rng, dim, lo, hi):
    """nx, ny, nz and the cells per diameter: the body fits with room around it"""
    n = _logint(rng, lo, hi)
    nx = n
    ny = max(lo, int(n * rng.uniform(0.45, 1.0)))
    nz = max(lo, int(n * rng.uniform(0.45, 1.0))) if dim == 3 else 1
    small = min(nx, ny, nz) if dim == 3 else min(nx, ny)
    div = max(6, int(small / rng.uniform(5.0, 9.0)))
    return nx, ny, nz, div


def draw(rng):
    kind = rng.choice(["run"] * 6 + ["batch"] * 2 + ["gradient"] * 2 + ["body", "operators", "rhs"])
    gas = dict(mach=round(rng.uniform(0.2, 0.5), 3), re=round(rng.uniform(40.0, 300.0), 1))
    tw = round(rng.choice([rng.uniform(0.6, 0.85), rng.uniform(1.15, 1.8)]), 3)
    if kind == "batch":
        return dict(kind=kind, ncases=_logint(rng, 2, 64), nmax=_logint(rng, 130, 512),
                    layout=rng.randrange(10, 1000), fp=rng.choice([4, 4, 8]),
                    steps=rng.randrange(5, 21))
    dim = rng.choice([2, 3, 3])
    fp = rng.choice([4, 4, 4, 8])
    if kind == "gradient":
        hi = (96 if dim == 3 else 192) if fp == 8 else (128 if dim == 3 else 512)
        nx, ny, nz, div = _sizes(rng, dim, 48, hi)
        steps = rng.randrange(4, 11)
        return dict(kind=kind, dim=dim, nx=nx, ny=ny, nz=nz, fp=fp, div=div, tw=tw, steps=steps,
                    every=rng.choice([3, 5, steps]), **gas)
    hi = (96 if dim == 3 else 512) if fp == 8 else (224 if dim == 3 else 1024)
    nx, ny, nz, div = _sizes(rng, dim, 48, hi)
    base = dict(kind=kind, dim=dim, nx=nx, ny=ny, nz=nz, fp=fp, div=div, **gas)
    if kind == "rhs":
        return base
    base["tw"] = tw
    if kind in ("body", "operators"):
        return base
    moving = rng.choice([0, 0, 1])
    if moving:   # keep the weights' solve of a moving body within its usual size
        base["div"] = min(div, 14 if dim == 3 else 40)
    return dict(base, steps=2 * rng.randrange(2, 11 if dim == 2 else 6), graphs=rng.choice([0, 2, 4]),
                moving=moving, reading=rng.choice([0, 0, 0, 1]),
                stage_forcing=rng.choice([0, 0, 0, 0, 1]))


# ---- inputs ----------------------------------------------------------------

def _grid(c):
    dim, h = c["dim"], 1.0 / c["div"]
    n = (c["nx"], c["ny"], c["nz"] if dim == 3 else 1)
    lo = (-0.375 * n[0] * h, -0.5 * n[1] * h, -0.5 * n[2] * h if dim == 3 else 0.0)
    side = C.BC_SLIP
    return C.GridDesc(dim=dim, n=n, lo=lo, h=h, fp_bytes=c["fp"], Re=c["re"], Mach=c["mach"],
                      bc=(C.BC_FREESTREAM, C.BC_ZEROGRAD, side, side, side, side),
                      tile=(8, 8, 8) if dim == 3 else (16, 16, 1),
                      forcing_per_stage=c.get("stage_forcing", 0))


def _body(c, g, seed):
    """markers one cell apart on a circle or sphere whose centre moves a little
    with the seed, and their wall temperatures"""
    rng = np.random.Generator(np.random.PCG64(seed))
    if g.dim == 2:
        X = C.circle_markers(C.markers_at_arc_spacing(g.h))
    else:
        X = C.fibonacci_sphere_markers(C.markers_at_cell_spacing(g.h))
    X = X + g.h * rng.uniform(-0.5, 0.5, g.dim)
    Tw = c["tw"] * (1.0 + 0.02 * rng.uniform(-1.0, 1.0, len(X)))
    if c["fp"] == 4:   # design parameters in the grid's precision
        X, Tw = X.astype(np.float32).astype(np.float64), Tw.astype(np.float32).astype(np.float64)
    return X, Tw


def _motion(c):
    return C.Motion(amp=0.2, freq=0.2, axis=1) if c.get("moving") else None


def _state(g, seed, rough=0.0):
    """a stream carrying smooth waves in every variable and 1e-3 density noise;
    rough: noise of that size in every variable too"""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    rng = random.Random(seed)
    shape = tuple(reversed(g.n[: g.dim]))
    f8 = dict(device=DEV, dtype=torch.float64)
    axes = [(torch.arange(m, **f8) + 0.5) / m for m in g.n[: g.dim]]

    def waves(amp):
        out = torch.zeros(shape, **f8)
        for _ in range(3):
            w = torch.ones((), **f8)
            for d, x in enumerate(axes):
                k = 2.0 * math.pi * rng.randrange(1, 5)
                v = torch.sin(k * x + rng.uniform(0.0, 2.0 * math.pi))
                w = w * v.reshape([-1 if i == g.dim - 1 - d else 1 for i in range(g.dim)])
            out = out + amp * w
        return out

    rho = 1.0 + waves(0.02) + 1e-3 * torch.randn(shape, generator=gen, **f8)
    u = [(1.0 if d == 0 else 0.0) + waves(0.03) for d in range(g.dim)]
    p = (1.0 + waves(0.01)) / (g.gamma * g.Mach * g.Mach)
    if rough:
        def noise(s=rough):
            return s * torch.randn(shape, generator=gen, **f8)
        rho, u, p = rho + noise(), [v + noise() for v in u], p * (1.0 + noise())
    E = p / (g.gamma - 1.0) + 0.5 * rho * sum(v * v for v in u)
    U = torch.stack([rho] + [rho * v for v in u] + [E])
    return U.to(torch.float32 if g.fp_bytes == 4 else torch.float64).contiguous()


def _rough(c):
    """operators on fields are called on fields of any kind: rough ones"""
    return 0.03 if c["kind"] in ("rhs", "operators") else 0.0


def _batch_cases(c):
    m = c["nmax"]
    return C.batched_cylinders(c["ncases"], (m // 4, m // 2, (3 * m) // 4, m), c["layout"], c["fp"])


def _batch_tw(cs, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return [k.Tw * (1.0 + 0.02 * rng.uniform(-1.0, 1.0, len(k.Tw))) for k in cs]


def prepare(case, seed):
    c, s = case, {"case": case}
    if c["kind"] == "batch":
        cs = _batch_cases(c)
        b = ibm.Batch([k.grid for k in cs], [len(k.X) for k in cs])
        for k, gr, Tw in zip(cs, b.cases, _batch_tw(cs, seed)):
            gr.set_markers(k.X, Tw)
        s["batch"] = b
        s["U"] = [_state(k.grid, 1000 * seed + i) for i, k in enumerate(cs)]
        return s
    g = _grid(c)
    s["U"] = _state(g, seed, _rough(c))
    if c["kind"] == "rhs":
        s["desc"] = ibm.make_desc(g)
        s["L"] = torch.empty_like(s["U"])
        s["dt"] = torch.empty(1, dtype=torch.float64, device=DEV)
        return s
    X, Tw = _body(c, g, seed)
    s["grid"] = grid = ibm.Grid(g, max_markers=len(X), energy_reading=c.get("reading", 0))
    s["X"], s["Tw"] = X, Tw
    if c["kind"] == "gradient":
        t = torch.float32 if c["fp"] == 4 else torch.float64
        s["Xt"] = torch.from_numpy(X).to(t).requires_grad_(c["fp"] == 8)
        s["Twt"] = torch.from_numpy(Tw).to(t).requires_grad_()
        s["J"] = ibm.cd_nu_objective()
    elif c["kind"] in ("run", "operators"):
        grid.set_markers(X, Tw, motion=_motion(c))
        s["idx"] = grid.markers()[2]
        if c.get("graphs"):
            grid.use_graphs(c["graphs"])
    if c["kind"] == "operators":
        grid.set_state(s["U"])
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed + 1)
        s["R"] = torch.randn((grid.n_kept, g.dim + 1), generator=gen, device=DEV, dtype=torch.float64)
    return s


# ---- one pass ----------------------------------------------------------------

def _kept(c, v):
    """marker values of an FP32 grid, kept in its own precision"""
    return v.astype(np.float32) if c["fp"] == 4 else v


def _full(n, idx, v):
    """kept-marker values in the order of the input markers (0 where dropped)"""
    out = np.zeros((n,) + v.shape[1:], v.dtype)
    out[idx] = v
    return out


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "rhs":
        ibm.ibm_rhs_dt_noalloc(s["desc"], s["U"].data_ptr(), s["L"].data_ptr(), s["dt"].data_ptr(),
                               torch.cuda.current_stream().cuda_stream)
        return {"L": s["L"], "dt": s["dt"].to(s["U"].dtype)}
    if kind == "batch":
        b = s["batch"]
        for gr, U in zip(b.cases, s["U"]):
            gr.set_state(U)
        b.step(c["steps"])
        return {"forces": _kept(c, b.forces()[:, :2]),
                "state": torch.cat([gr.get_state().reshape(-1) for gr in b.cases])}
    grid = s["grid"]
    if kind == "run":
        grid.set_state(s["U"])
        grid.step(c["steps"])
        rho, F, Q = grid.marker_forcing()
        idx, n = s["idx"], len(s["X"])
        return {"rho": _full(n, idx, _kept(c, rho)), "F": _full(n, idx, _kept(c, F)),
                "Q": _full(n, idx, _kept(c, Q)), "state": grid.get_state()}
    if kind == "gradient":
        s["Xt"].grad = s["Twt"].grad = None
        J = s["J"].apply(s["Xt"], s["Twt"], grid, s["U"], c["steps"], 1.0, 0.5, c["every"])
        J.backward()
        if c["fp"] == 4:
            return {"dTw": s["Twt"].grad}
        return {"J": J.detach(), "dX": s["Xt"].grad, "dTw": s["Twt"].grad}
    if kind == "body":
        grid.set_markers(s["X"], s["Tw"])
        X, eps, idx = grid.markers()
        n = len(s["X"])
        return {"X": _full(n, idx, X), "eps": _full(n, idx, eps)}
    L = grid.rhs(s["U"])
    I = grid.interpolate(s["U"])
    S = grid.spread(s["R"])
    cp = grid.surface_pressure()
    _, _, idx = grid.markers()
    n = len(s["X"])
    return {"L": L, "I": _full(n, idx, _kept(c, I.cpu().numpy())), "S": S, "cp": _full(n, idx, cp)}


# ---- what a pass cannot do without -------------------------------------------

def _stage_flops(dim):
    """floating-point operations of one cell and stage: per face two limited
    slopes are shared with the neighbours (one per cell and axis), then the
    two states' fluxes and the viscous terms; conversion and update"""
    nc = dim + 2
    face = nc * (2 + 5 + 2) + 2 * (4 * dim + 12) + 6 * nc + (14 * dim + 20)
    return dim * face + 4 * nc + 12


def work(case):
    c = case
    if c["kind"] == "batch":
        N = sum(k.grid.ncells for k in _batch_cases(c))
        return {"bytes": c["steps"] * 2 * 4 * c["fp"] * N, "flops": c["steps"] * 2 * _stage_flops(2) * N}
    dim, nc = c["dim"], c["dim"] + 2
    N = c["nx"] * c["ny"] * c["nz"]
    ns = math.pi * (c["div"] ** (dim - 1))
    state = nc * c["fp"] * N
    if c["kind"] == "rhs":
        return {"bytes": 2 * state, "flops": (_stage_flops(dim) + 30) * N}
    if c["kind"] == "run":   # each step reads the state and writes the next
        return {"bytes": c["steps"] * 2 * state, "flops": c["steps"] * 2 * _stage_flops(dim) * N}
    if c["kind"] == "gradient":   # forward, then a reversed step of about three forward ones
        return {"bytes": c["steps"] * 6 * state, "flops": c["steps"] * 8 * _stage_flops(dim) * N}
    if c["kind"] == "body":   # positions and temperatures in, positions and weights out
        return {"bytes": ns * (2 * dim + 2) * 8, "flops": ns * 5 ** dim * 60}
    return {"bytes": 2 * state + (dim + 1) * c["fp"] * N + ns * (3 * dim + 4) * 8,
            "flops": _stage_flops(dim) * N}


# ---- 64-bit values -------------------------------------------------------------
# The method in plain torch: state (dim+2, [nz,] ny, nx), axis d of the grid is
# tensor dimension -(d + 1).

def _gas(g):
    R = 1.0 / (g.gamma * g.Mach ** 2)
    cv = R / (g.gamma - 1.0)
    return R, cv, g.gamma * cv, 1.0 / g.Re if g.Re > 0 else 0.0


def _ghosts(U, g):
    """two ghost layers per axis: free stream, zero gradient, mirror or periodic"""
    stream = [1.0, 1.0] + [0.0] * (g.dim - 1) + [1.0 / (g.gamma * g.Mach ** 2) / (g.gamma - 1.0) + 0.5]
    fs = None
    for d in range(g.dim):
        n = g.n[d]
        idx, sign, free = [], [], []
        for i in range(-2, n + 2):
            bc = -1 if 0 <= i < n else g.bc[2 * d + (i >= n)]
            mirror = -1 - i if i < 0 else 2 * n - 1 - i
            idx.append(i if bc < 0 else i % n if bc == C.BC_PERIODIC else mirror if bc == C.BC_SLIP
                       else min(max(i, 0), n - 1))
            sign.append(-1.0 if bc == C.BC_SLIP else 1.0)
            free.append(bc == C.BC_FREESTREAM)
        U = U.index_select(U.dim() - 1 - d, torch.tensor(idx, device=U.device))
        along = [-1 if e == d else 1 for e in reversed(range(g.dim))]
        sg = torch.tensor(sign, device=U.device, dtype=U.dtype).reshape(along)
        U = torch.stack([U[m] * sg if m == 1 + d else U[m] for m in range(g.dim + 2)])
        f = torch.tensor(free, device=U.device).reshape(along)
        fs = f if fs is None else fs | f
    return torch.stack([torch.where(fs, torch.full_like(U[m], stream[m]), U[m])
                        for m in range(g.dim + 2)])


def _limited(a, b):
    ab = a * b
    up = ab > 0
    return torch.where(up, 2.0 * ab / torch.where(up, a + b, torch.ones_like(a)), torch.zeros_like(a))


def _L(U, g):
    """rate of change: MUSCL/van Leer, Rusanov, central viscous and heat fluxes"""
    R, cv, cp, mu0 = _gas(g)
    dim = g.dim
    V = _ghosts(U, g)
    rho = V[0]
    vel = [V[1 + d] / rho for d in range(dim)]
    p = (g.gamma - 1.0) * (V[dim + 1] - 0.5 * rho * sum(v * v for v in vel))
    T = p / (rho * R)
    out = torch.zeros_like(U)
    for d in range(dim):
        def at(w, off, e=None, sh=0):
            """cells beside the faces of axis d (off 0: lower, 1: upper), shifted by sh along e"""
            for a in range(dim):
                start = 1 + off if a == d else 2 + (sh if a == e else 0)
                w = w.narrow(w.dim() - 1 - a, start, g.n[a] + (1 if a == d else 0))
            return w
        order = [rho] + vel + [p]
        wl, wr = [], []
        for w in order:
            am, a, b, bp = at(w, -1), at(w, 0), at(w, 1), at(w, 2)
            wl.append(a + 0.5 * _limited(a - am, b - a))
            wr.append(b - 0.5 * _limited(b - a, bp - b))

        def side(w):
            r, v, q = w[0], w[1:-1], w[-1]
            E = q / (g.gamma - 1.0) + 0.5 * r * sum(x * x for x in v)
            un = v[d]
            F = [r * un] + [r * x * un + (q if m == d else 0.0) for m, x in enumerate(v)] + [(E + q) * un]
            return [r] + [r * x for x in v] + [E], F, un.abs() + torch.sqrt(g.gamma * q / r)
        UL, FL, sL = side(wl)
        UR, FR, sR = side(wr)
        s = torch.maximum(sL, sR)
        F = [0.5 * (fl + fr) - 0.5 * s * (ur - ul) for fl, fr, ul, ur in zip(FL, FR, UL, UR)]
        if mu0 > 0.0:
            Ta, Tb = at(T, 0), at(T, 1)
            Tf = 0.5 * (Ta + Tb)
            mu = mu0 * Tf * torch.sqrt(Tf) * (1.0 + g.sutherland_S) / (Tf + g.sutherland_S)
            grad = [[None] * dim for _ in range(dim)]
            for m in range(dim):
                for e in range(dim):
                    if e == d:
                        grad[m][e] = (at(vel[m], 1) - at(vel[m], 0)) / g.h
                    else:
                        grad[m][e] = (at(vel[m], 0, e, 1) - at(vel[m], 0, e, -1) + at(vel[m], 1, e, 1) -
                                      at(vel[m], 1, e, -1)) / (4.0 * g.h)
            div = sum(grad[m][m] for m in range(dim))
            heat = mu * cp / g.Pr * (Tb - Ta) / g.h
            for m in range(dim):
                tau = mu * (grad[d][m] + grad[m][d])
                if m == d:
                    tau = tau - 2.0 / 3.0 * mu * div
                F[1 + m] = F[1 + m] - tau
                heat = heat + 0.5 * (at(vel[m], 0) + at(vel[m], 1)) * tau
            F[dim + 1] = F[dim + 1] - heat
        F = torch.stack(F)
        ax = F.dim() - 1 - d
        out = out - (F.narrow(ax, 1, g.n[d]) - F.narrow(ax, 0, g.n[d])) / g.h
    return out


def _dt(U, g):
    R, cv, cp, mu0 = _gas(g)
    rho = U[0]
    vel = [U[1 + d] / rho for d in range(g.dim)]
    p = (g.gamma - 1.0) * (U[g.dim + 1] - 0.5 * rho * sum(v * v for v in vel))
    T = p / (rho * R)
    mu = mu0 * T * torch.sqrt(T) * (1.0 + g.sutherland_S) / (T + g.sutherland_S)
    c = torch.sqrt(g.gamma * p / rho)
    s = (sum(v.abs() for v in vel) + g.dim * c) / g.h + \
        2.0 * g.dim * max(4.0 / 3.0, g.gamma / g.Pr) * mu / rho / g.h ** 2
    return (g.cfl / s.max()).detach()


def _phi(r):
    a = r.abs()
    one = torch.ones_like(a)
    inner = torch.where(a <= 0.5, 1.0 - 3.0 * a * a, one)
    b = 1.0 - a
    mid = (a > 0.5) & (a <= 1.5)
    outer = torch.where(mid, 1.0 - 3.0 * b * b, one)
    # the root is taken of positive numbers only, so its derivative is finite
    tail = (5.0 - 3.0 * a - torch.sqrt(outer.clamp_min(1e-300))) / 6.0
    return torch.where(a <= 0.5, (1.0 + torch.sqrt(inner)) / 3.0, torch.where(mid, tail, 0.0 * a))


def _owner(X, g):
    lo = torch.tensor(g.lo[: g.dim], device=X.device, dtype=X.dtype)
    return torch.floor((X - lo) / g.h).long()


def _keep(X, g):
    """one marker per cell: the one closest to the cell centre"""
    Xn = X.detach()
    cell = _owner(Xn, g).cpu().numpy()
    lo = np.array(g.lo[: g.dim])
    x = Xn.cpu().numpy()
    dist = ((x - (lo + (cell + 0.5) * g.h)) ** 2).sum(1)
    best = {}
    for k in range(len(x)):
        key = tuple(cell[k])
        if key not in best or dist[k] < dist[best[key]]:
            best[key] = k
    return torch.tensor(sorted(best.values()), device=X.device)


class _Body:
    """support weights and quadrature weights of markers at X (differentiable)"""

    def __init__(self, X, g):
        dim = g.dim
        cell = _owner(X.detach(), g)
        lo = torch.tensor(g.lo[:dim], device=X.device, dtype=X.dtype)
        frac = (X - lo) / g.h - cell
        o = torch.arange(-1, 2, device=X.device)
        w1 = _phi(o + 0.5 - frac[:, :, None])                 # (ns, dim, 3)
        A = None
        for d in range(dim):
            same = (cell[:, d, None, None, None] + o[None, None, :, None] ==
                    cell[None, :, d, None, None] + o[None, None, None, :]).to(X.dtype)
            a = torch.einsum("ki,klij,lj->kl", w1[:, d], same, w1[:, d])
            A = a if A is None else A * a
        self.eps = torch.linalg.solve(A, torch.ones(len(X), 1, device=X.device, dtype=X.dtype))[:, 0]
        w, j, stride = w1[:, 0], cell[:, 0, None] + o, g.n[0]
        for d in range(1, dim):
            w = (w1[:, d, :, None] * w[:, None, :]).reshape(len(X), -1)
            j = ((cell[:, d, None] + o)[:, :, None] * stride + j[:, None, :]).reshape(len(X), -1)
            stride *= g.n[d]
        self.w, self.j = w, j                                  # (ns, 3^dim)

    def interpolate(self, f):
        """(nc, N) -> (ns, nc)"""
        return (f[:, self.j.reshape(-1)].reshape(len(f), *self.j.shape) * self.w).sum(-1).T

    def spread(self, R, N):
        """(ns, nc) -> (nc, N)"""
        v = (R * self.eps[:, None]).T[:, :, None] * self.w
        return torch.zeros(R.shape[1], N, device=R.device, dtype=R.dtype).index_add(
            1, self.j.reshape(-1), v.reshape(len(v), -1))


def _force(U, b, Ub, Tw, g, reading):
    """the direct forcing of one state: (forced state, G = dt F, H = dt Q, rho_L)"""
    _, cv, _, _ = _gas(g)
    V = U.reshape(g.dim + 2, -1)
    rho, mom, E = V[0], V[1:-1], V[-1]
    re = E - (mom * mom).sum(0) / (2.0 * rho)
    at = b.interpolate(torch.cat([V[:-1], re[None]]))
    G = at[:, :1] * Ub - at[:, 1:-1]
    H = at[:, 0] * cv * Tw - at[:, -1]
    S = b.spread(torch.cat([G, H[:, None]], 1), V.shape[1])
    q = torch.maximum(S[-1], -0.9 * re)
    m2 = mom + S[:-1]
    E2 = E + q if reading else re + q + (m2 * m2).sum(0) / (2.0 * rho)
    return torch.cat([rho[None], m2, E2[None]]).reshape(U.shape), G, H, at[:, 0]


def _steps(U, X, Tw, motion, g, steps, reading, checkpoint=False):
    """k steps from U: (state, G, H, rho_L, dt, b) of the last one"""
    Ub = torch.zeros_like(X)
    b = None if motion else _Body(X, g)
    t = torch.zeros((), device=U.device, dtype=U.dtype)
    X0 = X
    for _ in range(steps):
        dt = _dt(U, g)
        t = t + dt
        if motion:
            w = 2.0 * math.pi * motion.freq
            e = torch.zeros(g.dim, device=U.device, dtype=U.dtype)
            e[motion.axis] = 1.0
            b = _Body(X0 + motion.amp * torch.sin(w * t) * e, g)
            Ub = (motion.amp * w * torch.cos(w * t) * e).expand_as(X0)

        def fluid(U, dt=dt, b=b, Ub=Ub):
            U1 = U + dt * _L(U, g)
            if g.forcing_per_stage:
                U1 = _force(U1, b, Ub, Tw, g, reading)[0]
            return 0.5 * U + 0.5 * (U1 + dt * _L(U1, g))
        if checkpoint:
            Us = torch.utils.checkpoint.checkpoint(fluid, U, use_reentrant=False)
        else:
            Us = fluid(U)
        U, G, H, rho = _force(Us, b, Ub, Tw, g, reading)
    return U, G, H, rho, dt, b


def _coefficients(G, H, Tw, dt, b, g):
    """(force on the body, Cd, Nu) from the last step's forcing"""
    hd = g.h ** g.dim
    F = -hd * (b.eps[:, None] * G).sum(0) / dt
    Q = hd * (b.eps * H).sum() / dt
    _, _, cp, mu0 = _gas(g)
    lref = g.D if g.dim == 2 else math.pi * g.D ** 2 / 4.0
    area = math.pi * g.D if g.dim == 2 else math.pi * g.D ** 2
    return F, 2.0 * F[0] / lref, Q * g.D / (mu0 * cp / g.Pr * area * (Tw.mean() - 1.0))


def _exact_batch(c, seed):
    cs = _batch_cases(c)
    forces, states = [], []
    for i, (k, Tw) in enumerate(zip(cs, _batch_tw(cs, seed))):
        g = k.grid
        X = torch.from_numpy(k.X).to(DEV)
        keep = _keep(X, g)
        T = torch.from_numpy(Tw).to(DEV)[keep]
        U, G, H, _, dt, b = _steps(_state(g, 1000 * seed + i).double(), X[keep], T, None, g,
                                   c["steps"], 0)
        forces.append(_coefficients(G, H, T, dt, b, g)[0])
        states.append(U.reshape(-1))
    return {"forces": torch.stack(forces), "state": torch.cat(states)}


def exact(case, seed):
    c = case
    if c["kind"] == "batch":
        with torch.no_grad():
            return _exact_batch(c, seed)
    g = _grid(c)
    U = _state(g, seed, _rough(c)).double()
    if c["kind"] == "rhs":
        return {"L": _L(U, g), "dt": _dt(U, g).reshape(1)}
    X, Tw = (torch.from_numpy(v).to(DEV) for v in _body(c, g, seed))
    keep = _keep(X, g)
    n = len(X)

    def full(v):
        return torch.zeros((n,) + v.shape[1:], device=DEV, dtype=v.dtype).index_copy(0, keep, v)

    if c["kind"] == "run":
        with torch.no_grad():
            U, G, H, rho, dt, _ = _steps(U, X[keep], Tw[keep], _motion(c), g, c["steps"], c["reading"])
        return {"rho": full(rho), "F": full(G / dt), "Q": full(H / dt), "state": U}
    if c["kind"] == "gradient":
        X.requires_grad_()
        Tw.requires_grad_()
        _, G, H, _, dt, b = _steps(U, X[keep], Tw[keep], None, g, c["steps"], 0, checkpoint=True)
        _, cd, nu = _coefficients(G, H, Tw[keep], dt, b, g)
        J = cd + 0.5 * nu
        dX, dTw = torch.autograd.grad(J, (X, Tw))
        return {"dTw": dTw} if c["fp"] == 4 else {"J": J.detach(), "dX": dX, "dTw": dTw}
    b = _Body(X[keep], g)
    if c["kind"] == "body":
        return {"X": full(X[keep]), "eps": full(b.eps)}
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed + 1)
    R = torch.randn((len(keep), g.dim + 1), generator=gen, device=DEV, dtype=torch.float64)
    V = U.reshape(g.dim + 2, -1)
    p = (g.gamma - 1.0) * (V[-1] - (V[1:-1] ** 2).sum(0) / (2.0 * V[0]))
    cp = 2.0 * (b.interpolate(p[None])[:, 0] - 1.0 / (g.gamma * g.Mach ** 2))
    S = b.spread(R, V.shape[1]).reshape((g.dim + 1,) + U.shape[1:])
    return {"L": _L(U, g), "I": full(b.interpolate(V)), "S": S, "cp": full(cp)}
