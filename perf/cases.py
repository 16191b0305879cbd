"""What a user of this framework has it do, as cases that can be timed and compared.

A case names a kind of call, a precision and a grid; every kind goes through the package's public
entry points (``Plan``, ``BatchPlan``, ``ProjectionFn``).  The grids are the channel of the solver
(periodic x and z with Lx = 2 pi and Lz = pi, tanh-stretched walls at y = -1 and 1), the inputs
seeded fields of the kinds a simulation meets: the divergence of a random staggered velocity as a
right-hand side, the laminar profile plus noise as a flow state, uniform weights as the gradient of
a loss.

``exact`` restates every kind in plain torch FP64 (library FFTs, a tridiagonal elimination
vectorised over the modes, rolled neighbour differences) and uses nothing of the package.
"""
import math

import numpy as np
import torch

import paper_2104_08863_gb300 as P

LX, LZ = 2.0 * math.pi, math.pi
NU = 1.0 / 550.0
FX = 2.0 * NU
F64, F32, REFINED = "f64", "f32", "refined"
PRECISION = {F64: P.PP_FP64, F32: P.PP_FP32, REFINED: P.PP_FP32_REFINED}
BATCH_NX_NZ = (64, 96, 128, 192, 256, 384)
BATCH_NY = (48, 64, 96, 128, 192)


def listed():
    return [
        # the smallest call: one small channel's pressure, where launches and latency are the time
        dict(name="solve_f64_32", kind="solve", prec=F64, nx=32, ny=32, nz=32, stretch=1.5, thomas=True),
        # a laminar or start-up run on a small grid: whole timesteps in a loop
        dict(name="timestep_f64_64", kind="timestep", prec=F64, nx=64, ny=64, nz=64, stretch=1.5),
        # grids that are no power of two in any direction (2^a 3^b lengths, any number of rows)
        dict(name="solve_f32_162x90x108", kind="solve", prec=F32, nx=162, ny=90, nz=108, stretch=1.7),
        dict(name="solve_f64_216x130x162", kind="solve", prec=F64, nx=216, ny=130, nz=162, stretch=1.7),
        # gradient of a loss through one FP64-accurate solve
        dict(name="adjoint_refined_192x96x192", kind="adjoint", prec=REFINED, nx=192, ny=96, nz=192, stretch=1.8, steps=2),
        # training through the projection: forward and hand-written backward under autograd
        dict(name="project_grad_f32_256x192x256", kind="grad", prec=F32, nx=256, ny=192, nz=256, stretch=1.8),
        # an ensemble of channels of uneven sizes, solved in one launch
        dict(name="batch_f32_64", kind="batch", prec=F32, count=64, sizes=5),
        # a single-precision run
        dict(name="timestep_f32_384x192x256", kind="timestep", prec=F32, nx=384, ny=192, nz=256, stretch=1.8),
        dict(name="solve_f32_768x384x512", kind="solve", prec=F32, nx=768, ny=384, nz=512, stretch=2.0),
        # the production timestep in FP64 (PDD with 8 blocks), and its FP64-accurate form on FP32 units
        dict(name="timestep_f64_512x384x512", kind="timestep", prec=F64, nx=512, ny=384, nz=512, stretch=2.0),
        dict(name="timestep_refined_512x384x512", kind="timestep", prec=REFINED, nx=512, ny=384, nz=512, stretch=2.0, steps=2),
        # the largest grid: the FP32 solve with one FP64-accurate correction
        dict(name="solve_refined_1536x768x1024", kind="solve", prec=REFINED, nx=1536, ny=768, nz=1024, stretch=2.2, steps=1),
    ]


# Most points of a drawn grid per (kind, precision), so that no draw costs more than the largest
# listed case.
CAP = {("solve", F64): 1.0e8, ("solve", F32): 9.0e8, ("solve", REFINED): 5.0e8,
       ("adjoint", F64): 9.0e7, ("adjoint", F32): 5.0e8, ("adjoint", REFINED): 2.0e8,
       ("grad", F64): 6.0e7, ("grad", F32): 2.5e8,
       ("timestep", F64): 5.0e7, ("timestep", F32): 2.0e8, ("timestep", REFINED): 8.0e7}


def _smooth(lo, hi, even):
    """Lengths of the form 2^a 3^b in [lo, hi] (twice such a length when even)."""
    out = set()
    for a in range(11):
        for b in range(7):
            n = 2 ** a * 3 ** b * (2 if even else 1)
            if lo <= n <= hi:
                out.add(n)
    return sorted(out)


def draw(rng):
    if rng.random() < 0.1:
        return dict(kind="batch", prec=F32, count=rng.randint(4, 48), sizes=rng.randint(0, 10 ** 6))
    kind, prec = rng.choice(sorted(CAP))
    target = math.exp(rng.uniform(math.log(3.0e4), math.log(0.98 * CAP[kind, prec])))
    while True:
        nx = rng.choice(_smooth(16, 1536, True))
        nz = rng.choice(_smooth(16, 1024, False))
        ny = int(round(target / (nx * nz)))
        if 16 <= ny <= 768 and nx * ny * nz <= CAP[kind, prec]:
            break
    if rng.random() < 0.6:
        ny += ny % 2 * (-1 if ny > 17 else 1)
    c = dict(kind=kind, prec=prec, nx=nx, ny=ny, nz=nz, stretch=round(rng.uniform(1.0, 2.2), 3))
    if prec == REFINED:
        c["steps"] = rng.randint(1, 2)
    return c


# ------------------------------------------------------------------------------ grid and inputs
class Grid:
    """Metrics of the stretched channel in FP64."""

    def __init__(self, nx, ny, nz, stretch):
        j = np.arange(ny + 1, dtype=np.float64)
        y = np.tanh(stretch * (2.0 * j / ny - 1.0)) / np.tanh(stretch)
        y[0], y[-1] = -1.0, 1.0
        yc = 0.5 * (y[1:] + y[:-1])
        self.nx, self.ny, self.nz, self.faces, self.centres = nx, ny, nz, y, yc
        self.dx, self.dz, self.dy = LX / nx, LZ / nz, np.diff(y)
        self.h = np.zeros(ny + 1)
        self.h[1:ny] = np.diff(yc)

    def rows(self, a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()[:, None, None]


def _grid(c):
    return Grid(c["nx"], c["ny"], c["nz"], c["stretch"])


def _batch_sizes(c):
    rng = np.random.default_rng(c["sizes"])
    out = []
    for _ in range(c["count"]):
        nx, nz, ny = int(rng.choice(BATCH_NX_NZ)), int(rng.choice(BATCH_NX_NZ)), int(rng.choice(BATCH_NY))
        out.append(dict(nx=nx, ny=ny, nz=nz, stretch=float(rng.uniform(1.0, 2.5))))
    return out


def _dtype(c):
    return torch.float32 if c["prec"] == F32 else torch.float64


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(gen, shape, scale=1.0):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64).mul_(scale)


def _rhs(g, gen):
    """The divergence of a N(0, 1) staggered velocity (one field at a time, to save memory)."""
    cell, face = (g.ny, g.nz, g.nx), (g.ny + 1, g.nz, g.nx)
    u = _normal(gen, cell)
    f = (torch.roll(u, -1, 2) - u).div_(g.dx)
    del u
    w = _normal(gen, cell)
    f += (torch.roll(w, -1, 1) - w).div_(g.dz)
    del w
    v = _normal(gen, face)
    f += (v[1:] - v[:-1]).div_(g.rows(g.dy))
    return f


def _flow(g, gen):
    """Laminar profile plus N(0, 0.1^2) on every component, v = 0 on the walls."""
    u = _normal(gen, (g.ny, g.nz, g.nx), 0.1)
    u += g.rows(1.0 - g.centres ** 2)
    v = _normal(gen, (g.ny + 1, g.nz, g.nx), 0.1)
    v[0] = 0.0
    v[-1] = 0.0
    return u, v, _normal(gen, (g.ny, g.nz, g.nx), 0.1)


def _dt(g):
    """A stable explicit step: convection and the wall-normal diffusion limit, at most 1e-4."""
    return float(min(1e-4, 0.05 * min(g.dx, g.dz), 0.15 * g.dy.min() ** 2 / NU))


def _inputs(c, seed):
    """The arrays a call reads, in the case's precision."""
    gen, dt = _gen(seed), _dtype(c)
    if c["kind"] == "batch":
        return [_rhs(Grid(s["nx"], s["ny"], s["nz"], s["stretch"]), gen).to(dt) for s in _batch_sizes(c)]
    g = _grid(c)
    cell, face = (g.ny, g.nz, g.nx), (g.ny + 1, g.nz, g.nx)
    if c["kind"] == "solve":
        return [_rhs(g, gen).to(dt)]
    if c["kind"] == "adjoint":
        return [torch.rand(cell, generator=gen, device="cuda", dtype=torch.float64).mul_(2).sub_(1).to(dt)]
    if c["kind"] == "timestep":
        return [a.to(dt) for a in _flow(g, gen)]
    fields = [_normal(gen, s).to(dt) for s in (cell, face, cell)]
    weights = [torch.rand(s, generator=gen, device="cuda", dtype=torch.float64).mul_(2).sub_(1).to(dt)
               for s in (cell, face, cell)]
    return fields + weights


# ------------------------------------------------------------------------------ the measured calls
def _plan(c):
    g = _grid(c)
    return P.Plan(c["nx"], c["ny"], c["nz"], g.faces, LX, LZ, precision=PRECISION[c["prec"]],
                  tridiag=P.PT_THOMAS if c.get("thomas") else P.PT_AUTO, refine_steps=c.get("steps", 1))


def prepare(case, seed):
    c = dict(case)
    x = _inputs(c, seed)
    s = dict(case=c, x=x)
    if c["kind"] == "batch":
        specs = [dict(nx=z["nx"], ny=z["ny"], nz=z["nz"],
                      y_faces=Grid(z["nx"], z["ny"], z["nz"], z["stretch"]).faces) for z in _batch_sizes(c)]
        s["plan"] = P.BatchPlan(specs, precision=PRECISION[c["prec"]])
        s["out"] = [torch.empty_like(r) for r in x]
        return s
    s["plan"] = _plan(c)
    if c["kind"] in ("solve", "adjoint"):
        s["out"] = torch.empty_like(x[0])
    elif c["kind"] == "timestep":
        s["dt"] = _dt(_grid(c))
        s["scratch"] = tuple(torch.empty_like(a) for a in x)
        # the FP32 step's pressure is not asked for: between two steps of nearly divergence-free
        # velocity it is the divergence's rounding, not a result
        s["p"] = None if c["prec"] == F32 else torch.empty_like(x[0])
    else:
        s["dt"] = 1e-3
        for a in x[:3]:
            a.requires_grad_(True)
    return s


def run(state):
    kind, x, plan = state["case"]["kind"], state["x"], state["plan"]
    if kind == "solve":
        return plan.solve(x[0], out=state["out"])
    if kind == "adjoint":
        return plan.solve_adjoint(x[0], out=state["out"])
    if kind == "batch":
        return plan.solve(x, out=state["out"])
    if kind == "timestep":   # in place, as a time loop runs it
        plan.timestep(x[0], x[1], x[2], state["dt"], NU, FX, p_out=state["p"], scratch=state["scratch"])
        return [x[0], x[1], x[2]] + ([] if state["p"] is None else [state["p"]])
    out = P.ProjectionFn.apply(x[0], x[1], x[2], plan, state["dt"])
    grads = torch.autograd.grad(out, x[:3], grad_outputs=x[3:])
    return [a.detach() for a in out] + list(grads)


# ------------------------------------------------------------------------------ size and tolerance
def _solve_flops(nx, ny, nz):
    n = nx * ny * nz
    return n * (2 * (2.5 * math.log2(nx) + 2.5 * math.log2(nz)) + 10.0)


def work(case):
    c = dict(case)
    es = 4 if c["prec"] == F32 else 8
    if c["kind"] == "batch":
        z = _batch_sizes(c)
        return dict(bytes=sum(2 * es * s["nx"] * s["ny"] * s["nz"] for s in z),
                    flops=sum(_solve_flops(s["nx"], s["ny"], s["nz"]) for s in z))
    n = c["nx"] * c["ny"] * c["nz"]
    solve = _solve_flops(c["nx"], c["ny"], c["nz"])
    if c["kind"] in ("solve", "adjoint"):
        return dict(bytes=2 * es * n, flops=solve)
    if c["kind"] == "timestep":   # velocity in and out, pressure out; two momentum stages, D, G
        return dict(bytes=(6 if c["prec"] == F32 else 7) * es * n, flops=solve + (188 + 18) * n)
    return dict(bytes=12 * es * n, flops=2 * (solve + 18 * n))


def tolerance(case):
    """About four times the largest error against ``exact`` seen over the listed and 60 drawn grids.

    Two FP64-accurate steps in a row: the second step's pressure is the divergence of a velocity
    that the first made divergence-free, over dt, so it carries the velocity's rounding over
    dt times the cell size: 2e-10 (FP64) and 2e-9 (refined) of it were seen."""
    step = case["kind"] == "timestep"
    if case["prec"] == F32:
        return {"rel": 2e-5, "max": 8e-4}
    if case["prec"] == F64:
        return {"rel": 1e-9, "max": 3e-9} if step else {"rel": 1e-13, "max": 1e-12}
    if step:
        return {"rel": 1e-8, "max": 4e-8}
    return {"rel": 1e-10, "max": 1.6e-9} if case["steps"] == 1 else {"rel": 1e-12, "max": 1e-11}


# ------------------------------------------------------------------------------ plain FP64 restatement
def _xm(a):
    return torch.roll(a, 1, 2)


def _xp(a):
    return torch.roll(a, -1, 2)


def _zm(a):
    return torch.roll(a, 1, 1)


def _zp(a):
    return torch.roll(a, -1, 1)


def _poisson(g, f):
    """p with L_h p = f - <f> and zero dy-weighted mean, all in FP64 (f is not kept)."""
    ny, m = g.ny, g.nx // 2 + 1
    lo, up = np.zeros(ny), np.zeros(ny)
    lo[1:] = 1.0 / (g.dy[1:] * g.h[1:ny])
    up[:-1] = 1.0 / (g.dy[:-1] * g.h[1:ny])
    lx = (2.0 / g.dx * np.sin(np.pi * np.arange(m) / g.nx)) ** 2
    lz = (2.0 / g.dz * np.sin(np.pi * np.arange(g.nz) / g.nz)) ** 2
    sigma = torch.from_numpy(lz[:, None] + lx[None, :]).cuda()
    sigma[0, 0] = 1.0   # the singular mode is done apart
    F = torch.empty((ny, g.nz, m), dtype=torch.complex128, device="cuda")
    rows = max(1, int(2 ** 27 // (g.nz * g.nx)))
    for j in range(0, ny, rows):
        F[j:j + rows] = torch.fft.rfft2(f[j:j + rows], dim=(1, 2))
    F0 = F[:, 0, 0].cpu().numpy().real.copy()
    # elimination with the pivot's excess over the upper coefficient carried, all terms positive
    rb = torch.empty((ny, g.nz, m), dtype=torch.float64, device="cuda")
    e = sigma.clone()
    for j in range(ny):
        if j:
            mult = rb[j - 1] * lo[j]
            e.mul_(mult).add_(sigma)
            F[j].add_(F[j - 1] * mult)
        torch.reciprocal(e + up[j], out=rb[j])
    for j in range(ny - 1, -1, -1):
        if j < ny - 1:
            F[j].add_(F[j + 1], alpha=-float(up[j]))
        F[j].mul_(rb[j]).neg_()
    # (0, 0): flux sums, then the pressure differences, in extended precision on the host
    dy, F0 = g.dy.astype(np.longdouble), F0.astype(np.longdouble)
    q = np.cumsum(dy * (F0 - np.sum(dy * F0) / np.sum(dy)))
    p0 = np.concatenate([[0.0], np.cumsum(g.h[1:ny].astype(np.longdouble) * q[:-1])])
    p0 = p0 - np.sum(dy * p0) / np.sum(dy)
    F[:, 0, 0] = torch.from_numpy(p0.astype(np.float64)).cuda().to(torch.complex128)
    del rb
    p = torch.empty((ny, g.nz, g.nx), dtype=torch.float64, device="cuda")
    for j in range(0, ny, rows):
        p[j:j + rows] = torch.fft.irfft2(F[j:j + rows], s=(g.nz, g.nx), dim=(1, 2))
    return p


def _divergence(g, u, v, w):
    return (_xp(u) - u) / g.dx + (v[1:] - v[:-1]) / g.rows(g.dy) + (_zp(w) - w) / g.dz


def _project(g, u, v, w, dt):
    p = _poisson(g, _divergence(g, u, v, w) / dt)
    v = v.clone()
    v[1:g.ny] -= dt * (p[1:] - p[:-1]) / g.rows(g.h[1:g.ny])
    return u - dt * (p - _xm(p)) / g.dx, v, w - dt * (p - _zm(p)) / g.dz, p


def _project_transposed(g, gu, gv, gw):
    """g - D^T S^T G^T g, with S^T r = W S(W^-1 r)."""
    r = (gu - _xp(gu)) / g.dx + (gw - _zp(gw)) / g.dz
    s = gv[1:g.ny] / g.rows(g.h[1:g.ny])
    r[1:] += s
    r[:-1] -= s
    q = _poisson(g, r / g.rows(g.dy))
    gv = gv.clone()
    gv[1:] -= q
    gv[:-1] += q
    q = q * g.rows(g.dy)
    return gu - (_xm(q) - q) / g.dx, gv, gw - (_zm(q) - q) / g.dz


def _wall_lap(g, q):
    grad = torch.zeros((g.ny + 1,) + tuple(q.shape[1:]), dtype=q.dtype, device=q.device)
    grad[1:g.ny] = (q[1:] - q[:-1]) / g.rows(g.h[1:g.ny])
    grad[0] = q[0] / (0.5 * g.dy[0])
    grad[g.ny] = -q[-1] / (0.5 * g.dy[-1])
    return (grad[1:] - grad[:-1]) / g.rows(g.dy)


def _lap_xz(g, q):
    return (_xp(q) - 2 * q + _xm(q)) / g.dx ** 2 + (_zp(q) - 2 * q + _zm(q)) / g.dz ** 2


def _rates(g, u, v, w):
    """Momentum right-hand side: divergence-form central advection, diffusion, body force."""
    ny, dy, hf = g.ny, g.rows(g.dy), g.rows(g.h[1:g.ny])
    uw = 0.25 * (_xm(w) + w) * (_zm(u) + u)          # at x-face, z-face
    uv, vw = torch.zeros_like(v), torch.zeros_like(v)  # at the y-faces, zero on the walls
    uv[1:ny] = 0.25 * (_xm(v[1:ny]) + v[1:ny]) * (u[:-1] + u[1:])
    vw[1:ny] = 0.25 * (_zm(v[1:ny]) + v[1:ny]) * (w[:-1] + w[1:])
    c = 0.5 * (u + _xp(u))
    ru = -((c ** 2 - _xm(c) ** 2) / g.dx + (uv[1:] - uv[:-1]) / dy + (_zp(uw) - uw) / g.dz)
    ru += NU * (_lap_xz(g, u) + _wall_lap(g, u)) + FX
    c = 0.5 * (w + _zp(w))
    rw = -((c ** 2 - _zm(c) ** 2) / g.dz + (vw[1:] - vw[:-1]) / dy + (_xp(uw) - uw) / g.dx)
    rw += NU * (_lap_xz(g, w) + _wall_lap(g, w))
    c = 0.5 * (v[1:] + v[:-1])
    vi = v[1:ny]
    rv = torch.zeros_like(v)
    rv[1:ny] = -((c[1:] ** 2 - c[:-1] ** 2) / hf + (_xp(uv[1:ny]) - uv[1:ny]) / g.dx + (_zp(vw[1:ny]) - vw[1:ny]) / g.dz)
    dvy = ((v[2:] - vi) / dy[1:] - (vi - v[:-2]) / dy[:-1]) / hf
    rv[1:ny] += NU * (_lap_xz(g, vi) + dvy)
    return ru, rv, rw


def _timestep(g, u, v, w, dt):
    r0 = _rates(g, u, v, w)
    r1 = _rates(g, *(a + dt * r for a, r in zip((u, v, w), r0)))
    return _project(g, *(a + 0.5 * dt * (x + y) for a, x, y in zip((u, v, w), r0, r1)), dt)


def exact(case, seed):
    c = dict(case)
    x = [a.double() for a in _inputs(c, seed)]
    if c["kind"] == "batch":
        return [_poisson(Grid(s["nx"], s["ny"], s["nz"], s["stretch"]), f) for s, f in zip(_batch_sizes(c), x)]
    g = _grid(c)
    if c["kind"] == "solve":
        return _poisson(g, x.pop())
    if c["kind"] == "adjoint":
        dy = g.rows(g.dy)
        return _poisson(g, x.pop() / dy) * dy
    if c["kind"] == "timestep":
        out = _timestep(g, x[0], x[1], x[2], _dt(g))
        return list(out[:3] if c["prec"] == F32 else out)
    return list(_project(g, x[0], x[1], x[2], 1e-3)[:3]) + list(_project_transposed(g, x[3], x[4], x[5]))
