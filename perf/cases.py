"""The workloads whose speed is measured, as a user's program runs them through the public
binding (paper_2309_12019_gb300.dgw / .adjoint), and what they return in 64 bits.

A case is a dict of plain values: its kind, the mesh, degree, precision and data.
  step      Context.rk_step on a device state (scalar laws and the Euler system, 1D and 2D)
  host      Context.rk_step_host: state in pinned host memory, copied in, stepped, copied out
  ensemble  Batch.rk_step on many independent meshes of uneven size and degree
  gradient  adjoint.rollout + adjoint.misfit and the backward pass (checkpointed adjoint)
  project   Context.project of sampled initial data and Context.mass of the result
"""
import math
import random

import numpy as np
import torch

from paper_2309_12019_gb300 import adjoint, dgw

PERIODIC = ("periodic",) * 4
# initial data by name: box, boundary sides, flux and its parameters, wave-speed bound that
# sets the step (per direction), threshold b where the workload departs from the default
DATA = {
    "mixed": dict(box=(0.0, 1.0, 0.0, 1.0), bc=PERIODIC, flux="advect", a=(1.0, 0.0), lam=1.0),
    "sine": dict(box=(0.0, 1.0, 0.0, 1.0), bc=PERIODIC, flux="burgers", a=(1.0, 0.0), lam=1.2),
    "rotation": dict(box=(0.0, 1.0, 0.0, 1.0), bc=("inflow_zero",) * 4, flux="rotation", lam=0.5),
    "kpp": dict(box=(-2.0, 2.0, -2.5, 1.5), bc=("outflow",) * 4, flux="kpp", lambda_nu=2.0, lam=1.0),
    "quadrants": dict(box=(0.0, 1.0, 0.0, 1.0), bc=PERIODIC, flux="burgers", a=(1.0, 1.0), lam=1.3),
    "fourier": dict(box=(0.0, 1.0, 0.0, 1.0), bc=PERIODIC, flux="burgers", a=(1.0, 1.0), lam=6.0, b=0.0),
    "sod": dict(box=(0.0, 1.0, 0.0, 1.0), bc=("reflect",) * 2 + PERIODIC[:2], flux="euler", lam=2.5),
    "sod_train": dict(box=(0.0, 1.0, 0.0, 1.0), bc=PERIODIC, flux="euler", lam=2.5),
    "kelvin_helmholtz": dict(box=(0.0, 1.0, 0.0, 1.0), bc=PERIODIC, flux="euler", lam=3.0),
    "triple_point": dict(box=(0.0, 7.0, 0.0, 3.0), bc=("reflect",) * 4, flux="euler", lam=3.0),
    "rarefaction": dict(box=(0.0, 1.0, 0.0, 1.0), bc=("outflow",) * 4, flux="euler", lam=3.0),
}


def _case(name, kind, data, dim, nx, ny, p, prec, steps, stab="weno", rk=3, **more):
    return dict(name=name, kind=kind, data=data, dim=dim, nx=nx, ny=ny, p=p, prec=prec, steps=steps, stab=stab,
                rk_order=rk, **more)


def listed():
    return [
        # 1D convergence studies and shock tubes at the paper's sizes: many short steps on a
        # mesh that occupies a corner of the GPU, so latency and launches are all of it
        _case("advect_1d_128_q2_f64", "step", "mixed", 1, 128, 1, 2, "fp64", 16),
        _case("sod_128_q2_f64", "step", "sod", 1, 128, 1, 2, "fp64", 16),
        # solid-body rotation at 256^2 in double, the reference precision of the 2D studies
        _case("rotation_256x256_q2_f64", "step", "rotation", 2, 256, 256, 2, "fp64", 2),
        # the KPP problem at 1024^2, the headline mesh, and the same from and to host memory
        _case("kpp_1024x1024_q3_f32", "step", "kpp", 2, 1024, 1024, 3, "fp32", 2),
        _case("kpp_1024x1024_q3_host_f32", "host", "kpp", 2, 1024, 1024, 3, "fp32", 1),
        # a scalar run on a mesh whose rows are no multiple of anything (ragged tiles), with
        # SSP-RK of order p + 1 as the paper integrates
        _case("burgers_333x217_q1_f32", "step", "quadrants", 2, 333, 217, 1, "fp32", 4, rk=2),
        # an ensemble of 512 uneven 1D Burgers and 2D advection instances, advanced together
        _case("ensemble_512_f32", "ensemble", "ensemble", 2, 0, 0, 0, "fp32", 1, count=512),
        # gradient of a final-time misfit through the checkpointed adjoint: forward and backward
        _case("gradient_burgers_512x512_q2_f32", "gradient", "fourier", 2, 512, 512, 2, "fp32", 8, every=4),
        # the Euler system: a long 1D train of shock tubes, the triple point between walls at
        # the paper's mesh (fits in L2) and Kelvin-Helmholtz at 2048^2 (does not)
        _case("sod_train_4194304_q2_f32", "step", "sod_train", 1, 1 << 22, 1, 2, "fp32", 2),
        _case("triple_point_896x384_q2_f32", "step", "triple_point", 2, 896, 384, 2, "fp32", 4),
        _case("kelvin_helmholtz_2048x2048_q2_f32", "step", "kelvin_helmholtz", 2, 2048, 2048, 2, "fp32", 2),
        # start of every run: initial data sampled at 8 x 8 points per cell, projected, and its mass
        _case("project_kpp_1024x1024_q3_f32", "project", "kpp", 2, 1024, 1024, 3, "fp32", 0),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["scalar1d", "scalar2d", "scalar2d", "euler1d", "euler2d", "euler2d", "host", "ensemble",
                       "gradient", "project"])
    p = rng.choice([1, 2, 3])
    rk = rng.choice([3, 3, p + 1])
    stab = rng.choice(["weno", "weno", "weno", "weno", "lo", "dg", "zhao"])
    if kind == "scalar1d":
        return _undressed(_case("", "step", rng.choice(["mixed", "sine"]), 1, size(16, 4096), 1, p,
                                rng.choice(["fp64", "fp64", "fp32"]), rng.choice([4, 8, 16]), stab, rk))
    if kind == "scalar2d":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        n = size(24, 1000 if prec == "fp32" else 320)
        data = rng.choice(["rotation", "kpp", "quadrants"])
        m = max(8, int(n * rng.uniform(0.5, 1.0)))
        return _undressed(_case("", "step", data, 2, n, m, p, prec, rng.choice([1, 2, 4]), stab, rk))
    if kind == "euler1d":
        prec = rng.choice(["fp32", "fp64"])
        if rng.random() < 0.5:
            return _undressed(_case("", "step", "sod", 1, size(64, 2048), 1, rng.choice([2, 3]), prec, 8, stab, rk))
        n = 64 * size(1, (1 << 22) // 64 if prec == "fp32" else (1 << 17) // 64)
        return _undressed(_case("", "step", "sod_train", 1, n, 1, rng.choice([2, 3]), prec, 2, stab, 3))
    if kind == "euler2d":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        n = size(32, 1500 if prec == "fp32" else 200)
        data = rng.choice(["kelvin_helmholtz", "triple_point", "rarefaction"])
        m = n if data != "triple_point" else max(3, (n // 7) * 3)
        n = n if data != "triple_point" else max(7, (n // 7) * 7)
        return _undressed(_case("", "step", data, 2, n, m, rng.choice([1, 2, 2]), prec, rng.choice([1, 2]), stab, 3))
    if kind == "host":
        n = size(64, 1000)
        data = rng.choice(["kpp", "rotation"])
        return _undressed(_case("", "host", data, 2, n, n, p, "fp32", rng.choice([1, 3]), "weno", 3))
    if kind == "ensemble":
        return _undressed(_case("", "ensemble", "ensemble", 2, 0, 0, 0, "fp32", rng.choice([1, 2]),
                                count=size(16, 256)))
    if kind == "gradient":
        # degree 3 in double: in float the derivative of its much smaller sensor ratios is noise
        prec = "fp64" if p == 3 else rng.choice(["fp32", "fp32", "fp64"])
        n = size(48, 500 if prec == "fp32" else 128)
        return _undressed(_case("", "gradient", "fourier", 2, n, n, p, prec, rng.choice([3, 6]),
                                rng.choice(["weno", "weno", "lo", "dg"]), 3, every=3))
    n = size(64, 1000)
    return _undressed(_case("", "project", rng.choice(["kpp", "kelvin_helmholtz"]), 2, n, n, p,
                            rng.choice(["fp32", "fp64"]), 0))


def _undressed(c):
    return {k: v for k, v in c.items() if k != "name"}


# ------------------------------------------------------------------------------------------
# Inputs: modal states projected from closed-form data in double, rounded to the precision
# ------------------------------------------------------------------------------------------
DEV = "cuda"
F64 = torch.float64


def _dtype(case):
    return F64 if case["prec"] == "fp64" else torch.float32


def _box(case):
    """The data's box, its upper side moved so that cells are square."""
    x0, x1, y0, y1 = DATA[case["data"]]["box"]
    h = (x1 - x0) / case["nx"]
    return (x0, x1, y0, y0 + h * case["ny"] if case["dim"] == 2 else y1)


def _h(case):
    b = _box(case)
    return (b[1] - b[0]) / case["nx"]


def _dt(case):
    # inside the stability interval of the stabilization at gamma = 1; directions add in 2D
    d = DATA[case["data"]]
    cfl = {1: 0.1, 2: 0.05, 3: 0.025}[case["p"]] * (0.5 if case["dim"] == 2 else 1.0)
    return cfl * _h(case) / max(d["lam"], d.get("lambda_nu", 0.0))


def _problem(case):
    d = DATA[case["data"]]
    more = {k: d[k] for k in ("a", "lambda_nu", "b") if k in d}
    return dgw.Problem(dim=case["dim"], nx=case["nx"], ny=case["ny"], p=case["p"], box=_box(case), bc=d["bc"],
                       flux=d["flux"], stab=case["stab"], prec=case["prec"], rk_order=case["rk_order"], **more)


def _points(dim, nx, ny, box, nq):
    """Sample points (ny, nx, nq, nq) (1D: (1, nx, 1, nq)), the last axis along x, and the
    cells' indices."""
    g = torch.tensor(np.polynomial.legendre.leggauss(nq)[0], dtype=F64, device=DEV)
    h = (box[1] - box[0]) / nx
    ix = torch.arange(nx, dtype=F64, device=DEV)
    iy = torch.arange(ny, dtype=F64, device=DEV)
    x = box[0] + (ix[:, None] + 0.5 + 0.5 * g[None, :]) * h
    gy = g if dim == 2 else torch.zeros(1, dtype=F64, device=DEV)
    y = box[2] + (iy[:, None] + 0.5 + 0.5 * gy[None, :]) * h
    return x[None, :, None, :], y[:, None, :, None], ix[None, :, None, None], iy[:, None, None, None]


def _samples(case, seed, nq):
    """The conserved variables at the Gauss points, (components, ny, nx, nq_y, nq_x)."""
    r = random.Random(seed)
    nx, ny, dim = case["nx"], case["ny"], case["dim"]
    x, y, ix, iy = _points(dim, nx, ny, _box(case), nq)
    ph = [r.uniform(0.0, 2.0 * math.pi) for _ in range(16)]
    name, pi = case["data"], math.pi
    if name == "mixed":         # square wave + Gaussian + part of a sine, moved around the period
        z = torch.remainder(x - r.random(), 1.0)
        u = ((z >= 0.2) & (z <= 0.4)).to(F64) + torch.exp(-300.0 * (z - 0.6) ** 2)
        u = u + torch.where((z >= 0.7) & (z <= 0.9), 0.5 * torch.sin(2.0 * pi * z), 0.0)
    elif name == "sine":
        u = torch.sin(2.0 * pi * x + ph[0]) + 0.1 * torch.sin(6.0 * pi * x + ph[1])
    elif name == "rotation":    # slotted cylinder, cone and hump, turned by some angle
        cs, sn = math.cos(ph[0]), math.sin(ph[0])
        xr = 0.5 + cs * (x - 0.5) + sn * (y - 0.5)
        yr = 0.5 - sn * (x - 0.5) + cs * (y - 0.5)
        cyl, cone, hump = (torch.hypot(xr - a, yr - b) for a, b in ((0.5, 0.75), (0.5, 0.25), (0.25, 0.5)))
        u = ((cyl <= 0.15) & (((xr - 0.5).abs() >= 0.025) | (yr >= 0.85))).to(F64)
        u = torch.where(cone <= 0.15, 1.0 - cone / 0.15, u)
        u = torch.where(hump <= 0.15, 0.25 + 0.25 * torch.cos(pi * hump / 0.15), u)
    elif name == "kpp":         # 7 pi / 2 in the unit disc, pi / 4 outside, slightly uneven
        inner = torch.hypot(x - r.uniform(-0.2, 0.2), y - r.uniform(-0.2, 0.2)) <= 1.0
        u = torch.where(inner, 3.5 * pi, 0.25 * pi)
        u = u + 0.05 * torch.sin(3.0 * x + ph[0]) * torch.cos(2.0 * y + ph[1])
    elif name == "quadrants":   # the four constant states of the 2D Burgers problem, periodic
        q = (torch.remainder(x - r.random(), 1.0) > 0.5).to(F64) + 2.0 * (torch.remainder(y - r.random(), 1.0) > 0.5)
        u = torch.where(q == 3, -1.0, torch.where(q == 2, -0.2, torch.where(q == 0, 0.5, 0.8)))
        u = u + 0.1 * torch.sin(2.0 * pi * x + ph[0]) * torch.sin(4.0 * pi * y + ph[1])
    elif name == "fourier":     # modes at all scales down to ten cells, and a step
        u = torch.zeros_like(x + y)
        for j in range(12):
            k, th = max(1.0, nx / 10.0) ** (j / 11.0), r.uniform(0.0, 2.0 * pi)
            kx, ky = round(k * math.cos(th)), round(k * math.sin(th))
            amp = r.uniform(0.5, 1.0) / math.sqrt(k)
            u = u + amp * torch.sin(2.0 * pi * ((kx if kx or ky else 1) * x + ky * y) + ph[j])
        u = u + ((torch.remainder(x - r.random(), 1.0) < 0.3) & (torch.remainder(y - r.random(), 1.0) < 0.25)).to(F64)
    else:
        # the Euler problems: states that jump on cell faces, the density slightly uneven
        if name in ("sod", "sod_train"):
            if name == "sod":
                left = ix < round(nx * r.uniform(0.45, 0.55))
            else:
                left = torch.remainder(ix - r.randrange(64), 64) < 32
            rho, pr = torch.where(left, 1.0, 0.125), torch.where(left, 1.0, 0.1)
            vx = vy = torch.zeros_like(rho)
        elif name == "kelvin_helmholtz":
            inner = ((iy + 0.5) / ny - 0.5).abs() < 0.25
            rho, vx = torch.where(inner, 2.0, 1.0), torch.where(inner, -0.5, 0.5)
            vy = 0.01 * torch.sin(2.0 * pi * x + ph[0])
            pr = torch.full_like(rho, 2.5)
        elif name == "triple_point":
            left, low = (ix + 0.5) * 7 < nx, (iy + 0.5) * 2 < ny
            rho = torch.where(left, 1.0, torch.where(low, 1.0, 0.125))
            pr = torch.where(left, 1.0, 0.1)
            vx = vy = torch.zeros_like(rho)
        else:
            east, north = (ix + 0.5) * 2 > nx, (iy + 0.5) * 2 > ny
            same = east == north
            rho, pr = torch.where(same, 1.0, 0.389), torch.where(same, 1.5, 0.4)
            vx, vy = torch.where(east, 0.6233, -0.6233), torch.where(north, 0.6233, -0.6233)
        rho = rho * (1.0 + 0.02 * torch.sin(2.0 * pi * x + ph[2]) * torch.cos(2.0 * pi * y + ph[3]))
        en = pr / 0.4 + 0.5 * rho * (vx * vx + vy * vy)
        u = [rho, rho * vx, rho * vy, en] if dim == 2 else [rho, rho * vx, en]
    full = (ny, nx, nq if dim == 2 else 1, nq)
    return torch.stack([v.to(F64).expand(full) for v in (u if isinstance(u, list) else [u])])


def _legendre(n, x):
    """P_0 .. P_{n-1} at the points x, (points, n)."""
    return np.polynomial.legendre.legvander(np.asarray(x), n - 1)


def _l2(f, p, dim, nq):
    """L2 projection of samples (C, ny, nx, qy, qx) onto the modes: (C, J, I, ny, nx)."""
    g, w = np.polynomial.legendre.leggauss(nq)
    M = _legendre(p + 1, g) * w[:, None] * (np.arange(p + 1) + 0.5)
    M = torch.tensor(M, dtype=F64, device=DEV)
    My = M if dim == 2 else torch.ones((1, 1), dtype=F64, device=DEV)
    return torch.einsum("bj,cyxbi->cjiyx", My, torch.einsum("cyxba,ai->cyxbi", f, M)).contiguous()


def _state(case, seed):
    """The initial modal state, rounded to the case's precision: (K, E)."""
    c = _l2(_samples(case, seed, 4), case["p"], case["dim"], 4)
    return c.reshape(-1, case["nx"] * case["ny"]).to(_dtype(case)).contiguous()


def _ensemble(case):
    """The instances of an ensemble (sizes, degrees, velocities), as the case fixes them."""
    r = random.Random(case["count"])
    out = []
    for i in range(case["count"]):
        dim = r.choice([1, 2])
        n = int(round(math.exp(r.uniform(math.log(64 if dim == 1 else 32), math.log(4096 if dim == 1 else 512)))))
        th = r.uniform(0.0, 2.0 * math.pi)
        out.append(dict(dim=dim, nx=n, ny=n if dim == 2 else 1, p=r.choice([1, 2, 3]),
                        flux="burgers" if dim == 1 else "advect",
                        a=(1.0, 0.0) if dim == 1 else (math.cos(th), math.sin(th))))
    for c in out:
        cfl = {1: 0.1, 2: 0.05, 3: 0.025}[c["p"]]
        c["dt"] = cfl / c["nx"] / (9.0 if c["dim"] == 1 else abs(c["a"][0]) + abs(c["a"][1]))
    return out


def _ensemble_state(inst, i, seed):
    """Instance i's initial state (K, E) in double: eight Fourier modes and up to three steps."""
    r = random.Random(seed * 100003 + i)
    dim, nx, ny = inst["dim"], inst["nx"], inst["ny"]
    x, y, _, _ = _points(dim, nx, ny, (0.0, 1.0, 0.0, 1.0), 4)
    u = 0.0
    for _ in range(8):          # a sin(kx x + ky y + phase), split along the axes
        kx, ky = (r.randint(1, 8), 0) if dim == 1 else (r.randint(1, 4), r.randint(-4, 4))
        a, ph = r.random(), r.uniform(0.0, 2.0 * math.pi)
        tx, ty = 2.0 * math.pi * kx * x + ph, 2.0 * math.pi * ky * y
        u = u + a * (torch.sin(tx) * torch.cos(ty) + torch.cos(tx) * torch.sin(ty))
    for _ in range(r.randint(0, 3)):
        s = torch.remainder(x - r.random(), 1.0) < r.uniform(0.05, 0.4)
        if dim == 2:
            s = s & (torch.remainder(y - r.random(), 1.0) < r.uniform(0.05, 0.4))
        u = u + s.to(F64)
    c = _l2(u.expand(ny, nx, 4 if dim == 2 else 1, 4)[None], inst["p"], dim, 4)
    return c.reshape(-1, nx * ny)


# ------------------------------------------------------------------------------------------
# What a program has in hand, and the pass
# ------------------------------------------------------------------------------------------
def prepare(case, seed):
    s = dict(kind=case["kind"], steps=case["steps"])
    if case["kind"] == "ensemble":
        insts = _ensemble(case)
        probs = [dgw.Problem(dim=d["dim"], nx=d["nx"], ny=d["ny"], p=d["p"], flux=d["flux"], a=d["a"]) for d in insts]
        b = dgw.Batch(probs, prec=case["prec"])
        b.set_dt([d["dt"] for d in insts])
        U = torch.zeros(b.total, dtype=b.dtype, device=DEV)
        for i, d in enumerate(insts):
            b.view(U, i).copy_(_ensemble_state(d, i, seed))
        return dict(s, batch=b, U=U)
    ctx = dgw.Context(_problem(case))
    s.update(ctx=ctx, dt=_dt(case))
    if case["kind"] == "project":
        s["samples"] = _samples(case, seed, 8).reshape(-1).contiguous()
        s["U"] = torch.empty((ctx.K, ctx.E), dtype=ctx.dtype, device=DEV)
        return s
    s["U"] = _state(case, seed)
    if case["kind"] == "host":
        s["U_in"] = s.pop("U").cpu().pin_memory()
        s["U_out"] = torch.empty_like(s["U_in"]).pin_memory()
    if case["kind"] == "gradient":
        s.update(target=_state(case, seed + 1), every=case["every"])
    return s


def run(s):
    if s["kind"] == "step":
        s["ctx"].rk_step(s["U"], s["dt"], s["steps"])
        return s["U"]
    if s["kind"] == "host":
        s["ctx"].rk_step_host(s["U_in"], s["U_out"], s["dt"], s["steps"])
        return s["U_out"]
    if s["kind"] == "ensemble":
        s["batch"].rk_step(s["U"], s["steps"])
        return s["U"]
    if s["kind"] == "gradient":
        U0 = s["U"].detach().requires_grad_(True)
        UN = adjoint.rollout(s["ctx"], U0, s["dt"], s["steps"], s["every"])
        J = adjoint.misfit(s["ctx"], UN, s["target"])
        J.backward()
        return {"grad": U0.grad, "state": UN.detach(), "misfit": J.detach().to(UN.dtype)}
    s["ctx"].project(s["samples"], s["U"])
    return {"state": s["U"], "mass": s["ctx"].mass(s["U"])}


# ------------------------------------------------------------------------------------------
# Bytes and operations a pass cannot do without
# ------------------------------------------------------------------------------------------
RK_STAGES = {2: 2, 3: 3, 4: 10}


def _cell_flops(dim, p, flux, stab):
    """Operations of one stage per cell: sum-factorised volume and face integrals, the
    sensor's candidates and seminorms, the stabilization and the update."""
    n, q = p + 1, p + 2
    C = dim + 2 if flux == "euler" else 1
    point = 12 * dim + 12 if flux == "euler" else (20 if flux == "kpp" else 4)
    if dim == 1:
        vol = C * 2 * 2 * n * q + q * point
        face = C * 4 * n + 3 * point
        sens = 2 * n * n + 3 * n * n + 6 * n
        rest = C * (n * n + 6 * n)
    else:
        vol = C * 2 * (n * n * q + n * q * q) * 3 + q * q * point
        face = 2 * (C * (4 * n * n + 3 * 2 * n * q) + q * 3 * point)
        sens = 4 * n * n * n + 6 * (n ** 4 // 4 + n * n) + 10 * n * n
        rest = C * (2 * n ** 3 + 8 * n * n)
    return vol + face + (sens if stab in ("weno", "zhao") else 0) + rest


def work(case):
    if case["kind"] == "ensemble":
        w = dict(bytes=0.0, flops=0.0)
        for d in _ensemble(case):
            E = d["nx"] * d["ny"]
            w["bytes"] += 2.0 * 4 * E * (d["p"] + 1) ** d["dim"]
            w["flops"] += 3.0 * case["steps"] * E * _cell_flops(d["dim"], d["p"], d["flux"], "weno")
        return w
    dim, p, flux = case["dim"], case["p"], DATA[case["data"]]["flux"]
    E, C = case["nx"] * case["ny"], dim + 2 if flux == "euler" else 1
    state = float(E * C * (p + 1) ** dim * (8 if case["prec"] == "fp64" else 4))
    if case["kind"] == "project":
        n = p + 1
        return dict(bytes=8.0 * C * E * 64 + state, flops=2.0 * C * E * (64 * n + 8 * n * n))
    stage = float(E * _cell_flops(dim, p, flux, case["stab"]))
    if case["kind"] == "gradient":      # U0 and the target in; the final state and the gradient out
        return dict(bytes=4.0 * state, flops=3.0 * case["steps"] * stage * 3.0)
    return dict(bytes=2.0 * state, flops=RK_STAGES[case["rk_order"]] * case["steps"] * stage)


# ------------------------------------------------------------------------------------------
# The scheme in 64 bits, in plain torch: states as (C, J, I, ny, nx); a 1D mesh is one row
# of cells with the single y-mode P_0
# ------------------------------------------------------------------------------------------
class _Scheme:
    def __init__(self, dim, nx, ny, p, flux, box, bc, a=(1.0, 0.0), lambda_nu=0.0, stab="weno", b=None):
        self.dim, self.nx, self.ny, self.p, self.flux, self.a = dim, nx, ny, p, flux, a
        self.stab, self.b = stab, (0.0 if flux == "euler" else 0.1) if b is None else b
        self.lambda_nu, self.bc = lambda_nu, bc
        self.h = (box[1] - box[0]) / nx
        n = p + 1
        g, w = np.polynomial.legendre.leggauss(p + 2)
        leg = np.polynomial.legendre
        eye = np.eye(n)
        B = _legendre(n, g)
        D = np.stack([leg.legval(g, leg.legder(eye[i])) if i else 0.0 * g for i in range(n)], 1)
        # derivative Gram matrices A^(a)_mn = int P_m^(a) P_n^(a), a = 0 .. p
        A = np.zeros((n, n, n))
        for k in range(n):
            d = np.stack([leg.legval(g, leg.legder(eye[i], k)) if i >= k else 0.0 * g for i in range(n)], 1)
            A[k] = d.T @ (w[:, None] * d)
        # P_m(xi +- 2) in the Legendre basis (neighbour on the minus / plus side)
        T = [(np.arange(n)[:, None] + 0.5) * (B.T @ (w[:, None] * _legendre(n, g + s))) for s in (2.0, -2.0)]
        T = [np.triu(t) for t in T]
        ny1 = n if dim == 2 else 1
        Ay = A if dim == 2 else np.concatenate([[[[2.0]]], np.zeros((p, 1, 1))])
        G = np.zeros((ny1 * n, ny1 * n))
        for kx in range(n):
            for ky in range(n):
                if 1 <= kx + ky <= p:
                    G += 2.0 ** (2 * (kx + ky) - 2) * np.einsum("jl,ik->jilk", Ay[ky], A[kx]).reshape(G.shape)
        K = np.einsum("jl,ik->jilk", Ay[0], A[1]) + np.einsum("jl,ik->jilk", Ay[1], A[0])
        m = np.arange(n) + 0.5
        self.M = dict(B=B, WB=B * w[:, None], WD=D * w[:, None], G=G, K=K.reshape(G.shape), T0=T[0], T1=T[1],
                      m=np.outer(m if dim == 2 else [0.5], m), g=g, sg=(-1.0) ** np.arange(n))
        one, two = np.ones((1, 1)), 2.0 * np.ones((1, 1))
        self.M.update(By=B if dim == 2 else one, WBy=B * w[:, None] if dim == 2 else two,
                      WDy=D * w[:, None] if dim == 2 else 0.0 * one)
        self.M = {k: torch.tensor(np.asarray(v), dtype=F64, device=DEV) for k, v in self.M.items()}
        self.xc = box[0] + (torch.arange(nx, dtype=F64, device=DEV) + 0.5) * self.h
        self.yc = box[2] + (torch.arange(ny, dtype=F64, device=DEV) + 0.5) * self.h

    def prim(self, u):
        rho, m, en = u[0], u[1:-1], u[-1]
        v = m / rho
        return rho, v, 0.4 * (en - 0.5 * (m * v).sum(0))

    def fluxes(self, u, x, y):
        """F along every axis, and |F'| (|v| + c)."""
        if self.flux == "euler":
            rho, v, pr = self.prim(u)
            F = []
            for d in range(self.dim):
                f = u * v[d]
                f[1 + d] = f[1 + d] + pr
                f[-1] = f[-1] + pr * v[d]
                F.append(f)
            return F, v.square().sum(0).sqrt() + (1.4 * pr / rho).sqrt()
        if self.flux == "kpp":
            return [torch.sin(u), torch.cos(u)], torch.ones_like(u[0])
        if self.flux == "rotation":
            v = [0.5 - y, x - 0.5]
        else:
            v = list(self.a[: self.dim])
        if self.flux == "burgers":
            return [s * 0.5 * u * u for s in v], math.hypot(*v) * u[0].abs()
        spd = sum(s * s for s in v)
        spd = spd.sqrt() if torch.is_tensor(spd) else torch.tensor(math.sqrt(spd), dtype=F64, device=DEV)
        return [s * u for s in v], spd.expand(u[0].shape)

    def llf(self, ax, uL, uR, x, y):
        """H along +e_ax, and the speed |F'| of each side's own value."""
        FL, sL = self.fluxes(uL, x, y)
        FR, sR = self.fluxes(uR, x, y)
        if self.flux == "euler":
            s = []
            for u in (uL, uR):
                rho, v, pr = self.prim(u)
                s.append(v[ax].abs() + (1.4 * pr / rho).sqrt())
            s = torch.maximum(*s)
        elif self.flux == "kpp":
            shift = 0.0 if ax == 0 else 0.5 * math.pi
            lo, hi = torch.minimum(uL, uR), torch.maximum(uL, uR)
            inside = torch.ceil((lo - shift) / math.pi) * math.pi + shift <= hi
            f = torch.cos if ax == 0 else torch.sin
            s = torch.where(inside, 1.0, torch.maximum(f(uL).abs(), f(uR).abs()))
        elif self.flux == "burgers":
            s = abs(self.a[ax]) * torch.maximum(uL.abs(), uR.abs())
        else:
            v = self.a[ax] if self.flux == "advect" else (0.5 - y if ax == 0 else x - 0.5)
            s = v.abs() if torch.is_tensor(v) else abs(v)
        return 0.5 * (FL[ax] + FR[ax]) - 0.5 * s * (uR - uL), sL, sR

    def faces(self, c, ax, acc, lam):
        """Adds the face terms of one axis to acc; returns lam with the faces' own speeds."""
        M = self.M
        # values at the face's Gauss points, (C, q, ny, nx): at xi = -1 and +1 of every cell
        if ax == 0:
            lo, hi = torch.einsum("i,cjiyx->cjyx", M["sg"], c), c.sum(2)
            Bf, WBf, dim = M["By"], M["WBy"], 3
        else:
            lo, hi = torch.einsum("j,cjiyx->ciyx", M["sg"], c), c.sum(1)
            Bf, WBf, dim = M["B"], M["WB"], 2
        lo, hi = (torch.einsum("qt,ctyx->cqyx", Bf, t) for t in (lo, hi))
        n = lo.shape[dim]
        first, last = lo.narrow(dim, 0, 1), hi.narrow(dim, n - 1, 1)
        hf = 0.5 * self.h
        if ax == 0:
            x = (self.xc[0] - hf + torch.arange(n + 1, dtype=F64, device=DEV) * self.h)[None, None, :]
            y = self.yc[None, :, None] + hf * M["g"][:, None, None] if self.dim == 2 else 0.0 * x
        else:
            y = (self.yc[0] - hf + torch.arange(n + 1, dtype=F64, device=DEV) * self.h)[None, :, None]
            x = self.xc[None, None, :] + hf * M["g"][:, None, None]

        def ghost(kind, inner, sign):
            if kind == "reflect":
                g = inner.clone()
                g[1 + ax] = -g[1 + ax]
                return g
            if kind == "inflow_zero":       # rotation only: F' does not depend on the state
                at = 0 if sign < 0 else n
                v = 0.5 - y if ax == 0 else x.narrow(2, 0, x.shape[2]) - 0.5
                v = v.expand(inner.shape[1:]) if v.shape[dim - 1] == 1 else v.narrow(dim - 1, at, 1)
                return torch.where(sign * v < 0.0, 0.0, inner)
            return inner

        if self.bc[2 * ax] == "periodic":
            gl, gr = last, first
        else:
            gl, gr = ghost(self.bc[2 * ax], first, -1.0), ghost(self.bc[2 * ax + 1], last, 1.0)
        uL, uR = torch.cat([gl, hi], dim), torch.cat([lo, gr], dim)
        H, sL, sR = self.llf(ax, uL, uR, x, y)
        own = torch.maximum(sL.narrow(dim - 1, 1, n), sR.narrow(dim - 1, 0, n)).amax(0)
        Hc = torch.einsum("qt,cqyx->ctyx", WBf, H)
        Hm, Hp = Hc.narrow(dim, 0, n), Hc.narrow(dim, 1, n)
        if ax == 0:
            acc = acc + M["sg"][None, None, :, None, None] * Hm[:, :, None] - Hp[:, :, None]
        else:
            acc = acc + M["sg"][None, :, None, None, None] * Hm[:, None] - Hp[:, None]
        return acc, torch.maximum(lam, own)

    def sensor(self, c):
        """gamma of every cell, (ny, nx), from the modes c (J, I, ny, nx)."""
        M = self.M
        shape = c.shape

        def norm2(v):
            v = v.reshape(-1, shape[2], shape[3])
            return (v * torch.einsum("kl,lyx->kyx", M["G"], v)).sum(0)

        cand, has = [], []
        for f in range(2 * self.dim):
            ax, plus = f // 2, f % 2
            d = 3 - ax
            nb = torch.roll(c, -1 if plus else 1, d)
            ok = torch.ones(shape[2:], dtype=F64, device=DEV)
            if self.bc[2 * ax] != "periodic":
                ok.select(d - 2, shape[d] - 1 if plus else 0).zero_()
            cand.append(torch.einsum("im,jmyx->jiyx" if ax == 0 else "jm,miyx->jiyx", M["T%d" % plus], nb))
            has.append(ok)
        me = sum(has)
        beta0 = norm2(c)
        lin0 = 1.0 - 0.01 * me
        w0 = lin0 / (1e-6 + beta0) ** 2
        w = [0.01 * ok / (1e-6 + norm2(q)) ** 2 for q, ok in zip(cand, has)]
        total = w0 + sum(w)
        if self.stab == "zhao":
            dev = (w0 / total / lin0 - 1.0).abs()
            for wl, ok in zip(w, has):
                dev = dev + ok * (wl / total / 0.01 - 1.0).abs()
            return torch.where(me > 0, dev / ((1.0 / 0.01 - 1.0) + me), 0.0)
        d = sum(wl / total * (c - q) for wl, q in zip(w, cand))
        num2 = norm2(d)
        live = (num2 > 1e-24) & (beta0 > 0.0)
        r = torch.where(live, num2, 1.0).sqrt() / torch.where(live, beta0, 1.0).sqrt()
        g = torch.where(r < self.b, 0.0, torch.clamp(r, max=1.0))
        return torch.where(live, g, torch.where(num2 > 1e-24, 1.0, 0.0))

    def residual(self, c):
        M = self.M
        u = torch.einsum("rj,cjqyx->crqyx", M["By"], torch.einsum("qi,cjiyx->cjqyx", M["B"], c))
        hf = 0.5 * self.h
        x = (self.xc[None, :] + hf * M["g"][:, None])[None, :, None, :]
        y = (self.yc[None, :] + hf * M["g"][:, None])[:, None, :, None] if self.dim == 2 else 0.0 * x
        F, spd = self.fluxes(u, x, y)
        lam = spd.amax((0, 1))
        acc = torch.einsum("rj,criyx->cjiyx", M["WBy"], torch.einsum("qi,crqyx->criyx", M["WD"], F[0]))
        if self.dim == 2:
            acc = acc + torch.einsum("rj,criyx->cjiyx", M["WDy"], torch.einsum("qi,crqyx->criyx", M["WB"], F[1]))
        del u, F
        for ax in range(self.dim):
            acc, lam = self.faces(c, ax, acc, lam)
        if self.stab != "dg":
            gamma = 1.0 if self.stab == "lo" else self.sensor(c[0])
            lam = self.lambda_nu if self.lambda_nu > 0.0 else lam
            kc = torch.einsum("kl,clyx->ckyx", M["K"], c.reshape(c.shape[0], -1, self.ny, self.nx)).reshape(c.shape)
            acc = acc - gamma * lam / self.p * kc
        return (2.0 / self.h) * M["m"][None, :, :, None, None] * acc

    def step(self, u, dt, order=3):
        L = self.residual
        if order == 2:
            s = u + dt * L(u)
            return 0.5 * u + 0.5 * (s + dt * L(s))
        if order == 3:
            s = u + dt * L(u)
            s = 0.75 * u + 0.25 * (s + dt * L(s))
            return u / 3.0 + 2.0 / 3.0 * (s + dt * L(s))
        q1, q2 = u, u
        for _ in range(5):
            q1 = q1 + dt / 6.0 * L(q1)
        q2 = q2 / 25.0 + 9.0 / 25.0 * q1
        q1 = 15.0 * q2 - 5.0 * q1
        for _ in range(4):
            q1 = q1 + dt / 6.0 * L(q1)
        return q2 + 0.6 * q1 + dt / 10.0 * L(q1)

    def modes(self, U):
        """(K, E) rows as (C, J, I, ny, nx)."""
        J = self.p + 1 if self.dim == 2 else 1
        return U.to(F64).reshape(-1, J, self.p + 1, self.ny, self.nx)


def _scheme(case):
    d = DATA[case["data"]]
    more = {k: d[k] for k in ("a", "lambda_nu", "b") if k in d}
    return _Scheme(case["dim"], case["nx"], case["ny"], case["p"], d["flux"], _box(case), d["bc"], stab=case["stab"],
                   **more)


def exact(case, seed):
    if case["kind"] == "ensemble":
        out = []
        for i, d in enumerate(_ensemble(case)):
            S = _Scheme(d["dim"], d["nx"], d["ny"], d["p"], d["flux"], (0.0, 1.0, 0.0, 1.0), PERIODIC, a=d["a"])
            u = S.modes(_ensemble_state(d, i, seed).to(_dtype(case)))
            for _ in range(case["steps"]):
                u = S.step(u, d["dt"])
            out.append(torch.nn.functional.pad(u.reshape(-1), (0, -u.numel() % 4)))
        return torch.cat(out)
    if case["kind"] == "project":
        c = _l2(_samples(case, seed, 8), case["p"], case["dim"], 8)
        U = c.reshape(-1, case["nx"] * case["ny"])
        return {"state": U, "mass": float(U[0].to(_dtype(case)).to(F64).sum()) * _h(case) ** 2}
    S, dt = _scheme(case), _dt(case)
    u = S.modes(_state(case, seed))
    rows = (-1, case["nx"] * case["ny"])
    if case["kind"] != "gradient":
        for _ in range(case["steps"]):
            u = S.step(u, dt, case["rk_order"])
        return u.reshape(rows) if case["kind"] != "host" else u.reshape(rows).cpu()
    path = [u]
    for _ in range(case["steps"]):
        path.append(S.step(path[-1], dt))
    i = torch.arange(case["p"] + 1, dtype=F64, device=DEV)
    mass = S.h / (2.0 * i + 1.0)
    d = path[-1] - S.modes(_state(case, seed + 1))
    lam = (mass[:, None] * mass[None, :])[None, :, :, None, None] * d
    misfit = 0.5 * (lam * d).sum()
    end = path.pop()
    while path:
        v = path.pop().requires_grad_(True)
        (lam,) = torch.autograd.grad(S.step(v, dt), v, lam)
    return {"grad": lam.reshape(rows), "state": end.reshape(rows), "misfit": misfit}
