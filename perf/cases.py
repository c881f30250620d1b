"""What a program that uses this library asks of it, as cases that can be timed.

The library analyses the oil film of axial-piston pumps: a program assembles the
Reynolds equation for a joint batch of working conditions, solves it, integrates
loads, takes Picard steps of a march, or serves such steps for many clients.  The
cases run from the smallest batch (one condition on 64 x 32 cells, where launches
and latency are the cost) to the largest one that the benchmark names (9 conditions
on 2048 x 1024 cells, 18.9 million unknowns), in FP64 (the default) and in mixed
precision, with each criterion, preconditioner and entry point that is used.

Solves ask for a relative residual of 1e-12 (the tolerance of the accuracy
references), so that what comes back is set by the problem and not by where an
iteration happened to stop; steps whose finite-difference Jacobian comes back too ask
for 1e-13 in mixed precision.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2511_06824_gb300 import gmaf

# Piston radius, gap length, clearance [m], viscosity [Pa s], sliding speed [m/s],
# chamber and case pressure [Pa]: the physical set of the repository's workloads.
PHYS = (0.010, 0.040, 20e-6, 0.04, 5.0, 20e6, 0.1e6)
DIMPLE = (1.0, 0.5e-3, 5e-6, 0.2)       # kind, radius, depth [m], area density
DT = (60.0 / 600.0) / 360.0             # one degree of shaft angle at 600 rpm
D_E = 1e-3 * PHYS[2]                    # eccentricity difference of the Jacobian
D_EDOT = 1e-4                           # rate difference: the rates' own scale (A is affine in them)
F_EXT = (30.0, -15.0, 6.0, -3.0)
OMEGA = 1.2


def listed():
    return [
        # one condition on the coarsest configured grid: a real-time model's call, all latency
        _solve("solve_fp64_64x32_k1", 64, 32, 1, textured=False),
        # a whole general Picard step on a coarse grid, as a design sweep takes them by the thousand
        _picard("picard_fp64_96x48", 96, 48, precision=0),
        # an odd column count (no vector loads), a batch of three unrelated working conditions
        _solve("solve_fp64_255x97_k3", 255, 97, 3),
        # the asynchronized criterion: nine independent recurrences on the smallest served grid
        _solve("solve_async_256x128_k9", 256, 128, 9, criterion=1),
        # a mixed-precision Picard step on the smallest served grid
        _picard("picard_mixed_256x128", 256, 128, precision=1),
        # the smooth 9-condition batch in FP64, from L2
        _solve("solve_fp64_512x256_k9", 512, 256, 9, textured=False),
        # the same size in mixed precision, a whole step
        _picard("picard_mixed_512x256", 512, 256, precision=1),
        # a march's solve: started from the previous shaft step's fields
        _solve("solve_warm_mixed_1024x512_k9", 1024, 512, 9, precision=1, warm=True),
        # the benchmark's batch, the largest
        _solve("solve_mixed_2048x1024_k9", 2048, 1024, 9, precision=1),
        # a burst of requests of uneven grids at the continuous-batching server
        _server("server_burst_of_6", 6, 1024),
        # assembly alone (the coefficients handed to another solver), textured
        _assemble("assemble_1024x512_k9", 1024, 512, 9),
        # loads alone, from pressure fields that the program holds
        _loads("loads_1024x512_k9", 1024, 512, 9),
    ]


def _solve(name, n_theta, n_z, n_cond, precision=0, precond=1, criterion=0, textured=True,
           warm=False, noalloc=False):
    return dict(name=name, kind="solve", n_theta=n_theta, n_z=n_z, n_cond=n_cond,
                precision=precision, precond=precond, criterion=criterion, textured=textured,
                warm=warm, noalloc=noalloc, eps=1e-12)


def _picard(name, n_theta, n_z, precision, textured=True, simplified=False):
    return dict(name=name, kind="picard", n_theta=n_theta, n_z=n_z,
                n_cond=5 if simplified else 9, precision=precision, textured=textured,
                simplified=simplified, eps=1e-13 if precision else 1e-12)


def _server(name, requests, largest):
    return dict(name=name, kind="server", requests=requests, largest=largest, eps=1e-13)


def _assemble(name, n_theta, n_z, n_cond, textured=True):
    return dict(name=name, kind="assemble", n_theta=n_theta, n_z=n_z, n_cond=n_cond,
                textured=textured)


def _loads(name, n_theta, n_z, n_cond, textured=True):
    return dict(name=name, kind="loads", n_theta=n_theta, n_z=n_z, n_cond=n_cond,
                textured=textured)


def draw(rng):
    """A case of the same ranges: grids of 24 to 512 axial cells, odd ones among them."""

    def grid(lo, hi, multiple=1):
        n_z = round(math.exp(rng.uniform(math.log(lo), math.log(hi))))
        n_theta = round(2 * n_z * rng.uniform(0.75, 1.25))
        return max(multiple, n_theta // multiple * multiple), n_z

    kind = rng.choice(["fp64", "fp64", "async", "noalloc", "mixed", "mixed", "warm", "picard",
                       "picard", "server", "assemble", "loads"])
    textured = rng.random() < 0.7
    precond = rng.choice([1, 1, 1, 1, 0, 2])
    if kind == "fp64":
        g = grid(24, 384, rng.choice([1, 2, 4]))
        c = _solve("", *g, rng.choice([1, 2, 3, 5, 9, 9]), precond=precond, textured=textured)
    elif kind == "async":
        c = _solve("", *grid(24, 192, rng.choice([1, 2])), rng.choice([3, 5, 9, 9]), criterion=1,
                   precond=precond, textured=textured)
    elif kind == "noalloc":
        c = _solve("", *grid(24, 200, rng.choice([1, 2])), rng.choice([1, 5, 9]), noalloc=True,
                   textured=textured)
    elif kind in ("mixed", "warm"):
        g = grid(32, 512, rng.choice([1, 4, 4, 4]))
        c = _solve("", *g, rng.choice([1, 3, 5, 9, 9, 9]), precision=1, textured=textured,
                   precond=1 if kind == "warm" else precond, warm=kind == "warm")
    elif kind == "picard":
        p = rng.choice([0, 1])
        c = _picard("", *grid(32, 256, 4), precision=p, textured=textured,
                    simplified=rng.random() < 0.3)
    elif kind == "server":
        c = _server("", rng.randint(2, 8), rng.choice([256, 512]))
    elif kind == "assemble":
        c = _assemble("", *grid(32, 512), rng.choice([1, 3, 9, 9]), textured)
    else:
        c = _loads("", *grid(32, 512), rng.choice([1, 3, 9, 9]), textured)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs


def _texture(rng, textured):
    o = (rng.uniform(0.0, 2.0 * math.pi * PHYS[0]), rng.uniform(0.0, PHYS[1]))
    return DIMPLE + o if textured else (0.0,) * 6


def _state(rng):
    return np.concatenate([rng.uniform(0.0, 0.5 * PHYS[2], 4), rng.uniform(-1e-4, 1e-4, 4)])


def _fan_out(base, simplified=False):
    """The conditions of a Picard step: the base and its finite-difference neighbours."""
    conds = [base.copy() for _ in range(5 if simplified else 9)]
    for j in range(4):
        if simplified:
            conds[1 + j][4 + j] += D_EDOT
        else:
            conds[1 + j][j] += D_E
            conds[5 + j][4 + j] += D_EDOT
    return conds


def _inputs(case, seed):
    """Texture and condition states: a step's fan-out for 9 conditions, else unrelated states."""
    rng = np.random.default_rng(seed)
    tex = _texture(rng, case["textured"])
    k = case["n_cond"]
    if case["kind"] == "picard":
        conds = _fan_out(_state(rng), case["simplified"])
    else:
        conds = _fan_out(_state(rng)) if k == 9 else [_state(rng) for _ in range(k)]
    return tex, conds


def _requests(case, seed):
    """(n_theta, n_z, texture, state) of a burst over the served grids, half of them textured."""
    rng = np.random.default_rng(seed)
    grids = [(nt, nt // 2) for nt in (256, 512, 1024) if nt <= case["largest"]]
    out = []
    for i in range(case["requests"]):
        nt, nz = grids[i % len(grids)]
        out.append((nt, nz, _texture(rng, i % 2 == 0), _state(rng)))
    return out


_kept = {}


def _context():
    """The one context that a program keeps for its device and stream."""
    if "ctx" not in _kept:
        _kept["ctx"] = gmaf.Context()
    return _kept["ctx"].handle


def _the_server():
    if "server" not in _kept:
        _kept["server"] = gmaf.Server(_context(), 4 << 30)
    return _kept["server"]


def _device(n):
    return torch.empty(n, dtype=torch.float64, device="cuda")


def _system(case, tex, conds):
    n = len(conds) * case["n_theta"] * case["n_z"]
    arrays = [_device(n) for _ in range(4)]
    gmaf.gmaf_assemble(_context(), case["n_theta"], case["n_z"], PHYS, tex, conds, *arrays)
    return arrays


def _options(case, **more):
    return gmaf.solver_opts(precond=case.get("precond", 1), omega=OMEGA, eps=case["eps"],
                            precision=case.get("precision", 0),
                            criterion=case.get("criterion", 0), **more)


def prepare(case, seed):
    if case["kind"] == "server":
        reqs = [gmaf.request(nt, nz, PHYS, tex, st, st[:4], DT, F_EXT, D_E, D_EDOT, omega=OMEGA,
                             eps=case["eps"])
                for nt, nz, tex, st in _requests(case, seed)]
        return dict(case=case, server=_the_server(), requests=reqs)
    tex, conds = _inputs(case, seed)
    s = dict(case=case, ctx=_context(), tex=tex, conds=conds)
    n = len(conds) * case["n_theta"] * case["n_z"]
    if case["kind"] == "picard":
        s["opts"] = _options(case)
        s["fields"] = torch.zeros(9 * case["n_theta"] * case["n_z"], dtype=torch.float64,
                                  device="cuda")
    elif case["kind"] == "assemble":
        s["out"] = [_device(n) for _ in range(4)]
    elif case["kind"] == "loads":
        s["p"] = _pressure(case, seed)
        s["loads"] = _device(12 * len(conds))
    else:
        s["system"] = _system(case, tex, conds)
        s["p"] = _device(n)
        s["opts"] = _options(case, zero_init=0 if case["warm"] else 1)
        if case["warm"]:
            # the fields of the shaft step before: the same gap, moved by one step
            before = [c.copy() for c in conds]
            for c in before:
                c[:4] -= DT * c[4:]
            s["start"] = torch.zeros_like(s["p"])
            gmaf.gmaf_solve_joint(s["ctx"], case["n_theta"], case["n_z"], len(conds),
                                  *_system(case, tex, before), s["start"],
                                  gmaf.solver_opts(omega=OMEGA, eps=1e-10, precision=1))
    return s


def _pressure(case, seed):
    """Smooth pressure fields such as the solver leaves: axial drop plus a circumferential wave."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    k, nt, nz = case["n_cond"], case["n_theta"], case["n_z"]
    f64 = dict(dtype=torch.float64, device="cuda")
    a = torch.rand(k, 2, 1, 1, generator=g, **f64)
    th = (torch.arange(nt, **f64) + 0.5) * (2.0 * math.pi / nt)
    z = (torch.arange(nz, **f64).reshape(-1, 1) + 0.5) / nz
    p = PHYS[5] * (1.0 - z) + PHYS[6] * z
    return (p + 5e6 * a[:, 0] * torch.sin(math.pi * z) * torch.cos(th + 6.0 * a[:, 1])).reshape(-1)


# ------------------------------------------------------------------ one pass


def run(state):
    case = state["case"]
    if case["kind"] == "server":
        return _run_server(state)
    nt, nz, ctx = case["n_theta"], case["n_z"], state["ctx"]
    if case["kind"] == "assemble":
        gmaf.gmaf_assemble(ctx, nt, nz, PHYS, state["tex"], state["conds"], *state["out"])
        return dict(zip(("D", "aE", "aN", "S"), state["out"]))
    if case["kind"] == "loads":
        gmaf.gmaf_integrate_loads(ctx, nt, nz, PHYS, state["tex"], state["conds"], state["p"],
                                  state["loads"])
        return state["loads"]
    if case["kind"] == "picard":
        base = state["conds"][0]
        if case["simplified"]:
            r = gmaf.gmaf_picard_step_simplified(ctx, nt, nz, PHYS, state["tex"], base, DT, F_EXT,
                                                 D_EDOT, state["opts"])
        else:
            r = gmaf.gmaf_picard_step(ctx, nt, nz, PHYS, state["tex"], base, base[:4], DT, F_EXT,
                                      D_E, D_EDOT, state["opts"])
        gmaf.gmaf_last_fields(ctx, nt, nz, state["fields"])
        return dict(loads=r["loads"], J=r["J"], G=r["G"], state=r["state"],
                    fields=state["fields"][:case["n_cond"] * nt * nz])
    p = state["p"]
    if case["warm"]:
        p.copy_(state["start"])
    if case["noalloc"]:
        gmaf.gmaf_solve_joint_noalloc(nt, nz, case["n_cond"], *state["system"], p, state["opts"])
    else:
        gmaf.gmaf_solve_joint(ctx, nt, nz, case["n_cond"], *state["system"], p, state["opts"])
    return p


def _run_server(state):
    server, results = state["server"], {}
    ids = [server.submit(r) for r in state["requests"]]
    while len(results) < len(ids):
        server.run(64)
        for r in server.poll():
            results[r["id"]] = r
    out = [results[i] for i in ids]
    return [{k: r[k] for k in ("status", "loads", "J", "G", "state")} for r in out]


# ------------------------------------------------------------------ work


def _iterations(case, n_theta, n_z):
    """PCG iterations of a solve: they grow with the finer direction's cell count."""
    it = 1.9 * max(n_theta, 2 * n_z) * (1.0 if case["textured"] else 0.9)
    return it * {0: 1.85, 1: 1.0, 2: 1.9}[case.get("precond", 1)]


def work(case):
    """Inputs read once and results written once; the arithmetic of the iterations."""
    if case["kind"] == "server":
        total = {"bytes": 0.0, "flops": 0.0}
        for nt, nz, _, _ in _requests(case, 0):
            w = work(_picard("", nt, nz, precision=1))
            total = {k: total[k] + w[k] for k in total}
        return total
    nt, nz, k = case["n_theta"], case["n_z"], case["n_cond"]
    n = nt * nz
    if case["kind"] == "assemble":
        return {"bytes": 32.0 * k * n, "flops": 70.0 * k * n}
    if case["kind"] == "loads":
        return {"bytes": 8.0 * k * n, "flops": 70.0 * k * n}
    # x, r, u, A u (five points), both sweeps of M^-1, three dot products: 36 flops an unknown
    flops = 36.0 * k * n * _iterations(case, nt, nz)
    if case["kind"] == "picard":
        return {"bytes": 8.0 * k * n, "flops": flops + 140.0 * k * n}
    return {"bytes": 8.0 * k * n * (6 if case["warm"] else 5), "flops": flops}


# ------------------------------------------------------------------ the same in plain torch


def _arange(n):
    return torch.arange(n, dtype=torch.float64, device="cuda")


def _depth(tex, x, z):
    """Dimple depth at unwrapped positions x (row) and z (column)."""
    shape = torch.zeros(z.shape[0], x.shape[1], dtype=torch.bool, device="cuda")
    if not tex[0]:
        return shape.double()
    radius, depth, density, o_x, o_z = tex[1:]
    round_ = 2.0 * math.pi * PHYS[0]
    columns = max(1.0, round(round_ / (radius * math.sqrt(2.0 * math.pi / (math.sqrt(3.0) * density)))))
    a_x = round_ / columns
    a_z = math.pi * radius * radius / (density * a_x)
    k0 = torch.floor((z - o_z) / a_z)
    for dk in (-1.0, 0.0, 1.0, 2.0):
        k = k0 + dk
        dz = z - (o_z + k * a_z)
        u = (x - o_x) - torch.where(torch.remainder(k, 2.0) == 1.0, 0.5 * a_x, 0.0)
        m = torch.floor(u / a_x)
        for q in (0.0, 1.0):
            dx = u - (m + q) * a_x
            shape |= dx * dx + dz * dz < radius * radius
    return shape.double() * depth


def _film(cond, th, z):
    """Cartesian offsets, their length and the smooth film thickness at angles th and heights z."""
    r_k, length, c = PHYS[:3]
    t = z / length
    x = (r_k + c) * torch.cos(th) - (cond[0] + (cond[2] - cond[0]) * t)
    y = (r_k + c) * torch.sin(th) - (cond[1] + (cond[3] - cond[1]) * t)
    rho = torch.sqrt(x * x + y * y)
    return x, y, rho, rho - r_k


def _equations(tex, conds, nt, nz):
    """D, aE, aN, S of every condition, [n_cond][n_z][n_theta]."""
    r_k, length, _, mu, v, p_ch, p_case = PHYS
    dth = 2.0 * math.pi / nt
    dx, dz = r_k * dth, length / nz
    thc, the = ((_arange(nt) + 0.5) * dth).reshape(1, -1), ((_arange(nt) + 1.0) * dth).reshape(1, -1)
    zc, zf = ((_arange(nz) + 0.5) * dz).reshape(-1, 1), (_arange(nz + 1) * dz).reshape(-1, 1)
    deep_e, deep_f = _depth(tex, r_k * the, zc), _depth(tex, r_k * thc, zf)
    out = []
    for cond in conds:
        cond = [float(v) for v in cond]
        h_e = _film(cond, the, zc)[3] + deep_e
        h_f = _film(cond, thc, zf)[3] + deep_f
        x, y, rho, _ = _film(cond, thc, zc)
        t = zc / length
        h_dot = -(x * (cond[4] * (1 - t) + cond[6] * t) + y * (cond[5] * (1 - t) + cond[7] * t)) / rho
        east = h_e ** 3 / (12.0 * mu) * dz / dx
        face = h_f ** 3 / (12.0 * mu) * dx / dz
        face[0] *= 2.0
        face[nz] *= 2.0
        source = (v / 2.0) * (h_f[1:] - h_f[:-1]) * dx - h_dot * dx * dz
        source[0] += face[0] * p_ch
        source[-1] += face[nz] * p_case
        diag = east + east.roll(1, 1) + face[1:] + face[:-1]
        north = face[1:].clone()
        north[-1] = 0.0
        out.append((diag, east, north, source))
    return [torch.stack(x) for x in zip(*out)]


def _solution(diag, east, north, source):
    """The pressure fields by conjugate gradients, each condition with its own scalars."""
    west, south = east.roll(1, 2), torch.zeros_like(north)
    south[:, 1:] = north[:, :-1]

    def times(p):
        q = diag * p - east * p.roll(-1, 2) - west * p.roll(1, 2)
        q[:, :-1] -= north[:, :-1] * p[:, 1:]
        q[:, 1:] -= south[:, 1:] * p[:, :-1]
        return q

    def dot(a, b):
        return (a * b).sum((1, 2), keepdim=True)

    p, norm = torch.zeros_like(source), torch.sqrt(dot(source, source))
    for _ in range(3):                  # restarts take away what the recurrence has drifted
        r = source - times(p)
        u = z = r / diag
        d = dot(r, z)
        for i in range(40 * max(source.shape)):
            if i % 64 == 0 and bool((torch.sqrt(dot(r, r)) <= 2e-15 * norm).all()):
                break
            q = times(u)
            a = d / dot(u, q).clamp_min(1e-300)
            p = p + a * u
            r = r - a * q
            z = r / diag
            d, last = dot(r, z), d
            u = z + d / last.clamp_min(1e-300) * u
    return p


def _integrals(tex, conds, p, nt, nz):
    """Pressure and shear forces and moments of every condition, [n_cond][12]."""
    r_k, length, _, mu, v, p_ch, p_case = PHYS
    dth, dz = 2.0 * math.pi / nt, length / nz
    thc, the = ((_arange(nt) + 0.5) * dth).reshape(1, -1), ((_arange(nt) + 1.0) * dth).reshape(1, -1)
    nodes = torch.cat([_arange(1), (_arange(nz) + 0.5) * dz, _arange(1) + length]).reshape(-1, 1)
    step, mid = nodes[1:] - nodes[:-1], 0.5 * (nodes[1:] + nodes[:-1])
    weight = torch.zeros_like(nodes)
    weight[1:] += 0.5 * step
    weight[:-1] += 0.5 * step
    deep = _depth(tex, r_k * the, mid)
    out = []
    for cond, field in zip(conds, p):
        f = torch.cat([torch.full_like(field[:1], p_ch), field, torch.full_like(field[:1], p_case)])
        fx, fy = -f * torch.cos(thc) * weight * r_k * dth, -f * torch.sin(thc) * weight * r_k * dth
        rx, ry = r_k * torch.cos(thc), r_k * torch.sin(thc)
        row = [fx, fy, 0.0 * fx, -nodes * fy, nodes * fx, rx * fy - ry * fx]
        h = _film([float(c) for c in cond], the, mid)[3] + deep
        east = f.roll(-1, 1)
        along = ((f[1:] + east[1:]) - (f[:-1] + east[:-1])) / (2.0 * step)
        around = ((east[:-1] + east[1:]) - (f[:-1] + f[1:])) / (2.0 * dth)
        area = r_k * dth * step
        tz, tt = -(h / 2.0) * along - mu * v / h, -(h / 2.0) * around / r_k
        sx, sy, sz = -tt * torch.sin(the) * area, tt * torch.cos(the) * area, tz * area
        rx, ry = r_k * torch.cos(the), r_k * torch.sin(the)
        row += [sx, sy, sz, ry * sz - mid * sy, mid * sx - rx * sz, rx * sy - ry * sx]
        out.append(torch.stack([x.sum() for x in row]))
    return torch.stack(out)


def _step(tex, base, nt, nz, simplified=False):
    """A Picard step: loads, Jacobian, generalized force, new state, pressure fields."""
    conds = _fan_out(base, simplified)
    p = _solution(*_equations(tex, conds, nt, nz))
    loads = _integrals(tex, conds, p, nt, nz).cpu().numpy()
    total = loads[:, :6] + loads[:, 6:]
    jac = np.zeros((6, 8))
    for c in range(4):
        if simplified:
            jac[:, 4 + c] = (total[1 + c] - total[0]) / D_EDOT
        else:
            jac[:, c] = (total[1 + c] - total[0]) / D_E
            jac[:, 4 + c] = (total[5 + c] - total[0]) / D_EDOT
    tilt = np.zeros((4, 6))
    tilt[0, 0] = tilt[1, 1] = 1.0
    tilt[0, 4] = tilt[3, 3] = -1.0 / PHYS[1]
    tilt[1, 3] = tilt[2, 4] = 1.0 / PHYS[1]
    force = tilt @ total[0] + np.array(F_EXT)
    j_e, j_d = tilt @ jac[:, :4], tilt @ jac[:, 4:]
    e, rate = base[:4], base[4:]
    if simplified:
        delta = np.linalg.solve(j_d, -force)
        new = np.concatenate([e + DT * delta, rate + delta])
    else:
        delta = np.linalg.solve(j_d + DT * j_e, -force - j_e @ (DT * rate))
        new = np.concatenate([e + DT * (rate + delta), rate + delta])
    return dict(loads=loads[0], J=jac, G=force, state=new, fields=p.reshape(-1))


def exact(case, seed):
    if case["kind"] == "server":
        out = []
        for nt, nz, tex, st in _requests(case, seed):
            r = _step(tex, st, nt, nz)
            out.append({"status": None, **{k: r[k] for k in ("loads", "J", "G", "state")}})
        return out
    tex, conds = _inputs(case, seed)
    nt, nz = case["n_theta"], case["n_z"]
    if case["kind"] == "loads":
        p = _pressure(case, seed).reshape(len(conds), nz, nt)
        return _integrals(tex, conds, p, nt, nz).reshape(-1)
    if case["kind"] == "picard":
        return _step(tex, conds[0], nt, nz, case["simplified"])
    if len(conds) * nt * nz > 6e6 and case["kind"] == "solve":
        return None
    eqs = _equations(tex, conds, nt, nz)
    if case["kind"] == "assemble":
        return dict(zip(("D", "aE", "aN", "S"), (x.reshape(-1) for x in eqs)))
    return _solution(*eqs).reshape(-1)
