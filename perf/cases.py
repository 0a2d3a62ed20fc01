"""What the speed of this framework is measured on: FR solver runs through its Python entry points.

A case is a dict of plain values; `prepare` builds the mesh handle and the solver that a user's program keeps and sets a
seeded start, `run` makes one pass (a few Runge-Kutta steps with their samples, a residual, a restart) and returns what
such a program takes out of it.  A mixed-precision solver holds its flow in FP32, so its fields are handed on as FP32
tensors on the GPU (where post-processing reads them); a plain FP64 solver's stay the FP64 host arrays of the calls.

Meshes (all sizes come from bench.py and the tests): periodic boxes, a flat-plate channel of the cavity proxy's size,
O-meshes of uneven size around thin elliptic sections (the candidates of one poll) and a spanwise-extruded O-mesh around
a cylinder.  `exact` is a plain numpy FP64 solver for the periodic boxes.
"""
from __future__ import annotations

import atexit
import functools
import math
import os
import tempfile
from types import SimpleNamespace

import numpy as np
import torch

from paper_2312_14167_gb300 import fr

GAMMA, PR = 1.4, 0.71
PERIODIC, WALL, FARFIELD, INFLOW, OUTFLOW = 1, 2, 3, 4, 5

TUNE_CACHE = os.path.join(tempfile.gettempdir(), "fr_cases_tune_%d.json" % os.getpid())
atexit.register(lambda: os.path.exists(TUNE_CACHE) and os.unlink(TUNE_CACHE))


def listed():
    return [
        # the smallest run: the isentropic vortex (256 quads, Euler, RK4, plain FP64), 100 steps and the state out
        dict(name="vortex_16_p2_fp64", kind="box", n=16, dim=2, p=2, viscous=False, precision="fp64", rk="rk4",
             mach=0.5, steps=100),
        # a small mixed-precision run (4,096 quads, Navier-Stokes): latency and launches count
        dict(name="box_64_p3_fp32", kind="box", n=64, dim=2, p=3, viscous=True, precision="fp32", rk="lsrk45",
             mach=0.3, steps=20),
        # one design of the cavity proxy's size (31,722 quads), inflow, outflow, wall and far field, one observer:
        # 50 steps between two looks at the flow
        dict(name="channel_31722_p3_fp32", kind="channel", nx=311, ny=102, p=3, precision="fp32", mach=0.15, re=1500.0,
             steps=50),
        # the main use: the 32 candidates of a poll (uneven, 849k curved quads in all) advance together
        dict(name="poll_32_p3_fp32", kind="poll", n_inst=32, e_lo=8000, e_hi=45000, p=3, precision="fp32", mach=0.2,
             re=23000.0, steps=20),
        # the same with the far-field sponge of lower degrees (P3 to P0, mortar faces), 8 candidates
        dict(name="poll_8_sponge_p3_fp32", kind="poll", n_inst=8, e_lo=8000, e_hi=45000, p=3, sponge=True,
             precision="fp32", mach=0.2, re=23000.0, steps=20),
        # 8 candidates with adaptive steps
        dict(name="poll_8_adaptive_p3_fp32", kind="poll", n_inst=8, e_lo=8000, e_hi=45000, p=3, rk="bs32",
             precision="fp32", mach=0.2, re=23000.0, steps=20),
        # the other schemes in use: LDG and Roe, degree 4, one design
        dict(name="section_ldg_roe_p4_fp32", kind="poll", n_inst=1, e_lo=26000, e_hi=26000, p=4, scheme="ldg",
             flux="roe", precision="fp32", mach=0.2, re=23000.0, steps=20),
        # restart from a host checkpoint, one step, checkpoint again (what a driver that owns the states does)
        dict(name="restart_8_p3_fp32", kind="poll", n_inst=8, e_lo=8000, e_hi=45000, p=3, restart=True,
             precision="fp32", mach=0.2, re=23000.0, steps=1),
        # the plain path: one design in FP64
        dict(name="section_26k_p3_fp64", kind="poll", n_inst=1, e_lo=26000, e_hi=26000, p=3, precision="fp64", mach=0.2,
             re=23000.0, steps=5),
        # Taylor-Green hexes, mixed precision
        dict(name="tgv_48_p3_fp32", kind="box", n=48, dim=3, p=3, viscous=True, precision="fp32", rk="lsrk45", mach=0.1,
             steps=5),
        # a spanwise-extruded cylinder mesh, curved hexes of degree 4, 16 layers, wall forces and spanwise observers
        dict(name="cylinder_57k_p4_fp32", kind="span", n_theta=102, n_r=35, n_z=16, p=4, precision="fp32", mach=0.2,
             re=1000.0, steps=4),
        # one residual evaluation and the conservation check of a hex mesh in FP64
        dict(name="residual_tgv_16_p3_fp64", kind="box", n=16, dim=3, p=3, viscous=True, precision="fp64",
             rk="lsrk45", mach=0.1, residual=True, steps=0),
    ]


def draw(rng):
    """One more case of the ranges above."""
    kind = rng.choice(["box2", "box3", "channel", "poll", "poll", "sponge", "adaptive", "scheme", "restart", "fp64",
                       "span", "residual"])
    size = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    poll = dict(kind="poll", precision="fp32", mach=0.2, re=23000.0)
    if kind == "box2":
        visc = rng.random() < 0.7
        return dict(kind="box", n=size(5, 200), dim=2, p=rng.choice([1, 2, 3, 4]), viscous=visc,
                    precision=rng.choice(["fp32", "fp64"]), rk=rng.choice(["rk4", "lsrk45"]), mach=0.3,
                    steps=rng.choice([10, 20, 40]))
    if kind == "box3":
        return dict(kind="box", n=size(5, 44), dim=3, p=rng.choice([1, 2, 3, 3]), viscous=True, precision="fp32",
                    rk=rng.choice(["lsrk45", "rk4"]), mach=0.1, steps=rng.choice([2, 5]))
    if kind == "channel":
        return dict(kind="channel", nx=size(30, 300), ny=rng.randint(20, 110), p=rng.choice([2, 3, 4]),
                    precision="fp32", mach=0.15, re=1500.0, steps=rng.choice([10, 50]))
    if kind == "poll":
        lo = size(500, 9000)
        return dict(poll, n_inst=rng.randint(2, 16), e_lo=lo, e_hi=4 * lo, p=rng.choice([2, 3, 3, 4]), steps=10)
    if kind == "sponge":
        lo = size(500, 8000)
        return dict(poll, n_inst=rng.randint(2, 8), e_lo=lo, e_hi=4 * lo, p=rng.choice([2, 3, 4]), sponge=True,
                    steps=10)
    if kind == "adaptive":
        lo = size(500, 8000)
        return dict(poll, n_inst=rng.randint(2, 8), e_lo=lo, e_hi=4 * lo, p=rng.choice([2, 3]), rk="bs32", steps=10)
    if kind == "scheme":
        e = size(1000, 40000)
        return dict(poll, n_inst=1, e_lo=e, e_hi=e, p=rng.choice([2, 3, 4]), scheme=rng.choice(["ldg", "br2"]),
                    flux=rng.choice(["roe", "rusanov"]), steps=rng.choice([10, 20]))
    if kind == "restart":
        lo = size(500, 8000)
        return dict(poll, n_inst=rng.randint(2, 8), e_lo=lo, e_hi=4 * lo, p=rng.choice([2, 3]), restart=True, steps=1)
    if kind == "fp64":
        e = size(1000, 20000)
        return dict(poll, n_inst=1, e_lo=e, e_hi=e, p=rng.choice([2, 3, 4]), precision="fp64", steps=rng.choice([2, 5]))
    if kind == "span":
        return dict(kind="span", n_theta=rng.randint(24, 100), n_r=rng.randint(9, 34), n_z=rng.choice([4, 7, 16]),
                    p=rng.choice([2, 3, 4, 4]), precision="fp32", mach=0.2, re=1000.0, steps=rng.choice([2, 4]))
    return dict(kind="box", n=size(4, 24), dim=3, p=rng.choice([1, 2, 3]), viscous=True,
                precision=rng.choice(["fp64", "fp32"]), rk="lsrk45", mach=0.1, residual=True, steps=0)


# ------------------------------------------------------------------ meshes

def box_mesh(n, dim):
    """Uniform periodic box of n^dim elements, side 2 pi (3-D) or 10 (2-D), centred in 2-D."""
    side, lo = (10.0, -5.0) if dim == 2 else (2 * math.pi, 0.0)
    x = lo + side * np.arange(n + 1) / n
    grid = np.meshgrid(*[x] * dim, indexing="ij")
    xyz = np.stack([g.T.ravel() for g in grid], 1)
    tags = np.zeros([n] * dim + [2 * dim], np.int32)
    for d in range(dim):
        at = np.moveaxis(tags, dim - 1 - d, 0)
        at[0, ..., 2 * d] = PERIODIC
        at[-1, ..., 2 * d + 1] = PERIODIC
    return SimpleNamespace(dim=dim, xyz=xyz, elem_vert=lattice(*[n] * dim), face_tag=tags.reshape(-1, 2 * dim),
                           periodic_shift=side * np.eye(dim), geo_order=1, geo_nodes=None)


def lattice(*cells, wrap=False):
    """Corner vertices of a structured block of cells (x fastest); `wrap` closes the first direction."""
    e = np.meshgrid(*[np.arange(c) for c in cells], indexing="ij")
    e = [a.T.ravel() for a in e]
    verts = [cells[0] if wrap else cells[0] + 1] + [c + 1 for c in cells[1:]]
    out = []
    for corner in range(2 ** len(cells)):
        idx, step = 0, 1
        for d, a in enumerate(e):
            v = a + (corner >> d & 1)
            idx = idx + step * (v % verts[d] if d == 0 and wrap else v)
            step *= verts[d]
        out.append(idx)
    return np.stack(out, 1).astype(np.int64)


def channel_mesh(nx, ny):
    """Flat-plate channel, stretched off the plate; inflow left, outflow right, far field above."""
    x = 3.0 * np.arange(nx + 1) / nx
    y = np.cumsum(np.concatenate([[0.0], 1.05 ** np.arange(ny)]))
    y = 3.0 * y / y[-1]
    gx, gy = np.meshgrid(x, y, indexing="ij")
    tags = np.zeros((ny, nx, 4), np.int32)
    tags[:, 0, 0], tags[:, -1, 1], tags[0, :, 2], tags[-1, :, 3] = INFLOW, OUTFLOW, WALL, FARFIELD
    return SimpleNamespace(dim=2, xyz=np.stack([gx.T.ravel(), gy.T.ravel()], 1), elem_vert=lattice(nx, ny),
                           face_tag=tags.reshape(-1, 4), periodic_shift=np.zeros((0, 2)), geo_order=1, geo_nodes=None)


def o_mesh(n_t, n_r, thick, angle, q, radius=20.0, first=1e-3):
    """Curved O-mesh of n_t x n_r quads around an elliptic section (chord 1 about the origin, relative thickness
    `thick`, pitched by `angle`), radially stretched from a first cell `first` to a circle of `radius`."""
    length = radius - 0.5
    a, b = 1.0 + 1e-9, 3.0
    for _ in range(80):
        r = 0.5 * (a + b)
        a, b = (r, b) if first * (r ** n_r - 1) / (r - 1) < length else (a, r)
    t = np.concatenate([[0.0], np.cumsum(first * a ** np.arange(n_r))])
    t = t / t[-1]
    c, s = math.cos(angle), math.sin(angle)

    def place(th, ta):
        sx, sy = 0.5 * np.cos(th), 0.5 * thick * np.sin(th)
        sx, sy = c * sx + s * sy, -s * sx + c * sy
        return np.stack([sx + ta * (radius * np.cos(th) - sx), sy + ta * (radius * np.sin(th) - sy)], -1)

    th = -2 * math.pi * np.arange(n_t) / n_t
    xyz = place(th[None, :], t[:, None]).reshape(-1, 2)
    f = np.arange(q + 1) / q
    tn = -2 * math.pi * (np.arange(n_t)[:, None] + f) / n_t                     # (n_t, q + 1)
    rn = t[:-1, None] + f * (t[1:] - t[:-1])[:, None]                           # (n_r, q + 1)
    nodes = place(tn[None, :, None, :], rn[:, None, :, None]).reshape(n_r * n_t, (q + 1) ** 2, 2)
    tags = np.zeros((n_r, n_t, 4), np.int32)
    tags[0, :, 2], tags[-1, :, 3] = WALL, FARFIELD
    return SimpleNamespace(dim=2, xyz=xyz, elem_vert=lattice(n_t, n_r, wrap=True), face_tag=tags.reshape(-1, 4),
                           periodic_shift=np.zeros((0, 2)), geo_order=q, geo_nodes=nodes, thick=thick, angle=angle)


def span_mesh(n_t, n_r, n_z, q=2):
    """The O-mesh around a circular cylinder extruded over a periodic span of pi diameters."""
    m = o_mesh(n_t, n_r, 1.0, 0.0, q, radius=15.0, first=8e-3)
    nv, span = m.xyz.shape[0], math.pi
    z = span * np.arange(n_z + 1) / n_z
    xyz = np.concatenate([np.tile(m.xyz, (n_z + 1, 1)), np.repeat(z, nv)[:, None]], 1)
    ev = np.concatenate([np.concatenate([m.elem_vert + k * nv, m.elem_vert + (k + 1) * nv], 1) for k in range(n_z)])
    f = np.arange(q + 1) / q
    n2 = m.geo_nodes.shape[1]
    nodes = np.empty((n_z, ev.shape[0] // n_z, q + 1, n2, 3))
    nodes[..., :2] = m.geo_nodes[None, :, None]
    nodes[..., 2] = (span * (np.arange(n_z)[:, None] + f) / n_z)[:, None, :, None]
    tags = np.zeros((n_z, ev.shape[0] // n_z, 6), np.int32)
    tags[..., :4] = m.face_tag
    tags[0, :, 4], tags[-1, :, 5] = PERIODIC, PERIODIC
    return SimpleNamespace(dim=3, xyz=xyz, elem_vert=ev, face_tag=tags.reshape(-1, 6),
                           periodic_shift=np.array([[0.0, 0.0, span]]), geo_order=q,
                           geo_nodes=nodes.reshape(-1, (q + 1) * n2, 3), thick=1.0, angle=0.0)


@functools.lru_cache(maxsize=4)
def handles(kind, p, sponge, *sizes):
    """The mesh handles of a case, their shortest edge and their observers; a program builds them once per design."""
    rng = np.random.default_rng(2312)
    if kind == "box":
        meshes = [box_mesh(*sizes)]
    elif kind == "channel":
        meshes = [channel_mesh(*sizes)]
    elif kind == "span":
        meshes = [span_mesh(*sizes)]
    else:
        n_inst, e_lo, e_hi = sizes
        meshes = []
        for _ in range(n_inst):
            n_r = max(6, int(round(math.sqrt(rng.uniform(e_lo, e_hi) / 4.0))))
            meshes.append(o_mesh(4 * n_r + int(rng.integers(0, 5)), n_r, rng.uniform(0.08, 0.16),
                                 math.radians(rng.uniform(0.0, 6.0)), 3))
    edge, found = math.inf, []
    for m in meshes:
        v = m.xyz[m.elem_vert]
        for a, b in ((0, 1), (0, 2), (1, 3), (2, 3)) if m.dim == 2 else ((0, 1), (0, 2), (0, 4)):
            edge = min(edge, float(np.linalg.norm(v[:, a] - v[:, b], axis=1).min()))
        degree = p
        if sponge:
            rc = np.linalg.norm(m.geo_nodes.mean(1), axis=1)
            degree = np.maximum(p - np.searchsorted([4.0, 8.0, 12.0], rc, side="right"), 0)
        found.append(fr.Mesh(m, degree))
    if kind == "poll":
        seen = [[(0.5, -2.0)]] * len(meshes)
    elif kind == "span":
        seen = [[(0.0, 2.0, math.pi * (k + 0.5) / 16) for k in range(16)]]
    elif kind == "channel":
        seen = [[(1.5, 0.3)]]
    else:
        seen = [[]]
    return found, meshes, edge, seen


# ------------------------------------------------------------------ the case

def start(case, x, mesh, seed, inst):
    """Seeded start at the points x (an FP64 tensor): Taylor-Green field plus perturbations, isentropic vortex, or the
    free stream with smooth perturbations, the velocity damped towards the walls."""
    rng = np.random.default_rng([seed, inst])
    dim, mach = x.shape[-1], case["mach"]
    box = case["kind"] == "box"
    length = 10.0 if dim == 2 else 2 * math.pi
    at = [x[..., d] for d in range(dim)]
    modes = []
    for _ in range(dim + 2):
        acc = 0.0
        for _ in range(3):
            k = 2 * math.pi / length * rng.integers(-2, 3, dim) if box else rng.uniform(0.2, 1.5, dim)
            phase = sum(float(kd) * xd for kd, xd in zip(k, at)) + rng.uniform(0, 2 * math.pi)
            acc = acc + rng.uniform(0.1, 0.33) * torch.sin(phase)
        modes.append(acc)
    rho, vel, p = 1.0 + 0.02 * modes[0], [0.02 * m for m in modes[1:-1]], 1.0 + 0.02 * modes[-1]
    p_inf = 1.0 / (GAMMA * mach * mach)
    if box and dim == 3:
        X, Y, Z = at
        vel[0] = vel[0] + torch.sin(X) * torch.cos(Y) * torch.cos(Z)
        vel[1] = vel[1] - torch.cos(X) * torch.sin(Y) * torch.cos(Z)
        p = p_inf * (1.0 + 0.1 * (p - 1.0)) + (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0) / 16.0
        rho = 1.0 + 0.1 * (rho - 1.0)
    elif box and not case["viscous"]:
        p_inf = 1.0
        f = torch.exp(0.5 * (1.0 - at[0] ** 2 - at[1] ** 2))
        T = 1.0 - (GAMMA - 1.0) * 25.0 / (8.0 * GAMMA * math.pi ** 2) * f * f
        rho, p = rho * T ** 2.5, p * T ** 3.5
        vel[0] = vel[0] + mach * math.sqrt(GAMMA) - 5.0 / (2 * math.pi) * at[1] * f
        vel[1] = vel[1] + 5.0 / (2 * math.pi) * at[0] * f
    else:
        vel[0] = vel[0] + 1.0
        p = p_inf * p
    if case["kind"] == "channel":
        vel = [v * torch.tanh(3.0 * at[1] / 0.2) for v in vel]
    elif not box:
        c, s = math.cos(mesh.angle), math.sin(mesh.angle)
        xl, yl = c * at[0] - s * at[1], s * at[0] + c * at[1]
        off = torch.sqrt((2 * xl) ** 2 + (2 * yl / mesh.thick) ** 2) - 1.0
        vel = [v * (1.0 - torch.exp(-torch.clamp(off, min=0.0) / 0.2)) for v in vel]
    ke = 0.5 * rho * sum(v * v for v in vel)
    return torch.stack([rho] + [rho * v for v in vel] + [p / (GAMMA - 1.0) + ke], -1)


def time_step(case, edge, p):
    c = math.sqrt(GAMMA) if case["kind"] == "box" and not case["viscous"] else 1.0 / case["mach"]
    return 0.3 * edge / ((1.0 + c) * (p + 1) ** 2)


def viscosity(case):
    if case["kind"] == "box":
        return (0.02 if case["dim"] == 2 else 1.0 / 1600.0) if case["viscous"] else 0.0
    return 1.0 / case["re"]


def plan(case):
    c = dict(viscous=True, rk="lsrk45", scheme="br2", flux="rusanov", sponge=False, restart=False, residual=False)
    c.update(case)
    c["sizes"] = {"box": lambda: (c["n"], c["dim"]), "channel": lambda: (c["nx"], c["ny"]),
                  "span": lambda: (c["n_theta"], c["n_r"], c["n_z"]),
                  "poll": lambda: (c["n_inst"], c["e_lo"], c["e_hi"])}[c["kind"]]()
    return c


def prepare(case, seed):
    c = plan(case)
    found, meshes, edge, seen = handles(c["kind"], c["p"], c["sponge"], *c["sizes"])
    dim, mixed = meshes[0].dim, c["precision"] == "fp32"
    still = c["kind"] == "box" and dim == 3
    vortex = c["kind"] == "box" and not c["viscous"]
    free = (0.0,) * dim if still else (c["mach"] * math.sqrt(GAMMA) if vortex else 1.0,) + (0.0,) * (dim - 1)
    p_inf = 1.0 if vortex else 1.0 / (GAMMA * c["mach"] ** 2)
    dt = time_step(c, edge, c["p"])
    cfg = fr.make_config(
        dim, gamma=GAMMA, prandtl=PR, mu=viscosity(c), rho_inf=1.0, v_inf=free, p_inf=p_inf, dt=dt,
        viscous=c["viscous"], inflow_delta=0.2, inflow_ywall=0.0,
        rk={"rk4": fr.FR_RK4, "lsrk45": fr.FR_LSRK45, "bs32": fr.FR_BS32}[c["rk"]],
        precision=fr.FR_FP32 if mixed else fr.FR_FP64,
        flux=fr.FR_FLUX_ROE if c["flux"] == "roe" else fr.FR_FLUX_RUSANOV,
        viscous_scheme=fr.FR_VISC_LDG if c["scheme"] == "ldg" else fr.FR_VISC_BR2,
        rtol=1e-6, atol=[1e-6] * (dim + 1) + [1e-6 * p_inf / (GAMMA - 1.0)])
    sol = fr.Solver(found, cfg)
    if mixed and not c["residual"]:
        sol.tune(TUNE_CACHE)            # measured once per shape, then looked up
    sizes = sol.state_sizes()
    host = torch.empty(sum(sizes), dtype=torch.float64, pin_memory=True)
    at = 0
    for i, (m, h) in enumerate(zip(meshes, found)):
        points = torch.from_numpy(h.sol_coords()).cuda()
        host[at:at + sizes[i]] = start(c, points, m, seed, i).reshape(-1).cpu()
        at += sizes[i]
    sol.set_states(host.numpy())
    probes = [sol.probe_add(i, np.array(x)) for i, pts in enumerate(seen) for x in pts]
    back = torch.empty(sum(sizes), dtype=torch.float64, pin_memory=True) if c["restart"] else host
    wall = any((m.face_tag == WALL).any() for m in meshes)
    return SimpleNamespace(case=c, sol=sol, host=host, back=back, probes=probes, wall=wall, mixed=mixed,
                           sums=dim + 2, out=np.empty(found[0].state_shape + (dim + 2,)) if c["residual"] else None)


def run(state):
    c, sol = state.case, state.sol
    if c["residual"]:
        r = sol.residual(0, state.out)
        return dict(residual=np.float32(r)) if state.mixed else dict(residual=r)
    if c["restart"]:
        sol.set_states(state.host.numpy())
    sol.rk_step(c["steps"])
    sol.get_states(state.back.numpy())
    if not state.mixed:
        return dict(state=state.back)
    out = dict(state=state.back.to("cuda").float())
    if state.probes:
        out["pressure"] = np.float32([sol.probe_pressure(i) for i in state.probes])
    if state.wall and c["rk"] != "bs32":
        out["force"] = np.float32([sol.forces(i) for i in range(len(sol.meshes))])
    return out


# ------------------------------------------------------------------ what a pass cannot do without

def degrees(c):
    """(elements, degree) of each part of a case, near enough for a count."""
    if c["kind"] == "box":
        return [(c["n"] ** c["dim"], c["p"])], c["dim"]
    if c["kind"] == "channel":
        return [(c["nx"] * c["ny"], c["p"])], 2
    if c["kind"] == "span":
        return [(c["n_theta"] * c["n_r"] * c["n_z"], c["p"])], 3
    found, _, _, _ = handles(c["kind"], c["p"], c["sponge"], *c["sizes"])
    every = np.concatenate([h.elem_p for h in found])
    return [(int((every == d).sum()), int(d)) for d in np.unique(every)], 2


def work(case):
    c = plan(case)
    parts, dim = degrees(c)
    s, V = 4 if c["precision"] == "fp32" else 8, dim + 2
    stages = 1 if c["residual"] else c["steps"] * {"rk4": 4, "lsrk45": 5, "bs32": 3}[c["rk"]]
    nbytes = flops = 0
    for elements, p in parts:
        n = p + 1
        points, faces = elements * n ** dim, elements * 2 * dim * n ** (dim - 1)
        # a stage: state and register in and out, the metric terms; per flux point its normal, its partner's index and
        # state, and for viscous flow the partner's viscous flux
        nbytes += stages * (points * (4 * V * s + (dim * dim + 1) * s) +
                            faces * (dim * s + 4 + V * s * (2 if c["viscous"] else 1)))
        lines = 2 * dim * n * V                       # one derivative along every direction
        per_point = lines + dim * 2 * V + 2 * dim * dim * V + 20 * V
        per_point += 2 * dim * dim * V + lines + 40 * V if c["viscous"] else 0
        per_face = 2 * n * V + 30 * V + ((2 * n + 4) * dim * V + 30 * V if c["viscous"] else 0)
        flops += stages * (points * per_point + faces * per_face)
        nbytes += points * V * 8 * (2 if c["restart"] else 1)
    return dict(bytes=nbytes, flops=flops)


# ------------------------------------------------------------------ FP64 reference on uniform periodic boxes

def exact(case, seed):
    c = plan(case)
    if c["kind"] != "box":
        return None                                   # curved meshes: minutes in plain numpy
    n, dim, p = c["n"], c["dim"], c["p"]
    evaluations = 1 if c["residual"] else c["steps"] * (4 if c["rk"] == "rk4" else 5)
    if n ** dim * (p + 1) ** dim * evaluations * (dim + 2) * (p + 2) > (3.5e8 if c["viscous"] else 1.2e9):
        return None
    length = 10.0 if dim == 2 else 2 * math.pi
    h = length / n
    ref = Reference(n, dim, p, h, viscosity(c))
    lo = -5.0 if dim == 2 else 0.0
    grid = np.indices([n] * dim).reshape(dim, -1)[::-1].T                     # element index, x first
    node = np.indices([p + 1] * dim).reshape(dim, -1)[::-1].T
    x = lo + h * (grid[:, None, :] + 0.5 * (1.0 + ref.xi[node])[None])
    u = start(c, torch.from_numpy(x), None, seed, 0).numpy()
    shape = u.shape
    u = u.reshape([n] * dim + [p + 1] * dim + [dim + 2])
    if c["residual"]:
        return dict(residual=ref.residual(u).reshape(shape))
    dt = time_step(c, h, p)
    for _ in range(c["steps"]):
        u = ref.rk4(u, dt) if c["rk"] == "rk4" else ref.lsrk45(u, dt)
    return dict(state=u.ravel())


class Reference:
    """Flux Reconstruction (DG-recovery correction, Gauss points, Rusanov, BR2) on a uniform periodic box in plain
    numpy FP64.  Arrays are [ez][ey][ex][k][j][i][v]; axis(d) of direction d counts from the back."""

    def __init__(self, n, dim, p, h, mu):
        self.dim, self.mu, self.scale = dim, mu, 2.0 / h
        leg = np.polynomial.legendre
        xi, _ = leg.leggauss(p + 1)
        self.xi = xi
        vand = np.stack([leg.legval(xi, np.eye(p + 1)[k]) for k in range(p + 1)], 1)
        inv = np.linalg.inv(vand)
        der = np.stack([leg.legval(xi, leg.legder(np.eye(p + 1)[k])) if k else 0 * xi for k in range(p + 1)], 1)
        self.D = der @ inv
        self.end = np.stack([np.array([s ** k for k in range(p + 1)], float) @ inv for s in (-1, 1)])
        radau = (-1.0) ** (p + 1) / 2 * (np.eye(p + 2)[p + 1] - np.eye(p + 2)[p])   # 1 at -1, 0 at +1
        gl = leg.legval(xi, leg.legder(radau))
        self.g = np.stack([gl, -gl[::-1]])

    def axis(self, d):
        return -2 - d, -2 - self.dim - d              # points, elements

    def along(self, mat, u, d):
        return np.moveaxis(np.tensordot(u, mat, axes=(self.axis(d)[0], 1)), -1, self.axis(d)[0])

    def ends(self, u, d):
        a = self.axis(d)[0]
        return [np.tensordot(u, self.end[s], axes=(a, 0)) for s in (0, 1)]

    def spread(self, jump, s, d):
        """g' of side s times a face jump, at every point of the line."""
        a = self.axis(d)[0] + 1
        shape = [1] * (jump.ndim + 1)
        shape[self.axis(d)[0]] = -1
        return np.expand_dims(jump, a - 1 if a < 0 else a) * self.g[s].reshape(shape)

    def euler(self, u, d):
        rho, m, E = u[..., 0], u[..., 1:-1], u[..., -1]
        v = m / rho[..., None]
        p = (GAMMA - 1.0) * (E - 0.5 * (m * v).sum(-1))
        F = u * v[..., d:d + 1]
        F[..., 1 + d] += p
        F[..., -1] += p * v[..., d]
        return F, v[..., d], np.sqrt(GAMMA * p / rho)

    def viscous(self, u, grad, d):
        """Viscous flux in direction d; grad[j] = du/dx_j."""
        rho = u[..., 0]
        v = u[..., 1:-1] / rho[..., None]
        gv = [(g[..., 1:-1] - g[..., :1] * v) / rho[..., None] for g in grad]
        gE = (grad[d][..., -1] - grad[d][..., 0] * u[..., -1] / rho) / rho
        div = sum(gv[i][..., i] for i in range(self.dim))
        out = np.zeros_like(u)
        for i in range(self.dim):
            tau = self.mu * (gv[d][..., i] + gv[i][..., d] - (2.0 / 3.0 * div if i == d else 0.0))
            out[..., 1 + i] = tau
            out[..., -1] += v[..., i] * tau
        out[..., -1] += self.mu / PR * GAMMA * (gE - (v * gv[d]).sum(-1))
        return out

    def residual(self, u):
        sc, dims = self.scale, range(self.dim)
        roll = lambda a, d, k: np.roll(a, k, axis=self.axis(d)[1] + 1)  # noqa: E731  (face arrays lack the point axis)
        raw = [sc * self.along(self.D, u, d) for d in dims] if self.mu else None
        grad = list(raw) if self.mu else None
        faces = []
        for d in dims:
            low, high = self.ends(u, d)
            left, right = high, roll(low, d, -1)      # the face above each element
            FL, vL, cL = self.euler(left, d)
            FR, vR, cR = self.euler(right, d)
            lam = np.maximum(np.abs(vL) + cL, np.abs(vR) + cR)[..., None]
            common = 0.5 * (FL + FR) - 0.5 * lam * (right - left)
            if self.mu:
                mean = 0.5 * (left + right)
                eta = 2.0 * self.dim
                sides = []
                for s, own in ((1, left), (0, right)):
                    Q = [self.ends(g, d)[s] if s == 1 else roll(self.ends(g, d)[0], d, -1) for g in raw]
                    Q[d] = Q[d] + eta * sc * (self.end[s] @ self.g[s]) * (mean - own)
                    sides.append(self.viscous(own, Q, d))
                common = common - 0.5 * (sides[0] + sides[1])
                grad[d] = grad[d] + sc * (self.spread(mean - left, 1, d) + self.spread(roll(mean, d, 1) - low, 0, d))
            faces.append(common)
        r = 0.0
        for d in dims:
            F = self.euler(u, d)[0]
            if self.mu:
                F = F - self.viscous(u, grad, d)
            low, high = self.ends(F, d)
            r = r - sc * (self.along(self.D, F, d) + self.spread(faces[d] - high, 1, d) +
                          self.spread(roll(faces[d], d, 1) - low, 0, d))
        return r

    def rk4(self, u, dt):
        a = self.residual(u)
        b = self.residual(u + 0.5 * dt * a)
        c = self.residual(u + 0.5 * dt * b)
        d = self.residual(u + dt * c)
        return u + dt / 6.0 * (a + 2 * b + 2 * c + d)

    def lsrk45(self, u, dt):
        """Carpenter and Kennedy's five-stage fourth-order 2N-storage scheme."""
        A = (0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238, -3550918686646 / 2091501179385,
             -1275806237668 / 842570457699)
        B = (1432997174477 / 9575080441755, 5161836677717 / 13612068292357, 1720146321549 / 2090206949498,
             3134564353537 / 4481467310338, 2277821191437 / 14882151754819)
        du = 0.0
        for a, b in zip(A, B):
            du = a * du + dt * self.residual(u)
            u = u + b * du
        return u
