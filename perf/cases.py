"""The work a user of this framework has it do, as measured cases.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw``
one more of the same ranges, ``prepare`` what a program holds before the call
(fields in device memory and the solver it keeps), ``run`` one pass through the
public entry points, ``work`` what a pass cannot do without, ``exact`` the same
outputs from plain torch in 64 bits.

Kinds:
  run       a simulation: initial fields in, n steps, final fields out
            (physical fields, or the raw state of a checkpoint for 16-bit storage)
  batch     many 2D cavities advanced together
  gradient  a differentiable rollout, forward and backward
"""
import math
import random

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1901_02716_gb300 import adjoint
from paper_1901_02716_gb300 import maclab as M

PRECISION = {"f64": M.F64, "f32": M.F32, "bf16": M.BF16_STORE, "f16": M.F16_STORE}
# The most node updates a drawn run may take (three quarters of the largest listed run).
MOST_UPDATES = 1.0e9


def listed():
    def run(name, flow, nx, ny, nz, precision, steps, re=0.0, monitor=0):
        return {"name": name, "kind": "run", "flow": flow, "nx": nx, "ny": ny, "nz": nz, "precision": precision,
                "steps": steps, "re": re, "monitor": monitor}

    return [
        # the 2D Taylor-Green vortex in double precision: a small validation run, all launches and latency
        run("tgv2d_64_f64", "tgv", 64, 64, 1, "f64", 100),
        # 2D lid-driven cavities: the two sizes of the standard workload, and the paper's 400 x 400
        # intervals (401 nodes a side, an odd width)
        run("cavity2d_256_f32", "cavity", 256, 256, 1, "f32", 200, re=1000.0),
        run("cavity2d_401_f32", "cavity", 401, 401, 1, "f32", 100, re=1000.0),
        run("cavity2d_1024_f32", "cavity", 1024, 1024, 1, "f32", 100, re=1000.0),
        # the same flow in double precision
        run("cavity2d_256_f64", "cavity", 256, 256, 1, "f64", 50, re=1000.0),
        # 3D lid-driven cavities: the headline size, the paper's 250^3 intervals (251 nodes a side), and a
        # state far larger than the L2
        run("cavity3d_128_f32", "cavity", 128, 128, 128, "f32", 100, re=100.0),
        run("cavity3d_251_f32", "cavity", 251, 251, 251, "f32", 20, re=400.0),
        run("cavity3d_512_f32", "cavity", 512, 512, 512, "f32", 10, re=400.0),
        # 16-bit storage, returned as the raw state that a checkpoint holds
        run("cavity3d_128_bf16", "cavity", 128, 128, 128, "bf16", 20, re=100.0),
        # an obstacle flow (spinning sphere, per-node wall values, body force) with its diagnostics logged
        # every ten steps
        run("sphere_128x128x256_f32", "sphere", 128, 128, 256, "f32", 50, monitor=10),
        # many cavities of different sizes at once
        {"name": "batch_64_cavities_f32", "kind": "batch", "count": 64, "low": 64, "high": 512, "layout": 4,
         "precision": "f32", "steps": 200},
        # training through the solver: a rollout and the gradients of its inputs and of the viscosity
        {"name": "gradient_tgv3d_96_f32", "kind": "gradient", "nx": 96, "ny": 96, "nz": 96, "precision": "f32",
         "steps": 32},
    ]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def _width(rng, low, high):
    """A size of the range: as often any number as a multiple of 4 or of 32."""
    n = _log_int(rng, low, high)
    step = rng.choice([1, 1, 4, 32])
    return max(low, n // step * step)


def draw(rng):
    kind = rng.choice(["2d", "2d", "2d", "3d", "3d", "3d", "batch", "gradient"])
    if kind == "batch":
        return {"kind": "batch", "count": _log_int(rng, 8, 64), "low": 64, "high": rng.choice([256, 512]),
                "layout": rng.randrange(1 << 20), "precision": "f32", "steps": rng.randrange(50, 201)}
    if kind == "gradient":
        return {"kind": "gradient", "nx": _width(rng, 24, 112), "ny": _width(rng, 24, 112),
                "nz": _width(rng, 24, 112), "precision": "f32", "steps": rng.randrange(8, 33)}
    case = {"kind": "run", "flow": rng.choice(["cavity", "cavity", "tgv"]), "monitor": 0}
    if kind == "2d":
        case["nx"] = _width(rng, 40, 4096)
        case["ny"] = case["nx"] if rng.random() < 0.5 else max(40, min(4096, int(case["nx"] * rng.uniform(0.4, 2.5))))
        case["nz"] = 1
        case["precision"] = rng.choice(["f32", "f32", "f32", "f64"])
        if case["precision"] == "f64":
            case["nx"], case["ny"] = min(case["nx"], 1024), min(case["ny"], 1024)
        steps = rng.randrange(20, 201)
    else:
        case["nx"] = _width(rng, 32, 400)
        for axis in ("ny", "nz"):
            case[axis] = case["nx"] if rng.random() < 0.5 else max(32, min(512, int(case["nx"] * rng.uniform(0.4, 2.0))))
        case["precision"] = rng.choice(["f32", "f32", "f32", "bf16", "f16"])
        if rng.random() < 0.2:
            case["flow"] = "sphere"
        if rng.random() < 0.25 and case["precision"] == "f32":
            case["monitor"] = 10
        steps = rng.randrange(10, 21) if case["precision"] in ("bf16", "f16") else rng.randrange(10, 101)
    updates = case["nx"] * case["ny"] * case["nz"]
    case["steps"] = int(max(4, min(steps, MOST_UPDATES // updates // (16 if case["precision"] == "f64" else 1))))
    case["re"] = round(math.exp(rng.uniform(math.log(100.0), math.log(1000.0))), 1) if case["flow"] == "cavity" else 0.0
    return case


# ------------------------------------------------------------------ the flows

def _grid(case):
    return (case["ny"], case["nx"]) if case["nz"] == 1 else (case["nz"], case["ny"], case["nx"])


def _axes(grid):
    return torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.float64) for n in grid], indexing="ij")


def _walls(flow, grid):
    """(node types [grid] uint8 on the host or None, wall id count, periodic bits)."""
    d = len(grid)
    if flow == "tgv":
        return None, 0, (1 << d) - 1
    nt = np.zeros(grid, dtype=np.uint8)
    for axis in range(d):
        if flow == "sphere" and axis == 0:
            continue  # periodic along the channel
        edge = [slice(None)] * d
        for i in (0, grid[axis] - 1):
            edge[axis] = i
            nt[tuple(edge)] = 1
    if flow == "cavity":
        nt[(grid[0] - 1,) + (slice(1, -1),) * (d - 1)] = 2  # the lid, strictly between the side walls
        return nt, 2, 0
    (xc, yc, zc), r = _sphere(grid)
    z, y, x = np.ogrid[tuple(slice(n) for n in grid)]
    nt[((x - xc) ** 2 + (y - yc) ** 2 + (z - zc) ** 2 <= r * r) & (nt == 0)] = 2
    return nt, 2, 0b100


def _sphere(grid):
    nz, ny, nx = grid
    return ((nx - 1) / 2.0, (ny - 1) / 2.0, nz / 4.0), min(nx, ny) / 8.0


def _lid(case):
    """Lattice lid speed for the Reynolds number (lattice viscosity 1/6), at most 0.3."""
    return min(0.3, case["re"] / (6.0 * (case["nx"] - 1)))


def _fields(case, seed, grid, generator=None):
    """A developing flow in lattice units, in 64 bits on the GPU: seeded large-scale modes
    (a Taylor-Green field for the periodic flows) and a little noise."""
    d = len(grid)
    host = random.Random(seed)
    gen = generator or torch.Generator(device="cuda").manual_seed(seed)
    ax = [a * (2.0 * math.pi / n) for a, n in zip(_axes(grid), grid)][::-1]  # x first
    phase = [host.uniform(0.0, 2.0 * math.pi) for _ in range(3 * d + 3)]
    amp = 0.05 * host.uniform(0.6, 1.0)
    u = torch.empty((d,) + tuple(grid), device="cuda", dtype=torch.float64)
    if case.get("flow", "tgv") == "tgv":
        rest = torch.cos(ax[2]) if d == 3 else 1.0
        u[0] = amp * torch.sin(ax[0] + phase[0]) * torch.cos(ax[1] + phase[1]) * rest
        u[1] = -amp * torch.cos(ax[0] + phase[0]) * torch.sin(ax[1] + phase[1]) * rest
        if d == 3:
            u[2] = 0.2 * amp * torch.sin(ax[0] + phase[2])
    else:
        for i in range(d):
            u[i] = amp * torch.sin(ax[(i + 1) % d] + phase[i]) * torch.sin(2.0 * ax[i] + phase[d + i])
    u += 1e-3 * torch.randn(u.shape, generator=gen, device="cuda", dtype=torch.float64)
    rho = 1.0 + 0.005 * torch.sin(ax[0] + phase[3 * d]) * torch.sin(ax[1] + phase[3 * d + 1])
    return rho, u


def _output_gradients(rho, u):
    """Gradients of a loss by the final fields, as smooth as a fit to measured fields has them: the
    pressure pattern, its slopes and the velocity field."""
    slope = [10.0 * (torch.roll(rho, -1, -1 - i) - torch.roll(rho, 1, -1 - i)) for i in range(u.shape[0])]
    return rho - 1.0, u + torch.stack(slope)


def _force(case):
    return (0.0, 0.0, 1e-5) if case["flow"] == "sphere" else None


def _spin(grid):
    """Wall velocities: the sphere spins about the channel axis at 0.01 per lattice spacing, the side walls rest."""
    (xc, yc, _), _ = _sphere(grid)
    _, y, x = _axes(grid)
    body = torch.from_numpy(_walls("sphere", grid)[0]).cuda() == 2
    return torch.stack([-0.01 * (y - yc), 0.01 * (x - xc), torch.zeros_like(x)]) * body


def _sides(case):
    r = random.Random(case["layout"])
    sides = [r.randrange(case["low"], case["high"] + 1, 32) for _ in range(case["count"])]
    lids = [min(1.0 / 6.0, math.exp(r.uniform(math.log(100.0), math.log(3200.0))) / (6.0 * (n - 1))) for n in sides]
    return sides, lids


# ------------------------------------------------------------------ preparation and one pass

def _config(flow, grid, precision, lid=0.0, force=None):
    nt, ids, periodic = _walls(flow, grid)
    wall_u = None
    if ids:
        wall_u = np.zeros((ids, len(grid)))
        wall_u[1, 0] = lid
    return dict(lattice=M.D2Q9 if len(grid) == 2 else M.D3Q19, dims=tuple(reversed(grid)), dx=1.0, nu=1.0 / 6.0,
                precision=PRECISION[precision], periodic=periodic, node_type=nt, wall_u=wall_u, body_force=force)


def prepare(case, seed):
    if case["kind"] == "batch":
        return _prepare_batch(case, seed)
    grid = _grid(case)
    rho, u = _fields(case, seed, grid)
    dtype = torch.float64 if case["precision"] == "f64" else torch.float32
    if case["kind"] == "gradient":
        s = {"kind": "gradient", "rho": rho.to(dtype).requires_grad_(), "u": u.to(dtype).requires_grad_()}
        s["nu"] = torch.tensor(1.0 / 6.0, dtype=torch.float64, requires_grad=True)
        s["g_rho"], s["g_u"] = (g.to(dtype) for g in _output_gradients(rho, u))
        s["spec"] = adjoint.RolloutSpec(M.D3Q19, tuple(reversed(grid)), 1.0, case["steps"], 0b111,
                                        precision=PRECISION[case["precision"]])
        return s
    solver = M.Solver(**_config(case["flow"], grid, case["precision"], _lid(case) if case["re"] else 0.0,
                                _force(case)))
    s = {"kind": "run", "solver": solver, "steps": case["steps"], "monitor": case["monitor"], "rho": rho.to(dtype),
         "u": u.to(dtype), "spin": _spin(grid).to(dtype) if case["flow"] == "sphere" else None}
    s["ones"] = torch.ones_like(s["rho"]) if s["spin"] is not None else None
    if case["monitor"]:
        s["log"] = torch.zeros((case["steps"] // case["monitor"], 9), dtype=torch.float64, device="cuda")
    if case["precision"] in ("bf16", "f16"):
        s["raw"] = torch.empty(solver.state_bytes(), dtype=torch.uint8, device="cuda")
        s["storage"] = torch.bfloat16 if case["precision"] == "bf16" else torch.float16
    else:
        s["rho_out"], s["u_out"] = torch.empty_like(s["rho"]), torch.empty_like(s["u"])
    return s


def _prepare_batch(case, seed):
    sides, lids = _sides(case)
    batch = M.Batch([_config("cavity", (n, n), case["precision"], v) for n, v in zip(sides, lids)])
    batch.tune()
    gen = torch.Generator(device="cuda").manual_seed(seed)
    fields = [_fields({"flow": "cavity"}, seed + k, (n, n), gen) for k, n in enumerate(sides)]
    return {"kind": "batch", "batch": batch, "steps": case["steps"],
            "fields": [(r.float(), u.float()) for r, u in fields],
            "raw": [torch.empty(m.state_bytes(), dtype=torch.uint8, device="cuda") for m in batch.members],
            "shapes": [(3, n, n) for n in sides]}


def run(state):
    if state["kind"] == "batch":
        batch = state["batch"]
        for member, (rho, u) in zip(batch.members, state["fields"]):
            member.set_state(rho, u)
        batch.step(state["steps"])
        for member, raw in zip(batch.members, state["raw"]):
            member.get_lattice_state(raw)
        return [raw.view(torch.float32).view(shape) for raw, shape in zip(state["raw"], state["shapes"])]
    if state["kind"] == "gradient":
        rho_t, u_t = adjoint.rollout(state["rho"], state["u"], None, state["nu"], state["spec"])
        g = torch.autograd.grad((rho_t, u_t), (state["rho"], state["u"], state["nu"]), (state["g_rho"], state["g_u"]))
        return {"rho": rho_t.detach(), "u": u_t.detach(), "grad_rho": g[0], "grad_u": g[1], "grad_nu": g[2].float()}
    s = state["solver"]
    s.set_state(state["rho"], state["u"])
    if state["spin"] is not None:
        s.set_wall_state(state["ones"], state["spin"])
    if state["monitor"]:
        for k in range(state["log"].shape[0]):
            s.step(state["monitor"])
            M.maclab_diagnostics_device(s.handle, state["log"][k])
        s.step(state["steps"] - state["monitor"] * state["log"].shape[0])
    else:
        s.step(state["steps"])
    if "raw" in state:
        s.get_lattice_state(state["raw"])
        return {"state": state["raw"].view(state["storage"])}
    s.get_state_into(state["rho_out"], state["u_out"])
    out = {"rho": state["rho_out"], "u": state["u_out"]}
    if state["monitor"]:
        out["log"] = state["log"].float()  # logged in 32 bits
    return out


def work(case):
    """Bytes: the fields in and out, once.  Operations: those of the update with each node's terms
    formed once (about 80 for nine directions, 200 for nineteen), the reverse step counted as two more."""
    if case["kind"] == "batch":
        nodes = sum(n * n for n in _sides(case)[0])
        return {"bytes": 2.0 * 12 * nodes, "flops": 80.0 * nodes * case["steps"]}
    nodes = case["nx"] * case["ny"] * case["nz"]
    d = 2 if case["nz"] == 1 else 3
    flops = (80.0 if d == 2 else 200.0) * nodes * case["steps"]
    if case["kind"] == "gradient":
        return {"bytes": 4.0 * 4 * (d + 1) * nodes, "flops": 3.0 * flops}
    inp = 8 if case["precision"] == "f64" else 4
    out = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}[case["precision"]]
    return {"bytes": float((inp + out) * (d + 1) * nodes), "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits

_VELOCITIES = {
    2: [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)],
    3: [(x, y, z) for x in (0, 1, -1) for y in (0, 1, -1) for z in (0, 1, -1) if abs(x) + abs(y) + abs(z) <= 2],
}


def _weight(c):
    n = sum(abs(v) for v in c)
    return (16, 4, 1)[n] / 36.0 if len(c) == 2 else (12, 2, 1)[n] / 36.0


def _exact_step(rho, u, wall=None, force=None):
    """One step in lattice units; u is a list of components, the grid the last len(u) axes."""
    d = len(u)
    axes = [-1 - i for i in range(d)]  # x, y, z
    half = 1.0 - 1.5 * sum(v * v for v in u)
    new, mom = 0.0, [0.0] * d
    for c in _VELOCITIES[d]:
        cu = sum(k * v for k, v in zip(c, u) if k)
        f = rho * (half + 3.0 * cu + 4.5 * cu * cu) * _weight(c) if any(c) else rho * half * _weight(c)
        moved = [(k, a) for k, a in zip(c, axes) if k]
        if moved:
            f = torch.roll(f, [k for k, _ in moved], [a for _, a in moved])
        new = new + f
        for i in range(d):
            if c[i]:
                mom[i] = mom[i] + c[i] * f
    vel = [m / new for m in mom]
    if force is not None:
        vel = [v + f if f else v for v, f in zip(vel, force)]
    if wall is not None:
        new = torch.where(wall, rho, new)
        vel = [torch.where(wall, v, w) for v, w in zip(u, vel)]
    return new, vel


def _storage(x):
    """Raw state order of the last axis: the two halves interleaved where its size is a multiple of 4."""
    n = x.shape[-1]
    return x if n % 4 else x.reshape(x.shape[:-1] + (2, n // 2)).transpose(-1, -2).reshape(x.shape)


def _with_walls(rho, u, nt, lid):
    wall = nt != 0
    rho = torch.where(wall, torch.ones_like(rho), rho)
    u = [torch.where(wall, torch.zeros_like(v), v) for v in u]
    u[0] = torch.where(nt == 2, torch.full_like(u[0], lid), u[0])
    return rho, u, wall


def exact(case, seed):
    if case["kind"] == "batch":
        return _exact_batch(case, seed)
    grid = _grid(case)
    d = len(grid)
    rho, u = _fields(case, seed, grid)
    dtype = torch.float64 if case["precision"] == "f64" else torch.float32
    gradients = [g.to(dtype).double() for g in _output_gradients(rho, u)] if case["kind"] == "gradient" else None
    rho, u = rho.to(dtype).double(), u.to(dtype).double()
    if gradients:
        return _exact_gradient(*gradients, case, rho, u)
    if case["nx"] * case["ny"] * case["nz"] * case["steps"] > 1.5e9:
        return None
    nt, _, _ = _walls(case["flow"], grid)
    u, wall = list(u), None
    if nt is not None:
        nt = torch.from_numpy(nt).cuda()
        rho, u, wall = _with_walls(rho, u, nt, _lid(case) if case["re"] else 0.0)
        if case["flow"] == "sphere":
            u = [torch.where(wall, w, v) for v, w in zip(u, _spin(grid).to(dtype).double())]
    log = []
    for k in range(case["steps"]):
        last = u
        rho, u = _exact_step(rho, u, wall, _force(case))
        if case["monitor"] and (k + 1) % case["monitor"] == 0:
            fluid = torch.ones_like(rho) if wall is None else (~wall).double()
            uu = sum(v * v for v in u) * fluid
            sums = [((rho - 1.0) * fluid).sum(), (rho * uu).sum()] + [(rho * v * fluid).sum() for v in u]
            sums += [rho.new_zeros(())] * (3 - d)
            sums += [sum(((a - b) * fluid).square().sum() for a, b in zip(u, last)), uu.sum(), uu.max().sqrt(),
                     rho.new_zeros(())]
            log.append(torch.stack(sums))
    if case["precision"] in ("bf16", "f16"):
        return {"state": torch.stack([_storage(x) for x in [rho - 1.0] + u]).reshape(-1)}
    out = {"rho": rho, "u": torch.stack(u)}
    if case["monitor"]:
        out["log"] = torch.stack(log)
    return out


def _exact_batch(case, seed):
    sides, lids = _sides(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    fields = [_fields({"flow": "cavity"}, seed + k, (n, n), gen) for k, n in enumerate(sides)]
    out = [None] * len(sides)
    for n in sorted(set(sides)):  # equal sides together
        members = [k for k, m in enumerate(sides) if m == n]
        nt = torch.from_numpy(_walls("cavity", (n, n))[0]).cuda()
        start = [_with_walls(fields[k][0].float().double(), list(fields[k][1].float().double()), nt, lids[k])
                 for k in members]
        rho, wall = torch.stack([s[0] for s in start]), start[0][2]
        u = [torch.stack([s[1][i] for s in start]) for i in range(2)]
        for _ in range(case["steps"]):
            rho, u = _exact_step(rho, u, wall)
        for i, k in enumerate(members):
            out[k] = torch.stack([_storage(rho[i] - 1.0), _storage(u[0][i]), _storage(u[1][i])])
    return out


def _exact_gradient(g_rho, g_u, case, rho0, u0):
    rho0, u0 = rho0.requires_grad_(), u0.requires_grad_()
    nu = torch.tensor(1.0 / 6.0, dtype=torch.float64, device="cuda", requires_grad=True)
    e = 6.0 * nu
    state = (rho0,) + tuple(v / e for v in u0)

    def step(*s):
        r, v = _exact_step(s[0], list(s[1:]))
        return (r,) + tuple(v)

    for _ in range(case["steps"]):
        state = checkpoint(step, *state, use_reentrant=False)
    rho_t, u_t = state[0], e * torch.stack(state[1:])
    g = torch.autograd.grad((rho_t, u_t), (rho0, u0, nu), (g_rho, g_u))
    return {"rho": rho_t.detach(), "u": u_t.detach(), "grad_rho": g[0], "grad_u": g[1], "grad_nu": g[2]}
