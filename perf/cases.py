"""The work a user of the library has it do, as cases that can be timed.

A case is one pass through the public entry points: a run of time steps from
a state the program holds (`steps`), the same with conservation sums and the
steady-state residual read between the runs (`steady`), the start of a run
from macroscopic fields (`start`), an ensemble of uneven grids stepped
together (`batch`), and a training step, i.e. K steps forward and the
gradients of a loss back (`adjoint`).  The flows are those of workloads.py.

`exact` repeats a pass in FP64 with plain torch operations: the step as the
paper writes it (dense products with M and its inverse), none of the
library's kernels.
"""
import functools
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1106_0785_gb300 import autograd, mrtlb, workloads
from paper_1106_0785_gb300.mrtlb import Config
from paper_1106_0785_gb300.simulation import Batch, Simulation

# flops of one node update (a fused multiply-add counts two), as the test
# suite counts them from the step's templates
FLOPS = {"fp32": 539, "fp64": 521}


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the Sod tube of the configurations in its default precision: a thin
        # strip, where launches and latency are all there is
        {"name": "sod_400x4_fp64", "path": "steps", "flow": "sod", "nx": 400, "ny": 4, "precision": "fp64",
         "version": 1, "steps": 200},
        # the thermal Couette channel: the smallest grid, with walls refilled
        # before every step
        {"name": "couette_4x200_fp32", "path": "steps", "flow": "couette", "nx": 4, "ny": 200,
         "precision": "fp32", "version": 1, "steps": 200},
        # the same channel on its way to the steady state: sums and residual
        # read every 50 steps, as a run that stops at a residual does
        {"name": "couette_4x200_fp64_steady", "path": "steady", "flow": "couette", "nx": 4, "ny": 200,
         "precision": "fp64", "version": 1, "steps": 50, "reads": 4},
        # the paper's shock-bubble channel: an ordinary grid that stays in the
        # caches; inflow, outflow and reflecting sides
        {"name": "bubble_600x100_fp32", "path": "steps", "flow": "bubble", "nx": 600, "ny": 100,
         "precision": "fp32", "version": 1, "steps": 128},
        # Richtmyer-Meshkov at a quarter of its resolution in FP64
        {"name": "rm_1024x256_fp64", "path": "steps", "flow": "rm", "nx": 1024, "ny": 256,
         "precision": "fp64", "version": 1, "steps": 16},
        # an odd periodic grid under the equilibrium version with exponentials
        {"name": "waves_1501x701_fp32_v3", "path": "steps", "flow": "waves", "nx": 1501, "ny": 701,
         "precision": "fp32", "version": 3, "steps": 24},
        # the Richtmyer-Meshkov run of the benchmark, the largest single grid
        {"name": "rm_4096x1024_fp32", "path": "steps", "flow": "rm", "nx": 4096, "ny": 1024,
         "precision": "fp32", "version": 1, "steps": 64},
        # what a run does before its first step on that grid: the state from
        # the fields, its conserved totals, the distributions for a restart file
        {"name": "start_4096x1024_fp32", "path": "start", "flow": "rm", "nx": 4096, "ny": 1024,
         "precision": "fp32", "version": 1},
        # the ensemble of 64 uneven tubes and channels (10.3 million nodes)
        {"name": "batch_64_fp32", "path": "batch", "count": 64, "first": 0, "nx_max": 2048, "ny_max": 256,
         "precision": "fp32", "steps": 64},
        # gradients of the Couette temperature misfit: the smallest training step
        {"name": "couette_adjoint_4x200_fp64", "path": "adjoint", "flow": "couette", "nx": 4, "ny": 200,
         "precision": "fp64", "version": 1, "steps": 71},
        # a training step on the grid the configurations train on
        {"name": "rm_adjoint_512x128_fp32", "path": "adjoint", "flow": "rm", "nx": 512, "ny": 128,
         "precision": "fp32", "version": 1, "steps": 64},
        # the benchmark's forward + adjoint run
        {"name": "rm_adjoint_4096x1024_fp32", "path": "adjoint", "flow": "rm", "nx": 4096, "ny": 1024,
         "precision": "fp32", "version": 1, "steps": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_grid(rng, flow, most):
    """Sizes of a flow, most nodes at the utmost."""
    for _ in range(1000):
        if flow == "sod":
            nx, ny = _log_int(rng, 128, 4096), _log_int(rng, 3, 256)
        elif flow == "couette":
            nx, ny = _log_int(rng, 4, 2048), _log_int(rng, 20, 400)
        elif flow == "slip":
            nx, ny = _log_int(rng, 40, 1000), _log_int(rng, 3, 300)
        elif flow == "bubble":
            nx, ny = _log_int(rng, 560, 2400), _log_int(rng, 60, 500)
        elif flow == "rm":
            nx, ny = _log_int(rng, 200, 4096), _log_int(rng, 50, 1024)
        else:
            nx, ny = _log_int(rng, 24, 3000), _log_int(rng, 24, 1400)
        if nx * ny <= most:
            return nx, ny
    return 200, 50


def draw(rng):
    path = rng.choice(["steps"] * 6 + ["steady", "start", "batch", "adjoint", "adjoint"])
    precision = rng.choice(["fp32", "fp32", "fp32", "fp64"])
    if path == "batch":
        n = _log_int(rng, 4, 48)
        case = {"path": path, "count": n, "first": rng.randrange(10000), "precision": precision,
                "nx_max": rng.randint(256, 2048 if precision == "fp32" else 600),
                "ny_max": rng.randint(8, 256 if precision == "fp32" else 48)}
        # an even count of steps: the state is set again in the same buffer
        case["steps"] = 2 * rng.randint(4, 16) if precision == "fp32" else 2 * rng.randint(2, 4)
        return case
    flows = ["sod", "couette", "slip", "bubble", "rm", "rm", "waves", "waves"]
    flow = rng.choice(flows if path == "steps" else ["couette", "slip", "sod"] if path == "steady" else ["rm", "bubble", "waves"]
                      if path == "start" else ["couette", "rm", "waves"])
    version = rng.choice([1, 1, 1, 1, 2, 3])
    most = {"fp32": 4096 * 1024, "fp64": 512 * 512}[precision]
    if path == "steady":
        precision, most = "fp64", 64 * 1024
    if path == "adjoint":
        most = {"fp32": 2048 * 512, "fp64": 128 * 128}[precision]
    nx, ny = _draw_grid(rng, flow, most)
    case = {"path": path, "flow": flow, "nx": nx, "ny": ny, "precision": precision, "version": version}
    if path == "start":
        return case
    updates = {"fp32": 64 * 4096 * 1024, "fp64": 4 * 1024 * 1024}[precision]  # node updates a pass may take
    if path == "steady":
        case["reads"] = rng.randint(2, 4)
        case["steps"] = max(1, min(_log_int(rng, 10, 70), updates // (nx * ny * case["reads"])))
    elif path == "adjoint":
        case["steps"] = max(2, min(_log_int(rng, 8, 100), updates // (4 * nx * ny)))
    else:
        case["steps"] = max(2, min(_log_int(rng, 8, 250), updates // (nx * ny)))
    return case


def work(case):
    """Every step reads its state once and writes the next one once (16 values
    a node); an adjoint step reads the state and the adjoint and writes the
    adjoint."""
    size = 4 if case["precision"] == "fp32" else 8
    flops = FLOPS[case["precision"]]
    if case["path"] == "batch":
        nodes = sum(cfg.nx * cfg.ny for cfg in _batch_configs(case))
    else:
        nodes = case["nx"] * case["ny"]
    if case["path"] == "start":
        # four FP64 fields in, the state out, read for the sums and once more
        # for the dense copy (the previous temperatures are written too)
        return {"bytes": nodes * (32 + 8 + 16 * size * 4), "flops": nodes * 300}
    steps = case["steps"] * case.get("reads", 1)
    if case["path"] == "adjoint":
        return {"bytes": nodes * steps * 16 * size * 5, "flops": nodes * steps * 3 * flops}
    return {"bytes": nodes * steps * 16 * size * 2, "flops": nodes * steps * flops}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _smooth(shape, rng, modes=3):
    """A low-mode random field of size about one on the GPU."""
    ny, nx = shape
    x = torch.arange(nx, dtype=torch.float64, device="cuda") / nx
    y = torch.arange(ny, dtype=torch.float64, device="cuda") / ny
    out = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for _ in range(modes):
        kx, ky = (int(k) for k in rng.integers(0, 3, size=2))
        out += rng.uniform(-1, 1) * torch.cos(2 * math.pi * (kx * x[None, :] + ky * y[:, None]) + rng.uniform(0, 2 * math.pi))
    return out / modes


def _flow(case, rng):
    """Configuration and initial fields of a single-grid case.  The seed picks
    the states of the flow and a smooth 1% disturbance of density and
    temperature."""
    flow, nx, ny, prec = case["flow"], case["nx"], case["ny"], case["precision"]
    if flow == "sod":
        cfg, fields = workloads.sod(nx=nx, ny=ny, precision=prec, right=(0.125, rng.uniform(0.5, 0.9)))
    elif flow == "couette":
        cfg, fields = workloads.couette(Pr=rng.uniform(0.5, 2.0), nx=nx, ny=ny, precision=prec, U=rng.uniform(0.4, 0.8))
    elif flow == "slip":
        cfg, fields = workloads.slip_couette(nx=nx, ny=ny, precision=prec, U=rng.uniform(0.1, 0.2))
    elif flow == "bubble":
        cfg, fields = workloads.shock_bubble(nx=nx, ny=ny, precision=prec, radius=rng.uniform(15.0, 30.0))
    elif flow == "rm":
        cfg, fields = workloads.richtmyer_meshkov(nx=nx, ny=ny, precision=prec, amplitudes=rng.uniform(0, 0.02, 3))
    else:
        d = 1.0 / max(nx, ny)
        cfg = Config(nx=nx, ny=ny, dx=d, dy=d, dt=5e-6, s=workloads.rates(1e4, 1.5e4, 1e5), precision=prec)
        fields = (np.ones((ny, nx)), np.zeros((ny, nx)), np.zeros((ny, nx)), np.ones((ny, nx)))
    cfg.eq_version = case["version"]
    rho, ux, uy, T = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in fields)
    rho = rho * (1.0 + 0.01 * _smooth((ny, nx), rng))
    T = T * (1.0 + 0.01 * _smooth((ny, nx), rng))
    if flow == "waves":
        rho = rho * (1.0 + 0.1 * _smooth((ny, nx), rng))
        ux, uy = 0.3 * _smooth((ny, nx), rng), 0.3 * _smooth((ny, nx), rng)
        T = T * (1.0 + 0.1 * _smooth((ny, nx), rng))
    return cfg, (rho, ux, uy, T)


@functools.lru_cache(maxsize=4)
def _batch_instances(count, first, nx_max, ny_max, precision):
    """`count` instances of the ensemble's recipe (even: Sod-type tubes, odd:
    Couette channels), number `first` onwards."""
    first -= first % 2
    out = []
    for i in range(first, first + count):
        rng = np.random.default_rng(seed=i)
        nx, ny = int(rng.integers(128, nx_max + 1)), int(rng.integers(4, ny_max + 1))
        Pr = float(rng.uniform(0.3, 3.0))
        if i % 2 == 0:
            ratio = float(rng.uniform(2.0, 20.0))
            out.append(workloads.sod(nx=nx, ny=ny, precision=precision, right=(0.125, 8.0 / ratio), s_cond=Pr * 1.5e4))
        else:
            out.append(workloads.couette(Pr=Pr, nx=nx, ny=ny, precision=precision, U=float(rng.uniform(0.1, 0.8))))
    return out


def _batch_configs(case):
    return [cfg for cfg, _ in _batch_instances(case["count"], case["first"], case["nx_max"], case["ny_max"], case["precision"])]


def _batch_inputs(case, seed):
    """(configuration, dense state) of every instance."""
    rng = np.random.default_rng(seed)
    out = []
    for cfg, fields in _batch_instances(case["count"], case["first"], case["nx_max"], case["ny_max"], case["precision"]):
        rho, ux, uy, T = (torch.from_numpy(a).cuda() for a in fields)
        rho = rho * (1.0 + 0.01 * _smooth(rho.shape, rng))
        out.append((cfg, _equilibrium(rho, ux, uy, T, cfg.eq_version).to(_dtype(cfg))))
    return out


def _dtype(cfg):
    return torch.float32 if cfg.precision == "fp32" else torch.float64


def _adjoint_inputs(case, seed):
    """(configuration, fields, rates, target) of a training step: the fields
    (rho, ux, uy, T) as one parameter [4][ny][nx] and the rates, both in the
    precision of the run."""
    cfg, fields = _flow(case, np.random.default_rng(seed))
    fields = torch.stack(fields).to(_dtype(cfg))
    rates = torch.tensor(cfg.s, dtype=_dtype(cfg))
    y = torch.arange(cfg.ny, dtype=torch.float64, device="cuda") / max(1, cfg.ny - 1)
    target = (1.0 + 0.07 * y * (1.0 - y))[:, None].expand(cfg.ny, cfg.nx)
    return cfg, fields, rates, target


def _loss(case, cfg, T, target):
    """The misfit of the temperature to a profile, for the Richtmyer-Meshkov
    flow its integral (the benchmark's loss)."""
    if case["flow"] == "rm":
        return T.sum() * cfg.dx * cfg.dy
    return ((T - target) ** 2).sum() * cfg.dx * cfg.dy


def prepare(case, seed):
    path = case["path"]
    if path == "batch":
        inputs = _batch_inputs(case, seed)
        sims = [Simulation(cfg) for cfg, _ in inputs]
        states = [f for _, f in inputs]
        for sim, f in zip(sims, states):
            sim.set_f(f)
        batch = Batch(sims)
        batch.tune()
        return {"case": case, "sims": sims, "states": states, "batch": batch}
    if path == "adjoint":
        cfg, fields, rates, target = _adjoint_inputs(case, seed)
        return {"case": case, "cfg": cfg, "sim": Simulation(cfg), "fields": fields, "rates": rates, "target": target}
    cfg, fields = _flow(case, np.random.default_rng(seed))
    state = {"case": case, "cfg": cfg, "sim": Simulation(cfg)}
    if path == "start":
        state["fields"] = fields
    else:
        state["f"] = _equilibrium(*fields, cfg.eq_version).to(_dtype(cfg))
    return state


# ---------------------------------------------------------------------------
# A pass
# ---------------------------------------------------------------------------
def run(state):
    case = state["case"]
    path = case["path"]
    if path == "batch":
        for sim, f in zip(state["sims"], state["states"]):
            sim.set_f(f)
        state["batch"].step(case["steps"])
        sizes = [f.numel() for f in state["states"]]
        out = torch.empty(sum(sizes), dtype=state["states"][0].dtype, device="cuda")
        for sim, part in zip(state["sims"], out.split(sizes)):
            mrtlb.mrtlb_get_f(sim.ctx, part, True)
        return out
    sim = state["sim"]
    if path == "steps":
        sim.set_f(state["f"])
        sim.step(case["steps"])
        return sim.get_f(on_device=True)
    if path == "steady":
        sim.set_f(state["f"])
        reads = []
        for _ in range(case["reads"]):
            sim.step(case["steps"])
            reads.append(sim.reduce())
        return {"f": sim.get_f(on_device=True), "reads": reads}
    if path == "start":
        sim.init_equilibrium(*state["fields"])
        return {"sums": sim.reduce(), "f": sim.get_f(on_device=True)}
    fields, rates = state["fields"].requires_grad_(), state["rates"].requires_grad_()
    T = autograd.run(sim, *fields, rates, case["steps"])[3]
    loss = _loss(case, state["cfg"], T, state["target"])
    g_fields, g_rates = torch.autograd.grad(loss, [fields, rates])
    return {"loss": loss.detach().to(rates.dtype), "fields": g_fields, "rates": g_rates}


# ---------------------------------------------------------------------------
# The same pass in FP64 with torch
# ---------------------------------------------------------------------------
_V = [(c * a, c * b) for c, ring in ((1, ((1, 0), (0, 1), (-1, 0), (0, -1))), (1, ((1, 1), (-1, 1), (-1, -1), (1, -1))),
                                     (2, ((1, 0), (0, 1), (-1, 0), (0, -1))), (2, ((1, 1), (-1, 1), (-1, -1), (1, -1))))
      for a, b in ring]


@functools.lru_cache(maxsize=None)
def _matrices():
    """M (its rows are polynomials of the velocities) and its inverse."""
    rows = []
    for x, y in _V:
        v2, m9, m10 = x * x + y * y, x ** 3 - 3 * x * y * y, 3 * x * x * y - y ** 3
        rows.append([1, x, y, v2 / 2, x * x - y * y, x * y, v2 * x / 2, v2 * y / 2, m9, m10, v2 * v2 / 4,
                     x ** 4 - 6 * x * x * y * y + y ** 4, v2 * (x * x - y * y), v2 * x * y, v2 * m9, v2 * m10])
    M = np.array(rows, dtype=np.float64).T
    return torch.from_numpy(M.copy()).cuda(), torch.from_numpy(np.linalg.inv(M)).cuda()


def _times(A, f):
    return (A @ f.reshape(f.shape[0], -1)).reshape(A.shape[0], *f.shape[1:])


def _primitive(m):
    rho, jx, jy, e = m[0], m[1], m[2], m[3]
    ux, uy = jx / rho, jy / rho
    return rho, ux, uy, e / rho - 0.5 * (ux * ux + uy * uy)


def _equilibrium_moments(rho, ux, uy, T, version):
    e, x2, y2 = rho * (T + 0.5 * (ux * ux + uy * uy)), ux * ux, uy * uy
    u2, w, zero = x2 + y2, 6 * e - 2 * rho * (x2 + y2), torch.zeros_like(rho)
    m = [rho, rho * ux, rho * uy, e, rho * (x2 - y2), rho * ux * uy, (e + rho * T) * ux, (e + rho * T) * uy,
         rho * ux * (x2 - 3 * y2), rho * uy * (3 * x2 - y2), 2 * e * e / rho - 0.25 * rho * u2 * u2, zero,
         w * (x2 - y2), w * ux * uy, zero, zero]
    if version == 2:
        m[14] = rho * ux * (-4 + 10 * T + 5 * x2 - 5 * y2)
        m[15] = rho * uy * (4 - 10 * T + 5 * x2 - 5 * y2)
    elif version == 3:
        g = torch.stack([rho / (2 * math.pi * T) * torch.exp(-((x - ux) ** 2 + (y - uy) ** 2) / (2 * T)) for x, y in _V])
        m[11], m[14], m[15] = _times(_matrices()[0][[11, 14, 15]], g)
    return torch.stack(m)


def _equilibrium(rho, ux, uy, T, version):
    return _times(_matrices()[1], _equilibrium_moments(rho, ux, uy, T, version))


def _side_state(side, like):
    one = torch.ones_like(like)
    return (side[4] if len(side) > 4 else 1.0) * one, side[1] * one, side[2] * one, side[3] * one


def _wall(fluid, side, version):
    """The wall layer from the fluid layer beside it (non-equilibrium extrapolation)."""
    rho, ux, uy, T = _primitive(_times(_matrices()[0], fluid))
    _, wx, wy, wT = _side_state(side, rho)
    return _equilibrium(rho, wx, wy, wT, version) + fluid - _equilibrium(rho, ux, uy, T, version)


def _walls(f, cfg):
    kinds = [s[0] for s in cfg.bc]
    if kinds[2] == "wall":
        f = torch.cat([_wall(f[:, 1:2], cfg.bc[2], cfg.eq_version), f[:, 1:]], 1)
    if kinds[3] == "wall":
        f = torch.cat([f[:, :-1], _wall(f[:, -2:-1], cfg.bc[3], cfg.eq_version)], 1)
    return f


def _ghost(edge, side, axis, sign, cfg):
    """The ghost layer beside the edge layer `edge` of a side that is not periodic."""
    kind = side[0]
    if kind == "reflect":
        flip = [(-x, y) if axis == 0 else (x, -y) for x, y in _V]
        return edge[[_V.index(v) for v in flip]]
    if kind == "inflow":
        return _equilibrium(*_side_state(side, edge[0]), cfg.eq_version)
    if kind == "diffuse":
        d = cfg.dx if axis == 0 else cfg.dy
        v = torch.tensor([c[axis] for c in _V], dtype=torch.float64, device=edge.device)
        a, b = v * cfg.dt / (2 * d), 0.5 * (v * cfg.dt / d) ** 2
        ghost_w, edge_w = (b + a, b - a) if sign < 0 else (b - a, b + a)  # weights of the ghost here, of the edge there
        enters = (-sign * v > 0).double()[:, None, None]
        _, wx, wy, wT = _side_state(side, edge[0])
        e = _equilibrium(torch.ones_like(wx), wx, wy, wT, cfg.eq_version)
        num = (edge_w[:, None, None] * edge).sum(0) - (ghost_w[:, None, None] * (1 - enters) * edge).sum(0)
        den = (ghost_w[:, None, None] * enters * e).sum(0)
        return enters * (num / den) * e + (1 - enters) * edge
    return edge


def _step(f, s, cfg):
    """One time step of the state f [16][ny][nx] with the rates s."""
    M, Minv = _matrices()
    f = _walls(f, cfg)
    if cfg.bc[0][0] == "periodic":
        W, E = f[:, :, -1:], f[:, :, :1]
    else:
        W, E = _ghost(f[:, :, :1], cfg.bc[0], 0, -1, cfg), _ghost(f[:, :, -1:], cfg.bc[1], 0, 1, cfg)
    if cfg.bc[2][0] == "periodic":
        S, N = f[:, -1:], f[:, :1]
    else:
        S, N = _ghost(f[:, :1], cfg.bc[2], 1, -1, cfg), _ghost(f[:, -1:], cfg.bc[3], 1, 1, cfg)
    fx, fy = torch.cat([W, f, E], 2), torch.cat([S, f, N], 1)
    m = _times(M, f)
    rho, ux, uy, T = _primitive(m)
    _, gx_ux, gx_uy, _ = _primitive(_times(M[:4], fx))
    _, gy_ux, gy_uy, _ = _primitive(_times(M[:4], fy))
    c = s[:, None, None] * (m - _equilibrium_moments(rho, ux, uy, T, cfg.eq_version))
    if cfg.modified:
        dx2, dy2 = 2 * cfg.dx, 2 * cfg.dy
        shear = (gx_ux[:, 2:] - gx_ux[:, :-2]) / dx2 - (gy_uy[2:] - gy_uy[:-2]) / dy2
        strain = (gx_uy[:, 2:] - gx_uy[:, :-2]) / dx2 + (gy_ux[2:] - gy_ux[:-2]) / dy2
        p = rho * T
        c6 = (s[6] / s[4] - 1) * p * ux * shear + (s[6] / s[5] - 1) * p * uy * strain
        c7 = (s[7] / s[5] - 1) * p * ux * strain + (s[7] / s[4] - 1) * p * uy * shear
        zero = torch.zeros_like(p)
        c = c + torch.stack([zero] * 6 + [c6, c7] + [zero] * 8)
    v = torch.tensor(_V, dtype=torch.float64, device=f.device)
    ax, ay = v[:, 0, None, None] * cfg.dt / cfg.dx, v[:, 1, None, None] * cfg.dt / cfg.dy
    new = f - cfg.dt * _times(Minv, c)
    new = new - 0.5 * ax * (fx[:, :, 2:] - fx[:, :, :-2]) + 0.5 * ax * ax * (fx[:, :, 2:] - 2 * f + fx[:, :, :-2])
    new = new - 0.5 * ay * (fy[:, 2:] - fy[:, :-2]) + 0.5 * ay * ay * (fy[:, 2:] - 2 * f + fy[:, :-2])
    return _walls(new, cfg)


def _rates(cfg):
    s = torch.tensor(cfg.s, dtype=torch.float64, device="cuda")
    return torch.cat([torch.zeros(4, dtype=torch.float64, device="cuda"), s[4:]])


def _run(f, s, cfg, steps):
    for _ in range(steps):
        f = _step(f, s, cfg)
    return f


def _sums(f, before):
    """Totals of the conserved moments and the largest change of T."""
    m = _times(_matrices()[0], f)
    T = _primitive(m)[3]
    change = (T - before).abs().max() if before is not None else torch.zeros((), dtype=torch.float64, device="cuda")
    return torch.cat([m[:4].sum((1, 2)), change[None]]), T


def exact(case, seed):
    path = case["path"]
    if path == "adjoint":
        cfg, fields, rates, target = _adjoint_inputs(case, seed)
        fields, rates = fields.double().requires_grad_(), rates.double().requires_grad_()
        s = torch.cat([torch.zeros(4, dtype=torch.float64), rates[4:]]).cuda()
        f = _walls(_equilibrium(*fields, cfg.eq_version), cfg)
        for _ in range(case["steps"]):
            f = checkpoint(_step, f, s, cfg, use_reentrant=False)
        loss = _loss(case, cfg, _primitive(_times(_matrices()[0], f))[3], target)
        g_fields, g_rates = torch.autograd.grad(loss, [fields, rates])
        return {"loss": loss.detach(), "fields": g_fields, "rates": g_rates}
    with torch.no_grad():
        if path == "batch":
            done = []
            for cfg, f in _batch_inputs(case, seed):
                done.append(_run(_walls(f.double(), cfg), _rates(cfg), cfg, case["steps"]).reshape(-1))
            return torch.cat(done)
        cfg, fields = _flow(case, np.random.default_rng(seed))
        f = _equilibrium(*fields, cfg.eq_version)
        if path == "start":
            f = _walls(f, cfg)
            # the totals are those of the state in the precision it is kept in
            return {"sums": _sums(f.to(_dtype(cfg)).double(), None)[0], "f": f}
        f = _walls(f.to(_dtype(cfg)).double(), cfg)
        if path == "steps":
            return _run(f, _rates(cfg), cfg, case["steps"])
        reads, T = [], None
        for _ in range(case["reads"]):
            f = _run(f, _rates(cfg), cfg, case["steps"])
            r, T = _sums(f, T)
            reads.append(r)
        return {"f": f, "reads": reads}
