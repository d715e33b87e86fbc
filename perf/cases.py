"""The work that users of this framework have it do, as cases that can be timed and compared.

Every kind of case goes through the framework's public entry points (solver.Hierarchy and its
steppers, captured coarse steps, regridding, host-resident steps, adjoint.rollout) after the
autotuner chose the tilings, as bench.py and measure.py run them:

  grid      one level, uniform medium: one step of the one-launch stepper
  medium    one level, cell-wise density and bulk modulus: one step of the one-launch stepper
  swe       one level, shallow water (Roe solvers): one step of the one-launch stepper
  amr       a hierarchy, uniform medium: two coarse steps as one captured graph
  swe_amr   the same for shallow water
  batch     many two-level runs with their own media: two coarse steps as one captured graph
  regrid    two coarse steps with eager launches, then the fine levels rebuilt from the flags
  host      the state in pinned host memory: steps that copy it in and out
  gradient  a rollout in a cell-wise medium and its reverse sweep

Initial states: ring pulses (the workload of the paper's Sec. 4.1) with seeded centre, radius and
height over a smooth seeded field, at rest or moving.  Domains are closed by walls, so that a
state that is stepped on stays a state with waves in it.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1808_02638_gb300 import inputs, tune
from paper_1808_02638_gb300.adjoint import rollout
from paper_1808_02638_gb300.solver import Hierarchy

MINMOD, SUPERBEE, VANLEER, MC = 1, 2, 3, 4
EXTRAP, PERIODIC, WALL = 0, 1, 2
RHO0, K0, GRAV, CFL = 1.0, 4.0, 1.0, 0.9
DEV = "cuda"


def listed():
    return [
        # the smallest call: a 100 x 100 grid in one box, where the launch and one tile's latency count
        {"name": "grid_100", "kind": "grid", "nx": 100, "ny": 100, "patch": 0, "limiter": MC},
        # the benchmark's workload: 2048 x 2048 as 4096 patches of 32 x 32
        {"name": "grid_2048", "kind": "grid", "nx": 2048, "ny": 2048, "patch": 32, "limiter": MC},
        # an ordinary grid whose patches do not divide it, with the paper's limiter
        {"name": "grid_ragged", "kind": "grid", "nx": 1001, "ny": 604, "patch": 64, "limiter": VANLEER},
        # 3-level AMR, ratio 4 twice, 64 x 64 base: many substeps of small levels
        {"name": "amr_3level", "kind": "amr", "base": 64, "ratio": 4, "nlev": 3, "limiter": MC, "reflux": False},
        # the paper's settings: ratio 2, van Leer, the conservation fix at the level interfaces
        {"name": "amr_fix", "kind": "amr", "base": 128, "ratio": 2, "nlev": 3, "limiter": VANLEER, "reflux": True},
        # the paper's run loop on a small base: coarse steps and a regrid
        {"name": "regrid_cycle", "kind": "regrid", "base": 240, "limiter": VANLEER},
        # heterogeneous medium, one grid (the inversion workload's forward step)
        {"name": "medium_256", "kind": "medium", "nx": 256, "ny": 256, "limiter": MC},
        # a batch of independent heterogeneous two-level runs in one launch per level-step
        {"name": "batch_16", "kind": "batch", "runs": 16, "first": 4000, "limiter": MC},
        # its gradient: forward rollout with checkpoints and the reverse sweep
        {"name": "gradient_256", "kind": "gradient", "nx": 256, "ny": 256, "steps": 20, "every": 10, "limiter": MC},
        # the second system at the benchmark's size, and through the AMR path
        {"name": "swe_2048", "kind": "swe", "nx": 2048, "ny": 2048, "patch": 32, "limiter": MC},
        {"name": "swe_amr", "kind": "swe_amr", "base": 64, "ratio": 4, "nlev": 3, "limiter": MC, "reflux": False},
        # the state kept in host memory
        {"name": "host_1024", "kind": "host", "nx": 1024, "ny": 1024, "patch": 32, "steps": 4, "limiter": MC},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid", "grid", "amr", "regrid", "medium", "batch", "gradient", "swe", "swe_amr", "host"])
    lim = rng.choice([MC, MC, VANLEER, MINMOD, SUPERBEE])
    if kind in ("grid", "swe"):
        patch = rng.choice([0, 0, 24, 32, 50, 64])
        return {"kind": kind, "nx": _log(rng, 40, 2048), "ny": _log(rng, 40, 2048), "patch": patch, "limiter": lim}
    if kind == "medium":
        return {"kind": kind, "nx": _log(rng, 40, 512), "ny": _log(rng, 40, 512), "limiter": lim}
    if kind == "gradient":
        n = _log(rng, 40, 256)
        return {"kind": kind, "nx": n, "ny": n + rng.randrange(-9, 1), "steps": rng.randrange(4, 21),
                "every": rng.choice([4, 7, 10]), "limiter": lim}
    if kind in ("amr", "swe_amr"):
        ratio, nlev = rng.choice([(4, 3), (4, 2), (2, 3), (2, 2)])
        base = 4 * rng.randrange(8, 17 if ratio == 4 and nlev == 3 else 33)
        return {"kind": kind, "base": base, "ratio": ratio, "nlev": nlev, "limiter": lim,
                "reflux": rng.random() < 0.5}
    if kind == "regrid":
        return {"kind": kind, "base": 8 * rng.randrange(10, 31), "limiter": lim}
    if kind == "batch":
        return {"kind": kind, "runs": rng.randrange(1, 17), "first": 4000 + rng.randrange(48), "limiter": lim}
    return {"kind": "host", "nx": 32 * rng.randrange(4, 33), "ny": 32 * rng.randrange(4, 33), "patch": 32,
            "steps": rng.randrange(1, 5), "limiter": lim}


# ------------------------------------------------------------------------------- inputs

def _waves(seed, amp=0.5):
    """(ring pulses, Fourier modes) of a seed: parameters of a state on [-1, 1]^2"""
    r = random.Random(seed)
    rings = [(r.uniform(-0.3, 0.3), r.uniform(-0.3, 0.3), r.uniform(0.2, 0.4), r.uniform(0.08, 0.15),
              amp * r.uniform(0.6, 1.0)) for _ in range(2)]
    modes = [(r.uniform(0.2, 4.0), r.uniform(-4.0, 4.0), r.uniform(0.0, 6.28), r.uniform(0.01, 0.04)) for _ in range(9)]
    return rings, modes


def _state(x, y, seed, swe, lib):
    """(p, u, v) or (h, hu, hv) at points x, y; lib: torch or numpy"""
    rings, modes = _waves(seed)
    f = [1.0 + 0.0 * x, 0.0 * x, 0.0 * x]
    for cx, cy, r0, w, a in rings:
        d = lib.sqrt((x - cx) ** 2 + (y - cy) ** 2) - r0
        f[0] = f[0] + lib.where(abs(d) < w, 0.5 * a * (1.0 + lib.cos(math.pi / w * d)), 0.0 * x)
    for n, (kx, ky, ph, a) in enumerate(modes):
        f[n % 3] = f[n % 3] + a * lib.cos(math.pi * (kx * x + ky * y) + ph)
    return [f[0], f[0] * f[1], f[0] * f[2]] if swe else f


def _boxes(nx, ny, patch):
    if patch == 0:
        return [(0, 0, nx, ny)]
    return [(i, j, min(patch, nx - i), min(patch, ny - j)) for j in range(0, ny, patch) for i in range(0, nx, patch)]


def _grid_run(case):
    """a run with one level over [-1, 1]^2"""
    nx, ny = case["nx"], case["ny"]
    bc = EXTRAP if case["kind"] == "gradient" else WALL
    run = inputs.Run(*inputs.PULSE_DOMAIN, limiter=case["limiter"], bc=(bc,) * 4, cfl=CFL)
    run.levels = [inputs.Level(nx, ny, 2.0 / nx, 2.0 / ny, _boxes(nx, ny, case.get("patch", 0)))]
    return run


def _grid_field(case, seed, swe=False):
    """(3, ny, nx) initial state on the device"""
    nx, ny = case["nx"], case["ny"]
    x = -1.0 + (torch.arange(nx, dtype=torch.float64, device=DEV) + 0.5) * (2.0 / nx)
    y = -1.0 + (torch.arange(ny, dtype=torch.float64, device=DEV) + 0.5) * (2.0 / ny)
    return torch.stack(_state(x[None, :].expand(ny, nx), y[:, None].expand(ny, nx), seed, swe, torch))


def _grid_media(case, seed):
    """smooth positive density and bulk modulus, (ny, nx) on the device"""
    r = random.Random(seed + 77)
    nx, ny = case["nx"], case["ny"]
    x = -1.0 + (torch.arange(nx, dtype=torch.float64, device=DEV) + 0.5) * (2.0 / nx)
    y = -1.0 + (torch.arange(ny, dtype=torch.float64, device=DEV) + 0.5) * (2.0 / ny)
    out = []
    for lo, hi in ((0.5, 2.0), (1.0, 8.0)):
        f = torch.zeros(ny, nx, dtype=torch.float64, device=DEV)
        for _ in range(6):
            kx, ky, ph = r.uniform(0.5, 6.0), r.uniform(-6.0, 6.0), r.uniform(0.0, 6.28)
            f = f + torch.cos(math.pi * (kx * x[None, :] + ky * y[:, None]) + ph)
        out.append(lo + (hi - lo) * (f + 6.0) / 12.0)
    return out


def _pool_index(lev, ncomp=3):
    """(ncomp, NY, NX) positions of the level's cells in its pool of `ncomp` planes per box"""
    idx = np.empty((ncomp, lev.NY, lev.NX), dtype=np.int64)
    for (i, j, nx, ny), off in zip(lev.boxes.tolist(), (lev.qoff if ncomp == 3 else lev.coff).tolist()):
        w, h = nx + 4, ny + 4
        cell = off + (np.arange(ny)[:, None] + 2) * w + np.arange(nx)[None, :] + 2
        for m in range(ncomp):
            idx[m, j:j + ny, i:i + nx] = cell + m * w * h
    return torch.from_numpy(idx).to(DEV)


def _hierarchy_run(case):
    run = inputs.Run(*inputs.PULSE_DOMAIN, limiter=case["limiter"], bc=(WALL,) * 4, cfl=CFL)
    annuli = [(0.2, 0.45), (0.25, 0.35)][:case["nlev"] - 1]
    run.levels = inputs.amr_levels(run, case["base"], case["ratio"], annuli, [2002, 2003])
    return run


def _hierarchy_state(run, seed, swe=False):
    """per level the pool of a seed's state (numpy)"""
    out = []
    for lev in run.levels:
        pool = np.zeros(lev.qsize)
        for n, b in enumerate(lev.boxes):
            x, y = inputs.cell_centres(run, lev, b)
            inputs.box_view(pool, lev.qoff[n], int(b[2]), int(b[3]), 3)[...] = np.stack(_state(x, y, seed, swe, np))
        out.append(pool)
    return out


# ------------------------------------------------------------------------------- prepare

def prepare(case, seed):
    return {"grid": _prepare_grid, "medium": _prepare_grid, "swe": _prepare_grid, "amr": _prepare_amr,
            "swe_amr": _prepare_amr, "batch": _prepare_batch, "regrid": _prepare_regrid, "host": _prepare_host,
            "gradient": _prepare_gradient}[case["kind"]](case, seed)


def _prepare_grid(case, seed):
    run = _grid_run(case)
    lev = run.levels[0]
    swe = case["kind"] == "swe"
    q0 = [[np.zeros(lev.qsize)]]
    if case["kind"] == "medium":
        rho, K = _grid_media(case, seed)
        H = Hierarchy([run], q0, [[inputs.coef_pool(lev, rho.cpu().numpy(), 1)]],
                      [[inputs.coef_pool(lev, K.cpu().numpy(), 1)]])
    elif swe:
        H = Hierarchy([run], q0, system="shallow_water", grav=GRAV)
    else:
        H = Hierarchy([run], q0, rho0=RHO0, K0=K0)
    idx, q = _pool_index(lev), _grid_field(case, seed, swe)

    def start():
        H.q[0][H.cur[0]][idx] = q
        H.init_dt()

    start()
    tune.tune_level(H, 0, pull=True)
    stepper = H.fused_stepper()   # its captures take steps of their own
    start()
    H.q[0][1 - H.cur[0]].zero_()
    return {"case": case, "H": H, "stepper": stepper}


def _prepare_amr(case, seed):
    run = _hierarchy_run(case)
    swe = case["kind"] == "swe_amr"
    q0 = _hierarchy_state(run, seed, swe)
    kw = dict(system="shallow_water", grav=GRAV) if swe else dict(rho0=RHO0, K0=K0)
    return _captured(case, Hierarchy([run], [q0], reflux=case["reflux"], **kw))


def _prepare_batch(case, seed):
    runs, q0, rhos, Ks = [], [], [], []
    for k in range(case["runs"]):
        s = inputs.Stream(case["first"] + k)
        N = 4 * s.randint(16, 64)
        run = inputs.Run(*inputs.PULSE_DOMAIN, limiter=case["limiter"], bc=(WALL,) * 4, cfl=CFL)
        run.levels = inputs.amr_levels(run, N, 4, [(0.2, 0.45)], [case["first"] + k])
        rho, K = (a.cpu().numpy() for a in _grid_media({"nx": N, "ny": N}, seed + 1000 * k))
        runs.append(run)
        q0.append(_hierarchy_state(run, seed + 1000 * k))
        rhos.append([inputs.coef_pool(lev, rho, 4 ** L) for L, lev in enumerate(run.levels)])
        Ks.append([inputs.coef_pool(lev, K, 4 ** L) for L, lev in enumerate(run.levels)])
    return _captured(case, Hierarchy(runs, q0, rhos, Ks))


def _captured(case, H):
    """the hierarchy with tuned tilings and a graph of two coarse steps, at its initial state"""
    first = [H.q[L][0].clone() for L in range(H.nlev)]
    H.init_dt()
    for L in range(H.nlev):
        tune.tune_level(H, L)
    H.coarse_step()   # eager ones first: tensor maps and kernel attributes of the captured launches
    H.coarse_step()
    graph = H.capture(2)
    for L in range(H.nlev):
        H.q[L][H.cur[L]].copy_(first[L])
    H.smax.zero_()
    H.init_dt()
    return {"case": case, "H": H, "graph": graph}


REGRID = dict(tol=0.02, buffer=2, cutoff=0.7, max_size=260, nest=2)


def _prepare_regrid(case, seed):
    base, ratio, nlev = case["base"], 2, 3
    run = inputs.Run(*inputs.PULSE_DOMAIN, limiter=case["limiter"], bc=(WALL,) * 4, cfl=CFL)
    half = base // 2
    run.levels = [inputs.Level(base, base, 2.0 / base, 2.0 / base, _boxes(base, base, half))]
    for L in range(1, nlev):
        n = base * ratio ** L
        run.levels.append(inputs.Level(n, n, 2.0 / n, 2.0 / n, np.zeros((0, 4), dtype=np.int32), ratio))
    H = Hierarchy([run], [_hierarchy_state(run, seed)], rho0=RHO0, K0=K0, reflux=True,
                  tiling=((32, 16, 2, 256), (16, 16, 1, 128)))
    for _ in range(nlev - 1):   # the fine levels are built one by one from the flags
        H.regrid(**REGRID)
    for L, pool in enumerate(_hierarchy_state(run, seed)):
        H.q[L][H.cur[L]][:pool.size] = torch.from_numpy(pool).to(DEV)
    H.init_dt()
    out = [torch.zeros(3 * lev.NX * lev.NY, dtype=torch.float64, device=DEV) for lev in run.levels]
    return {"case": case, "H": H, "out": out}


def _prepare_host(case, seed):
    run = _grid_run(case)
    lev = run.levels[0]
    H = Hierarchy([run], [[np.zeros(lev.qsize)]], rho0=RHO0, K0=K0)
    H.q[0][0][_pool_index(lev)] = _grid_field(case, seed)
    H.init_dt()
    tune.tune_level(H, 0, pull=True)
    src = H.pack().cpu().pin_memory()
    return {"case": case, "H": H, "src": src, "dst": torch.empty_like(src).pin_memory()}


def _prepare_gradient(case, seed):
    run = _grid_run(case)
    lev = run.levels[0]
    nx, ny = case["nx"], case["ny"]
    rho, K = _grid_media(case, seed)
    pools = [inputs.coef_pool(lev, a.cpu().numpy(), 1) for a in (rho, K)]
    H = Hierarchy([run], [[np.zeros(lev.qsize)]], [[pools[0]]], [[pools[1]]])
    q = torch.zeros_like(H.q[0][0])
    q[_pool_index(lev)] = _grid_field(case, seed)
    leaf = [t.detach().clone().requires_grad_(True) for t in (q, H.rho[0], H.K[0])]
    H.init_dt()
    tune.tune_level(H, 0, pull=True)

    def inner(pool, n):
        return pool[:n * (nx + 4) * (ny + 4)].view(n, ny + 4, nx + 4)[:, 2:-2, 2:-2]

    return {"case": case, "H": H, "leaf": leaf, "inner": inner, "weight": _weight(case)}


def _weight(case):
    """the misfit's weight of every cell: two smooth receivers"""
    nx, ny = case["nx"], case["ny"]
    x = -1.0 + (torch.arange(nx, dtype=torch.float64, device=DEV) + 0.5) * (2.0 / nx)
    y = -1.0 + (torch.arange(ny, dtype=torch.float64, device=DEV) + 0.5) * (2.0 / ny)
    w = torch.zeros(ny, nx, dtype=torch.float64, device=DEV)
    for cx, cy in ((0.5, 0.0), (-0.2, 0.3)):
        w = w + torch.exp(-((x[None, :] - cx) ** 2 + (y[:, None] - cy) ** 2) / 0.1)
    return w


# ------------------------------------------------------------------------------- run

def run(s):
    case, H = s["case"], s["H"]
    kind = case["kind"]
    if kind in ("grid", "medium", "swe"):
        s["stepper"].step()
        return H.q[0][H.cur[0]]
    if kind in ("amr", "swe_amr", "batch"):
        s["graph"].replay()
        return [H.pack(L) for L in range(H.nlev)] + [H.dt]
    if kind == "regrid":
        H.coarse_step()
        H.coarse_step()
        H.regrid(**REGRID)
        for L in range(H.nlev):   # the boxes change from pass to pass: buffers that hold any of them
            if len(H.boxes[L]):
                H.pack(L, s["out"][L])
        return s["out"] + [H.dt]
    if kind == "host":
        out = H.steps_from_host(s["src"], s["dst"], case["steps"])
        s["src"], s["dst"] = out, s["src"] if out is s["dst"] else s["dst"]
        return out
    q, rho, K = s["leaf"]
    out = rollout(H, [q], [rho], [K], ncoarse=case["steps"], every=case["every"])
    p = s["inner"](out[0], 3)[0]
    grads = torch.autograd.grad(0.5 * (s["weight"] * p * p).sum(), (q, rho, K))
    return [s["inner"](out[0].detach(), 3)] + [s["inner"](g, n) for g, n in zip(grads, (3, 1, 1))]


# ------------------------------------------------------------------------------- work

def _cells(case):
    """cells advanced by one pass (every substep of every level)"""
    kind = case["kind"]
    if kind in ("grid", "medium", "swe"):
        return case["nx"] * case["ny"]
    if kind in ("host", "gradient"):
        return case["nx"] * case["ny"] * case["steps"]
    if kind == "regrid":   # the refined rings cover about a third of the domain, twice and four times finer
        return 2 * case["base"] ** 2 * (1 + 8 // 3 + 64 // 3)
    runs = [_hierarchy_run(case)] if kind != "batch" else []
    for k in range(case.get("runs", 0)):
        run = inputs.Run(*inputs.PULSE_DOMAIN)
        N = 4 * inputs.Stream(case["first"] + k).randint(16, 64)
        run.levels = inputs.amr_levels(run, N, 4, [(0.2, 0.45)], [case["first"] + k])
        runs.append(run)
    total = 0
    for run in runs:
        sub = 1
        for lev in run.levels:
            sub *= lev.ratio
            total += 2 * sub * lev.ncells
    return total


def work(case):
    """q read and written (48 B a cell-update; the cell-wise medium's two coefficients 16 B more;
    the reverse sweep reads the state and its adjoint and writes the adjoint and two gradients)
    and the method's operations of a cell-update: 59 with a uniform medium, about 110 cell-wise,
    about 450 for the Roe solvers; the reverse sweep about twice its forward"""
    n = _cells(case)
    kind = case["kind"]
    per = {"medium": (64, 110), "batch": (64, 110), "swe": (48, 450), "swe_amr": (48, 450),
           "gradient": (64 + 120, 330)}.get(kind, (48, 59))
    return {"bytes": float(n * per[0]), "flops": float(n * per[1])}


# ------------------------------------------------------------------------------- exact

def exact(case, seed):
    """One-level cases: the pass in plain torch, 64 bits, on the whole grid.  Hierarchies: None."""
    kind = case["kind"]
    if kind in ("amr", "swe_amr", "batch", "regrid"):
        return None
    lev = _grid_run(case).levels[0]
    swe = kind == "swe"
    q = _grid_field(case, seed, swe)
    if kind == "gradient":
        return _exact_gradient(case, seed, q)
    if swe:
        g = _ghosts(q, WALL)
        c = torch.sqrt(GRAV * g[0])
        g, c = g[:, 1:-1, 1:-1], c[1:-1, 1:-1]
        s = float(torch.maximum((g[1] / g[0]).abs() + c, (g[2] / g[0]).abs() + c).max())
        q = _swe_step(_ghosts(q, WALL), CFL * min(lev.dx, lev.dy) / s, lev.dx, lev.dy, case["limiter"])
    else:
        if kind == "medium":
            rho, K = _grid_media(case, seed)
        else:
            rho, K = (torch.full_like(q[0], a) for a in (RHO0, K0))
        rho, K = (_clamped(a) for a in (rho, K))
        dt = CFL * min(lev.dx, lev.dy) / float(torch.sqrt(K / rho).max())
        for _ in range(case.get("steps", 1)):
            q = _acoustics_step(_ghosts(q, WALL), rho, K, dt, lev.dx, lev.dy, case["limiter"])
    if kind == "host":   # packed interiors, box after box
        return torch.cat([q[:, j:j + ny, i:i + nx].reshape(-1) for i, j, nx, ny in lev.boxes.tolist()])
    pool = torch.zeros((lev.qsize + 31) // 32 * 32, dtype=torch.float64, device=DEV)
    pool[_pool_index(lev)] = q
    return pool


def _exact_gradient(case, seed, q):
    rho, K = _grid_media(case, seed)
    leaf = [t.detach().clone().requires_grad_(True) for t in (q, rho, K)]
    dx, dy = 2.0 / case["nx"], 2.0 / case["ny"]
    dt = CFL * min(dx, dy) / float(torch.sqrt(K / rho).max())
    r, k, s = _clamped(leaf[1]), _clamped(leaf[2]), leaf[0]
    for _ in range(case["steps"]):
        s = _acoustics_step(_ghosts(s, EXTRAP), r, k, dt, dx, dy, case["limiter"])
    grads = torch.autograd.grad(0.5 * (_weight(case) * s[0] * s[0]).sum(), leaf)
    return [s.detach(), grads[0], grads[1][None], grads[2][None]]


def _index(n, bc):
    i = torch.arange(-2, n + 2, device=DEV)
    if bc == WALL:
        return torch.where(i < 0, -1 - i, torch.where(i >= n, 2 * n - 1 - i, i))
    return i.clamp(0, n - 1)


def _clamped(a):
    ny, nx = a.shape
    return a[_index(ny, EXTRAP)[:, None], _index(nx, EXTRAP)[None, :]]


def _ghosts(q, bc):
    """two ghost layers: walls mirror the cells and turn the normal velocity, extrapolation repeats"""
    ny, nx = q.shape[1:]
    out = q[:, _index(ny, bc)[:, None], _index(nx, bc)[None, :]]
    if bc == WALL:
        sx, sy = (torch.ones(n + 4, dtype=q.dtype, device=q.device) for n in (nx, ny))
        sx[:2] = sx[-2:] = sy[:2] = sy[-2:] = -1.0
        out = torch.stack([out[0], out[1] * sx[None, :], out[2] * sy[:, None]])
    return out


def _limited(a, b, limiter):
    """phi(b / a) a"""
    m, t = a.abs(), torch.where(a < 0, -b, b)
    zero = torch.zeros_like(a)
    if limiter == MC:
        w = torch.minimum(0.5 * (m + t), 2.0 * torch.minimum(m, t))
    elif limiter == MINMOD:
        w = torch.minimum(m, t)
    elif limiter == SUPERBEE:
        w = torch.maximum(torch.minimum(m, 2.0 * t), torch.minimum(2.0 * m, t))
    else:
        ok = (m > 0) & (t > 0)
        w = torch.where(ok, 2.0 * m * t / torch.where(ok, m + t, torch.ones_like(m)), zero)
    w = torch.where((m > 0) & (t > 0), w, zero)
    return torch.where(a < 0, -w, w)


def _acoustics_sweep(p, u, rho, K, lam, limiter):
    """normal fluctuations and fluxes along the last axis: (update of p, of u, transverse pressure
    input D) for the cells 2 .. n-3 of every row"""
    c = torch.sqrt(K / rho)
    Z = rho * c
    dp, du = p[:, 1:] - p[:, :-1], u[:, 1:] - u[:, :-1]
    zl, zr, cl, cr = Z[:, :-1], Z[:, 1:], c[:, :-1], c[:, 1:]
    a1, a2 = (zr * du - dp) / (zl + zr), (zl * du + dp) / (zl + zr)
    i = slice(1, -1)   # edges with both neighbours
    f1 = (zl[:, 2:] * zl[:, i] + 1.0) / (zl[:, i] ** 2 + 1.0)
    f2 = (zr[:, :-2] * zr[:, i] + 1.0) / (zr[:, i] ** 2 + 1.0)
    m1 = _limited(a1[:, i], a1[:, 2:] * f1, limiter)
    m2 = _limited(a2[:, i], a2[:, :-2] * f2, limiter)
    a1, a2, zl, zr, cl, cr = (t[:, i] for t in (a1, a2, zl, zr, cl, cr))
    e1, e2 = 0.5 * cl * (1.0 - lam * cl) * m1, 0.5 * cr * (1.0 - lam * cr) * m2
    fp, fu = zr * e2 - zl * e1, e1 + e2
    lp, lu, rp, ru = cl * zl * a1, -cl * a1, cr * zr * a2, cr * a2   # A-dQ, A+dQ
    up = rp[:, :-1] - fp[:, :-1] + lp[:, 1:] + fp[:, 1:]
    uu = ru[:, :-1] - fu[:, :-1] + lu[:, 1:] + fu[:, 1:]
    d = rp[:, :-1] - 2.0 * fp[:, :-1] + lp[:, 1:] + 2.0 * fp[:, 1:]
    return up, uu, d


def _acoustics_transverse(d, rho, K, lam):
    """fluxes that the inputs d of the rows put on the edges between them (first axis)"""
    c = torch.sqrt(K / rho)
    Z = rho * c
    w = -0.5 * lam / (Z[:-1] + Z[1:])
    return w * (K[1:] * d[:-1] - K[:-1] * d[1:]), w * (c[1:] * d[:-1] + c[:-1] * d[1:])


def _acoustics_step(g, rho, K, dt, dx, dy, limiter):
    """one unsplit step (second order, full transverse corrections) of the padded state g"""
    lx, ly = dt / dx, dt / dy
    xp, xu, D = _acoustics_sweep(g[0], g[1], rho, K, lx, limiter)
    yp, yv, E = (t.T for t in _acoustics_sweep(g[0].T, g[2].T, rho.T, K.T, ly, limiter))
    gp, gv = _acoustics_transverse(D[1:-1], rho[1:-1, 2:-2], K[1:-1, 2:-2], lx)
    fp, fu = (t.T for t in _acoustics_transverse(E[:, 1:-1].T, rho[2:-2, 1:-1].T, K[2:-2, 1:-1].T, ly))
    p = g[0, 2:-2, 2:-2] - lx * xp[2:-2] - ly * yp[:, 2:-2] - lx * (fp[:, 1:] - fp[:, :-1]) - ly * (gp[1:] - gp[:-1])
    u = g[1, 2:-2, 2:-2] - lx * xu[2:-2] - lx * (fu[:, 1:] - fu[:, :-1])
    v = g[2, 2:-2, 2:-2] - ly * yv[:, 2:-2] - ly * (gv[1:] - gv[:-1])
    return torch.stack([p, u, v])


def _swe_sweep(h, n, t, lam, limiter):
    """normal update of (h, n, t) and the transverse fluxes below / above each cell, along the last
    axis, for the cells 2 .. len-3 of every row"""
    sh = torch.sqrt(h)
    den = sh[:, :-1] + sh[:, 1:]
    un = (n[:, :-1] / sh[:, :-1] + n[:, 1:] / sh[:, 1:]) / den
    ut = (t[:, :-1] / sh[:, :-1] + t[:, 1:] / sh[:, 1:]) / den
    c = torch.sqrt(0.5 * GRAV * (h[:, :-1] + h[:, 1:]))
    dh, dn, dt = h[:, 1:] - h[:, :-1], n[:, 1:] - n[:, :-1], t[:, 1:] - t[:, :-1]
    one, nil = torch.ones_like(un), torch.zeros_like(un)
    a1, a3 = ((un + c) * dh - dn) / (2.0 * c), (dn - (un - c) * dh) / (2.0 * c)
    waves = [(a1, a1 * (un - c), a1 * ut), (nil, nil, dt - ut * dh), (a3, a3 * (un + c), a3 * ut)]
    speeds = [un - c, un, un + c]
    i, lo, hi = slice(1, -1), slice(None, -2), slice(2, None)
    am, ap, cq = [[torch.zeros_like(un[:, i]) for _ in range(3)] for _ in range(3)]
    for s, w in zip(speeds, waves):
        s1 = s[:, i]
        own = sum(x[:, i] * x[:, i] for x in w)
        up = sum(torch.where(s1 > 0, x[:, lo], x[:, hi]) * x[:, i] for x in w)
        phi = torch.where(own > 0, _limited(own, up, limiter) / torch.where(own > 0, own, one[:, i]), nil[:, i])
        k = s1.abs() * (1.0 - lam * s1.abs()) * phi
        for m in range(3):
            am[m] = am[m] + s1.clamp(max=0.0) * w[m][:, i]
            ap[m] = ap[m] + s1.clamp(min=0.0) * w[m][:, i]
            cq[m] = cq[m] + k * w[m][:, i]
    un, ut, c = un[:, i], ut[:, i], c[:, i]

    def split(d):   # (h, n, t) parts going down and up
        b = [((ut + c) * d[0] - d[2]) / (2.0 * c), d[1] - un * d[0], (d[2] - (ut - c) * d[0]) / (2.0 * c)]
        r = [(1.0, un, ut - c), (0.0, 1.0, 0.0), (1.0, un, ut + c)]
        sp = [ut - c, ut, ut + c]
        return [[sum(f(sp[q]) * b[q] * r[q][m] for q in range(3)) for m in range(3)]
                for f in (lambda a: a.clamp(max=0.0), lambda a: a.clamp(min=0.0))]

    left, right = split([am[m] + cq[m] for m in range(3)]), split([ap[m] - cq[m] for m in range(3)])
    upd = [ap[m][:, :-1] - 0.5 * cq[m][:, :-1] + am[m][:, 1:] + 0.5 * cq[m][:, 1:] for m in range(3)]
    down, upw = ([right[k][m][:, :-1] + left[k][m][:, 1:] for m in range(3)] for k in range(2))
    return upd, down, upw


def _swe_step(g, dt, dx, dy, limiter):
    lx, ly = dt / dx, dt / dy
    ux, dx_, px = _swe_sweep(g[0], g[1], g[2], lx, limiter)
    uy, dy_, py = _swe_sweep(g[0].T, g[2].T, g[1].T, ly, limiter)
    out = []
    for m, k in ((0, 0), (1, 2), (2, 1)):   # component m is component k of the y sweep
        G = -0.5 * lx * (dx_[m][2:-1] + px[m][1:-2])             # on the y-edges above rows 1 .. ny+1
        F = -0.5 * ly * (dy_[k][2:-1] + py[k][1:-2]).T
        out.append(g[m, 2:-2, 2:-2] - lx * ux[m][2:-2] - ly * uy[k][2:-2].T
                   - ly * (G[1:] - G[:-1]) - lx * (F[:, 1:] - F[:, :-1]))
    return torch.stack(out)
