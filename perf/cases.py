"""The work that a program using this package has it do, one case each, through the public entry
points: time steps of the solver (two- and three-dimensional, synchronous and asynchronous, both
precisions, both orders, the compact scheme, connected curvilinear blocks, the learned halo),
the training and the use of the halo network, and the diagnostics of a run.

A solver case is a run in progress: `prepare` builds the solver, gives it its delay schedule and
the ring of time levels a run holds at that point (a checkpoint), and `run` advances it and reads
the state back.  A pass of an asynchronous case is one time step from the checkpoint (the ring has
one spare level, so the step overwrites nothing that the next pass reads); a synchronous case
starts from its state again and takes a few steps.  The fields are the Taylor-Green vortex, the
isentropic vortex or the airfoil's initial flow with seeded phases and disturbances, and change
from level to level as a flow carried along does.

`exact` computes the same pass in plain 64-bit torch, written from the method's definition:
central or compact differences on every sub-domain with its own halo, Lagrange extrapolation and
the buffer updates of the low-storage Runge-Kutta stages, the tenth-order filter as a dense solve.
"""
from __future__ import annotations

import math
from fractions import Fraction

import numpy as np
import torch

from paper_2506_03027_gb300 import cfs
from paper_2506_03027_gb300 import inputs as I


def _cart(name, dims, n, p, algo, **kw):
    """A periodic Cartesian block of n points per axis (an int, or one per axis) in p sub-domains
    per axis."""
    n = (n,) * dims if isinstance(n, int) else tuple(n)
    p = (p,) * dims if isinstance(p, int) else tuple(p)
    n, p = n + (1,) * (3 - dims), p + (1,) * (3 - dims)
    c = {"kind": "cart", "nx": n[0], "ny": n[1], "nz": n[2], "px": p[0], "py": p[1], "pz": p[2],
         "algo": algo, "L": 4, "kmax": {"SA": 0, "CAA": 3, "SAA": 3}[algo], "order": 4, "viscous": dims == 3,
         "visc_law": 0, "filter": dims == 3, "precision": 0, "compact": False, "steps": 1, "graph": True}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest run anyone starts with: the isentropic vortex on 64 x 64 points, synchronous,
        # Euler, no filter; a step is 15 launches on 4,096 points, so it is all latency
        _cart("vortex 64^2 SA", 2, 64, 2, "SA", steps=5),
        # the study of the asynchrony error: second-order schemes in two dimensions at large size
        _cart("study 1024^2 CAA order 2", 2, 1024, 16, "CAA", order=2, L=4, kmax=3),
        # a small three-dimensional run with ragged sub-domains (9, 9, 8, 8), as the tests take,
        # stepped without a graph
        _cart("tgv 34^3 SAA ragged", 3, 34, 4, "SAA", graph=False),
        # the benchmark's own run in FP64
        _cart("tgv 128^3 SAA", 3, 128, 4, "SAA"),
        # the synchronous algorithm it is compared with, on a grid that does not divide evenly
        _cart("tgv 100^3 SA", 3, 100, 3, "SA", steps=2),
        # the FP32-intermediate form at the size it is run at
        _cart("tgv 256^3 CAA fp32", 3, 256, 8, "CAA", precision=1),
        # the compact sixth-order scheme for the Euler equations
        _cart("compact euler 128^3 CAA", 3, 128, 4, "CAA", viscous=False, compact=True),
        # the airfoil C-grid (12 connected curvilinear blocks) in FP64 at half resolution
        {"name": "cgrid 2.8M SAA", "kind": "cgrid", "scale": 0.5, "precision": 0, "graph": True},
        # and in the FP32-intermediate form at three quarters of the full resolution
        {"name": "cgrid 9.3M SAA fp32", "kind": "cgrid", "scale": 0.75, "precision": 1, "graph": True},
        # the solver with the learned stage-0 halo
        {"name": "learned 128^3 SAA", "kind": "learned", "n": 128, "p": 4, "precision": 0, "graph": True},
        # training of the halo network at its usual batch: gradient and update, a few iterations
        {"name": "train 4096", "kind": "train", "batch": 4096, "iters": 4},
        # what a run prints as it goes: the diagnostics of a 128^3 state
        {"name": "diagnostics 128^3", "kind": "diag", "n": 128, "p": 4},
    ]


def draw(rng):
    """One more case of the same ranges."""
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["vortex", "study", "tgv", "tgv", "fp32", "fp32", "compact", "cgrid", "learned", "train", "predict", "diag"])
    if kind == "vortex":
        n = (logint(32, 512), logint(32, 512))
        return _cart(None, 2, n, [rng.randint(1, max(1, min(4, x // 12))) for x in n], "SA", steps=rng.randint(2, 5), graph=rng.random() < 0.5)
    if kind == "study":
        n = (logint(64, 1200), logint(64, 1200))
        return _cart(None, 2, n, [max(1, x // rng.randint(24, 72)) for x in n], rng.choice(["CAA", "SAA"]), order=2, kmax=3)
    if kind in ("tgv", "fp32"):
        algo = rng.choice(["SA", "CAA", "SAA"])
        hi = 128 if kind == "tgv" else 224
        n = [logint(24, hi)] * 3
        if rng.random() < 0.3:
            n = [max(24, int(x * rng.uniform(0.6, 1.0))) for x in n]
        w = rng.randint(9, 36)
        if kind == "fp32" and rng.random() < 0.5:  # the sub-domain size the form is used with
            n, w = [32 * max(1, round(x / 32)) for x in n], 32
        return _cart(None, 3, n, [max(1, x // w) for x in n], algo, precision=int(kind == "fp32"),
                     order=4 if kind == "fp32" else rng.choice([4, 4, 2]), visc_law=rng.choice([0, 0, 1]), steps=rng.randint(1, 3) if algo == "SA" else 1,
                     graph=rng.random() < 0.7)
    if kind == "compact":
        n = logint(32, 128)
        return _cart(None, 3, n, max(1, n // rng.randint(12, 40)), rng.choice(["SA", "CAA"]), viscous=False, compact=True)
    if kind == "cgrid":
        return {"kind": "cgrid", "scale": round(math.exp(rng.uniform(math.log(0.2), math.log(0.6))), 3), "precision": rng.randint(0, 1),
                "graph": rng.random() < 0.7}
    if kind == "learned":
        n = logint(32, 144)
        return {"kind": "learned", "n": n, "p": max(1, n // rng.randint(16, 40)), "precision": rng.randint(0, 1), "graph": rng.random() < 0.7}
    if kind == "train":
        return {"kind": "train", "batch": logint(256, 32768), "iters": rng.randint(1, 4)}
    if kind == "predict":
        return {"kind": "predict", "samples": logint(512, 400000)}
    n = logint(32, 192)
    return {"kind": "diag", "n": n, "p": max(1, n // 32)}


# ------------------------------------------------------------------------------- inputs

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _case_of(case):
    """The package's own description of a Cartesian case."""
    two = case["nz"] == 1
    length = 10.0 if two else 2 * math.pi
    c = I.Case(name="vortex" if two else "tgv", nx=case["nx"], ny=case["ny"], nz=case["nz"], px=case["px"], py=case["py"], pz=case["pz"],
               lx=length, ly=length, lz=1.0 if two else length, mach=0.5 if two else 0.1, viscous=case["viscous"],
               visc_law=case["visc_law"], order=case["order"], algo=case["algo"], caa_L=case["L"], kmax=case["kmax"],
               filter=case["filter"], compact=int(case["compact"]))
    h = min(c.dx, c.dy, c.dz if not two else c.dx)
    cfl = {"SA": 0.5, "CAA": 0.25, "SAA": 0.05}[case["algo"]]
    return c.replace(dt=cfl * h / (2 if two else 3) / (1.0 + 1.0 / c.mach))


def _phases(seed, count):
    return np.random.default_rng(seed).uniform(0.0, 2 * math.pi, count)


def _fields(c, seed, t):
    """The conserved state at time t: the case's vortex with seeded phases and disturbances."""
    d = _device()
    x = (c.dx * torch.arange(c.nx, dtype=torch.float64, device=d))[None, None, :]
    y = (c.dy * torch.arange(c.ny, dtype=torch.float64, device=d))[None, :, None]
    z = (c.dz * torch.arange(c.nz, dtype=torch.float64, device=d))[:, None, None]
    a = _phases(seed, 12)
    gm2 = c.gamma * c.mach ** 2
    if c.nz == 1:
        x0, y0 = c.lx * a[0] / (2 * math.pi), c.ly * a[1] / (2 * math.pi)
        xr = torch.remainder(x - x0 - t + c.lx / 2, c.lx) - c.lx / 2
        yr = torch.remainder(y - y0 + c.ly / 2, c.ly) - c.ly / 2
        eps = 4.0 + a[2] / (2 * math.pi)
        g = torch.exp(0.5 * (1.0 - xr * xr - yr * yr))
        s = eps / (2 * math.pi) / (c.mach * math.sqrt(c.gamma))
        T = 1.0 - (c.gamma - 1.0) * eps * eps / (8.0 * c.gamma * math.pi ** 2) * g * g
        rho = T ** (1.0 / (c.gamma - 1.0))
        u, v, w = 1.0 - s * yr * g, s * xr * g, torch.zeros_like(rho)
        p = rho * T / gm2
    else:
        sx, sy, sz = x + a[0] + t, y + a[1] + 0.7 * t, z + a[2] - 0.4 * t
        u = torch.sin(sx) * torch.cos(sy) * torch.cos(sz) + 0.1 * torch.sin(3 * sy + a[3]) * torch.cos(2 * sz + a[4])
        v = -torch.cos(sx) * torch.sin(sy) * torch.cos(sz) + 0.1 * torch.sin(3 * sz + a[5]) * torch.cos(2 * sx + a[6])
        w = 0.1 * torch.sin(3 * sx + a[7]) * torch.cos(2 * sy + a[8]) + torch.zeros_like(u)
        p = 1.0 / gm2 + (torch.cos(2 * sx) + torch.cos(2 * sy)) * (torch.cos(2 * sz) + 2.0) / 16.0
        rho = gm2 * p / (1.0 + 0.02 * torch.sin(sx + a[9]) * torch.sin(sy + a[10]) * torch.sin(2 * sz + a[11]))
    U = torch.empty((5, c.nz, c.ny, c.nx), dtype=torch.float64, device=d)
    U[0], U[1], U[2], U[3] = rho, rho * u, rho * v, rho * w
    U[4] = p / (c.gamma - 1.0) + 0.5 * rho * (u * u + v * v + w * w)
    return U


def _delays(c, seed, steps, nsub=None):
    return np.random.default_rng(seed + 1).integers(0, c.kmax + 1, size=(steps, c.nsub if nsub is None else nsub, 6), dtype=np.int8)


def _start_step(c):
    """The step index of the checkpoint: the first one whose every delay finds its levels."""
    return 0 if c.algo == "SA" else c.levels + c.kmax


def _solver(blocks, precision, graph, kmax):
    stream = torch.cuda.Stream() if graph else torch.cuda.current_stream()
    torch.cuda.current_stream().synchronize()
    return cfs.Solver(blocks, max_delay=kmax, precision=precision, stream=stream, graph=graph)


def _load_ring(s, n0, level):
    """Hand the solver its checkpoint: the levels n0 - R + 1 .. n0 (block states one after another)."""
    R = cfs.cfs_ring_depth(s.ctx)
    s.set_step(n0)
    points = sum(b.npts for b in s.blocks)
    ring = torch.empty((R, 5 * points), dtype=torch.float64, device="cuda")
    for i in range(R):
        ring[i] = level(n0 - R + 1 + i)
    torch.cuda.current_stream().synchronize()
    cfs.cfs_set_ring(s.ctx, ring.data_ptr(), cfs.DEVICE)


def _prepare_solver(case, seed, c, halo_model=None):
    s = _solver(c, case["precision"], case["graph"], c.kmax)
    n0 = _start_step(c)
    s.set_schedule(delays=_delays(c, seed, n0 + 1) if c.algo == "SAA" else None)
    state = {"case": case, "solver": s, "n0": n0, "out": [torch.empty((5, c.nz, c.ny, c.nx), dtype=torch.float64, device="cuda")]}
    if halo_model is not None:
        cfs.cfs_set_halo_model(s.ctx, *halo_model)
    if c.algo == "SA":
        state["start"] = _fields(c, seed, 0.0)
    else:
        _load_ring(s, n0, lambda n: _fields(c, seed, (n - n0) * c.dt).ravel())
    return state


def _cgrid(case):
    """The airfoil grid at a fraction of its full resolution, and the time step it runs with."""
    f = case["scale"]

    def r(x):
        return max(8, int(round(x * f)))
    sp = I.CGridSpec(wake=r(96), aft=r(160), fore=r(512), nj_in=r(192), nj_out=r(64), nz_in=2 * r(32), nz_out=r(32),
                     sub=(r(64), r(64), r(32)))
    mb = I.naca_cgrid(sp)
    return sp, mb.replace_all(dt=I.cgrid_dt(mb, 0.05))


def _cgrid_level(mb, sp, seed, t):
    """The initial flow of the airfoil grid (free stream slowed towards the wall) with a seeded
    disturbance carried along, every block's state one after another."""
    a = _phases(seed, 9)
    al = math.radians(sp.alpha_deg)
    parts = []
    rng = torch.Generator(device="cuda").manual_seed(seed)
    for b, c in enumerate(mb.blocks):
        xy = torch.from_numpy(np.ascontiguousarray(mb.xy[b][0])).cuda()
        x, y = xy[0][None], xy[1][None]
        z = (c.dz * torch.arange(c.nz, dtype=torch.float64, device="cuda"))[:, None, None]
        if b % 6 in (0, 5):
            dist = torch.hypot(x - 1.0, y)
        else:
            foot = torch.from_numpy(np.ascontiguousarray(mb.xy[b % 6][0][:, 0])).cuda()
            dist = torch.hypot(x - foot[0], y - foot[1])
        g = 1.0 - torch.exp(-((dist / sp.ramp) ** 2))
        noise = 2.0 * torch.rand((3, c.nz, c.ny, c.nx), generator=rng, dtype=torch.float64, device="cuda") - 1.0
        kz = 2 * math.pi / sp.span
        vel = []
        for q, base in enumerate((math.cos(al), math.sin(al), 0.0)):
            wave = torch.sin(3.0 * (x - t) + a[q]) * torch.cos(2.0 * y + a[3 + q]) * torch.cos(kz * z + a[6 + q])
            vel.append(g * (base + sp.perturb * (noise[q] + 5.0 * wave)))
        rho = 1.0 + 0.01 * g * torch.sin(2.0 * (x - t) + a[1]) * torch.cos(kz * z + a[2])
        p = rho / (c.gamma * c.mach ** 2)
        U = torch.empty((5, c.nz, c.ny, c.nx), dtype=torch.float64, device="cuda")
        U[0] = rho
        for q in range(3):
            U[1 + q] = rho * vel[q]
        U[4] = p / (c.gamma - 1.0) + 0.5 * rho * (vel[0] ** 2 + vel[1] ** 2 + vel[2] ** 2)
        parts.append(U.ravel())
    return torch.cat(parts)


def _prepare_cgrid(case, seed):
    sp, mb = _cgrid(case)
    s = _solver(mb, case["precision"], case["graph"], mb.case.kmax)
    n0 = _start_step(mb.case)
    s.set_schedule(delays=_delays(mb.case, seed, n0 + 1, mb.nsub))
    _load_ring(s, n0, lambda n: _cgrid_level(mb, sp, seed, (n - n0) * mb.case.dt))
    out = [torch.empty((5, c.nz, c.ny, c.nx), dtype=torch.float64, device="cuda") for c in mb.blocks]
    return {"case": case, "solver": s, "n0": n0, "out": out}


def _learned_case(case):
    n, p = case["n"], case["p"]
    c = _case_of(_cart(None, 3, n, p, "SAA", kmax=4))
    return c


def _network(seed):
    """Seeded parameters of the halo network (weights of the size training ends with) and scales."""
    rng = np.random.default_rng(seed + 2)
    parts = []
    for fan_in, count in ((65, 64), (64, 64), (64, 20)):
        parts.append(rng.uniform(-1, 1, size=fan_in * count) / math.sqrt(fan_in))
        parts.append(0.1 * rng.uniform(-1, 1, size=count))
    return np.concatenate(parts).astype(np.float32)


def _prepare_learned(case, seed):
    c = _learned_case(case)
    # features of order one, residuals of the size of a step's change
    step = 1.0 / c.dt
    scales = np.array([10 * step, step, step, step, step] + [5 * step] * 5 + [step * step] * 5)
    s = _prepare_solver(case, seed, c, (_network(seed), scales))
    return s


def _samples(seed, n):
    """Training pairs as the halo columns of a run give them: inputs of unit spread in BF16 with a
    one-hot delay, targets that depend on them."""
    g = torch.Generator(device=_device()).manual_seed(seed)
    x = torch.randn((n, 65), generator=g, device=_device())
    k = torch.randint(0, 5, (n,), generator=g, device=_device())
    x[:, 60:] = torch.nn.functional.one_hot(k, 5).float()
    x = x.to(torch.bfloat16)
    t = 0.3 * torch.randn((n, 20), generator=g, device=_device()) + (0.5 * x[:, :20] - 0.3 * x[:, 20:40]).float() * (1.0 + k[:, None]) * 0.4
    return x, t


def _train_setup(case, seed):
    n = case["batch"] * case["iters"]
    x, t = _samples(seed, n)
    rng = np.random.default_rng(seed + 3)
    params = torch.from_numpy(_network(seed))
    m = torch.from_numpy((1e-3 * rng.standard_normal(params.numel())).astype(np.float32))
    v = torch.from_numpy((1e-5 * (0.2 + rng.random(params.numel()))).astype(np.float32))
    return x, t, params, m, v


ADAM = dict(lr=2e-3, beta1=0.9, beta2=0.999, eps=1e-8, wd=1e-5)
FIRST_UPDATE = 100  # the training has been running for a while


def _prepare_train(case, seed):
    x, t, params, m, v = _train_setup(case, seed)
    work = torch.empty(cfs.cfs_mlp_workspace_bytes(case["batch"]) // 4 + 1, dtype=torch.float32, device="cuda")
    return {"case": case, "x": x.view(torch.int16), "t": t, "start": [q.cuda() for q in (params, m, v)],
            "now": [torch.empty_like(q, device="cuda") for q in (params, m, v)],
            "grad": torch.empty(params.numel(), device="cuda"), "loss": torch.empty(case["iters"], device="cuda"), "work": work}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "cart":
        return _prepare_solver(case, seed, _case_of(case))
    if kind == "cgrid":
        return _prepare_cgrid(case, seed)
    if kind == "learned":
        return _prepare_learned(case, seed)
    if kind == "train":
        return _prepare_train(case, seed)
    if kind == "predict":
        x, _ = _samples(seed, case["samples"])
        return {"case": case, "x": x.view(torch.int16), "params": torch.from_numpy(_network(seed)).cuda(),
                "y": torch.empty((case["samples"], 20), dtype=torch.float32, device="cuda")}
    c = _case_of(_cart(None, 3, case["n"], case["p"], "SA"))
    s = cfs.Solver(c)
    s.set_schedule()
    s.set_state(_fields(c, seed, 0.0))
    return {"case": case, "solver": s}


# ------------------------------------------------------------------------------- the pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("cart", "cgrid", "learned"):
        s = state["solver"]
        s.set_step(state["n0"])
        if "start" in state:
            s.set_state(state["start"])
        s.step(case.get("steps", 1))
        return {"U": [s.get_state(out=o, block=b) for b, o in enumerate(state["out"])]}
    if kind == "train":
        now, B = state["now"], case["batch"]
        for a, b in zip(now, state["start"]):
            a.copy_(b)
        st = torch.cuda.current_stream().cuda_stream
        p, m, v = (q.data_ptr() for q in now)
        for it in range(case["iters"]):
            cfs.cfs_mlp_grad(p, state["x"][it * B:].data_ptr(), state["t"][it * B:].data_ptr(), B, state["work"].data_ptr(),
                             state["grad"].data_ptr(), state["loss"][it:].data_ptr(), st)
            cfs.cfs_mlp_adamw(p, state["grad"].data_ptr(), m, v, FIRST_UPDATE + it, ADAM["lr"], ADAM["beta1"], ADAM["beta2"], ADAM["eps"],
                              ADAM["wd"], st)
        return {"params": now[0], "m": now[1], "v": now[2], "grad": state["grad"], "loss": state["loss"]}
    if kind == "predict":
        cfs.cfs_mlp_forward(state["params"].data_ptr(), state["x"].data_ptr(), state["y"].data_ptr(), case["samples"],
                            torch.cuda.current_stream().cuda_stream)
        return {"y": state["y"]}
    d = state["solver"].diagnostics()
    return {"mean": d[:2], "totals": d[2:7], "bad": d[7]}


# ------------------------------------------------------------------------------- work

def work(case):
    """Bytes and operations of one pass: the state read and written once per step and, on an
    asynchronous step, the delayed levels of the halo points; the operations of the differences,
    fluxes, updates and filter passes per point."""
    kind = case["kind"]
    if kind == "train":
        n = case["batch"] * case["iters"]
        return {"bytes": n * (130 + 80) + 7 * 4 * 9684 * case["iters"], "flops": 6 * 9536 * n}
    if kind == "predict":
        return {"bytes": case["samples"] * (130 + 80) + 4 * 9684, "flops": 2 * 9536 * case["samples"]}
    if kind == "diag":
        return {"bytes": 40 * case["n"] ** 3, "flops": 110 * case["n"] ** 3}
    if kind == "cgrid":
        f3 = case["scale"] ** 3
        pts, subs, width, steps, order, visc, filt, asyn = 22.0e6 * f3, 154, 64 * 64 * 32 * f3, 1, 4, True, True, True
        area = 2 * f3 ** (2 / 3) * (64 * 64 + 2 * 64 * 32)
        dims = 3
    else:
        c = _learned_case(case) if kind == "learned" else _case_of(case)
        dims = 2 if c.nz == 1 else 3
        pts, subs, steps, order, visc, filt, asyn = c.npts, c.nsub, case.get("steps", 1), c.order, c.viscous, c.filter, c.algo != "SA"
        wx, wy, wz = c.nx / c.px, c.ny / c.py, c.nz / c.pz
        area = 2 * (wx * wy * (dims == 3) + wx * wz + wy * wz)
    r = 2 if order == 4 else 1
    stages, levels = (5, 5) if order == 4 else (2, 3)
    halo = subs * area * (2 * r if visc else r) if asyn else 0
    per_stage = 20 + dims * (5 * (2.5 * r) + 15) + 20 + (90 + dims * 4 * 2.5 * r if visc else 0)
    bytes_ = steps * (80 * pts + 40 * levels * halo)
    flops = steps * (stages * (per_stage * pts + 10 * levels * halo) + (5 * dims * 21 * pts if filt else 0))
    if kind == "learned":
        flops += 2 * 9536 * subs * area
    return {"bytes": float(bytes_), "flops": float(flops)}


# ------------------------------------------------------------------------------- the exact pass

RK = {4: ((0.0, -0.4812317, -1.0495626, -1.6025296, -1.7782672), (0.09761835, 0.41225329, 0.44021696, 1.42631146, 0.19787605)),
      2: ((0.0, -0.5), (0.5, 1.0))}


def _lagrange(k, levels):
    """Weights of the levels 0, -1, ... (k steps back) for the value k steps ahead of the newest."""
    return [math.prod((k + j) / (j - l) for j in range(levels) if j != l) for l in range(levels)]


def _basis(k, l, levels):
    """Coefficients (of 1, t, t^2, ...) of the Lagrange polynomial that is 1 at -(k + l) and 0 at the
    other levels, as exact fractions."""
    q = [Fraction(1)]
    for j in range(levels):
        if j != l:  # times (t + k + j) / (j - l)
            q = [(Fraction(k + j) * u + v) / (j - l) for u, v in zip(q + [Fraction(0)], [Fraction(0)] + q)]
    return q


def _halo_weights(order, kmax):
    """W[k][m][l]: stage-m halo value from the levels n-k-l.  Stage 0 extrapolates; the following
    stages add the stage increments with time derivatives that match the Taylor series of the
    stage values (polynomials of the low-storage recursion) at the delayed levels."""
    A, B = RK[order]
    C = 5 if order == 4 else 3
    poly = [[1.0] + [0.0] * C]  # stage polynomials P_e(z) of y' = z y
    P, Q = poly[0][:], [0.0] * (C + 1)
    for a, b in zip(A, B):
        Q = [a * q + (P[j - 1] if j else 0.0) for j, q in enumerate(Q)]
        P = [p + b * q for p, q in zip(P, Q)]
        poly.append(P)
    W = []
    for k in range(kmax + 1):
        rows, acc = [np.array(_lagrange(k, C))], np.zeros(C)
        basis = [_basis(k, l, C) for l in range(C)]
        for m in range(1, len(A)):
            # the functional whose moments (of t^th / th!) are the stage polynomial's coefficients
            acc = A[m - 1] * acc + np.array([sum(float(q[th] * math.factorial(th)) * poly[m - 1][th - 1] for th in range(1, m + 1) if th < C)
                                             for q in basis])
            rows.append(rows[-1] + B[m - 1] * acc)
        W.append(rows)
    return W


def _split(n, p):
    base, rem = divmod(n, p)
    sizes = [base + (i < rem) for i in range(p)]
    return [(sum(sizes[:i]), sizes[i]) for i in range(p)]


def _diff(f, axis, h, order):
    """Central difference along a tensor axis (the ends lose the stencil's radius)."""
    r = 2 if order == 4 else 1
    n = f.shape[axis] - 2 * r

    def at(o):
        return f.narrow(axis, r + o, n)
    if order == 4:
        return (8.0 * (at(1) - at(-1)) - (at(2) - at(-2))) / (12.0 * h)
    return (at(1) - at(-1)) / (2.0 * h)


def _compact(f, axis, h, n):
    """Sixth-order compact derivative of a line of n points with 4 more on each side."""
    def at(o, count=n, first=4):
        return f.narrow(axis, first + o, count)
    rhs = (14.0 / 9.0) * (at(1) - at(-1)) / (2 * h) + (1.0 / 9.0) * (at(2) - at(-2)) / (4 * h)
    ends = []
    for i in (3, n + 4):
        e = (45.0 * (at(1, 1, i) - at(-1, 1, i)) - 9.0 * (at(2, 1, i) - at(-2, 1, i)) + (at(3, 1, i) - at(-3, 1, i))) / (60.0 * h)
        ends.append(e)
    rhs = rhs.clone()
    rhs.narrow(axis, 0, 1).sub_(ends[0] / 3.0)
    rhs.narrow(axis, n - 1, 1).sub_(ends[1] / 3.0)
    T = torch.eye(n, dtype=torch.float64, device=f.device) + (1.0 / 3.0) * (torch.diag(torch.ones(n - 1, dtype=torch.float64, device=f.device), 1)
                                                                           + torch.diag(torch.ones(n - 1, dtype=torch.float64, device=f.device), -1))
    return torch.movedim(torch.movedim(rhs, axis, -1) @ torch.linalg.inv(T).T, -1, axis)


def _rhs(c, E, G, Gz):
    """R(U) on the owned points of sub-domains stacked as E [5][sub][z][y][x] with halo."""
    dims = 3 if c.nz > 1 else 2
    r = 2 if c.order == 4 else 1
    axes = {0: -1, 1: -2, 2: -3}
    h = (c.dx, c.dy, c.dz)
    gm2 = c.gamma * c.mach ** 2
    rho = E[0]
    vel = [E[1] / rho, E[2] / rho, E[3] / rho]
    p = (c.gamma - 1.0) * (E[4] - 0.5 * (E[1] * vel[0] + E[2] * vel[1] + E[3] * vel[2]))
    depth = {0: G, 1: G, 2: Gz}

    def owned(f, keep=None, extra=0, had=0):
        """Cut every axis to the owned points; axis `keep` to the owned points and `extra` beyond.
        `had`: what is already missing of each end."""
        for a in range(dims):
            cut = depth[a] - had - (extra if a == keep else 0)
            if cut:
                f = f.narrow(axes[a], cut, f.shape[axes[a]] - 2 * cut)
        return f
    grads = None
    if c.viscous:
        T = gm2 * p / rho
        mu = T ** c.visc_exp if c.visc_law == 1 else torch.ones_like(T)

        def grad(f, a):  # every other axis cut alike
            d = _diff(f, axes[a], h[a], c.order)
            for b in range(dims):
                if b != a:
                    d = d.narrow(axes[b], r, d.shape[axes[b]] - 2 * r)
            return d
        grads = [[grad(f, a) for a in range(dims)] for f in vel + [T]]
    R = None
    kap = 1.0 / ((c.gamma - 1.0) * c.pr * c.mach ** 2)
    ext = 4 if c.compact else r
    for a in range(dims):
        def at(f):
            return owned(f, a, ext)
        ua = at(vel[a])
        F = [-at(E[1 + a])] + [-(at(E[1 + q]) * ua) for q in range(3)] + [-(at(E[4]) + at(p)) * ua]
        F[1 + a] = F[1 + a] - at(p)
        if c.viscous:
            D = [[owned(g, a, ext, r) for g in row] for row in grads]
            m = at(mu)
            div = sum(D[b][b] for b in range(dims))
            zero = torch.zeros_like(m)

            def d(i, j):
                return D[i][j] if j < dims else zero
            tau = [m * (d(a, i) + (D[i][a])) - (2.0 / 3.0 * m * div if i == a else 0.0) for i in range(3)]
            q = kap * m * D[3][a] + sum(at(vel[i]) * tau[i] for i in range(3))
            for i in range(3):
                F[1 + i] = F[1 + i] + tau[i] / c.re
            F[4] = F[4] + q / c.re
        F = torch.stack(F)
        n = F.shape[axes[a]] - 2 * ext
        dF = _compact(F, axes[a], h[a], n) if c.compact else _diff(F, axes[a], h[a], c.order)
        R = dF if R is None else R + dF
    return R


def _filter_line(F, axis, n, alpha):
    """Filtered values of lines of n points with 5 more on each side: the tenth-order filter as
    f + K T^-1 delta^10 f (its numerator has a five-fold zero at the smooth end), T = (alpha, 1,
    alpha), no change at the first point beyond each end."""
    d = F
    for _ in range(10):
        d = d.narrow(axis, 1, d.shape[axis] - 1) - d.narrow(axis, 0, d.shape[axis] - 1)
    one = torch.ones(n - 1, dtype=torch.float64, device=F.device)
    T = torch.eye(n, dtype=torch.float64, device=F.device) + alpha * (torch.diag(one, 1) + torch.diag(one, -1))
    x = torch.movedim(torch.movedim(d, axis, -1) @ torch.linalg.inv(T).T, -1, axis)
    # delta^10 of the shortest wave is -1024 f, which the filter has to remove: that fixes K
    return F.narrow(axis, 5, n) + (1.0 - 2.0 * alpha) / 1024.0 * x


def _exact_steps(c, seed, steps, n0):
    """The state after `steps` steps from the checkpoint, in 64 bits."""
    dims = 3 if c.nz > 1 else 2
    A, B = RK[c.order]
    C = c.levels
    r = 2 if c.order == 4 else 1
    G = 4 if c.compact else (2 * r if c.viscous else r)
    Gz = G if dims == 3 else 0
    dev = _device()
    levels = {0: _fields(c, seed, 0.0)}  # by how many steps back
    asyn = c.algo != "SA"
    if asyn:
        for j in range(1, c.kmax + C):
            levels[j] = _fields(c, seed, -j * c.dt)
    n3, p3 = (c.nx, c.ny, c.nz), (c.px, c.py, c.pz)
    cuts = [_split(n, p) for n, p in zip(n3, p3)]
    subs = [(i, j, k) for k in range(c.pz) for j in range(c.py) for i in range(c.px)]
    if c.algo == "SAA":
        table = _delays(c, seed, n0 + 1)[n0].astype(np.int64)
    elif c.algo == "CAA":
        table = np.full((len(subs), 6), (n0 - C) % c.caa_L)
    else:
        table = np.zeros((len(subs), 6), dtype=np.int64)
    table = np.clip(table, 0, max(0, n0 - C + 1))
    groups = {}  # sub-domains of one shape, a bounded number of points at a time
    for sid, ijk in enumerate(subs):
        shape = tuple(cuts[a][ijk[a]][1] for a in range(3))
        room = max(1, int(1.2e6 // ((shape[0] + 2 * G) * (shape[1] + 2 * G) * (shape[2] + 2 * Gz))))
        lists = groups.setdefault(shape, [[]])
        if len(lists[-1]) >= room:
            lists.append([])
        lists[-1].append(sid)

    def window(sids, depth, shape):
        """Index tensors of the sub-domains' points and those `depth` beyond, per axis, and the
        delay of the face that a point along the axis lies beyond (0 inside)."""
        idx, kd = [], []
        for a in range(3):
            o = torch.tensor([cuts[a][subs[s][a]][0] for s in sids], device=dev)
            t = torch.arange(-depth[a], shape[a] + depth[a], device=dev)
            idx.append(torch.remainder(o[:, None] + t[None, :], n3[a]))
            lo = torch.tensor(table[sids, 2 * a], device=dev)[:, None]
            hi = torch.tensor(table[sids, 2 * a + 1], device=dev)[:, None]
            kd.append(torch.where(t[None] < 0, lo, torch.where(t[None] >= shape[a], hi, torch.zeros_like(lo))))
        return idx, kd

    def take(U, idx):
        return U[:, idx[2][:, :, None, None], idx[1][:, None, :, None], idx[0][:, None, None, :]]

    def ext_state(Ucur, sids, shape, depth, table_k):
        """The sub-domains' points and halos: the current values on synchronous steps, otherwise
        the halo from the delayed levels with the weights table_k[k][l]."""
        idx, kd = window(sids, depth, shape)
        E = take(Ucur, idx)
        if not asyn:
            return E
        k = torch.maximum(torch.maximum(kd[2][:, :, None, None], kd[1][:, None, :, None]), kd[0][:, None, None, :])
        H = torch.zeros_like(E)
        for back in range(c.kmax + C):
            wt = torch.tensor([table_k[kk][back - kk] if 0 <= back - kk < C else 0.0 for kk in range(c.kmax + 1)], dtype=torch.float64, device=dev)
            H += wt[k] * take(levels[back], idx)
        inner = (slice(None), slice(None)) + tuple(slice(depth[a], depth[a] + shape[a]) for a in (2, 1, 0))
        H[inner] = E[inner]
        return H

    def put(U, vals, sids, shape):
        idx, _ = window(sids, (0, 0, 0), shape)
        U[:, idx[2][:, :, None, None], idx[1][:, None, :, None], idx[0][:, None, None, :]] = vals

    W = _halo_weights(c.order, c.kmax)
    Wf = [_lagrange(k + 1, C) for k in range(c.kmax + 1)]
    U = levels[0]
    for _ in range(steps):
        Q = torch.zeros_like(U)
        for m in range(len(A)):
            R = torch.empty_like(U)
            for shape, lists in groups.items():
                for sids in lists:
                    E = ext_state(U, sids, shape, (G, G, Gz), [W[k][m] for k in range(c.kmax + 1)])
                    put(R, _rhs(c, E, G, Gz), sids, shape)
            Q = A[m] * Q + c.dt * R
            U = U + B[m] * Q
        if c.filter:
            for a in range(dims):
                V = torch.empty_like(U)
                for shape, lists in groups.items():
                    for sids in lists:
                        depth = [0, 0, 0]
                        depth[a] = 5
                        E = ext_state(U, sids, shape, depth, Wf)
                        put(V, _filter_line(E, -1 - a, shape[a], c.alpha_f), sids, shape)
                U = V
    return U


def _gelu(z):
    return 0.5 * z * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (z + 0.044715 * z ** 3)))


def _layers(p):
    cut = np.cumsum([64 * 65, 64, 64 * 64, 64, 20 * 64])
    w = torch.tensor_split(p, [int(q) for q in cut])
    return w[0].view(64, 65), w[1], w[2].view(64, 64), w[3], w[4].view(20, 64), w[5]


def _network_out(p, x):
    W1, b1, W2, b2, W3, b3 = _layers(p)
    h = _gelu(x @ W1.T + b1)
    h = _gelu(h @ W2.T + b2)
    return h @ W3.T + b3


def _exact_train(case, seed):
    x, t, p, m, v = _train_setup(case, seed)
    x, t = x.double(), t.double()
    p, m, v = (q.double().to(x.device) for q in (p, m, v))
    B, losses = case["batch"], []
    for it in range(case["iters"]):
        q = p.clone().requires_grad_(True)
        loss = ((_network_out(q, x[it * B:(it + 1) * B]) - t[it * B:(it + 1) * B]) ** 2).mean()
        g, = torch.autograd.grad(loss, q)
        losses.append(loss.detach())
        step = FIRST_UPDATE + it
        m = ADAM["beta1"] * m + (1 - ADAM["beta1"]) * g
        v = ADAM["beta2"] * v + (1 - ADAM["beta2"]) * g * g
        mh, vh = m / (1 - ADAM["beta1"] ** step), v / (1 - ADAM["beta2"] ** step)
        p = p - ADAM["lr"] * (mh / (torch.sqrt(vh) + ADAM["eps"]) + ADAM["wd"] * p)
    return {"params": p, "m": m, "v": v, "grad": g, "loss": torch.stack(losses)}


def _exact_diag(case, seed):
    c = _case_of(_cart(None, 3, case["n"], case["p"], "SA"))
    U = _fields(c, seed, 0.0)
    vel = [U[1 + q] / U[0] for q in range(3)]

    def d(f, axis, h):
        return (8.0 * (torch.roll(f, -1, axis) - torch.roll(f, 1, axis)) - (torch.roll(f, -2, axis) - torch.roll(f, 2, axis))) / (12.0 * h)
    wx = d(vel[2], 1, c.dy) - d(vel[1], 0, c.dz)
    wy = d(vel[0], 0, c.dz) - d(vel[2], 2, c.dx)
    wz = d(vel[1], 2, c.dx) - d(vel[0], 1, c.dy)
    K = 0.5 * (U[0] * (vel[0] ** 2 + vel[1] ** 2 + vel[2] ** 2)).mean()
    ens = 0.5 * (U[0] * (wx ** 2 + wy ** 2 + wz ** 2)).mean()
    # (the totals of the momentum cancel to nothing but rounding: they have no value to be held to)
    return {"mean": torch.stack([K, ens]), "totals": None, "bad": None}


def exact(case, seed):
    kind = case["kind"]
    if kind == "cart":
        c = _case_of(case)
        return {"U": [_exact_steps(c, seed, case["steps"], _start_step(c))]}
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "predict":
        x, _ = _samples(seed, case["samples"])
        return {"y": _network_out(torch.from_numpy(_network(seed)).double().to(x.device), x.double())}
    if kind == "diag":
        return _exact_diag(case, seed)
    return None
