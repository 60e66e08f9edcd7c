"""What a program has this library do, as cases that can be timed and compared.

A case is a box (or a batch of boxes) of cosmic rays, what it is loaded with,
and the calls one pass makes through the public entry points:

``run``      ``mhdpic_run``: the production loop, several steps with a sort
             every few of them, on the program's own stream;
``steps``    the same step stage by stage, with the corrector deposit and the
             four-velocities read back (a program that looks at its particles);
``subcycle`` several particle sub-steps per gas step with the gas in pinned
             host memory and the conserved totals asked for (a host MHD solver
             coupled to the push, App. A.4 of arXiv:1412.1087);
``coupled``  the predictor-corrector step with the plane-parallel gas model;
``inject``   the shock box with the open inflow face: front tracking and
             injection, then the step;
``diagnose`` what a run writes out now and then: spectra, the Lambda map and
             the charge and current densities at the present positions;
``noalloc``  the charge and current deposit for callers that may not allocate.

Sizes are those of the library's own workloads and tests, or smaller and
ragged ones between.  Inputs are drawn on the GPU from the seed.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1412_1087_gb300 import mhdpic as m

PERIODIC, REFLECT, WALL_OPEN = 0, 1, 2
DEV = "cuda:0"
ETA, E_FACTOR, GAMMA_GAS, INJ_SEED = 2e-3, 10.0, 5.0 / 3.0, 77
NBINS, N_MOMENT = 64, 6
CHUNK = 1 << 23   # particles the 64-bit evaluation holds at once


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _case(kind, load, n, ppc, **kw):
    c = {"kind": kind, "load": load, "ndim": 3 if n[2] > 1 else 2, "nx": n[0], "ny": n[1], "nz": n[2], "ppc": float(ppc),
         "boxes": 1, "fp64": False, "hall": load == "bell", "steps": 1, "every": 1, "nsub": 1}
    c.update(kw)
    return c


def listed():
    named = [
        # a small test box, the smallest call: launches and latency
        ("thermal 64x64", _case("run", "thermal", (64, 64, 1), 16, steps=8, every=4)),
        # a small 3-D box stepped stage by stage with read-back, ragged sides
        ("beam small, by stages", _case("steps", "beam", (26, 22, 30), 8)),
        # the production 3-D box
        ("beam 128^3", _case("run", "beam", (128, 128, 128), 32, steps=2, every=1)),
        # the Bell-instability box with the CR-Hall term, ragged sides
        ("bell 1000x700", _case("run", "bell", (1000, 700, 1), 64, steps=8, every=4)),
        # the shock-shaped load: most particles in a few crowded cells at the wall
        ("shock at the wall", _case("run", "wall", (4096, 128, 1), 40, steps=8, every=4)),
        # many independent boxes of very different sizes in one context
        ("ensemble of 24", _case("run", "ensemble", (32, 512, 1), 34, steps=6, every=3, boxes=24)),
        # front tracking and injection with the step that follows
        ("shock front, injection", _case("inject", "front", (2048, 96, 1), 24)),
        # the FP64 path, stage by stage
        ("beam FP64", _case("steps", "beam", (48, 48, 48), 16, fp64=True)),
        # sub-cycled particles under a host gas solver
        ("beam 64^3, 5 sub-steps", _case("subcycle", "beam", (64, 64, 64), 32, nsub=5)),
        # the predictor-corrector step with the CR-Hall term
        ("coupled 700x500", _case("coupled", "bell", (700, 500, 1), 16)),
        # output time of a run
        ("diagnostics", _case("diagnose", "bell", (512, 512, 1), 64)),
        # the deposit without allocations, ragged 3-D box
        ("deposit, no allocation", _case("noalloc", "beam", (60, 50, 56), 24)),
    ]
    return [dict(c, name=name) for name, c in named]


def draw(rng):
    def between(lo, hi):   # whole number, uniform over its logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["run", "run", "run", "steps", "subcycle", "coupled", "inject", "diagnose", "noalloc"])
    most = {"run": 40e6, "steps": 4e6, "subcycle": 8e6, "coupled": 8e6, "inject": 12e6, "diagnose": 20e6, "noalloc": 3e6}[kind]
    load = {"run": rng.choice(["thermal", "beam", "bell", "wall", "ensemble"]), "steps": rng.choice(["thermal", "beam", "bell", "wall"]),
            "subcycle": rng.choice(["beam", "bell"]), "coupled": "bell", "inject": "front", "diagnose": rng.choice(["bell", "beam"]),
            "noalloc": rng.choice(["thermal", "beam", "wall"])}[kind]
    ppc = between(4, 64)
    kw = {"fp64": rng.random() < {"run": 0.15, "steps": 0.4, "diagnose": 0.4, "noalloc": 0.4}.get(kind, 0.0)}
    if kw["fp64"]:
        most /= 4
    if load == "ensemble":
        n = (32, between(64, 384), 1)
        kw["boxes"] = max(2, min(between(4, 64), int(most / (0.2 * n[1] * n[1] * ppc))))
    else:
        cells = between(3000, max(3001, int(most / ppc)))
        if kind == "noalloc":
            cells = min(cells, 200000)
        if load == "beam":
            a, b = rng.uniform(0.7, 1.4), rng.uniform(0.7, 1.4)
            s = cells ** (1.0 / 3.0)
            n = (max(8, int(s * a)), max(8, int(s * b)), max(8, int(s / (a * b))))
        else:
            r = rng.uniform(8.0, 32.0) if load in ("wall", "front") else rng.uniform(0.5, 2.0)
            n = (max(64 if load in ("wall", "front") else 16, int(math.sqrt(cells * r))), max(8, int(math.sqrt(cells / r))), 1)
    if kind == "run":
        kw["every"] = rng.choice([1, 2, 3, 4]) if load != "beam" else rng.choice([1, 1, 2])
        kw["steps"] = 2 * kw["every"]
    if kind == "subcycle":
        kw["nsub"] = rng.choice([3, 5])
    if load == "bell" and kind not in ("coupled", "run"):
        kw["hall"] = rng.random() < 0.5
    return _case(kind, load, n, ppc, **kw)


def _sides(case):
    """(nx, ny, nz) and particles per cell of every box: an ensemble's sides run
    from nx to ny, evenly over their logarithm, the particles per cell beside them."""
    if case["load"] != "ensemble":
        return [((case["nx"], case["ny"], case["nz"]), case["ppc"])]
    out = []
    for b in range(case["boxes"]):
        u, w = math.modf(0.5 + b * 0.6180339887498949)[0], math.modf(0.25 + b * 0.7548776662466927)[0]
        side = int(round(case["nx"] * (case["ny"] / case["nx"]) ** u))
        out.append(((side, side, 1), max(2.0, float(int(case["ppc"] * (0.15 + 1.7 * w))))))
    return out


def _sizes(case):
    cells = sum(n[0] * n[1] * n[2] for n, _ in _sides(case))
    parts = sum(int(round(p * n[0] * n[1] * n[2])) for n, p in _sides(case))
    return parts, cells


def work(case):
    np_, nc = _sizes(case)
    d, kind = case["ndim"], case["kind"]
    part = 8 * (d + 3) if case["fp64"] else 32   # one particle's state
    nodes = 3 ** d
    push = nodes * 28 + 250                      # gather 6, deposit 8 channels, the step itself
    if kind == "noalloc":
        return {"bytes": np_ * part + 32 * nc, "flops": np_ * (nodes * 8 + 60)}
    if kind == "diagnose":   # two spectra, the map, the deposit
        vel = 24 if case["fp64"] else 16
        return {"bytes": np_ * (vel + 2 * part) + nc * (8 * 15 + 48), "flops": np_ * (nodes * 8 + 160)}
    steps = case["steps"] * case["nsub"]
    # every sub-step reads and writes the particles; every step reads the gas, writes what the feedback changes
    # and the moments
    cell = 96 + 32 + (64 if kind == "coupled" else 0)
    return {"bytes": 2 * part * np_ * steps + cell * nc * case["steps"], "flops": np_ * steps * push + 100 * nc * case["steps"]}


def tolerance(case):
    """About four times the error against 64 bits that the cases show."""
    if case["kind"] == "noalloc":   # double arithmetic, sums in 62-bit fixed point: 7e-15
        return {"rel": 1e-12}
    if case["fp64"]:   # the same, the corrector's scale sized by a bound: 5e-14
        return {"rel": 4e-13}
    # 32-bit positions, fields and push: 1e-7 to 4.5e-7 in the deposits
    return {"rel": 2e-6}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

LOADS = {   # C, |p| or its range, drift of the particles along x
    "thermal": (100.0, 10.0, 0.0), "beam": (300.0, 100.0, 10.0), "bell": (300.0, (10.0, 1e4), 0.5),
    "wall": (200.0, (1.0, 1e5), 0.0), "front": (200.0, (1.0, 1e5), 0.0), "ensemble": (100.0, 10.0, 0.0),
}


def _waves(gen, n, ndim, rms, modes=24):
    """Transverse waves of random phase on a periodic box, (3, cells), of the given rms amplitude."""
    dB = torch.zeros(3, n[2], n[1], n[0], dtype=torch.float64, device=DEV)
    x = [torch.arange(n[d], dtype=torch.float64, device=DEV) + 0.5 for d in range(3)]
    k = torch.randint(-4, 5, (modes, 3), generator=gen, device=DEV).cpu().numpy().astype(float)
    ph = torch.rand(modes, generator=gen, device=DEV, dtype=torch.float64).cpu().numpy() * 2 * np.pi
    for i in range(modes):
        kv = 2 * np.pi * k[i] / np.array(n)
        if ndim == 2:
            kv[2] = 0.0
        if not kv.any():
            kv[1] = 2 * np.pi / n[1]
        e = np.cross(kv, [1.0, 0.0, 0.0]) if ndim == 3 else np.array([0.0, 0.0, 1.0])
        e = e / np.linalg.norm(e) if np.linalg.norm(e) > 0 else np.array([0.0, 0.6, 0.8])
        w = torch.cos(kv[0] * x[0][None, None, :] + kv[1] * x[1][None, :, None] + kv[2] * x[2][:, None, None] + ph[i])
        for d in range(3):
            if e[d]:
                dB[d] += (rms * math.sqrt(2.0 / modes) * e[d]) * w
    return dB.reshape(3, -1)


def _momenta(gen, npart, load):
    C, mag, V = LOADS[load]
    g = torch.randn(3, npart, generator=gen, device=DEV, dtype=torch.float32).double()
    g /= g.square().sum(0).sqrt().clamp_min(1e-30)
    if isinstance(mag, tuple):   # dN/dp ~ p^-2
        u = torch.rand(npart, generator=gen, device=DEV, dtype=torch.float64)
        g *= 1.0 / (1.0 / mag[0] - u * (1.0 / mag[0] - 1.0 / mag[1]))
    else:
        g *= mag
    if V:   # the drift frame moves at V along x
        gam = (1.0 + g.square().sum(0) / (C * C)).sqrt()
        g[0] = (g[0] + V * gam) / math.sqrt(1.0 - V * V / (C * C))
    return g.float()


def _box(gen, case, n, ppc):
    """One box: sizes, boundaries, parameters, gas (float64) and particles (cell, offsets, four-velocity)."""
    load, ndim = case["load"], case["ndim"]
    nc = n[0] * n[1] * n[2]
    npart = int(round(ppc * nc))
    C = LOADS[load][0]
    f64 = dict(dtype=torch.float64, device=DEV)
    B = torch.zeros(3, nc, **f64)
    B[0] = 1.0
    rho = torch.ones(nc, **f64)
    vel = torch.zeros(3, nc, **f64)
    P = torch.ones(nc, **f64)
    xc = (torch.arange(nc, device=DEV) % n[0]).double() + 0.5
    if load in ("beam", "ensemble"):
        dB = _waves(gen, n, ndim, 0.1 if load == "beam" else 0.2)
        B, vel = B + dB, vel - dB
    elif load in ("thermal", "bell"):
        dB = _waves(gen, n, ndim, 0.05)
        B, vel = B + dB, vel + 0.3 * torch.randn(3, nc, generator=gen, **f64)
    elif load == "wall":
        vel[0] = -20.0
        vel = vel + 0.3 * torch.randn(3, nc, generator=gen, **f64)
    elif load == "front":   # strong-shock state behind x = nx/4, inflow at -20 ahead
        down = xc < 0.25 * n[0]
        rho = torch.where(down, 4.0, 1.0).double()
        vel[0] = torch.where(down, 0.0, -20.0).double()
        P = torch.where(down, 4.0 / 3.0 * 400.0, 1.0).double()
    egas = P / (GAMMA_GAS - 1.0) + 0.5 * rho * vel.square().sum(0) + 0.5 * B.square().sum(0)
    s = torch.rand(ndim, npart, generator=gen, device=DEV, dtype=torch.float32).double()
    s += 2.0 ** -25 * torch.rand(ndim, npart, generator=gen, device=DEV, dtype=torch.float32).double()
    if load in ("wall", "front"):   # 80% of the particles in the 5% of the cells at the wall
        dense = torch.rand(npart, generator=gen, device=DEV) < 0.8
        s[0] = torch.where(dense, 0.05 * s[0], 0.05 + 0.95 * s[0])
    idx, off = [], []
    for d in range(ndim):
        sd = s[d] * n[d]
        i = sd.floor()
        off.append((sd - i).float().clamp_max(1.0 - 2.0 ** -24))
        idx.append(i.long().clamp_max(n[d] - 1))
    cell = idx[0] + n[0] * idx[1] + (n[0] * n[1] * idx[2] if ndim == 3 else 0)
    off = torch.stack(off)
    p = _momenta(gen, npart, load)
    if load == "front":   # free slots for the injected particles
        free = npart // 4
        cell = torch.cat([cell, torch.full((free,), -1, device=DEV)])
        off = torch.cat([off, torch.zeros(ndim, free, device=DEV)], dim=1)
    gam = (1.0 + p.double().square().sum(0) / (C * C)).sqrt()
    dt = min(0.4 / float((p.double() / gam).abs().max()), 0.3 * float(gam.min()) / float(B.square().sum(0).max().sqrt()))
    if load == "front":
        p = torch.cat([p, torch.zeros(3, free, device=DEV)], dim=1)
    bc = ({"wall": REFLECT, "front": WALL_OPEN}.get(load, PERIODIC), PERIODIC, PERIODIC)
    return {"n": n, "bc": bc, "ndim": ndim, "C": C, "m": 1e-3 / ppc, "hall": int(case["hall"]), "dt": dt, "rho": rho,
            "mom": rho * vel, "egas": egas, "B": B, "cell": cell.int(), "off": off, "p": p}


def _inputs(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) * 7919 + 17)
    return [_box(gen, case, n, ppc) for n, ppc in _sides(case)]


# ---------------------------------------------------------------------------
# what a program holds: its buffers, its stream and the context over them
# ---------------------------------------------------------------------------

class State:
    def __init__(self, case, boxes):
        self.case, self.ctx = case, None
        nb, fp64 = len(boxes), case["fp64"]
        self.G, self.P = (m.Grid * nb)(), (m.Params * nb)()
        for g, p, b in zip(self.G, self.P, boxes):
            g.ndim = b["ndim"]
            for d in range(3):
                g.n[d], g.dx[d], g.x0[d], g.bc[d] = b["n"][d], 1.0, 0.0, b["bc"][d]
            p.qm_cr, p.qm_gas, p.C, p.m_cr, p.hall, p.shape = 1.0, 1.0, b["C"], b["m"], b["hall"], m.MHDPIC_SHAPE_TSC
        self.np = sum(b["cell"].shape[0] for b in boxes)
        self.nc = sum(b["rho"].shape[0] for b in boxes)
        self.start = np.concatenate([[0], np.cumsum([b["cell"].shape[0] for b in boxes])]).astype(np.int64)
        self.pos = self.vel = self.x = self.p64 = None
        if fp64:
            self.x = torch.cat([_positions(b) for b in boxes], dim=1)
            self.p64 = torch.cat([b["p"].double() for b in boxes], dim=1)
        else:
            self.pos = torch.zeros(self.np, 4, dtype=torch.int32, device=DEV)
            self.vel = torch.zeros(self.np, 4, dtype=torch.float32, device=DEV)
            for b, s, e in zip(boxes, self.start[:-1], self.start[1:]):
                self.pos[s:e, 0] = b["cell"]
                self.pos.view(torch.float32)[s:e, 1:1 + b["ndim"]] = b["off"].t()
                self.vel[s:e, :3] = b["p"].t()
        host = case["kind"] == "subcycle"
        gas = [torch.cat([b[k] for b in boxes], dim=-1) for k in ("rho", "mom", "egas", "B")]
        self.rho, self.mom, self.egas, self.B = [g.cpu().pin_memory() if host else g.contiguous() for g in gas]
        self.dt = min(b["dt"] for b in boxes)
        if case["kind"] == "noalloc":
            self.out = torch.empty(4, self.nc, dtype=torch.float64, device=DEV)
            return
        opt = m.Options()
        opt.precision = m.MHDPIC_PREC_FP64 if fp64 else m.MHDPIC_PREC_MIXED
        opt.memory = m.MHDPIC_MEM_HOST_GAS if host else m.MHDPIC_MEM_DEVICE
        parts = m.Particles()
        parts.np = self.np
        parts.box_start = self.start.ctypes.data_as(ctypes.POINTER(ctypes.c_int64))
        ptr = lambda t: None if t is None else t.data_ptr()  # noqa: E731
        parts.pos, parts.vel, parts.x, parts.p64 = ptr(self.pos), ptr(self.vel), ptr(self.x), ptr(self.p64)
        g = m.Gas(ptr(self.rho), ptr(self.mom), ptr(self.egas), ptr(self.B))
        # the production loop has a stream of its own (its steps are replayed
        # as a graph); the calls stage by stage share torch's
        self.stream = torch.cuda.Stream() if case["kind"] == "run" else torch.cuda.current_stream()
        torch.cuda.synchronize()
        self.ctx = m.mhdpic_init(nb, self.G, self.P, opt, parts, g, ctypes.c_void_p(self.stream.cuda_stream))
        f64 = dict(dtype=torch.float64, device=DEV)
        self.moments = torch.empty(4, self.nc, **f64)
        if case["kind"] in ("run", "steps", "subcycle"):
            m.mhdpic_set_sort_lookahead(self.ctx, 0.5 * self.dt)
        if case["kind"] == "subcycle":
            m.mhdpic_set_subcycle_sort(self.ctx, 1)
            self.totals = np.zeros(8 * nb)
        if case["kind"] == "steps":
            self.corr, self.v = torch.empty(4, self.nc, **f64), torch.empty(3, self.np, **f64)
        if case["kind"] == "diagnose":
            lo, hi = _spectrum_range(case)
            self.edges = np.geomspace(lo, hi, NBINS + 1)
            self.region = np.array([0.0, 0.5 * case["nx"], 0.25 * case["ny"], case["ny"], 0.0, case["nz"]], dtype=np.float64)
            self.counts = np.zeros((2, nb * NBINS), dtype=np.int64)
            self.sums = np.zeros((2, 2 * nb))
            self.lam = torch.empty(3, self.nc, **f64)

    def __del__(self):
        if self.ctx is not None:
            m.mhdpic_destroy(self.ctx)
            self.ctx = None


def _spectrum_range(case):
    return (5.0, 2e4) if case["load"] == "bell" else (40.0, 200.0)


def prepare(case, seed):
    return State(case, _inputs(case, seed))


def run(s):
    case, ctx, dt = s.case, s.ctx, s.dt
    kind = case["kind"]
    if kind == "run":
        m.mhdpic_run(ctx, dt, case["steps"], case["every"])
        m.mhdpic_get_deposits(ctx, 1, s.moments.data_ptr())
        return {"mom": s.mom, "egas": s.egas, "moments": s.moments}
    if kind == "steps":
        m.mhdpic_interp_push(ctx, dt, 1)
        m.mhdpic_get_deposits(ctx, 0, s.corr.data_ptr())
        m.mhdpic_get_deposits(ctx, 1, s.moments.data_ptr())
        m.mhdpic_apply_feedback(ctx)
        m.mhdpic_get_velocities(ctx, s.v.data_ptr())
        m.mhdpic_sort(ctx)
        return {"corr": s.corr, "mom": s.mom, "egas": s.egas, "moments": s.moments, "v": s.v}
    if kind == "subcycle":
        m.mhdpic_interp_push(ctx, dt, case["nsub"])
        m.mhdpic_apply_feedback(ctx, s.totals)
        m.mhdpic_sort(ctx)
        m.mhdpic_get_deposits(ctx, 1, s.moments.data_ptr())
        return {"mom": s.mom, "egas": s.egas, "moments": s.moments, "totals": s.totals}
    if kind == "coupled":
        m.mhdpic_gas_predict(ctx, dt, m.MHDPIC_GAS_LINEAR_X)
        m.mhdpic_interp_push(ctx, dt, 1)
        m.mhdpic_gas_correct(ctx, dt, m.MHDPIC_GAS_LINEAR_X)
        m.mhdpic_sort(ctx)
        m.mhdpic_get_deposits(ctx, 1, s.moments.data_ptr())
        return {"mom": s.mom, "egas": s.egas, "B": s.B, "moments": s.moments}
    if kind == "inject":
        n, xs, xt = m.mhdpic_inject(ctx, dt, ETA, E_FACTOR, GAMMA_GAS, INJ_SEED)
        m.mhdpic_interp_push(ctx, dt, 1)
        m.mhdpic_apply_feedback(ctx)
        m.mhdpic_get_deposits(ctx, 1, s.moments.data_ptr())
        return {"n": n, "front": xs, "tail": xt, "rho": s.rho, "mom": s.mom, "egas": s.egas, "moments": s.moments}
    if kind == "diagnose":
        m.mhdpic_spectrum(ctx, m.MHDPIC_SPEC_ENERGY, s.edges, None, N_MOMENT, s.counts[0], s.sums[0])
        m.mhdpic_spectrum(ctx, m.MHDPIC_SPEC_MOMENTUM, s.edges, s.region, 1, s.counts[1], s.sums[1])
        m.mhdpic_lambda_map(ctx, s.lam.data_ptr())
        m.mhdpic_deposit(ctx)
        m.mhdpic_get_deposits(ctx, 1, s.moments.data_ptr())
        return {"counts": s.counts, "sums": s.sums, "lambda": s.lam, "moments": s.moments}
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    ptr = lambda t: 0 if t is None else t.data_ptr()  # noqa: E731
    m.mhdpic_deposit_moments_noalloc(s.G[0], s.P[0], m.MHDPIC_PREC_FP64 if case["fp64"] else m.MHDPIC_PREC_MIXED, s.np,
                                     pos=ptr(s.pos), vel=ptr(s.vel), x=ptr(s.x), p64=ptr(s.p64), out=s.out.data_ptr(), stream=st)
    return {"moments": s.out}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _positions(b):
    n, c = b["n"], b["cell"].long()
    i = [c % n[0], (c // n[0]) % n[1], c // (n[0] * n[1])]
    x = torch.stack([i[d].double() + b["off"][d].double() for d in range(b["ndim"])])
    x[0, c < 0] = math.nan
    return x


def _fold(i, n, bc):
    """Stencil cells beyond the box: periodic image, mirror image at a wall, the last cell beyond an open face."""
    if bc == PERIODIC:
        return i % n
    i = torch.where(i < 0, -1 - i, i)
    return i.clamp_max(n - 1) if bc == WALL_OPEN else torch.where(i >= n, 2 * n - 1 - i, i)


def _stencil(b, x):
    """(cells, weights) of every node of the quadratic spline."""
    n, D = b["n"], b["ndim"]
    per = []
    for d in range(D):
        i = x[d].floor()
        o = x[d] - i
        w = (0.5 * (1 - o) ** 2, 0.75 - (o - 0.5) ** 2, 0.5 * o * o)
        per.append([(_fold(i.long() + k - 1, n[d], b["bc"][d]), w[k]) for k in range(3)])
    for cz in range(3 if D == 3 else 1):
        for iy, wy in per[1]:
            for ix, wx in per[0]:
                g, w = ix + n[0] * iy, wx * wy
                if D == 3:
                    g, w = g + n[0] * n[1] * per[2][cz][0], w * per[2][cz][1]
                yield g, w


def _gamma(b, v):
    return (b["C"] ** 2 + v.square().sum(0)).sqrt() / b["C"]


def _drift(b, x, v, g, dt):
    """Half a step with the particle boundaries; which particles reach the open face."""
    gone = torch.zeros(x.shape[1], dtype=torch.bool, device=x.device)
    for d in range(b["ndim"]):
        L = float(b["n"][d])
        xd = x[d] + 0.5 * dt * v[d] / g
        if b["bc"][d] == PERIODIC:
            xd = torch.remainder(xd, L)
            xd = torch.where(xd >= L, 0.0, xd)
        else:
            low = xd < 0
            xd = torch.where(low, -xd, xd)
            v[d] = torch.where(low, -v[d], v[d])
            high = xd >= L
            if b["bc"][d] == WALL_OPEN:
                gone |= high
            else:
                xd = torch.where(high, 2 * L - xd, xd)
                v[d] = torch.where(high, -v[d], v[d])
            xd = torch.where(xd >= L, math.nextafter(L, 0.0), xd)
        x[d] = xd
    return gone


def _deposit_moments(b, x, v, out):
    g = _gamma(b, v)
    q = b["m"] * torch.cat([torch.ones_like(g)[None], v / g]).t()
    for node, w in _stencil(b, x):
        out.index_add_(0, node, w[:, None] * q)


def _moments(b, x, v):
    out = torch.zeros(b["rho"].shape[0], 4, dtype=torch.float64, device=DEV)
    for a in range(0, x.shape[1], CHUNK):
        live = ~torch.isnan(x[0, a:a + CHUNK])
        _deposit_moments(b, x[:, a:a + CHUNK][:, live], v[:, a:a + CHUNK][:, live], out)
    return out


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


def _force(b, rho, mom, B, mo, hall):
    """E0, the force on the particles per volume and the energy handed over per volume and time."""
    n, J = mo[:, 0], mo[:, 1:].t()
    E0 = -_cross(mom / rho, B)
    R = n / (rho + n) if hall else torch.zeros_like(n)
    return E0, (1 - R) * (n * E0 + _cross(J, B)), (1 - R) * (J * E0).sum(0)


def _field(b, rho, mom, B, mo):
    E0, F, _ = _force(b, rho, mom, B, mo, b["hall"])
    return torch.cat([E0 - F / rho if b["hall"] else E0, B]).t().contiguous()


def _push(b, x, v, F, dt, last=True):
    """One particle step in the cell fields F: the corrector deposit and, with `last`, the moments; x and v in place."""
    nc = F.shape[0]
    corr = torch.zeros(nc, 4, dtype=torch.float64, device=DEV)
    mo = torch.zeros(nc, 4, dtype=torch.float64, device=DEV)
    for a in range(0, x.shape[1], CHUNK):
        live = (~torch.isnan(x[0, a:a + CHUNK])).nonzero()[:, 0] + a
        xs, vs = x[:, live], v[:, live]
        gone = _drift(b, xs, vs, _gamma(b, vs), dt)
        f = torch.zeros(xs.shape[1], 6, dtype=torch.float64, device=DEV)
        for node, w in _stencil(b, xs):
            f += w[:, None] * F[node]
        E, Bf = f[:, :3].t(), f[:, 3:].t()
        B2 = Bf.square().sum(0)
        E = E - torch.where(B2 > 0, (E * Bf).sum(0) / B2, 0.0) * Bf
        e = 0.5 * dt * E
        v0 = vs + e
        bb = 0.5 * dt * Bf / _gamma(b, v0)
        rot = 2.0 * _cross(v0 + _cross(v0, bb), bb) / (1.0 + bb.square().sum(0))
        v1 = v0 + rot
        vn = v1 + e
        dE = (e * (vn + v1)).sum(0) / (_gamma(b, vn) + _gamma(b, v1)) + (e * (v0 + vs)).sum(0) / (_gamma(b, v0) + _gamma(b, vs))
        q = -b["m"] * torch.cat([2 * e + rot, dE[None]]).t()
        for node, w in _stencil(b, xs):
            corr.index_add_(0, node, w[:, None] * q)
        gone |= _drift(b, xs, vn, _gamma(b, vn), dt)
        if last:
            _deposit_moments(b, xs[:, ~gone], vn[:, ~gone], mo)
        xs[0, gone] = math.nan
        x[:, live], v[:, live] = xs, vn
    return corr, mo


def _order(b):
    """The library's particle order: stable by 4x4x4 or 8x8 brick, then by cell in the brick."""
    n, D, c = b["n"], b["ndim"], b["cell"].long()
    i = [c % n[0], (c // n[0]) % n[1], c // (n[0] * n[1])]
    w = (4, 4, 4) if D == 3 else (8, 8, 1)
    nb = [(n[d] + w[d] - 1) // w[d] for d in range(3)]
    brick = (i[2] // w[2] * nb[1] + i[1] // w[1]) * nb[0] + i[0] // w[0]
    cell = (i[2] % w[2] * w[1] + i[1] % w[1]) * w[0] + i[0] % w[0]
    return torch.sort(brick * (w[0] * w[1] * w[2]) + cell, stable=True)[1]


def _philox(n, key):
    """Philox4x32-10 with counters (k, 0, 0, 0) as uniform numbers in (0, 1), (4, n)."""
    M = np.uint64(0xffffffff)
    x = [np.arange(n, dtype=np.uint64)] + [np.zeros(n, dtype=np.uint64) for _ in range(3)]
    k0, k1 = key & 0xffffffff, key >> 32
    for _ in range(10):
        a, c = x[0] * np.uint64(0xD2511F53), x[2] * np.uint64(0xCD9E8D57)
        x = [(c >> np.uint64(32)) ^ x[1] ^ np.uint64(k0), c & M, (a >> np.uint64(32)) ^ x[3] ^ np.uint64(k1), a & M]
        k0, k1 = (k0 + 0x9E3779B9) & 0xffffffff, (k1 + 0xBB67AE85) & 0xffffffff
    return (np.stack(x).astype(np.float64) + 0.5) / 4294967296.0


def _inject(b, dt):
    """Front, tail and the particles injected in the first call, the gas compensated in place."""
    nx, ny = b["n"][0], b["n"][1]
    rho, mom, egas, B = (b[k].cpu().numpy() for k in ("rho", "mom", "egas", "B"))
    vx = mom[0] / rho
    P = (GAMMA_GAS - 1) * (egas - 0.5 * (mom * mom).sum(0) / rho - 0.5 * (B * B).sum(0))
    ker = np.exp(-0.5 * np.arange(-12, 13) ** 2 / 16.0)
    norm = np.convolve(np.ones(nx), ker, "same")
    vx, r, P = (np.convolve(a.reshape(ny, nx).mean(0), ker, "same") / norm for a in (vx, rho, P))
    vup, rup = vx[-1], r[-1]
    i = int(np.nonzero(np.abs(vx[:-1]) <= 0.6 * abs(vup))[0].max())
    a, c = abs(vx[i]), abs(vx[i + 1])
    xs = i + 0.5 + (0.6 * abs(vup) - a) / (c - a)
    comp = (GAMMA_GAS + 1) / (GAMMA_GAS - 1)
    hit = np.nonzero(P[:i + 1] >= 2.0 / 3.0 * (comp / (comp - 1) * rup * vup * vup))[0]
    xt = hit.max() + 0.5 if hit.size else 0.0
    n = int(math.floor(ETA * rup * abs(vup) * dt * ny / b["m"]))
    u = _philox(n, INJ_SEED)
    C, Ek = b["C"], E_FACTOR * 0.5 * vup * vup
    mag = C * math.sqrt((1 + Ek / C ** 2) ** 2 - 1)
    mu, ph = 2 * u[2] - 1, 2 * np.pi * u[3]
    s = np.sqrt(1 - mu * mu)
    v = torch.from_numpy(mag * np.stack([mu, s * np.cos(ph), s * np.sin(ph)])).to(DEV)
    if n:
        xc = np.arange(nx) + 0.5
        cols = np.nonzero((xc >= xt) & (xc < xs))[0]
        cols = cols if cols.size else np.array([min(int(xs), nx - 1)])
        at = torch.from_numpy((np.arange(ny)[:, None] * nx + cols).reshape(-1)).to(DEV)
        share = b["m"] / at.numel()
        b["rho"][at] -= share * n
        for d in range(3):
            b["mom"][d, at] -= share * v[d].sum()
        b["egas"][at] -= share * (v.square().sum(0) / (_gamma(b, v) + 1)).sum()
    x = torch.from_numpy(np.stack([np.full(n, xs), u[0] * ny])).to(DEV)
    return n, xs, xt, x, v


def _spectra(b, case, x, v):
    lo, hi = _spectrum_range(case)
    edges = torch.from_numpy(np.geomspace(lo, hi, NBINS + 1)).to(DEV)
    v2 = v.square().sum(0)
    energy = v2 / ((b["C"] ** 2 + v2).sqrt() / b["C"] + 1)
    inside = (x[0] < 0.5 * case["nx"]) & (x[1] >= 0.25 * case["ny"])
    counts, sums = [], []
    for q, power in ((energy, N_MOMENT), (v2.sqrt()[inside], 1)):
        q = q[(q >= edges[0]) & (q < edges[-1])]
        counts.append(torch.bincount(torch.bucketize(q, edges, right=True) - 1, minlength=NBINS).cpu().numpy())
        sums.append([float((q ** (power + 1)).sum()), float((q ** power).sum())])
    return np.stack(counts), np.array(sums)


def exact(case, seed):
    boxes, kind = _inputs(case, seed), case["kind"]
    dt = min(b["dt"] for b in boxes)
    each = []
    for b in boxes:
        x, v = _positions(b), b["p"].double()
        if kind == "noalloc":
            return {"moments": _moments(b, x, v).t()}
        if kind == "diagnose":
            mo = _moments(b, x, v)
            counts, sums = _spectra(b, case, x, v)
            vA = (b["B"].square().sum(0) / b["rho"]).sqrt()
            lam = (mo[:, 1:].t() - mo[:, 0] * b["mom"] / b["rho"]) / ((b["rho"] + mo[:, 0]) * vA)
            return {"counts": counts, "sums": sums, "lambda": lam, "moments": mo.t()}
        o = _order(b) if kind == "steps" else None
        if o is not None:
            x, v = x[:, o].clone(), v[:, o].clone()
        rho, mom, egas, B = b["rho"], b["mom"], b["egas"], b["B"]
        mo = _moments(b, x, v)
        got = {}
        if kind == "inject":
            got["n"], got["front"], got["tail"], xi, vi = _inject(b, dt)
            live = ~torch.isnan(x[0])
            x, v = torch.cat([x[:, live], xi], dim=1), torch.cat([v[:, live], vi], dim=1)
            got["rho"] = rho
        for _ in range(case["steps"]):
            if kind == "coupled":
                E0, F, P = _force(b, rho, mom, B, mo, b["hall"])
                step = lambda f: 0.5 * (torch.roll(f.reshape(-1, b["n"][0]), -1, 1) - torch.roll(f.reshape(-1, b["n"][0]), 1, 1)).reshape(-1)  # noqa: E731

                def gas(mm, BB, H):
                    dm, dB, vg = torch.zeros_like(mm), torch.zeros_like(BB), mm / rho
                    for d in (1, 2):
                        dm[d], dB[d] = BB[0] * step(BB[d]), BB[0] * step(vg[d])
                    if b["hall"]:
                        dB[1] -= step(H[2])
                        dB[2] += step(H[1])
                    return dm, dB

                dm, dB = gas(mom, B, F / rho)
                mh, Bh = mom + 0.5 * dt * (dm - F), B + 0.5 * dt * dB
                corr, mo = _push(b, x, v, _field(b, rho, mh, Bh, mo), dt)
                dm, dB = gas(mh, Bh, -corr[:, :3].t() / dt / rho)
                mom, B, egas = mom + dt * dm + corr[:, :3].t(), B + dt * dB, egas + corr[:, 3]
                continue
            F, corr = _field(b, rho, mom, B, mo), 0.0
            for sub in range(case["nsub"]):
                part, mo = _push(b, x, v, F, dt, sub == case["nsub"] - 1)
                corr = corr + part
            mom, egas = mom + corr[:, :3].t(), egas + corr[:, 3]
        got.update(mom=mom, egas=egas, moments=mo.t())
        if kind == "coupled":
            got["B"] = B
        if kind == "steps":
            got.update(corr=corr.t(), v=v)
        if kind == "subcycle":
            kin = v.square().sum(0) / (_gamma(b, v) + 1)
            got["totals"] = torch.cat([mom.sum(1), egas.sum()[None], b["m"] * v.sum(1), (b["m"] * kin.sum())[None]])
        each.append(got)
    if len(each) == 1:
        return each[0]
    return {k: torch.cat([g[k] for g in each], dim=-1) for k in each[0]}
