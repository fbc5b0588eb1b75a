"""Performance cases of the framework: what its users have it do, through the
public entry points of paper_2403_17018_gb300.binding, over the range of
sizes, precisions and options that are used in earnest.

Every case is a dict of plain values; `kind` says which entry point it
drives. Implicit steps keep the length of the full workload (tau_0 = 1800 s
on level 0, halved per level; the paper's own field model 64 s); `nt0` is the
number of level-0 steps, so that a long horizon can be cut to a shorter one of
the same kind of steps.
"""
from __future__ import annotations

import math

import torch

from paper_2403_17018_gb300 import binding as hb
from paper_2403_17018_gb300.inputs import xi_batch, xi_halton

TAU0 = 1800.0          # level-0 step of the configurations [s]: 43200 s in 24 steps
TAU0_PAPER = 64.0      # level-0 step of the paper's own workload: 6016 s in 94 steps

# The multigrid schedules that the autotuner gives a user's program on this
# GPU, per precision and MLMC level 0, 1, ...: (vcycles, nu1, nu2,
# mg_small_cells, jac_lag, res_rows, mg_tb_cells, jac_keep)
TUNED = {
    "fp64": [(3, 2, 2, 128, 100, 0, 0, 1), (3, 2, 2, 128, 30, 0, 0, 0), (3, 2, 2, 512, 100, 0, 0, 1),
             (2, 2, 2, 512, 30, 2, 0, 1), (3, 2, 2, 512, 100, 0, 0, 1), (2, 2, 2, 512, 30, 0, 0, 1)],
    "fp32mg": [(3, 2, 2, 512, 100, 0, 0, 1), (3, 2, 2, 512, 30, 0, 2048, 0),
               (3, 2, 2, 512, 100, 0, 2048, 1), (2, 2, 2, 512, 30, 0, 2048, 1),
               (3, 2, 2, 512, 30, 0, 2048, 0), (2, 2, 2, 512, 30, 0, 2048, 1)],
}
SCHEDULE_FIELDS = ("vcycles", "nu1", "nu2", "mg_small_cells", "jac_lag", "res_rows", "mg_tb_cells",
                   "jac_keep")


def _case(kind, **kw):
    c = {"kind": kind, "nx0": 32, "ny0": 16, "nt0": 24, "level": 0, "batch": 1, "n_xi": 3,
         "precision": "fp64", "tuned": False, "field_model": 0, "krylov": 0}
    c.update(kw)
    return c


def listed():
    return [
        # a first deterministic solve with the default configuration: one
        # sample of the 32x16 grid over the whole horizon (latency)
        _case("solve", name="single-solve"),
        # the plain two-level configuration: 16 pairs on level 1 (64x32 and
        # 32x16), FP64, nothing tuned
        _case("pairs", name="two-level-pairs-fp64", level=1, batch=16),
        # the README's example: 64 pairs on level 2 (128x64 and 64x32) with
        # FP32 multigrid, nothing tuned
        _case("pairs", name="level2-pairs-fp32mg", level=2, batch=64, precision="fp32mg"),
        # one round of the four-level MLMC benchmark (1024/256/64/16 pairs)
        # and its level statistics, with tuned schedules, in both precisions
        _case("round", name="mlmc-round-fp64", levels=4, batch=1024, tuned=True),
        _case("round", name="mlmc-round-fp32mg", levels=4, batch=1024, precision="fp32mg", tuned=True),
        # level 4 (512x256) of the precision comparison, FP64 multigrid, tuned
        _case("solve", name="level4-solve-fp64", level=4, batch=16, nt0=2, tuned=True),
        # the finest pairs of the six-level MLMC run (1024x512 and 512x256),
        # six random variables, FP32 multigrid, tuned: operands beyond the L2
        _case("pairs", name="level5-pairs-fp32mg", level=5, batch=16, nt0=1, n_xi=6,
              precision="fp32mg", tuned=True),
        # backward: gradients of Q_S with respect to xi and the per-cell log K
        # of 256 samples on 128x64 cells, a checkpoint every 8 steps
        _case("adjoint", name="adjoint-level2", level=2, batch=256, nt0=4, precision="fp32mg", ckpt=8),
        # quasi-Monte Carlo with the paper's own field model: QoI time series
        # of Halton points on 128x64 cells
        _case("series", name="qmc-series-paper", level=2, batch=200, nt0=6, precision="fp32mg",
              field_model=1, every=8),
        # the paper's multiscale field with its own kind of linear solver,
        # BiCGStab preconditioned by multigrid, on 256x128 cells in FP64
        _case("solve", name="krylov-paper-level3", level=3, batch=16, nt0=1, field_model=1, krylov=2),
        # residual and exact Jacobian of given states (tools, other solvers)
        _case("resjac", name="residual-jacobian", nx0=512, ny0=256, batch=16),
        # statistics of a batch of 600 solved samples on 128x64 cells: QoI
        # moments, mean and variance fields, exceedance counts
        _case("stats", name="qmc-statistics", level=2, batch=600),
    ]


# Level-0 grids that coarsen to a direct solve, with cells of moderate aspect
_BASES = ((8, 4), (8, 3), (6, 3), (6, 4), (10, 3), (6, 5), (4, 3), (14, 2), (4, 2))


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("solve", "solve", "pairs", "pairs", "round", "adjoint", "series", "solve",
                       "resjac", "stats"))
    prec = rng.choice(("fp64", "fp32mg"))
    if kind == "resjac":
        nx, ny = 2 * _log_uniform(rng, 4, 300), _log_uniform(rng, 3, 300)
        return _case(kind, nx0=nx, ny0=ny, batch=max(1, min(200, _log_uniform(rng, 2 ** 9, 2 ** 21) // (nx * ny))),
                     precision="fp64")
    cx, cy = rng.choice(_BASES)
    if kind == "stats":
        level = rng.randint(0, 4)
        return _case(kind, nx0=4 * cx, ny0=4 * cy, level=level,
                     batch=max(2, min(4096, _log_uniform(rng, 2 ** 8, 2 ** 23) // (16 * cx * cy << (2 * level)))))
    k = rng.choice((1, 2, 2))
    nx0, ny0 = cx << k, cy << k
    cells0 = nx0 * ny0
    if kind == "round":
        levels = rng.randint(2, 4)
        top = cells0 << (2 * (levels - 1))
        # the benchmark's rule: a quarter of the samples on each finer level
        batch = max(4, min(1024, _log_uniform(rng, 2 ** 13, 2 ** 18) // cells0))
        return _case(kind, nx0=nx0, ny0=ny0, nt0=max(1, min(8, (1 << 19) // top)), levels=levels,
                     batch=batch, n_xi=rng.choice((3, 6)), precision=prec, tuned=True)
    most = 2 if kind == "adjoint" else 5
    level = rng.randint(1 if kind == "pairs" else 0, most)
    cells = cells0 << (2 * level)
    batch = max(1, min(1024, _log_uniform(rng, 2 ** 9, 2 ** 20) // cells))
    c = _case(kind, nx0=nx0, ny0=ny0, level=level, batch=batch, n_xi=rng.choice((3, 3, 6)),
              precision=prec, tuned=rng.random() < 0.5,
              nt0=max(1, min(24, rng.choice((32, 64, 96)) >> level)))
    if kind == "adjoint":
        c.update(nt0=max(1, min(4, 8 >> level)), ckpt=rng.choice((1, 4, 8)))
    if kind == "series":
        c.update(n_xi=3, field_model=1, every=rng.choice((1, 2, 8)), nt0=max(1, 16 >> level),
                 level=min(level, 3))
        c["batch"] = max(1, min(256, (1 << 18) // (cells0 << (2 * c["level"]))))
    if kind == "solve" and rng.random() < 0.25:
        c.update(krylov=2, tuned=False, nt0=max(1, 16 >> level))
    return c


# ---------------------------------------------------------------------------
# what a user's program has in hand
# ---------------------------------------------------------------------------
def _config(case, nlevels):
    paper = case["field_model"] == 1
    return hb.default_config(
        nlevels=nlevels, nx0=case["nx0"], ny0=case["ny0"], nt0=case["nt0"],
        T=case["nt0"] * (TAU0_PAPER if paper else TAU0), n_xi=case["n_xi"],
        field_model=case["field_model"], krylov_iters=case["krylov"],
        precision=hb.PREC_FP64 if case["precision"] == "fp64" else hb.PREC_FP32_MG)


def _context(case, nlevels):
    ctx = hb.Context(_config(case, nlevels))
    if case["tuned"]:
        for l in range(nlevels):
            t = TUNED[case["precision"]][min(l, 5)]
            ctx.set_schedule(l, **dict(zip(SCHEDULE_FIELDS, t)))
    return ctx


def _batches(case):
    return {l: max(1, case["batch"] >> (2 * l)) for l in range(case["levels"])}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "resjac":
        return _prepare_resjac(case, seed)
    if kind == "stats":
        return _prepare_stats(case, seed)
    dev = torch.device("cuda")
    if kind == "round":
        xis = {l: torch.from_numpy(xi_batch(l, 0, b, n_xi=case["n_xi"], seed=seed)).to(dev)
               for l, b in _batches(case).items()}
        return {"case": case, "ctx": _context(case, case["levels"]), "xis": xis}
    draw_xi = xi_halton(1 + seed % 1000003, case["batch"], 3) if kind == "series" else \
        xi_batch(case["level"], 0, case["batch"], n_xi=case["n_xi"], seed=seed)
    return {"case": case, "ctx": _context(case, case["level"] + 1),
            "xi": torch.from_numpy(draw_xi).to(dev)}


def _uniform(seed, *shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.rand(shape, generator=g, dtype=torch.float64, device="cuda")


def _wedge(u, ny, nx):
    """Salt mass fractions shaped like the solved ones: a salt wedge from the
    right side, wider at the bottom, with its toe and its front's thickness
    from u [B, 2] in [0, 1)."""
    x = (torch.arange(nx, dtype=torch.float64, device=u.device) + 0.5) * (2.0 / nx)
    y = (torch.arange(ny, dtype=torch.float64, device=u.device) + 0.5) * (1.0 / ny)
    front = (1.0 + 0.5 * u[:, 0, None] + 0.45 * y[None, :])[:, :, None]
    return torch.sigmoid((x[None, None, :] - front) / (0.03 + 0.05 * u[:, 1, None, None]))


def _prepare_resjac(case, seed):
    B, ny, nx = case["batch"], case["ny0"], case["nx0"]
    cfg = hb.default_config()
    xi = torch.from_numpy(xi_batch(0, 0, B, seed=seed)).cuda()
    phi, K, qin = _fields(cfg, xi, nx, ny)
    u = _uniform(seed, B, 2)
    c = _wedge(u, ny, nx)
    c_old = _wedge((u + 0.02).clamp(max=1.0), ny, nx)
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny
    p = cfg.rho1 * cfg.g * (1.0 - y)[None, :, None] + 40.0 * (_uniform(seed + 1, B, ny, nx) - 0.5)
    return {"case": case, "cfg": cfg, "tau": TAU0 * 32 / nx, "phi": phi, "K": K, "qin": qin,
            "p": p, "c": c, "c_old": c_old}


def _prepare_stats(case, seed):
    B = case["batch"]
    ctx = hb.Context(_config(case, case["level"] + 1))
    li = ctx.level_info(case["level"])
    u = _uniform(seed, B, 2)
    c = _wedge(u, li.ny, li.nx)
    q = 100.0 * _uniform(seed + 1, B, hb.NQ) + torch.arange(hb.NQ, device="cuda")
    # a few failed samples, as a batch of hundreds may have; they are skipped
    status = (_uniform(seed + 2, B) < 0.003).to(torch.int32)
    cells = li.ny * li.nx
    acc = hb.new_field_accumulator(1, cells)
    return {"case": case, "ctx": ctx, "q": q, "c": c.reshape(B, cells), "status": status,
            "acc": {k: v.reshape(cells) for k, v in acc.items()}, "stats": hb.LevelStats(),
            "count": torch.zeros(cells, dtype=torch.int64, device="cuda")}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "resjac":
        R, J = hb.residual_jacobian(state["cfg"], state["tau"], state["phi"], state["K"],
                                    state["qin"], state["p"], state["c"], state["c_old"])
        return {"R": R, "J": J}
    ctx, level = state["ctx"], case["level"]
    if kind == "solve":
        o = ctx.solve(level, state["xi"], want_c=True, want_p=True)
        return {k: o[k] for k in ("q", "c", "p", "status")}
    if kind == "pairs":
        return ctx.sample_pairs(level, state["xi"], want_c=True)
    if kind == "series":
        return ctx.solve_series(level, state["xi"], case["every"])
    if kind == "adjoint":
        return ctx.adjoint(level, state["xi"], qoi="Q_S", ckpt_every=case["ckpt"])
    if kind == "round":
        out = ctx.sample_levels(state["xis"], want_c=True)
        stats = {}
        for l, (qf, qc, _, _, st) in out.items():
            stats[l] = ctx.level_stats(l, qf, qc, st, hb.LevelStats()).numpy()
        return {"pairs": {l: list(o) for l, o in out.items()}, "stats": stats}
    # statistics: the batch merged into the running state, as between the
    # batches of a quasi-Monte Carlo run
    S = ctx.level_stats(level, state["q"], None, state["status"], state["stats"])
    acc = ctx.field_stats(level, state["c"], None, state["status"], state["acc"])
    ctx.field_exceedance(level, state["c"], state["status"], 0.5, state["count"])
    return {"qoi": S.numpy(), "n": acc["n"], "mean": acc["mean_f"], "m2": acc["m2_f"],
            "count": state["count"]}


# ---------------------------------------------------------------------------
# work that a pass cannot do without
# ---------------------------------------------------------------------------
def _solve_work(case, level, batch):
    """(bytes, flops) of one level's solves: xi read, QoIs and fields written;
    two defect-correction iterations per step (three residuals of 46
    operations per cell and, per V(2,2), four sweeps of 32 operations and a
    residual of 20 per cell, 4/3 for the coarser levels)."""
    cells = (case["nx0"] * case["ny0"]) << (2 * level)
    steps = case["nt0"] << level
    cyc = 2 if not case["krylov"] else 2 * case["krylov"]
    flops = batch * cells * steps * (3 * 46 + 2 * cyc * (4 * 32 + 20) * 4.0 / 3.0)
    return batch * (8.0 * case["n_xi"] + 8 * hb.NQ + 8 * cells), flops


def work(case):
    kind, B = case["kind"], case["batch"]
    if kind == "resjac":
        n = B * case["nx0"] * case["ny0"]
        return {"bytes": n * 8.0 * (5 + 22), "flops": n * 162.0}
    if kind == "stats":
        n = B * (case["nx0"] * case["ny0"] << (2 * case["level"]))
        return {"bytes": 8.0 * n + 8.0 * B * hb.NQ, "flops": 7.0 * n}
    parts = [(case["level"], B)]
    if kind == "pairs":
        parts.append((case["level"] - 1, B))
    if kind == "round":
        parts = [(l, b) for l, b in _batches(case).items()]
        parts += [(l - 1, b) for l, b in _batches(case).items() if l > 0]
    by, fl = (sum(v) for v in zip(*(_solve_work(case, l, b) for l, b in parts)))
    if kind == "series":        # the QoIs after every k-th step instead of the field
        by = 8.0 * B * (case["n_xi"] + hb.NQ * (1 + (case["nt0"] << case["level"]) // case["every"]))
    if kind == "adjoint":       # forward, and backward a transposed solve per step
        by, fl = 2 * by, 3 * fl
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# the same results in plain 64-bit torch
# ---------------------------------------------------------------------------
def _fields(cfg, xi, nx, ny):
    """Smooth random fields at the cell centres: phi, K [B, ny, nx], qin [B, ny]."""
    pi = math.pi
    x = ((torch.arange(nx, dtype=torch.float64, device=xi.device) + 0.5) * (cfg.Lx / nx))[None, None, :]
    y = ((torch.arange(ny, dtype=torch.float64, device=xi.device) + 0.5) * (cfg.Ly / ny))[None, :, None]
    z = [v[:, None, None] for v in xi.unbind(1)]
    a = 0.1 * z[0] * torch.cos(pi * x / 2) * torch.sin(pi * y)
    e = 0.5 * z[1] * torch.sin(pi * x / 2) * torch.cos(pi * y)
    q = 1.0 + 0.1 * z[2] + 0.0 * y
    if len(z) > 3:
        a = a + 0.05 * z[3] * torch.cos(pi * x) * torch.sin(2 * pi * y)
        e = e + 0.05 * z[4] * torch.sin(pi * x) * torch.cos(2 * pi * y)
        q = q + 0.05 * z[5] * torch.cos(pi * y)
    return ((cfg.phi0 * (1 + a)).contiguous(), (cfg.K0 * torch.exp(e)).contiguous(),
            (cfg.q0 * q)[:, :, 0].contiguous())


def _residual_jacobian(cfg, tau, phi, K, qin, p, c, c_old):
    """Residual [B, 2, ny, nx] of one implicit step and its Jacobian [B, 20,
    ny, nx] (blocks P, W, E, S, N of (pp, pc, cp, cc)), p the full pressure."""
    B, ny, nx = p.shape
    hx, hy = cfg.Lx / nx, cfg.Ly / ny
    r0, dr = cfg.rho0, cfg.rho1 - cfg.rho0
    rho = r0 + dr * c
    vt = hx * hy * phi / tau
    R = torch.stack([vt * dr * (c - c_old), vt * (rho * c - (r0 + dr * c_old) * c_old)], 1)
    J = torch.zeros((B, 20, ny, nx), dtype=torch.float64, device=p.device)
    J[:, 1] += vt * dr
    J[:, 3] += vt * (rho + dr * c)

    def flux(t, dco, pL, cL, pU, cU, gd):
        """(F, dF/du_L, dF/du_U): mass and salt flux from L to U."""
        rL, rU = r0 + dr * cL, r0 + dr * cU
        rb = 0.5 * (rL + rU)
        q = -t * ((pU - pL) + rb * gd)
        up = q >= 0
        a = torch.where(up, rL, rU)
        s = torch.where(up, rL * cL, rU * cU)
        qc = -t * gd * 0.5 * dr
        zero = torch.zeros_like(q)
        dif = -dco * 0.5 * dr * (cU - cL)
        aL, aU = torch.where(up, q * dr, zero), torch.where(up, zero, q * dr)
        sL = torch.where(up, q * (rL + dr * cL), zero)
        sU = torch.where(up, zero, q * (rU + dr * cU))
        F = (q * a, q * s - dco * rb * (cU - cL))
        dL = (t * a, qc * a + aL, t * s, qc * s + sL + dif + dco * rb)
        dU = (-t * a, qc * a + aU, -t * s, qc * s + sU + dif - dco * rb)
        return F, dL, dU

    def add(L, U, bLU, bUL, f):
        """A face's flux leaves cell slice L and enters U; bLU: the block of L
        for its neighbour U, bUL the reverse."""
        F, dL, dU = f
        for e in range(2):
            R[(slice(None), e) + L] += F[e]
            R[(slice(None), e) + U] -= F[e]
        for m in range(4):
            J[(slice(None), m) + L] += dL[m]
            J[(slice(None), 4 * bLU + m) + L] += dU[m]
            J[(slice(None), m) + U] -= dU[m]
            J[(slice(None), 4 * bUL + m) + U] -= dL[m]

    def mean(v, L, U):
        a, b = v[(slice(None),) + L], v[(slice(None),) + U]
        return 2 * a * b / (a + b)

    at = lambda v, s: v[(slice(None),) + s]
    L, U = (slice(None), slice(0, nx - 1)), (slice(None), slice(1, nx))
    add(L, U, 2, 1, flux(hy * mean(K, L, U) / (cfg.mu * hx), hy * mean(phi, L, U) * cfg.D / hx,
                         at(p, L), at(c, L), at(p, U), at(c, U), 0.0))
    if ny > 1:
        L, U = (slice(0, ny - 1), slice(None)), (slice(1, ny), slice(None))
        add(L, U, 4, 3, flux(hx * mean(K, L, U) / (cfg.mu * hy), hx * mean(phi, L, U) * cfg.D / hy,
                             at(p, L), at(c, L), at(p, U), at(c, U), cfg.g * hy))
    # left side: fresh-water inflow, diffusion to c = 0 at half a cell
    dco = 2 * hy * cfg.D / hx * phi[:, :, 0]
    cl, rl = c[:, :, 0], rho[:, :, 0]
    R[:, 0, :, 0] -= hy * r0 * qin
    R[:, 1, :, 0] += dco * 0.5 * (rl + r0) * cl
    J[:, 3, :, 0] += dco * (0.5 * dr * cl + 0.5 * (rl + r0))
    # right side: seawater hydrostatics and c = 1 at half a cell
    y = (torch.arange(ny, dtype=torch.float64, device=p.device) + 0.5) * hy
    pr, cr = p[:, :, -1], c[:, :, -1]
    F, dL, _ = flux(2 * hy / (cfg.mu * hx) * K[:, :, -1], 2 * hy * cfg.D / hx * phi[:, :, -1], pr, cr,
                    (cfg.rho1 * cfg.g * (cfg.Ly - y))[None, :].expand_as(pr), torch.ones_like(cr), 0.0)
    for e in range(2):
        R[:, e, :, -1] += F[e]
    for m in range(4):
        J[:, m, :, -1] += dL[m]
    return R, J


def _dense(J):
    """The Jacobian of one sample as a dense matrix, unknowns (p of all cells,
    c of all cells)."""
    _, ny, nx = J.shape
    n = ny * nx
    cell = torch.arange(n, device=J.device).reshape(ny, nx)
    A = torch.zeros((2 * n, 2 * n), dtype=torch.float64, device=J.device)
    every = slice(None)
    for b, own, other in ((0, (every, every), (every, every)),
                          (1, (every, slice(1, nx)), (every, slice(0, nx - 1))),
                          (2, (every, slice(0, nx - 1)), (every, slice(1, nx))),
                          (3, (slice(1, ny), every), (slice(0, ny - 1), every)),
                          (4, (slice(0, ny - 1), every), (slice(1, ny), every))):
        i, j = cell[own].reshape(-1), cell[other].reshape(-1)
        for m in range(4):
            A[i + n * (m // 2), j + n * (m % 2)] = J[4 * b + m][own].reshape(-1)
    return A


def _qois(cfg, phi, c):
    """The 22 quantities of interest of fields c [B, ny, nx]."""
    B, ny, nx = c.shape
    hx, hy = cfg.Lx / nx, cfg.Ly / ny
    edge = lambda n, h: torch.arange(n, dtype=torch.float64, device=c.device) * h
    x0, y0 = edge(nx, hx), edge(ny, hy)
    rho = cfg.rho0 + (cfg.rho1 - cfg.rho0) * c
    V = hx * hy
    q = [(c * rho).sum((1, 2)) * V, (phi * rho * c).sum((1, 2)) * V,
         (c * (cfg.Lx - (x0 + hx / 2))).sum((1, 2)) * V]
    for px, py in ((1.40, 0.05), (1.65, 0.25), (1.90, 0.50)):
        fx, fy = px / hx - 0.5, py / hy - 0.5
        i, j = min(max(int(math.floor(fx)), 0), nx - 2), min(max(int(math.floor(fy)), 0), ny - 2)
        tx, ty = min(max(fx - i, 0.0), 1.0), min(max(fy - j, 0.0), 1.0)
        q.append((1 - tx) * (1 - ty) * c[:, j, i] + tx * (1 - ty) * c[:, j, i + 1]
                 + (1 - tx) * ty * c[:, j + 1, i] + tx * ty * c[:, j + 1, i + 1])
    q.append((c <= 0.012178).double().sum((1, 2)) * V)
    for py in (0.05, 0.25, 0.50):
        oy = (torch.clamp(y0 + hy, max=py + 0.1) - torch.clamp(y0, min=py - 0.1)).clamp(min=0)
        for px in (0.90, 1.15, 1.40, 1.65, 1.90):
            ox = (torch.clamp(x0 + hx, max=px + 0.1) - torch.clamp(x0, min=px - 0.1)).clamp(min=0)
            q.append((c * rho * oy[None, :, None] * ox[None, None, :]).sum((1, 2)))
    return torch.stack(q, 1)


def _exact_solve(case, state):
    """Newton with dense direct solves, sample by sample (small grids)."""
    cfg = _config(case, 1)
    nx, ny, nt = case["nx0"], case["ny0"], case["nt0"]
    tau = cfg.T / nt
    phi, K, qin = _fields(cfg, state["xi"], nx, ny)
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) * (cfg.Ly / ny)
    ps, cs = [], []
    for b in range(case["batch"]):
        f = [v[b:b + 1] for v in (phi, K, qin)]
        p = (cfg.rho1 * cfg.g * (cfg.Ly - y))[None, :, None].expand(1, ny, nx).clone()
        c = torch.zeros_like(p)
        for _ in range(nt):
            c_old = c.clone()
            for _ in range(30):
                R, J = _residual_jacobian(cfg, tau, *f, p, c, c_old)
                d = torch.linalg.solve(_dense(J[0]), -R[0].reshape(-1)).reshape(2, ny, nx)
                p, c = p + d[0], c + d[1]
                if float(d[1].abs().max()) < 1e-13:
                    break
        ps.append(p)
        cs.append(c)
    p, c = torch.cat(ps), torch.cat(cs)
    return {"q": _qois(cfg, phi, c), "c": c, "p": p, "status": None}


def exact(case, seed):
    kind = case["kind"]
    if kind == "resjac":
        s = _prepare_resjac(case, seed)
        R, J = _residual_jacobian(s["cfg"], s["tau"], s["phi"], s["K"], s["qin"], s["p"], s["c"],
                                  s["c_old"])
        return {"R": R, "J": J}
    if kind == "stats":
        s = _prepare_stats(case, seed)
        ok = s["status"] == 0
        q, c = s["q"][ok], s["c"][ok]
        mq, mc = q.mean(0), c.mean(0)
        vq = ((q - mq) ** 2).sum(0) / max(q.shape[0] - 1, 1)
        return {"qoi": {"n": None, "mean_f": mq, "var_f": vq, "mean_d": mq, "var_d": vq},
                "n": None, "mean": mc, "m2": ((c - mc) ** 2).sum(0), "count": None}
    small = case["nx0"] * case["ny0"] <= 512 and case["level"] == 0
    if kind == "solve" and small and case["field_model"] == 0 and case["batch"] * case["nt0"] <= 48:
        return _exact_solve(case, prepare(case, seed))
    return None
