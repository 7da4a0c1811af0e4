"""Measured cases: what a program that uses this library has it do.

Every case goes through the public entry points of
``paper_2502_03223_gb300.sacra2d``.  Kinds:

  run     one hierarchy of levels (a star, Bondi flow, the shock tube): the
          program holds a saved state in pinned host memory, loads it into its
          context (set_initial_data), advances it by a few steps with the
          step's CUDA graph and saves the evolved state back (read_level), the
          segment of a run between two checkpoints.
  sweep   the same for a batch of independent stars (SacraBatch).
  stage   one RK stage of a single level by the stage-wise calls, with the
          right-hand side of every field read back.
  rates   the allocation-free hydro right-hand side on device arrays.
  train   training of the recovery's seed network.

Inputs come from the seed alone: the star's central density, a smooth
perturbation of the metric and a velocity bump are drawn from it.  exact()
restates the hydro and Z4c right-hand sides and the shock tube in plain numpy.
"""
import dataclasses
import functools
import math

import numpy as np
import torch

from paper_2502_03223_gb300 import sacra2d as S
from paper_2502_03223_gb300 import workloads as W

G = 8                       # padding cells on every side of a level


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call a program makes: the special-relativistic shock tube in the plane,
        # frozen flat metric, 20 steps of a few thousand cells: launches and latency
        {"name": "tube_400x4", "kind": "run", "what": "tube", "nx": 400, "nz": 4, "levels": 1, "rk": 0, "solver": 0,
         "precision": 0, "sub": 0, "steps": 20, "diag": False, "tune": False},
        # a coarse star as used while setting a run up: every level is a fraction of a wave
        {"name": "star_3x48", "kind": "run", "what": "stable", "nx": 48, "nz": 48, "levels": 3, "rk": 0, "solver": 0,
         "precision": 0, "sub": 0, "steps": 4, "diag": False, "tune": False},
        # hydro on a frozen black-hole metric, Berger-Oliger sub-cycling on every refined level
        {"name": "bondi_3x64_sub", "kind": "run", "what": "bondi", "nx": 64, "nz": 64, "levels": 3, "rk": 0,
         "solver": 1, "precision": 0, "sub": 1, "steps": 4, "diag": False, "tune": False},
        # the stable star of the benchmark, SSP-RK3, diagnostics of every step
        {"name": "stable_3x256", "kind": "run", "what": "stable", "nx": 256, "nz": 256, "levels": 3, "rk": 1,
         "solver": 0, "precision": 0, "sub": 0, "steps": 6, "diag": True, "tune": True},
        # the headline: the migrating star in FP64, diagnostics of every step
        {"name": "migration_5x512", "kind": "run", "what": "migration", "nx": 512, "nz": 512, "levels": 5, "rk": 0,
         "solver": 0, "precision": 0, "sub": 0, "steps": 3, "diag": True, "tune": True},
        # the same star in mixed precision
        {"name": "migration_5x512_mixed", "kind": "run", "what": "migration", "nx": 512, "nz": 512, "levels": 5,
         "rk": 0, "solver": 0, "precision": 7, "sub": 0, "steps": 6, "diag": True, "tune": True},
        # the largest: seven levels of 1024^2, the two finest sub-cycled, mixed precision
        {"name": "large_7x1024_mixed", "kind": "run", "what": "migration", "nx": 1024, "nz": 1024, "levels": 7,
         "rk": 0, "solver": 0, "precision": 7, "sub": 5, "steps": 1, "diag": False, "tune": True},
        # a parameter sweep: stars of unequal grids and level counts advanced together, mixed precision
        {"name": "sweep_6_mixed", "kind": "sweep", "stars": 6, "nmin": 64, "nmax": 256, "lmin": 2, "lmax": 4,
         "rk": 1, "precision": 7, "steps": 8, "pick": 11},
        # one stage by the stage-wise calls on one ragged level (numerics work, a host that drives the stages)
        {"name": "stage_181x133", "kind": "stage", "nx": 181, "nz": 133, "solver": 0, "precision": 0},
        # the hydro rates for a host framework that owns the device memory: the largest level it takes
        {"name": "rates_256x256", "kind": "rates", "nx": 256, "nz": 256, "solver": 0, "precision": 0},
        # training of the recovery's seed on tuples of a run
        {"name": "train_20k", "kind": "train", "tuples": 20000, "train_steps": 100, "blocks": 32},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "star", "star", "star", "bondi", "sweep", "stage", "rates", "train"])
    if kind == "tube":
        return {"kind": "run", "what": "tube", "nx": _log_int(rng, 64, 1600), "nz": rng.randint(4, 24), "levels": 1,
                "rk": rng.choice([0, 1]), "solver": rng.choice([0, 1]), "precision": 0, "sub": 0,
                "steps": rng.randint(8, 24), "diag": False, "tune": False}
    if kind == "star":
        n = 2 * _log_int(rng, 14, 300)
        levels = rng.randint(2, 6)
        sub = rng.randint(1, levels - 1) if rng.random() < 0.25 else 0
        work = n * n * levels * (1 << (levels - sub if sub else 0))
        steps = max(1, min(8, int(6e6 / work)))
        return {"kind": "run", "what": rng.choice(["stable", "migration"]), "nx": n, "nz": n, "levels": levels,
                "rk": rng.choice([0, 1]), "solver": rng.choice([0, 0, 0, 1]), "precision": rng.choice([0, 0, 7]),
                "sub": sub, "steps": steps, "diag": sub == 0 and rng.random() < 0.5, "tune": n >= 160}
    if kind == "bondi":
        n = 2 * _log_int(rng, 14, 128)
        levels = rng.randint(1, 4)
        return {"kind": "run", "what": "bondi", "nx": n, "nz": n, "levels": levels, "rk": 0,
                "solver": rng.choice([0, 1]), "precision": 0, "sub": rng.randint(0, levels - 1),
                "steps": rng.randint(2, 5), "diag": False, "tune": False}
    if kind == "sweep":
        lo = 2 * _log_int(rng, 16, 64)
        return {"kind": "sweep", "stars": rng.randint(2, 7), "nmin": lo, "nmax": lo * rng.choice([1, 2]), "lmin": 1,
                "lmax": rng.randint(2, 4), "rk": rng.choice([0, 1]), "precision": rng.choice([0, 7]),
                "steps": rng.randint(3, 8), "pick": rng.randint(1, 1 << 20)}
    if kind == "stage":
        return {"kind": "stage", "nx": _log_int(rng, 24, 300), "nz": _log_int(rng, 24, 300),
                "solver": rng.choice([0, 1]), "precision": 0}
    if kind == "rates":
        return {"kind": "rates", "nx": _log_int(rng, 16, 256), "nz": _log_int(rng, 16, 256),
                "solver": rng.choice([0, 1]), "precision": rng.choice([0, 0, 3])}
    return {"kind": "train", "tuples": _log_int(rng, 2000, 200000), "train_steps": rng.randint(20, 120),
            "blocks": rng.choice([8, 16, 32])}


# ------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=32)
def _star(rho_c):
    return W.tov_solve(100.0, 2.0, rho_c, dR=5e-3)


def _bump(cfg, d, level, rng, amp):
    """A smooth moving bump of matter around the star and a small smooth
    perturbation of every metric field with its parities, so that no part of
    the right-hand side vanishes by symmetry of the background."""
    if amp:
        d[:25] += W.random_metric_perturbation(cfg, level, rng, amp=amp)
    X, Z = W.cell_centres(cfg, level)
    x0, z0 = rng.uniform(2.0, 5.0, 2)
    b = np.exp(-((np.abs(X) - x0) ** 2 + (np.abs(Z) - z0) ** 2) / 6.0)
    d[26] = 0.05 * b * X / (np.abs(X) + 1.0)
    d[28] = 0.03 * b * Z / (np.abs(Z) + 1.0)
    d[27] = 0.02 * b * X / (np.abs(X) + 1.0)


def _inputs(case, seed):
    """The configuration and the padded level data (25 metric planes, then
    rho, u_x, u_y, u_z, P) of a hierarchy."""
    rng = np.random.default_rng([int(seed), 77])
    nx, nz, L = case["nx"], case["nz"], case.get("levels", 1)
    what = case.get("what", "stable")
    if what == "tube":
        cfg = W.shock_tube_config(nx, nz, solver=case["solver"], rk=case["rk"])
        # pressures and densities of the benchmark tube, the membrane and the left state drawn around them
        left = (10.0 * (1.0 + 0.05 * rng.uniform(-1, 1)), 13.33 * (1.0 + 0.05 * rng.uniform(-1, 1)), 0.0)
        return cfg, [W.shock_tube_data(cfg, left=left, x0=0.5 + 0.05 * rng.uniform(-1, 1))]
    if what == "bondi":
        sol = W.bondi_solve(R_c=8.0 * (1.0 + 0.02 * rng.uniform(-1, 1)))
        cfg, _ = W.bondi_config(N=nx, n_levels=L, solver=case["solver"], rk=case["rk"], sol=sol)
        cfg = dataclasses.replace(cfg, subcycle_from=case["sub"])
        return cfg, [W.bondi_level_data(cfg, sol, l) for l in range(L)]
    rho = (1.28e-3 if what == "stable" else 7.993e-3) * (1.0 + 0.01 * rng.uniform(-1, 1))
    # the finest box holds the star: 0.25 at 256 cells, 0.1 at 512, as in the benchmark configurations
    dx = 0.25 * max(1.0, 64.0 / nx) if what == "stable" else 0.1 * max(1.0, 160.0 / nx)
    cfg, tov = W.tov_config(case["kind"], rho_c=rho, n_levels=L, N=nx, dx_fine=dx, rk=case.get("rk", 0),
                            solver=case["solver"], tov=_star(rho))
    cfg = dataclasses.replace(cfg, nz=nz, precision=case["precision"], subcycle_from=case.get("sub", 0))
    datas = []
    for l in range(L):
        d = W.tov_level_data(cfg, tov, l, p_deplete=0.99 if what == "migration" else 1.0)
        # the single-level kinds carry the perturbed metric too; a run starts from the star
        _bump(cfg, d, l, rng, 1e-3 if case["kind"] in ("stage", "rates") else 0.0)
        datas.append(d)
    return cfg, datas


def _pinned(n):
    return torch.empty(n, dtype=torch.float64, pin_memory=True).numpy()


def _sweep_stars(case, seed):
    """Stars of a sweep: grids and level counts from the case's own pick, the
    central densities from the seed."""
    g = np.random.default_rng([case["pick"], 5])
    rng = np.random.default_rng([int(seed), 78])
    sizes = sorted({case["nmin"], (case["nmin"] + case["nmax"]) // 4 * 2, case["nmax"]})
    out = []
    for i in range(case["stars"]):
        n, L = int(g.choice(sizes)), int(g.integers(case["lmin"], case["lmax"] + 1))
        rho = float(rng.uniform(1e-3, 8e-3))
        tov = W.tov_solve(100.0, 2.0, rho, dR=2e-2)
        cfg, _ = W.tov_config("sweep_%02d" % i, rho_c=rho, n_levels=L, N=n, dx_fine=0.25, rk=case["rk"], tov=tov)
        cfg.precision = case["precision"]
        out.append((cfg, tov))
    return out


class State:
    """What the user's program keeps between calls."""


def prepare(case, seed):
    s = State()
    s.case = case
    kind = case["kind"]
    if kind == "run":
        s.cfg, datas = _inputs(case, seed)
        s.dt, s.steps = s.cfg.dt, case["steps"]
        s.sim = S.Sacra(s.cfg)
        for l, d in enumerate(datas):
            s.sim.set_initial_data(l, S.PRIM_METRIC, d)
        if case["tune"]:
            s.sim.tune(reps=2)
        n = 30 * s.cfg.px * s.cfg.pz
        s.saved = [s.sim.read_level(l, _pinned(n)) for l in range(s.cfg.n_levels)]
        s.out = [_pinned(n) for _ in range(s.cfg.n_levels)]
    elif kind == "sweep":
        stars = _sweep_stars(case, seed)
        s.cfgs = [c for c, _ in stars]
        s.dt, s.steps = min(c.dt for c in s.cfgs), case["steps"]
        s.sim = S.SacraBatch(s.cfgs)
        s.data = []
        for i, (c, t) in enumerate(stars):
            for l in range(c.n_levels):
                a = _pinned(30 * c.px * c.pz)
                a[:] = W.tov_level_data(c, t, l, p_deplete=0.99 if t.rho_c > 3.2e-3 else 1.0).ravel()
                s.sim.set_initial_data(i, l, S.PRIM_METRIC, a)
                s.data.append((i, l, a))
        s.sim.tune(reps=2)
    elif kind == "stage":
        s.cfg, (d,) = _inputs(case, seed)
        s.sim = S.Sacra(s.cfg)
        s.data = _pinned(d.size)
        s.data[:] = d.ravel()
        s.sim.set_initial_data(0, S.PRIM_METRIC, s.data)
        s.dt = s.cfg.dt
        s.out = [_pinned(d.size), _pinned(d.size)]
    elif kind == "rates":
        s.cfg, (d,) = _inputs(case, seed)
        U, P = _filled(s.cfg, d)
        s.U = torch.from_numpy(np.ascontiguousarray(np.concatenate([U, np.zeros_like(U[:5])]))).cuda()
        s.P = torch.from_numpy(np.ascontiguousarray(P)).cuda()
        s.rhs = torch.zeros((5,) + d.shape[1:], dtype=torch.float64, device="cuda")
    else:
        g = torch.Generator(device="cpu").manual_seed(int(seed))
        n = case["tuples"]
        x = torch.rand((n, 9), generator=g)
        # densities over decades, slow to fast flows, mild metrics: the ranges of the recovery's features
        t = torch.stack([-12 + 10 * x[:, 0], 0.3 * x[:, 1], x[:, 2] ** 2, 0.9 * x[:, 3] ** 2, -0.2 * x[:, 4],
                         0.01 * (x[:, 5] - 0.5), 0.01 * (x[:, 6] - 0.5), 1e-4 * x[:, 7], -4 + 3 * x[:, 8]], dim=1)
        y = t[:, 8] + 0.5 * torch.tanh(3 * t[:, 1] - t[:, 3]) + 0.05 * t[:, 0] * t[:, 2]
        s.tuples = torch.cat([t, y[:, None]], dim=1).to(torch.float32).cuda().contiguous()
        s.seed = int(seed) & 0xFFFF
    return s


# ------------------------------------------------------------------ one pass

def run(state):
    case = state.case
    kind = case["kind"]
    if kind == "run":
        sim = state.sim
        for l, a in enumerate(state.saved):
            sim.set_initial_data(l, S.RAW, a)
        out = {}
        if case["diag"]:
            # the last two columns count branches taken at thresholds (failed recoveries, fallbacks), not values
            out["diag"] = sim.step_constraints(state.dt, state.steps, use_graph=True)[:, :7]
        else:
            sim.step(state.dt, state.steps, use_graph=True)
        for l, a in enumerate(state.out):
            out["level%d" % l] = sim.read_level(l, a)
        return out
    if kind == "sweep":
        sim = state.sim
        for i, l, a in state.data:
            sim.set_initial_data(i, l, S.PRIM_METRIC, a)
        sim.step(state.dt, state.steps, use_graph=True)
        out = {}
        for i, l, a in state.data:
            out["star%d_level%d" % (i, l)] = np.stack([sim.read(i, l, S.STATE_STEP, f) for f in range(30)])
        return out
    if kind == "stage":
        sim = state.sim
        sim.set_initial_data(0, S.PRIM_METRIC, state.data)
        sim.fill(0, state.dt)
        sim.rk_stage(0, state.dt)
        return {"rhs": sim.read_level(0, state.out[0], S.RHS), "stage": sim.read_level(0, state.out[1], S.STATE_STAGE)}
    if kind == "rates":
        rc = S.hydro_rhs_noalloc(state.cfg, 0, state.U.data_ptr(), state.P.data_ptr(), state.rhs.data_ptr(),
                                 torch.cuda.current_stream().cuda_stream)
        if rc != S.SACRA_OK:
            raise S.SacraError("hydro_rhs_noalloc: %d" % rc)
        return state.rhs
    net, report, loss = S.mlp_train(state.tuples, steps=case["train_steps"], batch_blocks=case["blocks"],
                                    seed=state.seed, record_loss=True)
    return {"net": net, "loss": loss}


# ------------------------------------------------------------------ the work of one pass

# floating-point operations per unit of one RK stage in the method's plain minimal form: x-face, z-face, hydro
# sources, stage update with the recovery; cartoon terms, derivatives, pointwise Z4c
_HYDRO = 508 + 536 + 391 + 396
_Z4C = 591 + 2139 + 2001


def work(case):
    kind = case["kind"]
    if kind == "train":
        n = case["blocks"] * 128 * case["train_steps"]
        return {"bytes": case["tuples"] * 40 + 20000, "flops": n * 4865 * 6}
    if kind == "sweep":
        g = np.random.default_rng([case["pick"], 5])
        sizes = sorted({case["nmin"], (case["nmin"] + case["nmax"]) // 4 * 2, case["nmax"]})
        b = f = 0
        for _ in range(case["stars"]):
            n, L = int(g.choice(sizes)), int(g.integers(case["lmin"], case["lmax"] + 1))
            b += 2 * 30 * 8 * (n + 16) ** 2 * L
            f += (_HYDRO + _Z4C) * n * n * L * (4 if case["rk"] == 0 else 3) * case["steps"]
        return {"bytes": b, "flops": f}
    nx, nz = case["nx"], case["nz"]
    pad = (nx + 16) * (nz + 16)
    if kind == "rates":
        return {"bytes": 8 * (35 * pad + 5 * nx * nz), "flops": (508 + 536 + 391) * nx * nz}
    if kind == "stage":
        return {"bytes": 8 * 90 * pad, "flops": (_HYDRO + _Z4C) * nx * nz}
    L, sub = case["levels"], case["sub"]
    steps = sum((1 << (l - sub + 1)) if sub and l >= sub else 1 for l in range(L)) * case["steps"]
    per = _HYDRO + (_Z4C if case["what"] in ("stable", "migration") else 0)
    return {"bytes": 8 * 60 * pad * L, "flops": per * nx * nz * steps * (4 if case["rk"] == 0 else 3)}


# ------------------------------------------------------------------ the same in plain numpy

PAR_X = {f: -1.0 for f in (14, 15, 19, 20, 22, 23, 3, 5, 9, 11)}
PAR_Z = {f: -1.0 for f in (16, 21, 24, 3, 5, 9, 11)}
SYM = [[0, 1, 2], [1, 3, 4], [2, 4, 5]]
PAIRS = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]


class _Eos:
    """P = K rho^2 (or nothing, K = 0) plus a thermal Gamma law."""

    def __init__(self, cfg):
        self.K, self.G, self.Gth = cfg.K, cfg.Gamma, cfg.Gamma_th

    def pc(self, rho):
        return self.K * rho ** self.G if self.K else np.zeros_like(rho)

    def ec(self, rho):
        return self.K * rho ** (self.G - 1.0) / (self.G - 1.0) if self.K else np.zeros_like(rho)

    def eps(self, rho, P):
        return self.ec(rho) + (P - self.pc(rho)) / ((self.Gth - 1.0) * rho)

    def cs2(self, rho, P):
        h = 1.0 + self.eps(rho, P) + P / rho
        c = (self.G * self.pc(rho) + self.Gth * (P - self.pc(rho))) / (rho * h)
        return np.clip(np.where(c > 0, c, 0.0), 0.0, 1.0 - 1e-15)


def _filled(cfg, d):
    """State planes (25 metric) and primitives (6) of one cylindrical level
    with the ghosts of stage 0: mirrored at the axis and the equator, the
    primitives copied outwards from the last cells."""
    U, P = d[:25].copy(), np.zeros((6,) + d.shape[1:])
    P[:5] = d[25:30]
    P[5] = _Eos(cfg).eps(P[0], P[4])
    for a in (U, P):
        pm = a is P
        if pm:
            a[:, :, G + cfg.nx:] = a[:, :, G + cfg.nx - 1:G + cfg.nx]
            a[:, G + cfg.nz:, :] = a[:, G + cfg.nz - 1:G + cfg.nz, :]
        for f in range(a.shape[0]):
            sx = (-1.0 if f in (1, 2) else 1.0) if pm else PAR_X.get(f, 1.0)
            sz = (-1.0 if f == 3 else 1.0) if pm else PAR_Z.get(f, 1.0)
            a[f][:, :G] = sx * a[f][:, G:2 * G][:, ::-1]
            a[f][:G, :] = sz * a[f][G:2 * G, :][::-1, :]
    return U, P


def _mat3(h):
    """gt_ij from six planes h_ij, its inverse and determinant."""
    g = np.array([[h[SYM[i][j]] + (1.0 if i == j else 0.0) for j in range(3)] for i in range(3)])
    gi = np.empty_like(g)
    for i in range(3):
        for j in range(3):
            a, b = (i + 1) % 3, (i + 2) % 3
            c, e = (j + 1) % 3, (j + 2) % 3
            gi[j, i] = g[a, c] * g[b, e] - g[a, e] * g[b, c]
    det = sum(g[0, i] * gi[i, 0] for i in range(3))
    return g, gi / det, det


def _ppm(c):
    """Left and right states of the face between c[2] and c[3] of six cells."""
    def slope(am, a0, ap):
        dl, dr, dc = a0 - am, ap - a0, 0.5 * (ap - am)
        lim = np.minimum(np.abs(dc), np.minimum(2 * np.abs(dl), 2 * np.abs(dr)))
        return np.where(dl * dr <= 0, 0.0, np.where(dc > 0, lim, -lim))

    def limit(a0, aL, aR):
        flat = (aR - a0) * (a0 - aL) <= 0
        dd, d6 = (aR - aL) ** 2, (aR - aL) * (6.0 * (a0 - 0.5 * (aL + aR)))
        nL = np.where(d6 > dd, 3.0 * a0 - 2.0 * aR, aL)
        nR = np.where(-dd > d6, 3.0 * a0 - 2.0 * aL, aR)
        return np.where(flat, a0, nL), np.where(flat, a0, nR)

    s = [slope(c[i], c[i + 1], c[i + 2]) for i in range(4)]
    f = [c[i + 1] + 0.5 * (c[i + 2] - c[i + 1]) - (s[i + 1] - s[i]) / 6.0 for i in range(3)]
    return limit(c[2], f[0], f[1])[1], limit(c[3], f[1], f[2])[0]


def _flux(cfg, eos, ax, pl, pr, al, beta, Wf, h):
    """HLLC (with its TVDLF fallback) or TVDLF flux through faces normal to
    axis ax, alpha psi^6 times the Eulerian flux of (D, S_x, S_y, S_z, E)."""
    p = [0, 1, 2] if ax == 0 else [2, 0, 1]
    g0, gi0, _ = _mat3(h)
    m = np.array([[g0[p[i], p[j]] for j in range(3)] for i in range(3)])
    mi = np.array([[gi0[p[i], p[j]] for j in range(3)] for i in range(3)])
    bn = beta[ax]
    B, C = 1.0 / np.sqrt(mi[0, 0]), 1.0 / np.sqrt(m[2, 2])
    D = B * C

    def side(s):
        rho, P = s[0], s[4]
        u = [s[1 + q] for q in p]
        t0 = Wf * B * (mi[0, 0] * u[0] + mi[0, 1] * u[1] + mi[0, 2] * u[2])
        t1 = Wf * D * (m[2, 2] * u[1] - m[1, 2] * u[2])
        t2 = Wf * C * u[2]
        w = np.sqrt(1.0 + t0 * t0 + t1 * t1 + t2 * t2)
        hh = 1.0 + eos.eps(rho, P) + P / rho
        c2 = eos.cs2(rho, P)
        r = rho * hh * w
        v = t0 / w
        vv = (t0 * t0 + t1 * t1 + t2 * t2) / (w * w)
        disc = np.sqrt(np.maximum(c2 * (1 - vv) * (1 - vv * c2 - v * v * (1 - c2)), 0.0))
        q = np.array([rho * w, r * t0, r * t1, r * t2, r * w - P])
        f = np.array([q[0] * v, q[1] * v + P, q[2] * v, q[3] * v, q[1]])
        return q, f, P, v, (v * (1 - c2) - disc) / (1 - vv * c2), (v * (1 - c2) + disc) / (1 - vv * c2)

    qL, fL, PL, vL, lmL, lpL = side(pl)
    qR, fR, PR, vR, lmR, lpR = side(pr)
    lamL, lamR = np.minimum(lmL, lmR), np.maximum(lpL, lpR)
    sg = Wf * mi[0, 0] * B
    vi = bn / (al * sg)
    cm = np.maximum(np.abs(lamL - vi), np.abs(lamR - vi))
    F = 0.5 * ((fL - vi * qL) + (fR - vi * qR)) - 0.5 * cm * (qR - qL)
    if cfg.solver == 0:
        idl = 1.0 / (lamR - lamL)
        hll = lambda n: (lamR * qR[n] - lamL * qL[n] + fL[n] - fR[n]) * idl                      # noqa: E731
        hlf = lambda n: (lamR * fL[n] - lamL * fR[n] + lamR * lamL * (qR[n] - qL[n])) * idl      # noqa: E731
        E, Sx, FE, FS = hll(4), hll(1), hlf(4), hlf(1)
        b = E + FS
        disc = b * b - 4.0 * FE * Sx
        lc = 2.0 * Sx / (b + np.sqrt(np.maximum(disc, 0.0)))
        Pc = FS - lc * FE
        ok = (disc >= 0) & (lc >= lamL) & (lc <= lamR) & (Pc > 0)
        left = vi <= lc
        pick = lambda a, c: np.where(left, a, c)                                                 # noqa: E731
        q, f, P, v, lam = pick(qL, qR), pick(fL, fR), pick(PL, PR), pick(vL, vR), pick(lamL, lamR)
        fac, iden = lam - v, 1.0 / (lam - lc)
        qs = np.array([q[0] * fac, q[1] * fac + Pc - P, q[2] * fac, q[3] * fac, q[4] * fac + Pc * lc - P * v]) * iden
        H = f + lam * (qs - q) - vi * qs
        F = np.where(ok & np.isfinite(H).all(axis=0), H, F)
        F = np.where(lamL >= vi, fL - vi * qL, np.where(lamR <= vi, fR - vi * qR, F))
    F = np.where((pl == pr).all(axis=0), fL - vi * qL, F)
    pre = al / Wf ** 3 * sg
    s0 = (B * F[1] - D * mi[0, 1] * F[2] + C * m[0, 2] * F[3]) / Wf
    s1 = (D * mi[0, 0] * F[2] + C * m[1, 2] * F[3]) / Wf
    s2 = C * m[2, 2] * F[3] / Wf
    out = np.empty_like(F)
    out[0], out[4] = pre * F[0], pre * F[4]
    for a, sv in zip(p, (s0, s1, s2)):
        out[1 + a] = pre * sv
    return out


def _win(a, nx, nz, j0, j1, k0, k1, dj=0, dk=0):
    """Cells [j0, j1] x [k0, k1] of padded planes, shifted."""
    return a[..., k0 + dk + G - 1:k1 + dk + G, j0 + dj + G - 1:j1 + dj + G]


def _hydro_rhs(cfg, U, P):
    """d_t (q_D, q_Sx, q_Sy, q_Sz, q_E) of the interior cells."""
    nx, nz, dx, dz = cfg.nx, cfg.nz, cfg.dx0, cfg.dz0
    cyl = cfg.geometry == 1
    eos = _Eos(cfg)
    w6 = np.array([3.0, -25.0, 150.0, 150.0, -25.0, 3.0]) / 256.0
    fl = []
    for ax in range(2):
        reg = (0, nx, 1, nz) if ax == 0 else (1, nx, 0, nz)
        at = lambda a, n: _win(a, nx, nz, *reg, dj=n if ax == 0 else 0, dk=0 if ax == 0 else n)   # noqa: E731
        st = [_ppm([at(P[v], n) for n in range(-2, 4)]) for v in range(5)]
        pl, pr = np.array([s[0] for s in st]), np.array([s[1] for s in st])
        c0, c1 = at(P[:5], 0), at(P[:5], 1)
        pl = np.where((pl[0] > 0) & (pl[4] > 0), pl, c0)
        pr = np.where((pr[0] > 0) & (pr[4] > 0), pr, c1)
        face = lambda f: sum(w * at(U[f], n) for w, n in zip(w6, range(-2, 4)))                   # noqa: E731
        f = _flux(cfg, eos, 0 if ax == 0 else 2, pl, pr, face(18), [face(19 + i) for i in range(3)], face(0),
                  [face(1 + a) for a in range(6)])
        if ax == 0:
            xf = np.arange(0, nx + 1) * dx
            f *= (xf if cyl else 1.0) * dz
            if cyl:
                f[2] *= xf
        else:
            xc = (np.arange(1, nx + 1) - 0.5) * dx
            if cyl:
                f[[0, 1, 2, 4], 0] = 0.0
            f *= (xc if cyl else 1.0) * dx
            if cyl:
                f[2] *= xc
        fl.append(f)
    x = (np.arange(1, nx + 1) - 0.5) * dx * np.ones((nz, 1))
    vol = (x if cyl else 1.0) * dx * dz
    div = (fl[0][:, :, 1:] - fl[0][:, :, :-1] + fl[1][:, 1:, :] - fl[1][:, :-1, :]) / vol
    c = lambda a: _win(a, nx, nz, 1, nx, 1, nz)                                                   # noqa: E731
    g, gi, _ = _mat3(c(U[1:7]))
    Wc, al = c(U[0]), c(U[18])
    rho, P_ = c(P[0]), c(P[4])
    u = c(P[1:4])
    w = np.sqrt(1.0 + Wc ** 2 * np.einsum("ijkl,ikl,jkl->kl", gi, u, u))
    r2 = rho * (1.0 + c(P[5]) + P_ / rho) * w * w
    vd = u / w
    vu = Wc ** 2 * np.einsum("ijkl,jkl->ikl", gi, vd)
    gv = np.einsum("ijkl,jkl->ikl", gi, vd)
    vv = (vd * vu).sum(axis=0)

    def d1(f, ax):
        t = lambda n: _win(U[f], nx, nz, 1, nx, 1, nz, dj=n if ax == 0 else 0, dk=0 if ax == 0 else n)   # noqa: E731
        return (45 * (t(1) - t(-1)) - 9 * (t(2) - t(-2)) + t(3) - t(-3)) / (60.0 * (dx if ax == 0 else dz))

    src, dal = [], []
    for ax in range(2):
        da, dW = d1(18, ax), d1(0, ax)
        dal.append(da)
        vdb = sum(vd[i] * d1(19 + i, ax) for i in range(3))
        dg = np.array([[d1(1 + SYM[i][j], ax) for j in range(3)] for i in range(3)])
        vvdg = -np.einsum("ijkl,ikl,jkl->kl", dg, gv, gv)
        dalW = da / Wc ** 3 - 3.0 * al * dW / Wc ** 4
        src.append(P_ * dalW - r2 / Wc ** 3 * (da - vdb + 0.5 * Wc ** 2 * al * vvdg + al / Wc * vv * dW))
    if cyl:
        src[0] = src[0] + al / Wc ** 3 * (r2 * vd[1] * (vu[1] - c(U[20]) / al) + P_) / x
    K = c(U[13]) + 2.0 * c(U[17])
    Kd = np.array([[(c(U[7 + SYM[i][j]]) + g[i, j] * K / 3.0) / Wc ** 2 for j in range(3)] for i in range(3)])
    KS = r2 * np.einsum("ijkl,ikl,jkl->kl", Kd, vu, vu) + P_ * Wc ** 2 * np.einsum("ijkl,ijkl->kl", gi, Kd)
    sE = (al * KS - r2 * (vu[0] * dal[0] + vu[2] * dal[1])) / Wc ** 3
    return np.array([-div[0], src[0] - div[1], -div[2], src[1] - div[3], sE - div[4]])


def _y_derivs(cfg, U):
    """d_y and d_yy of every metric field by interpolating each row onto the
    planes y = +-m dx and rotating, on all rows and columns 1 .. nx + 4."""
    nx, dx = cfg.nx, cfg.dx0
    j = np.arange(1, nx + 5)
    x = j - 0.5
    planes = {0: U[:, :, G:G + nx + 4]}
    for m in (1, 2, 3):
        vp = np.sqrt(x * x + m * m)
        I = np.zeros_like(planes[0])
        for n in range(-4, 5):
            wgt = np.ones_like(x)
            for q in range(-4, 5):
                if q != n:
                    wgt = wgt * ((vp - x) - q) / (n - q)
            I += wgt * U[:, :, G + n:G + n + nx + 4]
        for sgn in (1, -1):
            c, s = x / vp, sgn * m / vp
            R = [[c, -s, 0.0], [s, c, 0.0], [0.0, 0.0, 1.0]]
            o = I.copy()
            for v in (14, 19, 22):
                for a in range(3):
                    o[v + a] = sum(R[a][b] * I[v + b] for b in range(3))
            for t in (1, 7):
                for a, (i, k) in enumerate(PAIRS):
                    o[t + a] = sum(R[i][p] * R[k][q] * I[t + SYM[p][q]] for p in range(3) for q in range(3))
            planes[sgn * m] = o
    p = planes
    dy = (45 * (p[1] - p[-1]) - 9 * (p[2] - p[-2]) + p[3] - p[-3]) / (60.0 * dx)
    dyy = (270 * (p[1] + p[-1] - 2 * p[0]) - 27 * (p[2] + p[-2] - 2 * p[0]) + 2 * (p[3] + p[-3] - 2 * p[0])) / (180.0 * dx * dx)
    return dy, dyy


def _z4c_rhs(cfg, U, P):
    """The 25 metric right-hand sides of the interior cells, one level."""
    nx, nz, dx = cfg.nx, cfg.nz, cfg.dx0
    dy, dyy = _y_derivs(cfg, U)
    # d_y of the columns left of the axis: the rotation by pi of column 1 - j
    par = np.array([PAR_X.get(f, 1.0) for f in range(25)])
    dyf = np.concatenate([-par[:, None, None] * dy[:, :, 2::-1], dy], axis=2)                     # columns -2 .. nx + 4
    cell = lambda a, dj=0, dk=0: _win(a, nx, nz, 1, nx, 1, nz, dj, dk)                            # noqa: E731
    yc = lambda dj=0, dk=0: dyf[:, G + dk:G + dk + nz, 3 + dj:3 + dj + nx]                        # noqa: E731
    c6 = lambda t, i: (45 * (t(1) - t(-1)) - 9 * (t(2) - t(-2)) + t(3) - t(-3)) * i               # noqa: E731
    s6 = lambda t, i: (270 * (t(1) + t(-1) - 2 * t(0)) - 27 * (t(2) + t(-2) - 2 * t(0))           # noqa: E731
                       + 2 * (t(3) + t(-3) - 2 * t(0))) * i
    i1, i2 = 1.0 / (60.0 * dx), 1.0 / (180.0 * dx * dx)
    F = cell(U)
    D = np.array([c6(lambda n: cell(U, n, 0), i1), yc(), c6(lambda n: cell(U, 0, n), i1)])
    DD = np.empty((3, 3) + F.shape)
    DD[0, 0] = s6(lambda n: cell(U, n, 0), i2)
    DD[1, 1] = dyy[:, G:G + nz, :nx]
    DD[2, 2] = s6(lambda n: cell(U, 0, n), i2)
    DD[0, 2] = DD[2, 0] = c6(lambda n: c6(lambda m: cell(U, n, m), i1), i1)
    DD[0, 1] = DD[1, 0] = c6(lambda n: yc(n, 0), i1)
    DD[1, 2] = DD[2, 1] = c6(lambda n: yc(0, n), i1)
    adv = F[20] * D[1]
    for ax, b in ((0, F[19]), (2, F[21])):
        t = lambda n: cell(U, n, 0) if ax == 0 else cell(U, 0, n)                                 # noqa: E731
        up = (2 * t(-2) - 24 * t(-1) - 35 * t(0) + 80 * t(1) - 30 * t(2) + 8 * t(3) - t(4)) * i1
        dn = -(2 * t(2) - 24 * t(1) - 35 * t(0) + 80 * t(-1) - 30 * t(-2) + 8 * t(-3) - t(-4)) * i1
        adv = adv + b * np.where(b > 0, up, dn)
        ko = t(4) + t(-4) - 8 * (t(3) + t(-3)) + 28 * (t(2) + t(-2)) - 56 * (t(1) + t(-1)) + 70 * t(0)
        adv = adv - cfg.eps_ko / 256.0 * ko / dx
    mat = lambda a: np.array([[a[SYM[i][j]] for j in range(3)] for i in range(3)])                # noqa: E731
    Wc, al, Kh, Th = F[0], F[18], F[13], F[17]
    g, gi, _ = _mat3(F[1:7])
    A = mat(F[7:13])
    es = functools.partial(np.einsum, optimize=True)
    dg = np.array([mat(D[k, 1:7]) for k in range(3)])                                             # [k, i, j]
    ddg = np.array([[mat(DD[k, l, 1:7]) for l in range(3)] for k in range(3)])                    # [k, l, i, j]
    Gl = 0.5 * (np.moveaxis(dg, 0, 1) + es("jkiab->kijab", dg) - dg)                              # Gt_{k,ij}
    G2 = es("klab,lijab->kijab", gi, Gl)
    Gd = es("jkab,ijkab->iab", gi, G2)
    dGt = D[:, 14:17]                                                                             # [j, k]: d_j Gt^k
    R = -0.5 * es("lmab,lmijab->ijab", gi, ddg)
    t = es("kiab,jkab->ijab", g, dGt) + es("kab,ijkab->ijab", Gd, Gl)
    R = R + 0.5 * (t + np.swapaxes(t, 0, 1))
    q = es("lmab,kliab,jkmab->ijab", gi, G2, Gl)
    R = R + q + np.swapaxes(q, 0, 1) + es("lmab,kimab,kljab->ijab", gi, G2, Gl)
    dW = D[:, 0]
    DDW = DD[:, :, 0] - es("kijab,kab->ijab", G2, dW)
    R = R + (DDW + g * es("ijab,ijab->ab", gi, DDW)) / Wc - 2.0 * g * es("ijab,iab,jab->ab", gi, dW, dW) / Wc ** 2
    Rs = Wc ** 2 * es("ijab,ijab->ab", gi, R)
    c = lambda a: _win(a, nx, nz, 1, nx, 1, nz)                                                   # noqa: E731
    rho, pr, u = c(P[0]), c(P[4]), c(P[1:4])
    w = np.sqrt(1.0 + Wc ** 2 * es("ijab,iab,jab->ab", gi, u, u))
    rh = rho * (1.0 + c(P[5]) + pr / rho)
    E = rh * w * w - pr
    Si = rh * w * u
    Sij = rh * u[:, None] * u[None, :] + pr * g / Wc ** 2
    x, z = (np.arange(1, nx + 1) - 0.5) * dx, (np.arange(1, nz + 1) - 0.5) * cfg.dz0
    fz = np.exp(-(x[None, :] ** 2 + z[:, None] ** 2) / cfg.r_z4 ** 2)
    K, kap, PI = Kh + 2.0 * Th, cfg.kappa * fz, math.pi
    db = D[:, 19:22]                                                                              # [j, i]: d_j beta^i
    divb = db[0, 0] + db[1, 1] + db[2, 2]
    da = D[:, 18]
    mix = da[:, None] * dW[None, :]
    DDa = (DD[:, :, 18] - es("kijab,kab->ijab", G2, da)
           + (mix + np.swapaxes(mix, 0, 1) - g * es("ijab,iab,jab->ab", gi, da, dW)) / Wc)
    Am = es("ilab,lkab->ikab", A, gi)
    Au = es("ilab,ljab->ijab", gi, Am)
    AA = es("ikab,kiab->ab", Am, Am)
    X = al * R - DDa - 8.0 * PI * al * Sij
    tr = es("ijab,ijab->ab", gi, X)
    out = np.empty((25, nz, nx))
    out[0] = Wc * (al * K - divb) / 3.0
    gb = es("ikab,jkab->ijab", g, db)
    Ab = es("kjab,ikab->ijab", A, db)
    sh = -2.0 * al * A - 2.0 / 3.0 * g * divb + gb + np.swapaxes(gb, 0, 1)
    sa = (Wc ** 2 * (X - g * tr / 3.0) + al * (K * A - 2.0 * es("ilab,ljab->ijab", Am, A)) - 2.0 / 3.0 * A * divb
          + Ab + np.swapaxes(Ab, 0, 1))
    for a, (i, k) in enumerate(PAIRS):
        out[1 + a], out[7 + a] = sh[i, k], sa[i, k]
    out[13] = (-Wc ** 2 * es("ijab,ijab->ab", gi, DDa) + al * (AA + K * K / 3.0)
               + 4.0 * PI * al * (Wc ** 2 * es("ijab,ijab->ab", gi, Sij) + E) + al * kap * Th)
    inn = (-es("ijab,jab->iab", gi, 2.0 * D[:, 13] + D[:, 17]) / 3.0 - 3.0 / Wc * es("ijab,jab->iab", Au, dW)
           - 8.0 * PI * es("ijab,jab->iab", gi, Si) + es("ijkab,jkab->iab", G2, Au))
    ddb = DD[:, :, 19:22]                                                                         # [j, k, i]
    Gt = F[14:17]
    s = (-2.0 * es("ijab,jab->iab", Au, da) - es("jab,jiab->iab", Gd, db) + 2.0 * al * inn + 2.0 / 3.0 * Gd * divb
         + es("jkab,jkiab->iab", gi, ddb) + es("ijab,kjkab->iab", gi, ddb) / 3.0 - 2.0 * al * kap * (Gt - Gd))
    out[14:17] = s
    out[22:25] = s - cfg.eta_B * F[22:25]
    out[17] = fz * (0.5 * al * (Rs - AA + 2.0 / 3.0 * K * K) - 8.0 * PI * al * E) - 2.0 * al * kap * Th
    out[18] = -2.0 * al * Kh
    out[19:22] = 0.75 * F[22:25]
    return out + adv


def _tube(cfg, d, steps):
    """The planar shock tube: the conserved planes after some steps."""
    eos = _Eos(cfg)
    nx, nz = cfg.nx, cfg.nz
    U = d[:25]
    P = np.concatenate([d[25:30], eos.eps(d[25], d[29])[None]])

    def cons(p):
        w = np.sqrt(1.0 + (p[1:4] ** 2).sum(axis=0))
        r = p[0] * (1.0 + p[5] + p[4] / p[0]) * w
        return np.array([p[0] * w, r * p[1], r * p[2], r * p[3], r * w - p[4]])

    def prims(q):
        """Root of z = r / h(z) by bisection."""
        D, E, r = q[0], q[4], np.sqrt((q[1:4] ** 2).sum(axis=0)) / q[0]
        qq = E / D - 1.0
        k = r / (1.0 + qq)
        lo, hi = 0.5 * k / np.sqrt(1.0 - 0.25 * k * k), k / np.sqrt(1.0 - k * k)

        def parts(z):
            w = np.sqrt(1.0 + z * z)
            eps = np.maximum(w * qq - z * r + z * z / (1.0 + w), 0.0)
            return w, eps, 1.0 + eps + (cfg.Gamma_th - 1.0) * eps
        for _ in range(70):
            mid = 0.5 * (lo + hi)
            up = mid - r / parts(mid)[2] > 0
            lo, hi = np.where(up, lo, mid), np.where(up, mid, hi)
        w, eps, h = parts(0.5 * (lo + hi))
        rho = D / w
        return np.array([rho, q[1] / (D * h), q[2] / (D * h), q[3] / (D * h), (cfg.Gamma_th - 1.0) * rho * eps, eps])

    def fill(p):
        inner = p[:, G:G + nz, G:G + nx]
        return np.pad(inner, ((0, 0), (G, G), (G, G)), mode="edge")

    def rate(p):
        return _hydro_rhs(cfg, U, fill(p))
    ins = (slice(None), slice(G, G + nz), slice(G, G + nx))
    dt = cfg.dt
    q = cons(P)[ins]

    def prim_of(qq):
        full = P.copy()
        full[ins] = prims(qq)
        return full
    p = P
    for _ in range(steps):
        k1 = rate(p)
        if cfg.rk == 0:
            k2 = rate(prim_of(q + 0.5 * dt * k1))
            k3 = rate(prim_of(q + 0.5 * dt * k2))
            last = q + dt * k3
            k4 = rate(prim_of(last))
            q = q + dt * (k1 / 6.0 + k2 / 3.0 + k3 / 3.0 + k4 / 6.0)
        else:
            q1 = q + dt * k1
            last = 0.75 * q + 0.25 * q1 + 0.25 * dt * rate(prim_of(q1))
            q = q / 3.0 + 2.0 / 3.0 * last + 2.0 / 3.0 * dt * rate(prim_of(last))
        p = prim_of(q)
    # the ghost cells hold what the fill before the last stage copied there
    out = np.concatenate([d[:25], fill(np.pad(last, ((0, 0), (G, G), (G, G))))])
    out[25:, G:G + nz, G:G + nx] = q
    return out.ravel()


def exact(case, seed):
    kind = case["kind"]
    if kind == "rates":
        cfg, (d,) = _inputs(case, seed)
        if cfg.precision:
            cfg = dataclasses.replace(cfg, precision=0)
        out = np.zeros((5,) + d.shape[1:])
        out[:, G:G + cfg.nz, G:G + cfg.nx] = _hydro_rhs(cfg, *_filled(cfg, d))
        return out
    if kind == "stage":
        cfg, (d,) = _inputs(case, seed)
        U, P = _filled(cfg, d)
        out = np.zeros_like(d)
        out[:25, G:G + cfg.nz, G:G + cfg.nx] = _z4c_rhs(cfg, U, P)
        out[25:, G:G + cfg.nz, G:G + cfg.nx] = _hydro_rhs(cfg, U, P)
        # the state of the stage also holds the recovery's and the constraints' choices: no plain value
        return {"rhs": out.ravel(), "stage": None}
    if kind == "run" and case["what"] == "tube":
        cfg, (d,) = _inputs(case, seed)
        return {"level0": _tube(cfg, d, case["steps"])}
    # whole runs of the coupled system, and the network's training, have no short plain form
    return None

