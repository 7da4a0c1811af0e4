"""The block fixed-point forms of the FP64 kernels where they can go wrong: cells
they hand back to the FP64 arithmetic (non-finite values), values at the ends of
the exponent range, and the smallest and ragged grids, against the CPU oracle."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2502_03223_gb300 import sacra2d as S
from paper_2502_03223_gb300 import workloads as W

from gpu_common import both, compare_level

pytestmark = pytest.mark.gpu
G = 8


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2502_03223_gb300 import build as B
    B.build()


def _perturbed(nx, nz, amp, seed=3):
    cfg, tov = W.tov_config("fx", rho_c=1.28e-3, n_levels=1, N=nx, dx_fine=0.5, rk=0)
    cfg = dataclasses.replace(cfg, nz=nz)
    rng = np.random.default_rng(seed)
    d = W.tov_level_data(cfg, tov, 0)
    d[:25] += W.random_metric_perturbation(cfg, 0, rng, amp=amp)
    X, Z = W.cell_centres(cfg, 0)
    b = np.exp(-((np.abs(X) - 4.0) ** 2 + (np.abs(Z) - 3.0) ** 2) / 4.0)
    d[26] = 0.1 * b * X / (np.abs(X) + 1.0)
    d[28] = 0.05 * b * Z / (np.abs(Z) + 1.0)
    return cfg, d


@pytest.mark.parametrize("nx,nz", [(8, 4), (17, 9), (33, 16), (130, 31)])
@pytest.mark.parametrize("amp", [1e-1, 1e-2])
def test_stage_rhs_matches_oracle(nx, nz, amp):
    """Edges and remainders of the tiles, strong and mild metric perturbations: every right-hand side
    within the per-stage bound of the parity tests (1e-11 of its group)."""
    cfg, d = _perturbed(nx, nz, amp)
    gpu, orc = both(cfg, [d])
    gpu.fill(0, cfg.dt); orc.fill(0, cfg.dt)
    gpu.rk_stage(0, cfg.dt); orc.stage(0, cfg.dt)
    compare_level(gpu, orc, 0, 1e-11, which=(S.RHS, S.STATE_STAGE))


@pytest.mark.parametrize("field,value", [(18, -np.inf), (0, np.nan), (19, 1e200), (3, 1e-320)])
def test_cells_outside_the_fixed_point_range(field, value):
    """One bad value: the right-hand sides of the cells it reaches are what the FP64 arithmetic gives
    (finite where the oracle's are, non-finite where they are not), all others are untouched by it."""
    cfg, d = _perturbed(24, 24, 1e-2)
    bad = d.copy()
    bad[field, G + 12, G + 11] = value
    out = []
    for x in (d, bad):
        g = S.Sacra(cfg)
        g.set_initial_data(0, S.PRIM_METRIC, x)
        g.fill(0, cfg.dt)
        g.rk_stage(0, cfg.dt)
        out.append(np.stack([g.read(0, S.RHS, f, padded=False) for f in range(25)]))
    o = O.Oracle(cfg)
    o.set_level(0, 0, bad)
    o.fill(0, cfg.dt)
    o.stage(0, cfg.dt)
    ref = np.stack([o.read(0, 3, f)[G:G + cfg.nz, G:G + cfg.nx] for f in range(25)])
    k, j = np.meshgrid(np.arange(cfg.nz), np.arange(cfg.nx), indexing="ij")
    far = (np.abs(k - 12) > 4) | (np.abs(j - 11) > 8)      # beyond the stencils (x: planes, then their x-derivative)
    assert np.array_equal(out[0][:, far], out[1][:, far])
    with np.errstate(all="ignore"):
        same = np.isfinite(ref) == np.isfinite(out[1])
    assert same.all(), np.argwhere(~same)[:10]
    ok = np.isfinite(ref)
    scale = np.maximum(np.abs(ref), np.nanmax(np.where(ok, np.abs(ref), 0.0), axis=(1, 2), keepdims=True))
    assert np.all(np.abs(out[1] - ref)[ok] <= 1e-9 * scale[ok] + 1e-12)


@pytest.mark.parametrize("eos", ["hybrid", "ideal", "pieces", "adiabatic"])
def test_recovery_of_slow_matter(eos):
    """The closed forms of the recovery (matter at rest, slow flow) and the iteration either side of
    their threshold r = 1e-4, thermal and cold branch, against the oracle's iteration on the same
    conserved state.  Bounds: the iteration closes its bracket to 1e-12 relative in z; eps comes from
    E / D - 1 (rounded alike on both sides), so it carries a few 1e-16 absolute."""
    kw = {"hybrid": dict(K=100.0, Gamma=2.0, Gamma_th=2.0), "ideal": dict(K=0.0, Gamma_th=5.0 / 3.0),
          "pieces": dict(K=100.0, Gamma=2.0, Gamma_th=1.8, pwp=((1e-5, 2.4),)),
          "adiabatic": dict(K=100.0, Gamma=2.0, Gamma_th=2.0, eos_adiabatic=1)}[eos]
    cfg = dataclasses.replace(W.shock_tube_config(96, 40), rho_atm=1e-13, **kw)
    rng = np.random.default_rng(11)
    shape = (cfg.pz, cfg.px)
    d = np.zeros((30,) + shape)
    d[0] = d[18] = 1.0
    rho = 10.0 ** rng.uniform(-8, -2, shape)
    u = 10.0 ** rng.uniform(-14, -2, shape) * (rng.random(shape) > 0.1)       # a tenth at rest
    phi = rng.uniform(0, 2 * np.pi, shape)
    d[25] = rho
    d[26], d[27], d[28] = u * np.cos(phi), 0.3 * u, u * np.sin(phi)
    pc = W.cold_P(W.cold_pieces(cfg.K, cfg.Gamma, cfg.pwp), rho) if cfg.K else 1e-3 * rho
    d[29] = pc * (1.0 + 10.0 ** rng.uniform(-2, 1, shape))
    g = S.Sacra(cfg)
    g.set_initial_data(0, S.PRIM_METRIC, d)
    raw = g.read_level(0, np.zeros(30 * cfg.px * cfg.pz)).reshape(30, *shape)
    if eos in ("hybrid", "pieces"):                                            # a third below the cold curve
        cold = rng.random(shape) < 0.33
        raw[29] = np.where(cold, raw[25] * (1.0 + 0.2 * (raw[29] / raw[25] - 1.0)), raw[29])
    g.set_initial_data(0, S.RAW, raw)
    o = O.Oracle(cfg)
    o.set_level(0, 1, raw)
    a = [g.read(0, S.PRIMS, f) for f in range(6)]
    b = [o.read(0, 2, f) for f in range(6)]
    assert np.array_equal(g.read(0, S.STATUS, 0).astype(int), o.read(0, 4, 0).astype(int))
    for f in (1, 2, 3):
        assert np.all(np.abs(a[f] - b[f]) <= 1e-11 * np.abs(b[f]) + 1e-300), (eos, f)
    assert np.all(np.abs(a[0] - b[0]) <= 1e-14 * b[0])
    assert np.all(np.abs(a[4] - b[4]) <= 1e-12 * b[4] + 1e-14 * b[0])
    assert np.all(np.abs(a[5] - b[5]) <= 1e-12 * b[5] + 1e-14)
