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
