"""FP64 right-hand sides on conformal metrics stretched in one direction (collapse,
the vicinity of a puncture), with shear: their rounding error against that of the
CPU oracle, both measured against the oracle in long double."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2502_03223_gb300 import sacra2d as S
from paper_2502_03223_gb300 import workloads as W

from extended_oracle import ExtendedOracle, build as build_extended

pytestmark = pytest.mark.gpu
G = 8


@pytest.fixture(scope="module")
def extended(tmp_path_factory):
    from paper_2502_03223_gb300 import build as B
    B.build()
    return build_extended(str(tmp_path_factory.mktemp("ext")))


@pytest.mark.parametrize("axis", ["x", "z"])
@pytest.mark.parametrize("stretch", [3.0, 10.0, 100.0, 1e4])
def test_stretched_metric(extended, stretch, axis):
    """gt = diag(s, s^-1/2, s^-1/2) along x or z, every component varied by 5 % of its scale: the largest
    error of each right-hand side at most ten times the oracle's (the same sums in FP64 in another order;
    with the stretch the FP64 error of the sums that cancel grows on both sides), or 2e-14 of the field's
    largest value where the oracle happens to be exact to a few units in the last place."""
    cfg, tov = W.tov_config("stretch", rho_c=1.28e-3, n_levels=1, N=16, dx_fine=0.5, rk=0)
    cfg = dataclasses.replace(cfg, nz=24)
    rng = np.random.default_rng(5)
    d = W.tov_level_data(cfg, tov, 0)
    noise = W.random_metric_perturbation(cfg, 0, rng, amp=0.05)
    d[:25] += noise
    g = np.array([stretch, stretch ** -0.5, stretch ** -0.5])
    if axis == "z":
        g = g[::-1]
    for q, (i, j) in enumerate(((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))):
        s = np.sqrt(g[i] * g[j])
        d[1 + q] = s * noise[1 + q] + (g[i] - 1.0 if i == j else 0.0)
        d[7 + q] = s * noise[7 + q]
    gpu, orc, ext = S.Sacra(cfg), O.Oracle(cfg), ExtendedOracle(extended, cfg)
    gpu.set_initial_data(0, S.PRIM_METRIC, d)
    gpu.fill(0, cfg.dt)
    gpu.rk_stage(0, cfg.dt)
    for o in (orc, ext):
        o.set_level(0, 0, d)
        o.fill(0, cfg.dt)
        o.stage(0, cfg.dt)
    sl = (slice(G, G + cfg.nz), slice(G, G + cfg.nx))
    for f in range(25):
        ref = ext.read(0, 3, f)[sl]
        eg = float(np.max(np.abs(gpu.read(0, S.RHS, f, padded=False) - ref)))
        eo = float(np.max(np.abs(orc.read(0, 3, f)[sl] - ref)))
        assert eg <= 10.0 * eo + 2e-14 * float(np.max(np.abs(ref))), (f, eg, eo)
