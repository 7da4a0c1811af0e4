"""Closed forms for matter at rest: when they may be taken, and what non-finite
values in the metric or the matter give, against the CPU oracle."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2502_03223_gb300 import sacra2d as S
from paper_2502_03223_gb300 import workloads as W

pytestmark = pytest.mark.gpu
G = 8


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2502_03223_gb300 import build as B
    B.build()


def _recover(adiabatic, change):
    """Both sides' primitives and status of one conserved state (flat, at rest but for `change`)."""
    cfg = dataclasses.replace(W.shock_tube_config(40, 16), rho_atm=1e-13, K=100.0, Gamma=2.0, Gamma_th=2.0,
                              eos_adiabatic=adiabatic)
    shape = (cfg.pz, cfg.px)
    raw = np.zeros((30,) + shape)
    raw[0] = raw[18] = 1.0
    raw[25] = 10.0 ** np.random.default_rng(4).uniform(-9, -3, shape)
    raw[29] = raw[25] * 1.3
    change(raw)
    g, o = S.Sacra(cfg), O.Oracle(cfg)
    g.set_initial_data(0, S.RAW, raw)
    o.set_level(0, 1, raw)
    sl = (slice(G, G + cfg.nz), slice(G, G + cfg.nx))
    return ([g.read(0, S.PRIMS, f, padded=False) for f in range(6)], [o.read(0, 2, f)[sl] for f in range(6)],
            g.read(0, S.STATUS, 0, padded=False).astype(int), o.read(0, 4, 0)[sl].astype(int))


@pytest.mark.parametrize("adiabatic", [0, 1])
def test_tiny_momenta_are_not_rest(adiabatic):
    """|S| below 1e-162: its square underflows, u_i = S_i / (D h) does not (a quotient of three roundings)."""
    def change(raw):
        raw[26], raw[28] = 1e-170, -3e-180
    a, b, sa, sb = _recover(adiabatic, change)
    assert np.array_equal(sa, sb)
    for f in (1, 3):
        assert np.all(np.abs(a[f] - b[f]) <= 1e-14 * np.abs(b[f])) and np.all(b[f] != 0.0)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("field", [1, 2, 5, 6])
@pytest.mark.parametrize("adiabatic", [0, 1])
def test_recovery_in_a_broken_metric(adiabatic, field, value):
    """Matter at rest in a cell whose h_ij is not finite: the same cells, and only those, lose their
    primitives and say so in their status."""
    def change(raw):
        raw[field, G + 3:G + 5, G + 10:G + 20] = value
    a, b, sa, sb = _recover(adiabatic, change)
    assert np.array_equal(sa, sb)
    for f in range(6):
        assert np.array_equal(np.isfinite(a[f]), np.isfinite(b[f])), f


def _at_rest(evolve):
    """A star at rest with a mildly varying metric and shift (16 x 12 cells), and its PRIM_METRIC planes."""
    cfg, tov = W.tov_config("rest", rho_c=1.28e-3, n_levels=1, N=16, dx_fine=0.9, rk=0)
    cfg = dataclasses.replace(cfg, nz=12, evolve_spacetime=evolve)
    d = W.tov_level_data(cfg, tov, 0)
    d[:25] += W.random_metric_perturbation(cfg, 0, np.random.default_rng(8), amp=1e-2)
    return cfg, d


def _rates(field, value):
    """Rates of the conserved variables, GPU and oracle, with one primitive set to `value`."""
    cfg, d = _at_rest(0)
    d[25 + field, G + 6, G + 7] = value
    g, o = S.Sacra(cfg), O.Oracle(cfg)
    g.set_initial_data(0, S.PRIM_METRIC, d)
    g.fill(0, cfg.dt)
    g.rk_stage(0, cfg.dt)
    o.set_level(0, 0, d)
    o.fill(0, cfg.dt)
    o.stage(0, cfg.dt)
    return (np.stack([g.read(0, S.RHS, f, padded=False) for f in range(25, 30)]),
            np.stack([o.read(0, 3, f)[G:G + cfg.nz, G:G + cfg.nx] for f in range(25, 30)]))


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("evolve,field", [(e, f) for e in (0, 1) for f in (0, 1, 3, 5, 9, 13, 18, 19, 20, 21)
                                          if (e, f) != (0, 20)])
def test_hydro_rates_in_a_broken_metric(evolve, field, value):
    """Matter at rest around one metric value that is not finite: the rates of the conserved variables
    are lost in the cells whose faces and sources read it, and in no other."""
    cfg, d = _at_rest(evolve)
    d[field, G + 6, G + 7] = value
    g, o = S.Sacra(cfg), O.Oracle(cfg)
    g.set_initial_data(0, S.PRIM_METRIC, d)
    g.fill(0, cfg.dt)
    g.rk_stage(0, cfg.dt)
    o.set_level(0, 0, d)
    o.fill(0, cfg.dt)
    o.stage(0, cfg.dt)
    for f in range(25, 30):
        a = np.isfinite(g.read(0, S.RHS, f, padded=False))
        b = np.isfinite(o.read(0, 3, f)[G:G + cfg.nz, G:G + cfg.nx])
        assert np.array_equal(a, b), (f, np.argwhere(a != b)[:8])


@pytest.mark.parametrize("field,value", [(0, np.nan), (0, np.inf), (4, np.nan), (4, np.inf)])
def test_hydro_rates_around_broken_matter(field, value):
    """A density or pressure that is not finite in matter at rest: the same rates are lost."""
    a, b = _rates(field, value)
    assert np.array_equal(np.isfinite(a), np.isfinite(b))


@pytest.mark.parametrize("field,value", [(1, np.nan), (2, np.nan), (3, np.nan), (1, np.inf), (3, -np.inf)])
def test_broken_velocities_reach_their_neighbours(field, value):
    """A velocity that is not finite in matter at rest: every rate of the cell and of the four next to it
    is lost (both states of a face between them are made with it), beyond them at most what the oracle loses."""
    a, b = _rates(field, value)
    for k, j in ((6, 7), (5, 7), (7, 7), (6, 6), (6, 8)):
        assert not np.isfinite(a[:, k, j]).any(), (k, j)
    assert not (~np.isfinite(a) & np.isfinite(b)).any()


@pytest.mark.parametrize("field,value", [(25, np.nan), (25, np.inf), (29, np.nan), (29, np.inf), (26, np.nan), (2, np.inf),
                                         (8, np.nan), (13, np.inf), (15, np.nan), (17, np.inf), (23, np.inf)])
def test_metric_rates_around_a_broken_value(field, value):
    """One metric value or primitive that is not finite: the rates of the metric are lost in the cells
    where the oracle loses them."""
    cfg, d = _at_rest(1)
    d[field, G + 6, G + 7] = value
    g, o = S.Sacra(cfg), O.Oracle(cfg)
    g.set_initial_data(0, S.PRIM_METRIC, d)
    g.fill(0, cfg.dt)
    g.rk_stage(0, cfg.dt)
    o.set_level(0, 0, d)
    o.fill(0, cfg.dt)
    o.stage(0, cfg.dt)
    for f in range(25):
        a = np.isfinite(g.read(0, S.RHS, f, padded=False))
        b = np.isfinite(o.read(0, 3, f)[G:G + cfg.nz, G:G + cfg.nx])
        assert np.array_equal(a, b), (f, np.argwhere(a != b)[:8])
