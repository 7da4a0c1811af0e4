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
