"""Quotients and roots on the integer units, on the device."""
import ctypes as C

import numpy as np
import pytest

from paper_2502_03223_gb300 import build as B

pytestmark = pytest.mark.gpu


def _values(rng, n, spread):
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    kind = rng.integers(0, 4, n)
    m = np.where(kind == 1, rng.integers(0, 4, n, dtype=np.uint64), m)
    m = np.where(kind == 2, np.uint64((1 << 52) - 1) - rng.integers(0, 4, n, dtype=np.uint64), m)
    e = rng.integers(1023 - spread, 1023 + spread + 1, n).astype(np.uint64)
    return ((e << np.uint64(52)) | m).view(np.float64)


def _same(x, y):
    return (x.view(np.uint64) == y.view(np.uint64)) | (np.isnan(x) & np.isnan(y))


def test_quotients_and_roots():
    """Division, reciprocal and square root bit for bit as NumPy's; the reciprocal root within 0.52 ulp,
    the reciprocal cube root within 0.52 (its residual is exact to 2^-70, the series to 2^-60)."""
    B.build()
    lib = C.CDLL(B.PROBE)
    dp = np.ctypeslib.ndpointer(np.float64, flags="C")
    lib.sacra_probe_quotients.argtypes = [dp, dp, C.c_int, dp]
    rng = np.random.default_rng(2)
    special = np.array([0.0, -0.0, 1.0, 3.0, np.inf, -np.inf, np.nan, 5e-324, -2.3e-308, 2.2250738585072014e-308,
                        1.7976931348623157e308, -1.0, 4.0, 2.0])
    sa, sb = (x.ravel() for x in np.meshgrid(special, special))
    a = np.concatenate([_values(rng, 1 << 20, 1000), _values(rng, 1 << 20, 3), sa])
    b = np.concatenate([_values(rng, 1 << 20, 1000), _values(rng, 1 << 20, 3), sb])
    b *= np.where(rng.random(b.size) < 0.5, -1.0, 1.0)
    n = a.size
    out = np.zeros(5 * n)
    assert lib.sacra_probe_quotients(a, b, n, out) == 0
    q, r, s, rs, rc = out.reshape(5, n)
    with np.errstate(all="ignore"):
        assert _same(q, a / b).all()
        assert _same(r, 1.0 / b).all()
        assert _same(s, np.sqrt(a)).all()
        x = a[1 << 20:1 << 21].astype(np.longdouble)
        for got, ref, bound in ((rs, 1.0 / np.sqrt(x), 0.52), (rc, 1.0 / np.cbrt(x), 0.52)):
            ulp = np.spacing(ref.astype(np.float64)).astype(np.longdouble)
            err = np.abs(got[1 << 20:1 << 21].astype(np.longdouble) - ref) / ulp
            assert float(err.max()) < bound, float(err.max())
