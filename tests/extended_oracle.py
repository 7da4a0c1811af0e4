"""The CPU oracle in long double (80 bits on x86, 128 on Arm): its C sources with
`double` replaced, for tests that compare the rounding errors of two FP64 results
with each other.  Much slower than the oracle: small grids only."""
import ctypes as C
import os
import re
import subprocess

import numpy as np

import oracle as O

SOURCES = ["eos_c2p.c", "stencil.c", "riemann.c", "z4c.c", "grid.c"]
LD = C.c_longdouble


class Params(C.Structure):
    _fields_ = [(n, t if t is C.c_int else (LD * t._length_ if hasattr(t, "_length_") else LD))
                for n, t in O.Params._fields_]


def build(folder) -> C.CDLL:
    src = os.path.dirname(os.path.abspath(O.__file__))
    number = re.compile(r"(?<![\w.])((?:\d+\.\d*|\.\d+)(?:[eE][+-]?\d+)?|\d+[eE][+-]?\d+)(?![\w.])")
    for f in SOURCES + ["orc.h"]:
        s = open(os.path.join(src, f)).read()
        s = number.sub(r"\1L", re.sub(r"\bdouble\b", "long double", s))
        s = re.sub(r"\bI\b", "I_", s)                    # tgmath.h brings complex.h's I
        with open(os.path.join(folder, f), "w") as out:
            out.write(("" if f == "orc.h" else "#include <tgmath.h>\n") + s)
    lib = os.path.join(folder, "libextended.so")
    subprocess.check_call(["gcc", "-std=gnu11", "-O2", "-ffp-contract=off", "-fopenmp", "-fPIC", "-shared", "-o", lib]
                          + [os.path.join(folder, f) for f in SOURCES] + ["-lm"])
    L = C.CDLL(lib)
    L.orc_create.restype = C.c_void_p
    L.orc_create.argtypes = [C.POINTER(Params)]
    L.orc_destroy.argtypes = [C.c_void_p]
    L.orc_set_level.argtypes = [C.c_void_p, C.c_int, C.c_int, C.c_void_p]
    L.orc_fill.argtypes = [C.c_void_p, C.c_int, LD]
    L.orc_stage.argtypes = [C.c_void_p, C.c_int, LD]
    L.orc_read.argtypes = [C.c_void_p, C.c_int, C.c_int, C.c_int, C.c_void_p]
    L.orc_stencil_init()
    return L


class ExtendedOracle:
    """The calls of oracle.Oracle that the tests use."""

    def __init__(self, lib, cfg):
        p, q = O.make_params(cfg), Params()
        for n, t in O.Params._fields_:
            v = getattr(p, n)
            if hasattr(t, "_length_"):
                for i in range(t._length_):
                    getattr(q, n)[i] = v[i]
            else:
                setattr(q, n, v)
        self._L, self.cfg = lib, cfg
        self._c = lib.orc_create(C.byref(q))
        assert self._c

    def __del__(self):
        if self._c:
            self._L.orc_destroy(self._c)

    def set_level(self, level, kind, data):
        a = np.ascontiguousarray(data, dtype=np.longdouble)
        self._L.orc_set_level(self._c, level, kind, a.ctypes.data)

    def fill(self, stage, dt):
        self._L.orc_fill(self._c, stage, dt)

    def stage(self, stage, dt):
        self._L.orc_stage(self._c, stage, dt)

    def read(self, level, which, field):
        out = np.zeros((self.cfg.pz, self.cfg.px), dtype=np.longdouble)
        self._L.orc_read(self._c, level, which, field, out.ctypes.data)
        return out
