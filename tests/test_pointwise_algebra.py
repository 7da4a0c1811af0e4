"""The FP64 pointwise Z4c algebra of the device (csrc/z4c_pass.cuh), compiled for
the host in double and in long double: its rounding error may not grow with the
anisotropy of the conformal metric, nor with the ratio of a cell's large and small
components."""
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
GI, GD = 25, 25 + 14          # pass A's gt^ij (xx, xy, xz, yy, yz, zz) and Gt_d^i


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("pw") / "pointwise_host")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-Wno-unknown-pragmas", "-I",
                           os.path.join(ROOT, "paper_2502_03223_gb300", "csrc"),
                           os.path.join(HERE, "pointwise_host.cpp"), "-o", exe])

    def run(stretch, shear, grad, offdiag=1.0):
        out = subprocess.check_output([exe, repr(stretch), repr(shear), repr(grad), repr(offdiag)], text=True)
        return np.array([[float(x) for x in line.split()] for line in out.splitlines()])
    return run


@pytest.mark.parametrize("stretch", [1.0, 3.0, 10.0, 100.0, 1e4, 1e6])
def test_stretched_metric(host, stretch):
    """Every right-hand side and every value pass A hands on: sums of up to 60 products of operands a few
    roundings old, 2^-53 each, so an r.m.s. error of a few 1e-16 of the r.m.s. value; 2e-15 allowed."""
    e = host(stretch, 0.1, 0.3)[:, 0]
    assert np.all(e <= 2e-15), (stretch, np.argmax(e), e.max())


@pytest.mark.parametrize("small", [1e-4, 1e-7, 1e-10])
def test_small_components_keep_their_digits(host, small):
    """Nearly flat cells: gt^ij off the diagonal is made of the small h_ij alone (two products, a
    reciprocal), Gt_d^i of the small derivatives; both relative to themselves.  Off-diagonal terms of
    d_t h_ij with off-diagonal shift gradients `small` times the diagonal ones: gt_xk d_y beta^k +
    gt_yk d_x beta^k holds nothing of order one where h_ij is small too."""
    e = host(1.0, small, small, 1.0)
    for q in (1, 2, 4):
        assert e[GI + q, 1] <= 1e-15, (q, e[GI + q])
    assert np.all(e[GD:GD + 3, 0] <= 2e-15), e[GD:GD + 3]
    e = host(1.0, small, 1.0, small)
    assert np.all(e[[1, 2, 3, 4, 5, 6], 0] <= 2e-15), e[1:7]
