"""Quotients and roots on the integer units (csrc/softfp.cuh), compiled for the host."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_correctly_rounded(tmp_path):
    """Quotient, reciprocal and square root equal the processor's bit for bit (random and extreme
    significands, near ties, zeros, infinities, NaN, subnormals), for seeds off by up to two units;
    the reciprocal root within 0.52 ulp."""
    exe = str(tmp_path / "quotients_host")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-Wno-unknown-pragmas", "-I",
                           os.path.join(ROOT, "paper_2502_03223_gb300", "csrc"),
                           os.path.join(HERE, "quotients_host.cpp"), "-o", exe])
    q, r, s, rs = subprocess.check_output([exe], text=True).split()
    assert (int(q), int(r), int(s)) == (0, 0, 0)
    assert float(rs) < 0.52
