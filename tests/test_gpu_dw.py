"""The double-word arithmetic as the GPU runs it (tests/dw_device): the
reciprocal and the division built on it, which test_dw_host.py cannot see (the
host compiles a correctly rounded reciprocal in their place), and the packed
fiber product against the scalar operations it stands for.

Bounds.  rcp: rcp.approx is within 2^-22 relative, one Newton step leaves its
square, 2^-44, and two roundings, of the residual (2^-24 of 2^-22) and of the
result (half an ulp, at most 2^-24): 1.01 units of 2^-24.  div: the bound of the
host check, 8 units of 2^-47.  The packed product rounds each lane as the scalar
one does in the same order: no output word differs.  (A compiler that contracted
a packed product with the sum after it would leave errors of 2^-27 there.)"""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_device_arithmetic(tmp_path):
    from paper_2504_07042_gb300 import build

    exe = str(tmp_path / "dw_device_check")
    subprocess.run([build._nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-I", build.CSRC, "-o", exe,
                                                   os.path.join(HERE, "dw_device", "dw_device_check.cu")],
                   check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    got = {k: float(v) for k, v in (line.split() for line in out.strip().splitlines())}
    print(got)
    assert 0.0 < got["rcp"] <= 1.01
    assert 0.0 < got["div"] <= 8.0
    assert all(got["product%d" % n] == 0 for n in range(2, 17, 2))
