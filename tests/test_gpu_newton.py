"""The update's reciprocal and square root (the hardware's approximation and
one Newton step) against 64 bits and against CUDA's 1/x and sqrt.

Bounds: the approximations are good to 1 ulp (rcp) and 2**-22.9 (rsqrt). A
Newton step squares that error: what is left, with the rounding of the
residual, is below 2**-43 of the result, 2**-19 of an ulp, beside the last
rounding's half. Below 2**-100 the root's residual runs out of exponents and
the step may bring nothing: 2**-22.9 and a rounding, under 4 ulp."""
import os
import subprocess

import pytest

from paper_1909_01092_gb300 import build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_reciprocal_and_root_bounds(tmp_path):
    exe = str(tmp_path / "newton")
    subprocess.run([build.nvcc(), *build.ARCH_FLAGS, "-O3", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC,
                    "-o", exe, os.path.join(HERE, "gpu_newton.cu")], check=True, capture_output=True, timeout=300)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    got = {w[0]: (float(w[2]), int(w[4])) for w in (line.split() for line in out.splitlines())}
    for name in ("recip_mantissas", "recip_range", "root_mantissas", "root_range"):
        assert got[name][0] <= 0.5 + 2.0 ** -18 and got[name][1] <= 1, out
    assert got["root_small"][0] <= 4.0, out
