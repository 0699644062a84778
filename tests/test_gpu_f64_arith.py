"""The FP64 kernels' products, reciprocals and roots (swe_f64.cuh), on the FP64
pipe (Hard) and on the integer unit (Soft).  Bounds, in units of 2^-52
relative: the last operation rounds by at most 1/2 and the corrections of the
hardware seed leave under 0.02, so reciprocal and root are within 0.52, the
FP64 pipe's inverse root, formed from the root, within 1.04, and the inverse
cube root within 0.52 plus 1/4 (a third of its cube's three roundings); the
reference itself is within 1/2 (quotient, root), 1 (inverse root) or 2
(inverse cube root, from cbrt's own bound of 1).  Products are exactly the
correctly rounded ones."""
import os
import subprocess

import pytest

from paper_2010_14416_gb300 import build as libbuild

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2010_14416_gb300", "csrc")


def test_fp64_reciprocal_and_roots_within_their_bounds(tmp_path):
    exe = str(tmp_path / "f64_arith_check")
    cmd = [libbuild.nvcc()] + libbuild.ARCH + ["-O3", "-std=c++17", "-I", CSRC,
                                                os.path.join(HERE, "cuda", "f64_arith_check.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    got = {k: float(v) for k, v in (line.split() for line in r.stdout.splitlines())}
    one = dict(rcp=1.02, rcp_negative=1.02, sqrt=1.02, sqrt_with_inverse=1.02, rsqrt=2.04, rcbrt=3.0)
    bounds = {**one, **{"soft_" + k: v for k, v in one.items()}, "soft_rsqrt": 1.52, "scale": 0, "mul": 0, "special": 0}
    assert got.keys() == bounds.keys()
    assert all(got[k] <= bounds[k] for k in bounds), got
