"""The scalars of the float32 conjugate gradients of the impact zones are
rounded divisions, by the source: no approximate division or reciprocal in the
solver, and no compiler flag that makes `/` one."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1409_2081_gb300")


def test_no_approximate_division():
    src = open(os.path.join(PKG, "csrc", "solve.cu")).read()
    src = re.sub(r"//[^\n]*", "", src)
    assert not re.findall(r"__fdividef|__frcp_\w+|rcp\.approx|div\.approx|div\.full", src)
    build = open(os.path.join(PKG, "build.py")).read()
    assert not re.findall(r"use_fast_math|prec-div|ftz", build)
