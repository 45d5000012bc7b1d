"""The second-order operator in the V-cycle (mg_definite, mg_omega_scale, make_mg_tables with
fd_n = 1): as a preconditioner of the CG's own stencil it must reach the plain-CG solution in as
many iterations as the V-cycle built on that stencil, at most one more.  Host only."""
import json
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2011_07209_gb300", "csrc")


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path_factory.mktemp("mglow") / "mg_low_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "tests"), os.path.join(ROOT, "tests", "mg_low_check.cpp"),
                    os.path.join(CSRC, "plan.cpp"), "-o", exe], check=True)
    return exe


# scale, two shears (1.1: coefficients of either sign), points, R_PE, half-width
@pytest.mark.parametrize("cell", [(14.7, 0.0, 0.0, 72, 5.0, 7.0, 3), (14.7, 0.1, 0.05, 72, 5.0, 7.0, 3),
                                  (14.7, 0.1, 0.05, 60, 5.0, 7.0, 2), (14.7, 0.1, 0.05, 60, 5.0, 7.0, 1),
                                  (14.7, 1.1, 0.0, 60, 4.0, 6.5, 3), (14.7, 0.1, 0.05, 24, 3.0, 6.0, 3)])
def test_second_order_vcycle(harness, cell):
    r = json.loads(subprocess.run([harness, *map(str, cell)], check=True, capture_output=True, text=True).stdout)
    assert r["definite"] == 1
    assert r["scale"] == pytest.approx({1: 1.0, 2: 16 / 15, 3: 272 / 245}[cell[-1]], rel=1e-6)
    assert 0 < r["low"] < r["plain"]
    if r["high"] > 0:   # -1: the sixth-order hierarchy reaches too far for the coarse boxes
        assert r["low"] <= r["high"] + 1
    # both stop at |b - A x| <= 1e-9 |b|: the solutions differ by at most 2e-9 cond(A)^(1/2)-like
    # factors in norm; the bound of the sixth-order V-cycle's own test
    assert r["rel_diff"] < 1e-8
    assert r["K1_low"] <= 27   # the coarse operators keep a 3 x 3 x 3 pattern
