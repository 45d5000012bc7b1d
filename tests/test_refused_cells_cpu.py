"""A solve at a cell that is refused (halo) or whose upload fails (memory) must leave the plan
consistent: the same cell and later cells with the same stencil directions are refused again, and
what reaches the kernels is always a layout of the stencil that goes with it.  api.cu and plan.cpp
run on the host over stand-ins for the CUDA runtime and the launches (tests/api_check.cpp)."""
import json
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2011_07209_gb300", "csrc")
OK, HALO, OOM = 0, 3, 8


def _cuda_include():
    nv = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nv))), "include")
    return d if os.path.exists(os.path.join(d, "cuda_runtime.h")) else None


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx, inc = shutil.which("g++") or shutil.which("c++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("no host C++ compiler or no CUDA headers")
    exe = str(tmp_path_factory.mktemp("api") / "api_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-x", "c++", "-I", inc, "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "api_check.cpp"), os.path.join(CSRC, "plan.cpp"), "-o", exe], check=True)
    return exe


def run(exe, *lines):
    out = subprocess.run([exe], input="\n".join(lines), capture_output=True, text=True, check=True).stdout
    return [json.loads(s) for s in out.splitlines()]


def cell(*shear, scale=1.0):
    a, b, c = shear or (0.0, 0.0, 0.0)
    return " ".join(repr(float(x)) for x in (11.0 * scale * np.array([[1, 0, 0], [a, 1, 0], [b, c, 1]])).ravel())


PLAN, WIDER = cell(), cell(scale=1.001)
SHEAR, SAME_DIRS = cell(0.02, 0.01, -0.015), cell(0.021, 0.012, -0.016)
TIGHT, ROOMY = 4.8, 6.0   # R_ME that holds the axes' stencil only, and one that holds the slanted directions'


def test_the_cells_are_what_they_should_be(harness):
    plan, shear, same = run(harness, *[f"layout {PLAN} 48 48 48 {c} 4.0 {TIGHT}" for c in (PLAN, SHEAR, SAME_DIRS)])
    assert plan == [OK] and shear[0] == same[0] == HALO and shear[1:] == same[1:] and len(shear) == 4
    roomy = run(harness, f"layout {PLAN} 48 48 48 {SHEAR} 4.0 {ROOMY}")[0]
    assert roomy[0] == OK


# frozen: 1 (directions of the cell), 0 (everything rebuilt for the cell); FP64 and mixed
@pytest.mark.parametrize("frozen", [1, 0])
@pytest.mark.parametrize("precision", [0, 1])
def test_refused_cells_stay_refused(harness, frozen, precision):
    r = run(harness, f"plan {PLAN} 48 48 48 4.0 {TIGHT} {frozen} {precision} 1", f"step {SHEAR}", f"step {SHEAR}",
            f"step {SAME_DIRS}", f"step {PLAN}", f"step {SAME_DIRS}", f"step {WIDER}", f"step {PLAN}")
    refused, solved = [HALO, None], [OK, True]
    assert r == [OK, refused, refused, refused, solved, refused, solved, solved]


@pytest.mark.parametrize("frozen", [1, 0])
@pytest.mark.parametrize("fail_at", [1, 2, 5, 9, 14])
def test_failed_upload_is_made_again(harness, frozen, fail_at):
    r = run(harness, f"plan {PLAN} 48 48 48 4.0 {ROOMY} {frozen} 1 1", f"oom {fail_at}", f"step {SHEAR}", "oom 0",
            f"step {SHEAR}", f"step {SAME_DIRS}", f"step {PLAN}")
    assert r == [OK, [OOM, None], [OK, True], [OK, True], [OK, True]]


@pytest.mark.parametrize("frozen", [1, 0])
def test_definiteness_is_asked_when_the_stencil_changes(harness, frozen):
    """A cell with a negative stencil coefficient: mg_definite scans 32^3 frequencies there."""
    sheared, other = cell(1.1, 0.0, 0.0), cell(1.102, 0.0, 0.0)
    r = run(harness, f"plan {sheared} 36 36 36 3.0 5.5 {frozen} 1 1", "scans", f"step {sheared}", f"step {sheared}", "scans",
            f"step {other}", "scans", f"step {other}", "scans", f"plan {sheared} 36 36 36 3.0 5.5 {frozen} 1 0",
            f"step {other}", "scans")
    solved = [OK, True]
    # once for a plan, not at all for its solves, once for another cell, never without the preconditioner
    assert r == [OK, 1, solved, solved, 0, solved, 1, solved, 0, OK, solved, 0]
