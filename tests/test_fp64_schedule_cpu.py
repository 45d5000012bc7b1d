"""The schedule of an FP64 plan says what its solves run and can be set like a mixed plan's
(host only: api.cu over stand-ins for CUDA, see test_refused_cells_cpu.py); the byte count of the
benchmark for that path."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402
from test_refused_cells_cpu import PLAN, harness, run  # noqa: E402,F401

FP64, MIXED = 0, 1
ERR_ARG = 1
TO_SECOND_ORDER = 272 / 245   # Jacobi weight of the second-order operator per weight of the sixth-order one


@pytest.mark.parametrize("precision", [FP64, MIXED])
def test_schedule_is_what_runs(harness, precision):  # noqa: F811
    solve, weight = f"step {PLAN}", lambda om: pytest.approx(om * TO_SECOND_ORDER, abs=1e-4)
    r = run(harness, f"plan {PLAN} 48 48 48 4.0 6.0 0 {precision} 1", "get", solve, "seen", "set 0 0.8", solve, "seen", "get",
            "set 1 0.6", solve, "seen", "get")
    assert r[1] == [0, 1, 0.8, 14, 0.0] and r[3] == [1, weight(0.8)]    # as created: the V-cycle
    assert r[4] == 0 and r[6][0] == 0 and r[7] == [0, 0, 0.8, 14, 0.0]  # plain CG as asked
    assert r[8] == 0 and r[10] == [1, weight(0.6)] and r[11] == [0, 1, 0.6, 14, 0.0]


@pytest.mark.parametrize("precision", [FP64, MIXED])
def test_no_hierarchy_no_preconditioner(harness, precision):  # noqa: F811
    r = run(harness, f"plan {PLAN} 48 48 48 4.0 6.0 0 {precision} 0", "get", "set 1 0.8", f"step {PLAN}", "seen", "set 0 0.8")
    assert r[1][:2] == [0, 0] and r[2] == ERR_ARG and r[4][0] == 0 and r[5] == 0


def test_autotune_of_an_fp64_plan_keeps_its_schedule(harness):  # noqa: F811
    r = run(harness, f"plan {PLAN} 48 48 48 4.0 6.0 0 {FP64} 1", "auto", "get", f"step {PLAN}", "seen")
    assert r[1] == r[2] == [0, 1, 0.8, 14, 0.0] and r[4][0] == 1


def test_algorithmic_bytes_fp64_multigrid():
    n_pairs, it, ref, n_pe, n_me = 2, 15, 3, 1000, 2500
    per_pair = 2 * n_me * 8 + 2 * n_me * 16 + 8 * n_pe
    # 7 FP64 and 7 FP32 accesses per fine point-iteration, 8 FP32 per coarse point
    assert bench.algorithmic_bytes(n_pairs, it, ref, n_pe, n_me, 8, [1000, 140, 20]) == \
        it * (7 * n_pe * 8 + 7 * n_pe * 4 + 8 * 4 * 160) + ref * 24 * n_pe + n_pairs * per_pair
