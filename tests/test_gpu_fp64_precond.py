"""GPU: the FP64 path with the V-cycle and with plain CG (as created, and as set by a schedule):
the same discrete solution as the oracle's, from far fewer iterations; also at a second cell of a
frozen plan, whose hierarchy is the first cell's."""
import numpy as np
import pytest

import oracle
import paper_2011_07209_gb300.synth as synth
from test_gpu_parity import _compare, _oracle, _small_triclinic, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cell", ["cubic", "triclinic"])
def test_fp64_with_and_without_the_vcycle(ctx, cell):  # noqa: F811
    from paper_2011_07209_gb300 import driver, exx
    if cell == "cubic":
        ws, rp = synth.make_config(1), (8.0, 6.0, 8.0)
    else:
        ws, rp = _small_triclinic(), (7.0, 5.0, 6.5)
    outs = {}
    for name, pc in (("mg", exx.PRECOND_MG), ("plain", exx.PRECOND_NONE), ("plain by schedule", exx.PRECOND_MG)):
        p = exx.make_params(r_pair=rp[0], r_pe=rp[1], r_me=rp[2], tol=1e-10, precision=exx.FP64, precond=pc)
        cr = driver.prepare(ctx, ws, p)
        if name == "plain by schedule":
            cr.plan.set_schedule(exx.PRECOND_NONE, 0.8)
        g = driver.run(ctx, cr)
        g["dxx"] = cr.dxx.cpu().numpy()
        assert g["status"] == 0 and cr.plan.schedule()["precond"] == ("mg" if name == "mg" else "none")
        outs[name] = g
    o = _oracle(ws, *rp, 1e-10, cr.dbox, cr.dbox_lo_np)
    for g in outs.values():
        _compare(g, o, "fp64")
    mg, plain, by_schedule = outs["mg"], outs["plain"], outs["plain by schedule"]
    assert by_schedule["total_cg_iter"] == plain["total_cg_iter"] and by_schedule["e_xx"] == plain["e_xx"]
    # the bound of the mixed path's own comparison (a V-cycle replaces about ten plain iterations)
    assert mg["total_cg_iter"] < 0.25 * plain["total_cg_iter"], (mg["total_cg_iter"], plain["total_cg_iter"])


def test_fp64_second_cell_of_a_frozen_plan(ctx):  # noqa: F811
    from paper_2011_07209_gb300 import driver, exx
    ws0 = _small_triclinic()
    ws1 = synth.strained(ws0, np.array([[0.004, 0.002, -0.001], [0.002, -0.003, 0.001], [-0.001, 0.001, 0.002]]))
    p = exx.make_params(r_pair=7.0, r_pe=5.0, r_me=6.5, tol=1e-10, precision=exx.FP64, frozen=True)
    plan = exx.Plan(ctx, ws0.lattice, ws0.n, p, ws0.n_orb, ws0.box)
    out = {}
    for pc in (exx.PRECOND_MG, exx.PRECOND_NONE):
        plan.set_schedule(pc, 0.8)
        driver.run(ctx, driver.prepare(ctx, ws0, p, plan=plan))
        cr = driver.prepare(ctx, ws1, p, plan=plan)
        out[pc] = driver.run(ctx, cr)
        out[pc]["dxx"] = cr.dxx.cpu().numpy()
    po = oracle.make_params(r_pair=7.0, r_pe=5.0, r_me=6.5, tol=1e-10, lattice0=ws0.lattice)
    o = oracle.exx(ws1, po, dbox=cr.dbox, dbox_lo=cr.dbox_lo_np)
    for g in out.values():
        assert g["status"] == 0
        _compare(g, o, "fp64")
    assert out[exx.PRECOND_MG]["total_cg_iter"] < 0.25 * out[exx.PRECOND_NONE]["total_cg_iter"]
