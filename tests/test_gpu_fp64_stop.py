"""GPU: what the FP64 path accepts is |b - A v| <= cg_tol |b| on the true residual, with and without
the preconditioner: at the starting guess and at the last allowed iteration too."""
import numpy as np
import pytest

import paper_2011_07209_gb300.synth as synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def solve():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_07209_gb300 import driver, exx
    ctx = exx.Context(0)
    ws = synth.gaussian_set(np.diag([11.0] * 3), (40,) * 3, np.array([[5.0, 5.2, 4.9]]))   # one pair: one iteration count

    def go(tol, cap, precond):
        p = exx.make_params(r_pair=6.0, r_pe=4.0, r_me=5.5, tol=tol, max_iter=cap, precision=exx.FP64, precond=precond)
        cr = driver.prepare(ctx, ws, p, want_d=False)
        return driver.run(ctx, cr, pair_outputs=False, check=False)

    yield go
    ctx.close()


def test_last_allowed_iteration(solve):
    from paper_2011_07209_gb300 import exx
    for tol in np.geomspace(1e-4, 1e-10, 25):
        # the iteration after which the preconditioned CG's residual is at most tol |b| (it goes on to a fifth of the bound)
        n = solve(5.0 * tol, 1000, exx.PRECOND_MG)["max_cg_iter"]
        assert n > 1
        r = solve(tol, n, exx.PRECOND_MG)
        assert r["status"] == exx.OK and r["max_cg_iter"] <= n, (tol, n, r["status"])
    # one iteration is not enough for 1e-10
    assert solve(1e-10, 1, exx.PRECOND_MG)["status"] == exx.ERR_CG


def test_guess_that_meets_the_bound(solve):
    from paper_2011_07209_gb300 import exx
    seen = set()
    for tol in np.geomspace(0.004, 0.5, 16):
        plain, mg = solve(tol, 100, exx.PRECOND_NONE), solve(tol, 100, exx.PRECOND_MG)
        assert plain["status"] == mg["status"] == exx.OK
        assert (plain["total_cg_iter"] == 0) == (mg["total_cg_iter"] == 0), tol
        seen.add(plain["total_cg_iter"] == 0)
    assert seen == {True, False}   # the range holds the guess's residual
