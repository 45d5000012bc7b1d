"""GPU: a cell whose stencil does not fit the halo is refused every time, also after other cells,
and leaves the plan's own cell as it was.  (What reaches the kernels: test_refused_cells_cpu.py.)"""
import numpy as np
import pytest

import paper_2011_07209_gb300.synth as synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("frozen", [True, False])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_refused_cell_leaves_the_plan_as_it_was(frozen, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_07209_gb300 import driver, exx
    lat = np.diag([11.0] * 3)
    shear = 11.0 * np.array([[1, 0, 0], [0.02, 1, 0], [0.01, -0.015, 1]])
    same_dirs = 11.0 * np.array([[1, 0, 0], [0.021, 1, 0], [0.012, -0.016, 1]])
    ws = synth.gaussian_set(lat, (48,) * 3, np.array([[5.0, 5.0, 5.0], [6.0, 5.5, 4.5]]))
    ctx = exx.Context(0)
    try:
        # R_ME - R_PE holds three grid steps along the axes (0.69 bohr), not along the slanted directions
        p = exx.make_params(r_pair=6.0, r_pe=4.0, r_me=4.8, tol=1e-10, frozen=frozen,
                            precision=exx.FP64 if precision == "fp64" else exx.MIXED)
        cr = driver.prepare(ctx, ws, p)
        first = driver.run(ctx, cr)
        d_first = cr.dxx.cpu().numpy()
        assert first["status"] == exx.OK and first["e_xx"] != 0.0
        for c in (shear, shear, same_dirs):
            assert driver.run(ctx, cr, lattice=c, pair_outputs=False, check=False)["status"] == exx.ERR_HALO
        again = driver.run(ctx, cr)
        # the same plan and inputs: equal up to the order of the atomic sums into D
        assert again["e_xx"] == first["e_xx"] and np.array_equal(again["stress"], first["stress"])
        assert np.abs(cr.dxx.cpu().numpy() - d_first).max() < 1e-12 * np.abs(d_first).max()
        assert driver.run(ctx, cr, lattice=same_dirs, pair_outputs=False, check=False)["status"] == exx.ERR_HALO
    finally:
        ctx.close()
