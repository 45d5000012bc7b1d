"""The pair list where its CTAs change shape (one, two and four rows per CTA: rows that fill a
CTA in part, survivor lists that are emptied on the way) and over the cells of a batch, row for
row against the rule in numpy float64."""
import numpy as np
import pytest

from test_gpu_pair_screen import SKEW, _hinv, _rule

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def exx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_07209_gb300 import exx
    return exx


# cutoffs: about one pair in twenty, and all of them (lists of 1024 overflow into the rule from 769 on)
@pytest.mark.parametrize("m, cell, r_pair", [(303, "cubic", 3.3), (304, "skew", 3.3), (305, "flat", 3.0), (305, "skew", 60.0),
                                             (1001, "cubic", 60.0), (1215, "skew", 3.3), (1216, "flat", 2.5),
                                             (1217, "skew", 60.0), (1219, "cubic", 3.3)])
def test_list_at_the_edges_of_its_ctas(exx, m, cell, r_pair):
    import torch
    rng = np.random.default_rng(m)
    lat, n = 14.7 * SKEW[cell], (48, 47, 45)
    cen = rng.random((m, 3)) @ lat
    cap = m * (m + 1) // 2
    rows = torch.full((cap + 1, 8), -7, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert exx.pair_list_noalloc(lat, n, torch.tensor(cen, device="cuda"), m, r_pair, rows[:cap], cnt) == exx.OK
    k, h = int(cnt), lat.T
    want = _rule(h, _hinv(h), n, cen, r_pair)
    assert k == len(want) and np.array_equal(rows[:k].cpu().numpy(), want)
    assert bool((rows[k:] == -7).all())


@pytest.mark.parametrize("sizes", [(5, 1, 0, 7), (150, 0, 151, 1, 7), (401, 0, 403, 2, 411)])
def test_lists_of_a_batch(exx, sizes):
    """Orbital counts that leave CTAs part filled before another cell begins; one, two and four rows per CTA."""
    import torch
    ctx = exx.Context(0)
    try:
        rng = np.random.default_rng(sum(sizes))
        p = exx.make_params(r_pair=1.6, r_pe=1.5, r_me=3.6, tol=1e-3, precision=exx.MIXED)
        plans, cells, orbs, results, keep, cens = [], [], [], [], [], []
        for c, m in enumerate(sizes):
            lat, n, box = (8.0 + 0.3 * c) * SKEW["cubic"], (16, 16, 16), (4, 4, 4)
            cen = rng.random((m, 3)) @ lat
            t = [torch.tensor(cen, device="cuda"), torch.zeros((m, 3), dtype=torch.int32, device="cuda"),
                 torch.tensor(rng.random((m, 4, 4, 4)), device="cuda")]
            keep.append(t)
            cens.append(cen)
            plans.append(exx.Plan(ctx, lat, n, p, max(m, 1), box))
            cells.append((lat, n))
            orbs.append(exx.make_orbitals(m, box, *(t if m else (None, None, None))))
            results.append(exx.make_result())
        exx.solve_batch(ctx, plans, cells, orbs, results)
        for (lat, n), plan, cen, r in zip(cells, plans, cens, results):
            h = lat.T
            want = _rule(h, _hinv(h), n, cen, 1.6) if len(cen) else np.zeros((0, 8), np.int32)
            assert r.n_pairs == len(want)
            assert np.array_equal(np.asarray(plan.pair_list()).reshape(-1, 8), want)
    finally:
        ctx.close()
