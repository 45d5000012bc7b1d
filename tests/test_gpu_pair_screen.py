"""The screened pair list (FP32 screen, then the rule on the survivors) against the rule itself
in numpy float64, row for row: both entry points' kernels share it, so the allocation-free one
stands for both here (test_zz_no_alloc.py compares the two).  Sizes at the edges of its CTAs (4 rows,
256 columns, survivor lists of 1024), centres far outside the cell and on exact half-cell
distances, skewed cells, cutoffs from zero to beyond the cell."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _round(x):   # half away from zero
    t = np.trunc(x)
    return np.where(np.abs(x - t) >= 0.5, t + np.sign(x), t)


def _dot(r, a, b, c):
    return (r[0] * a + r[1] * b) + r[2] * c


def _hinv(h):
    """make_metric's h^-1: adjugate over determinant, in its operation order."""
    c00 = h[1][1] * h[2][2] - h[1][2] * h[2][1]
    c01 = h[1][0] * h[2][2] - h[1][2] * h[2][0]
    c02 = h[1][0] * h[2][1] - h[1][1] * h[2][0]
    det = h[0][0] * c00 - h[0][1] * c01 + h[0][2] * c02
    return np.array([[c00, h[0][2] * h[2][1] - h[0][1] * h[2][2], h[0][1] * h[1][2] - h[0][2] * h[1][1]],
                     [h[1][2] * h[2][0] - h[1][0] * h[2][2], h[0][0] * h[2][2] - h[0][2] * h[2][0],
                      h[0][2] * h[1][0] - h[0][0] * h[1][2]],
                     [c02, h[0][1] * h[2][0] - h[0][0] * h[2][1], h[0][0] * h[1][1] - h[0][1] * h[1][0]]]) / det


def _rule(h, hinv, n, cen, r_pair):
    s = np.stack([_dot(hinv[a], cen[:, 0], cen[:, 1], cen[:, 2]) for a in range(3)], 1)
    rows = []
    for i in range(len(cen)):
        d = s[i:] - s[i]
        ds = d - _round(d)
        best = np.full(len(ds), np.inf)
        kb = np.zeros((len(ds), 3), int)
        for k in np.ndindex(3, 3, 3):
            k = np.array(k) - 1
            t = ds + k
            x = [_dot(h[a], t[:, 0], t[:, 1], t[:, 2]) for a in range(3)]
            dd = (x[0] * x[0] + x[1] * x[1]) + x[2] * x[2]
            new = dd < best
            best[new] = dd[new]
            kb[new] = k
        q = np.nonzero(best <= r_pair * r_pair)[0]
        g = np.stack([_round(np.float64(n[a]) * (s[i, a] + (ds[q, a] + kb[q, a]) * 0.5)) % n[a] for a in range(3)], 1)
        rows.append(np.concatenate([np.full((len(q), 1), i), (i + q)[:, None], kb[q], g], 1))
    return np.concatenate(rows).astype(np.int32)


SKEW = {"cubic": np.eye(3), "skew": np.array([[1, 0, 0], [0.9, 1, 0], [-0.8, 0.7, 1]], float),
        "flat": np.array([[1, 0, 0], [0.1, 1, 0], [0.05, -0.08, 0.21]])}


@pytest.mark.parametrize("m, cell, r_pair, spread", [
    (1, "cubic", 8.0, 1.0), (3, "skew", 8.0, 1.0), (4, "flat", 3.0, 1.0), (5, "cubic", 0.0, 1.0), (255, "skew", 6.0, 1.0),
    (257, "cubic", 6.0, 40.0), (516, "flat", 4.0, 1.0), (1300, "cubic", 100.0, 1.0), (300, "cubic", 7.35, 0.0),
    (300, "skew", 9.0, -1.0)])
def test_screened_list_is_the_rule(m, cell, r_pair, spread):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_07209_gb300 import exx
    rng = np.random.default_rng(m)
    lat = 14.7 * SKEW[cell]
    n = (48, 47, 45)
    f = rng.random((m, 3)) * max(spread, 1.0) - (0.5 * spread if spread > 1 else 0.0)
    if spread <= 0.0:   # multiples of 1/8: image distances tie, differences hit +-1/2
        f = np.round(f * 8) / 8
    if spread < 0.0:    # and coincident centres
        f[::2] = f[0]
    cen = f @ lat
    h = lat.T
    cap = m * (m + 1) // 2
    rows = torch.zeros((cap, 8), dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    c = torch.tensor(cen, device="cuda")
    assert exx.pair_list_noalloc(lat, n, c, m, r_pair, rows, cnt) == exx.OK
    got = rows[:int(cnt)].cpu().numpy()
    assert np.array_equal(got, _rule(h, _hinv(h), n, cen, r_pair))
