"""What is measured: exact-exchange evaluations as a user of the library runs them.

Every case goes through the public binding (``exx.Context``, ``exx.Plan``, ``exx.solve``,
``exx.solve_batch``, ``exx.pair_list_noalloc``) on water-like sets of localized orbitals
(the recipe of ``synth.py``, sampled on the GPU).  A case's ``kind`` is "solve" (one cell per
call, or two MD steps of one plan), "batch" (several cells in one launch) or "list" (the
pair list alone).  Sizes are those of the package's configurations (``synth.CONFIGS``,
``synth.BATCH_CELLS``), of its smoke run and of its benchmark, or subsets of their orbitals.
"""
import math

import numpy as np
import torch

from paper_2011_07209_gb300 import exx, synth

_CTX = []


def _ctx():
    # one context per process, as a program keeps it
    if not _CTX:
        _CTX.append(exx.Context(0))
    return _CTX[0]


def _solve(name, shape, length, n, mol, **more):
    c = dict(name=name, kind="solve", shape=shape, length=length, n=n, mol=mol, orbitals=4 * mol, precision="mixed",
             r_pair=8.0, r_pe=6.0, r_me=8.0, tol=1e-9, steps=1, warm=False, host=False, pairs_out=False, dxx=True,
             stress=exx.STRESS_FULL)
    c.update(more)
    return c


def listed():
    return [
        # the pair list of the 1024-orbital cell alone (an engine that sizes its buffers, or re-lists every step)
        dict(name="list_1024", kind="list", shape="triclinic37", length=37.3, n=190, orbitals=1024, r_pair=8.0),
        # one molecule: the smallest evaluation, fewer pairs than the GPU has SMs (latency)
        _solve("water1_triclinic11", "triclinic", 11.0, 40, 1, r_pair=6.0, r_pe=4.0, r_me=5.5, tol=1e-10),
        # four molecules in full FP64: the configuration for small reference calculations
        _solve("water4_fp64", "cubic", 14.7, 48, 4, precision="fp64", tol=1e-10),
        # the same cell on the mixed path, with the per-pair energies and stresses handed out
        _solve("water4_mixed", "cubic", 14.7, 48, 4, tol=1e-10, pairs_out=True),
        # FP64 at production spacing: the reference arm on the first orbitals of the 128-molecule cell
        _solve("triclinic128_first32_fp64", "triclinic", 29.6, 150, 128, orbitals=32, precision="fp64"),
        # liquid water, 32 molecules, the smaller Poisson radius, simple-cubic pressure instead of the stress integrals
        _solve("water32_rpe5", "cubic", 18.6, 93, 32, r_pe=5.0, r_me=7.0, stress=exx.STRESS_CUBIC),
        # end to end from pinned host buffers: orbitals in, D_xx out
        _solve("water32_host", "cubic", 18.6, 93, 32, host=True),
        # two MD steps of one frozen plan, each pair's CG started from the step before (warm start)
        _solve("triclinic128_first128_md_warm", "triclinic", 29.6, 150, 128, orbitals=128, steps=2, warm=True),
        # liquid water, 64 molecules
        _solve("water64", "cubic", 23.5, 120, 64),
        # two MD steps of one frozen plan in the 256-molecule triclinic cell (its first 256 orbitals)
        _solve("traj256_first256_md", "triclinic37", 37.3, 190, 256, orbitals=256, steps=2),
        # uneven cells in one launch, with Poisson radii from 5 to 7 bohr
        dict(name="batch3", kind="batch", sizes="32,64,96", radii="6,7,5", tol=1e-9),
        # 128 molecules in a triclinic cell: the largest evaluation
        _solve("triclinic128", "triclinic", 29.6, 150, 128),
    ]


def draw(rng):
    u = rng.random()
    if u < 0.12:
        m = round(math.exp(rng.uniform(math.log(16), math.log(1024))))
        length = max(11.0, 5.88 * m ** (1 / 3)) * rng.uniform(1.0, 1.1)
        return dict(kind="list", shape=rng.choice(["cubic", "ortho", "mono", "triclinic"]), length=round(length, 3),
                    n=max(24, round(length / 0.2)), orbitals=4 * m - rng.randrange(4), r_pair=rng.choice([6.0, 8.0, 10.0]))
    if u < 0.22:
        sizes = [round(math.exp(rng.uniform(math.log(4), math.log(40)))) for _ in range(rng.choice([2, 3]))]
        return dict(kind="batch", sizes=",".join(map(str, sizes)), tol=1e-9,
                    radii=",".join(rng.choice(["5", "6", "7"]) for _ in sizes))
    fp64 = rng.random() < 0.2
    mol = round(math.exp(rng.uniform(0.0, math.log(5 if fp64 else 80))))
    r_pe = rng.choice([4.0, 5.0, 6.0, 6.0, 7.0])
    if mol < 4:
        r_pe = min(r_pe, 5.0)
    length = max(2 * r_pe + 2.7, 5.88 * mol ** (1 / 3)) * rng.uniform(1.0, 1.12)
    spacing = rng.uniform(0.19, 0.32) if mol < 8 else rng.uniform(0.19, 0.22)
    shape = rng.choice(["cubic", "ortho", "mono", "triclinic", "triclinic37"])
    # MD steps in a cell that is already skew, whose strained steps keep the plan's stencil directions
    steps = 2 if not fp64 and mol < 40 and shape.startswith("triclinic") and rng.random() < 0.6 else 1
    stress = rng.choice([exx.STRESS_FULL, exx.STRESS_FULL, exx.STRESS_ISOTROPIC])
    return dict(kind="solve", shape=shape, length=round(length, 3), n=round(length / spacing), mol=mol,
                orbitals=max(1, 4 * mol - rng.choice([0, 0, 1, 3])), precision="fp64" if fp64 else "mixed",
                r_pair=rng.choice([6.0, 8.0]), r_pe=r_pe, r_me=r_pe + 2.0, tol=rng.choice([1e-9, 1e-9, 1e-10]),
                steps=steps, warm=steps == 2 and rng.random() < 0.5, host=rng.random() < 0.15,
                pairs_out=rng.random() < 0.2, dxx=rng.random() < 0.9, stress=stress)


# ---------------------------------------------------------------- inputs
_SHAPES = {
    "cubic": [[1, 0, 0], [0, 1, 0], [0, 0, 1]],
    "ortho": [[1, 0, 0], [0, 1, 0], [0, 0, 1.045]],
    "mono": [[1, 0, 0], [0, 1, 0], [0.12, 0, 1]],
    "triclinic": [[1, 0, 0], [0.1, 1, 0], [0.05, -0.08, 1]],
    "triclinic37": [[1, 0, 0], [0.08, 1, 0], [0.04, 0.06, 1]],
}


def _cell(shape, length, n):
    lat = length * np.array(_SHAPES[shape], float)
    grid = [round(n * float(np.linalg.norm(v)) / length) for v in lat] if shape == "ortho" else [n] * 3
    return lat, np.array(grid, np.int32)


def _sites(lat, mol, rng, sep=synth.MIN_SEP):
    """Random sequential sites at least `sep` apart (minimum image), the separation eased if they do not fit."""
    h = lat.T
    img = np.array([(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1)], float) @ h.T
    got, tries = np.empty((0, 3)), 0
    while len(got) < mol:
        tries += 1
        if tries % 4000 == 0:
            sep *= 0.97
        s = rng.random(3)
        if len(got):
            d = got - s
            d = (d - np.round(d)) @ h.T
            if ((d[:, None, :] + img) ** 2).sum(-1).min() < sep * sep:
                continue
        got = np.vstack([got, s])
    return got @ h.T


def _centres(lat, mol, rng):
    oxy = _sites(lat, mol, rng)
    q = rng.normal(size=(mol, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    rot = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w), 2 * (x * y + z * w),
                    1 - 2 * (x * x + z * z), 2 * (y * z - x * w), 2 * (x * z - y * w), 2 * (y * z + x * w),
                    1 - 2 * (x * x + y * y)], -1).reshape(mol, 3, 3)
    tetra = np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]]) / math.sqrt(3.0)
    return (oxy[:, None, :] + synth.D_OC * np.einsum("mab,tb->mta", rot, tetra)).reshape(-1, 3)


def _orbitals(lat, n, cen, a, box=None):
    """exp(-d^2 / 2s^2) (1 + a.d) on each orbital's box, normalized on the grid; FP64 on the GPU."""
    hw = synth.box_halfwidth(lat, n, synth.R_PHI)
    box = np.minimum(2 * hw + 1, n).astype(np.int32) if box is None else box
    frac = cen @ np.linalg.inv(lat)
    frac -= np.floor(frac)
    lo = (np.floor(frac * n + 0.5).astype(np.int64) - box // 2).astype(np.int32)
    h = torch.tensor(lat.T / n, dtype=torch.float64, device="cuda")
    u = torch.meshgrid(*[torch.arange(int(b), device="cuda", dtype=torch.float64) for b in box], indexing="ij")
    grid = torch.stack(u, -1).reshape(-1, 3) @ h.T
    shift = torch.tensor(lo / n @ lat - frac @ lat, device="cuda")
    av = torch.tensor(a, device="cuda")
    phi = torch.empty((len(cen), len(grid)), dtype=torch.float64, device="cuda")
    for i in range(len(cen)):
        d = grid + shift[i]
        f = torch.exp(d.square().sum(1) * (-0.5 / synth.BOHR_S**2)) * (1.0 + d @ av[i])
        phi[i] = f
    dv = abs(np.linalg.det(lat)) / float(np.prod(n.astype(float)))
    phi /= (phi.square().sum(1, keepdim=True) * dv).sqrt()
    return box, lo, phi.reshape(len(cen), *[int(b) for b in box])


def _params(c):
    return exx.make_params(r_pair=c["r_pair"], r_pe=c["r_pe"], r_me=c["r_me"], tol=c["tol"],
                           precision=exx.FP64 if c["precision"] == "fp64" else exx.MIXED, frozen=c["steps"] > 1,
                           stress_mode=c["stress"], warm_start=c["warm"])


def _steps(c, seed):
    """The MD steps of a case: (lattice, n, centres, box, box_lo, phi) each."""
    rng = np.random.default_rng([seed, c["n"]])
    lat, n = _cell(c["shape"], c["length"], c["n"])
    cen = _centres(lat, c["mol"], rng)[:c["orbitals"]]
    a = rng.normal(scale=synth.A_SIGMA, size=cen.shape)
    box, out = None, []
    for k in range(c["steps"]):
        if k:
            e = rng.normal(scale=1e-3, size=(3, 3))
            f = np.eye(3) + 0.5 * (e + e.T)
            lat = (f @ lat.T).T
            # a warm-started run takes small steps; otherwise the trajectory of the benchmark
            cen = cen @ f.T + rng.normal(scale=0.01 if c["warm"] else 0.05, size=cen.shape)
        box, lo, phi = _orbitals(lat, n, cen, a, box)
        out.append((lat, n, cen, box, lo, phi))
    return out


def _buffers(c, step, params):
    """The call's orbitals and result descriptors, with the buffers that they point to."""
    lat, n, cen, box, lo, phi = step
    m = len(cen)
    dbox, dlo = exx.dbox_layout(lat, n, cen, params)
    host = c["host"]

    def put(x):
        t = torch.as_tensor(np.ascontiguousarray(x))
        return t.pin_memory() if host else t.cuda()

    def zeros(shape, dt=torch.float64):
        return torch.zeros(shape, dtype=dt, pin_memory=True) if host else torch.zeros(shape, dtype=dt, device="cuda")

    b = dict(lat=lat, n=n, cen=put(cen), lo=put(lo), phi=phi.cpu().pin_memory() if host else phi, dbox=dbox,
             dlo=put(dlo), dxx=zeros([m] + [int(x) for x in dbox]) if c["dxx"] else None, m=m, box=box, host=host,
             cap=m * (m + 1) // 2 if c["pairs_out"] else 0)
    if b["cap"]:
        b["pair_e"], b["pair_sig"] = zeros(b["cap"]), zeros((b["cap"], 3, 3))
    return b


def _descriptors(b):
    mem = exx.MEM_HOST if b["host"] else exx.MEM_DEVICE
    orb = exx.make_orbitals(b["m"], b["box"], b["cen"], b["lo"], b["phi"], mem)
    res = exx.make_result(b["dxx"], b["dbox"], b["dlo"] if b["dxx"] is not None else None, mem, b["cap"],
                          b.get("pair_e"), b.get("pair_sig"))
    return orb, res


def _batch_cells(c):
    """The cells of a batch: liquid density, spacing 0.2, one shape after the other."""
    shapes = ["cubic", "ortho", "mono"]
    out = []
    for k, (mol, r_pe) in enumerate(zip(c["sizes"].split(","), c["radii"].split(","))):
        mol, r_pe = int(mol), float(r_pe)
        length = round(max(2 * r_pe + 2.7, 5.88 * mol ** (1 / 3)), 2)
        out.append(_solve("", shapes[k], length, round(length / 0.2), mol, r_pe=r_pe, r_me=r_pe + 2.0, tol=c["tol"]))
    return out


def prepare(case, seed):
    if case["kind"] == "list":
        rng = np.random.default_rng([seed, case["orbitals"]])
        lat, n = _cell(case["shape"], case["length"], case["n"])
        m = case["orbitals"]
        mol = -(-m // 4)
        # sites on a jittered lattice: the list depends on the centres alone
        k = math.ceil(mol ** (1 / 3))
        s = np.array([(i, j, l) for i in range(k) for j in range(k) for l in range(k)], float)
        s = (s[np.sort(rng.permutation(len(s))[:mol])] + rng.random((mol, 3))) / k
        cen = (s @ lat)[:, None, :] + synth.D_OC * rng.normal(size=(mol, 4, 3)) / math.sqrt(3.0)
        cap = m * (m + 1) // 2 if m < 1024 else 256 * m
        return dict(kind="list", lat=lat, n=n, m=m, r_pair=case["r_pair"],
                    cen=torch.tensor(cen.reshape(-1, 3)[:m].copy(), device="cuda"),
                    rows=torch.zeros((cap, 8), dtype=torch.int32, device="cuda"),
                    count=torch.zeros(1, dtype=torch.int32, device="cuda"))
    ctx = _ctx()
    cells = _batch_cells(case) if case["kind"] == "batch" else [case]
    state = dict(kind=case["kind"], ctx=ctx, plans=[], calls=[])
    for k, c in enumerate(cells):
        p = _params(c)
        steps = _steps(c, seed + 1000 * k)
        lat, n, cen, box = steps[0][:4]
        state["plans"].append(exx.Plan(ctx, lat, n, p, len(cen), box))
        state["calls"].append([_buffers(c, s, p) for s in steps])
    return state


# ---------------------------------------------------------------- one pass
def _outputs(res, b):
    r = exx.result_dict(res)
    out = {"e_xx": r["e_xx"], "dedh": r["dedh"], "stress": r["stress"], "p_int": r["p_int"], "n_pairs": r["n_pairs"]}
    if b["dxx"] is not None:
        out["dxx"] = b["dxx"]
    if b["cap"]:
        out["pair_e"], out["pair_sig"] = b["pair_e"], b["pair_sig"]
    return out


def run(state):
    if state["kind"] == "list":
        code = exx.pair_list_noalloc(state["lat"], state["n"], state["cen"], state["m"], state["r_pair"],
                                     state["rows"], state["count"])
        assert code == exx.OK, code
        return {"rows": state["rows"], "n_pairs": state["count"]}
    if state["kind"] == "batch":
        bs = [calls[0] for calls in state["calls"]]
        d = [_descriptors(b) for b in bs]
        results = [r for _, r in d]
        exx.solve_batch(state["ctx"], state["plans"], [(b["lat"], b["n"]) for b in bs], [o for o, _ in d], results)
        return [_outputs(r, b) for r, b in zip(results, bs)]
    out = []
    for b in state["calls"][0]:
        orb, res = _descriptors(b)
        exx.solve(state["ctx"], state["plans"][0], b["lat"], b["n"], orb, res)
        out.append(_outputs(res, b))
    return out


# ---------------------------------------------------------------- work
def _pairs(c):
    """Expected unique pairs: each orbital's neighbours within R_pair at the cell's orbital density."""
    lat, _ = _cell(c["shape"], c["length"], c["n"])
    m, v = c["orbitals"], abs(np.linalg.det(lat))
    near = min(1.0, 4.0 / 3.0 * math.pi * c["r_pair"] ** 3 / v)
    return m + 0.5 * m * (m - 1) * near


def work(case):
    if case["kind"] == "list":
        m = case["orbitals"]
        rows = _pairs(case)
        return {"bytes": 24.0 * m + 32.0 * rows, "flops": 0.5 * m * (m + 1) * 30.0}
    total = {"bytes": 0.0, "flops": 0.0}
    for c in (_batch_cells(case) if case["kind"] == "batch" else [case]):
        lat, n = _cell(c["shape"], c["length"], c["n"])
        dv = abs(np.linalg.det(lat)) / float(np.prod(n.astype(float)))
        box = np.minimum(2 * synth.box_halfwidth(lat, n, synth.R_PHI) + 1, n)
        dbox = np.minimum(2 * exx.dbox_halfwidth(lat, n, _params(c)) + 1, n)
        pe = 4.0 / 3.0 * math.pi * c["r_pe"] ** 3 / dv
        me = 4.0 / 3.0 * math.pi * c["r_me"] ** 3 / dv
        stcl = {"cubic": 19, "ortho": 19, "mono": 25}.get(c["shape"], 37)
        # orbitals read and D_xx written once; per pair the density, the moments, the operator applied once (what the
        # stopping rule needs at the solution), the energy and stress integrals, and D_xx on PE and shell
        flops = _pairs(c) * (pe * (1 + 2 * 49 + 2 * stcl + 2 + 9 * 8) + (me - pe) * 2 * 49 + 4 * me)
        total["bytes"] += c["steps"] * 8.0 * c["orbitals"] * (float(np.prod(box)) + (float(np.prod(dbox)) if c["dxx"] else 0.0))
        total["flops"] += c["steps"] * flops
    return total


# ---------------------------------------------------------------- the same in plain FP64 torch
def _harmonics(x, y, z, lmax=6):
    """r^l Y_lm (real, orthonormal), [(lmax + 1)^2, points]."""
    a, b = [torch.ones_like(x)], [torch.zeros_like(x)]
    for m in range(lmax):
        a, b = a + [x * a[m] - y * b[m]], b + [x * b[m] + y * a[m]]
    r2, rows = x * x + y * y + z * z, {}
    for m in range(lmax + 1):
        q = {m: torch.full_like(x, float(np.prod(np.arange(1, 2 * m, 2))) if m else 1.0)}
        for l in range(m + 1, lmax + 1):
            q[l] = ((2 * l - 1) * z * q[l - 1] - ((l + m - 1) * r2 * q[l - 2] if l > m + 1 else 0.0)) / (l - m)
        for l in range(m, lmax + 1):
            c = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m))
            if m == 0:
                rows[l * l + l] = c * q[l]
            else:
                rows[l * l + l + m], rows[l * l + l - m] = math.sqrt(2) * c * q[l] * a[m], math.sqrt(2) * c * q[l] * b[m]
    return torch.stack([rows[k] for k in range((lmax + 1) ** 2)])


def _offsets(lat0, n, r_pe, r_me):
    h = lat0.T / n
    hw = synth.box_halfwidth(lat0, n, r_me)
    m = np.stack(np.meshgrid(*[np.arange(-w, w + 1) for w in hw], indexing="ij"), -1).reshape(-1, 3)
    d2 = ((m @ h.T) ** 2).sum(1)
    return m[d2 <= r_pe * r_pe], m[(d2 > r_pe * r_pe) & (d2 <= r_me * r_me)]


def _directions(lat, n):
    """Directions and coefficients of the Laplacian: G_ab = N_a N_b (h^-1 h^-T)_ab split into pure second derivatives."""
    hi = np.linalg.inv(lat.T) * n[:, None]
    g = hi @ hi.T
    dirs, coef, diag = [np.eye(3, dtype=int)[k] for k in range(3)], [], np.diag(g).copy()
    tiny = 1e-12 * diag.max()
    pairs = [(0, 1), (0, 2), (1, 2)]
    if sum(abs(g[p]) > tiny for p in pairs) > 1:
        use = pairs
    else:
        use = [p for p in pairs if abs(g[p]) > tiny]
    for a, b in use:
        s = 1 if g[a, b] > 0 else -1
        d = np.zeros(3, int)
        d[a], d[b] = 1, s
        dirs.append(d)
        coef.append(s * g[a, b])
        diag[a] -= s * g[a, b]
        diag[b] -= s * g[a, b]
    return dirs, list(diag) + coef


def _exact_step(c, lat0, step):
    lat, n, cen, box, lo, phi = step
    dev, m = phi.device, len(cen)
    h = lat.T
    hinv = np.linalg.inv(h)
    dv = abs(np.linalg.det(lat)) / float(np.prod(n.astype(float)))
    # pair list
    s = cen @ hinv.T
    img = np.array([(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1)], float)
    ii, jj, gg = [], [], []
    for i in range(m):
        ds = s[i:] - s[i]
        ds = ds - np.round(ds)
        t = ds[:, None, :] + img
        d2 = ((t @ h.T) ** 2).sum(-1)
        k = d2.argmin(1)
        near = np.nonzero(d2[np.arange(len(k)), k] <= c["r_pair"] ** 2)[0]
        x = n * (s[i] + 0.5 * t[near, k[near]])
        gg.append(np.mod(np.floor(np.abs(x) + 0.5) * np.sign(x), n).astype(np.int64))
        ii.append(np.full(len(near), i))
        jj.append(near + i)
    ii, jj, gg = np.concatenate(ii), np.concatenate(jj), np.concatenate(gg)
    pe, sh = _offsets(lat0, n, c["r_pe"], c["r_me"])
    me = np.concatenate([pe, sh])
    dirs, coef = _directions(lat, n)
    w2, w1 = [-49.0 / 18, 1.5, -0.15, 1.0 / 90], [0.0, 0.75, -0.15, 1.0 / 60]
    # dense box of every point that a stencil reaches from PE
    half = np.abs(pe).max(0) + 3
    size = [int(2 * w + 1) for w in half]
    stride = np.array([size[1] * size[2], size[2], 1])
    pe_at = torch.tensor((pe + half) @ stride, device=dev)
    inside = (np.abs(sh) <= half).all(1)
    sh_at, sh_in = torch.tensor((sh[inside] + half) @ stride, device=dev), torch.tensor(np.nonzero(inside)[0], device=dev)
    mask = torch.zeros(int(np.prod(size)), dtype=torch.float64, device=dev)
    mask[pe_at] = 1.0
    mask = mask.reshape(size)
    xyz = torch.tensor(me @ (h / n).T, device=dev)
    harm = _harmonics(xyz[:, 0], xyz[:, 1], xyz[:, 2])
    r = xyz.square().sum(1).sqrt()
    deg = torch.tensor([l for l in range(7) for _ in range(2 * l + 1)], device=dev, dtype=torch.float64)
    far = harm[:, len(pe):] * (4 * math.pi / (2 * deg + 1))[:, None] / r[None, len(pe):] ** (2 * deg + 1)[:, None]
    harm = harm[:, :len(pe)].contiguous()
    met = torch.tensor(me, device=dev)
    nt, bt, lot = (torch.tensor(np.asarray(v), device=dev).long() for v in (n, box, lo))
    dbox, dlo = exx.dbox_layout(lat, n, cen, _params(c)) if c["dxx"] else (None, None)
    dxx = torch.zeros((m, int(np.prod(dbox))), dtype=torch.float64, device=dev) if c["dxx"] else None
    flat = phi.reshape(m, -1)
    core = tuple(slice(3, z - 3) for z in size)
    mcore = mask[core]

    def lap(v, out):
        """The stencil at the points of the box without its margin."""
        out.copy_(v[(slice(None),) + core]).mul_(sum(k * w2[0] for k in coef))
        for d, k in zip(dirs, coef):
            for q in (1, 2, 3):
                for sg in (1, -1):
                    o = v[(slice(None),) + tuple(slice(3 + sg * q * int(e), z - 3 + sg * q * int(e)) for e, z in zip(d, size))]
                    out.add_(o, alpha=k * w2[q])
        return out

    es, sg = [], []
    chunk = max(1, int(2.5e8 // np.prod(size)))
    ul = lat / np.linalg.norm(lat, axis=1, keepdims=True)
    jac = np.linalg.inv(ul.T).T                                       # J[a][alpha] = |L_alpha| hinv[alpha][a]
    dxi = np.linalg.norm(lat, axis=1) / n
    for p0 in range(0, len(ii), chunk):
        i, j = torch.tensor(ii[p0:p0 + chunk], device=dev), torch.tensor(jj[p0:p0 + chunk], device=dev)
        g = torch.tensor(gg[p0:p0 + chunk], device=dev)

        def at(o, los, ext):
            u = torch.remainder(g[:, None, :] + met[None] - los[o][:, None, :], nt)
            ok = (u < ext).all(-1)
            return torch.where(ok, (u[..., 0] * ext[1] + u[..., 1]) * ext[2] + u[..., 2], 0), ok

        def value(o):
            k, ok = at(o, lot, bt)
            return torch.where(ok, torch.gather(flat[o], 1, k), 0.0)

        fi, fj = value(i), value(j)
        rho = (fi * fj)[:, :len(pe)]
        q = (rho @ harm.T) * dv
        vfar = q @ far
        v = torch.zeros([len(i)] + size, dtype=torch.float64, device=dev)
        v.view(len(i), -1)[:, sh_at] = vfar[:, sh_in]
        b = torch.zeros_like(v)
        b.view(len(i), -1)[:, pe_at] = 4 * math.pi * rho
        rr = torch.empty([len(i)] + [z - 6 for z in size], dtype=torch.float64, device=dev)
        res = (lap(v, rr) + b[(slice(None),) + core]) * mcore
        bn = res.square().sum((1, 2, 3)).sqrt()
        x, pv, ap = torch.zeros_like(res), torch.zeros_like(v), torch.empty_like(res)
        pc = pv[(slice(None),) + core]
        pc.copy_(res)
        r2 = res.square().sum((1, 2, 3))
        for _ in range(2000):
            lap(pv, ap).mul_(mcore).neg_()
            al = torch.where(r2 > 0, r2 / (pc * ap).sum((1, 2, 3)), 0.0)[:, None, None, None]
            x += al * pc
            res -= al * ap
            new = res.square().sum((1, 2, 3))
            if bool((new.sqrt() <= 1e-13 * bn).all()):
                break
            pc.mul_(torch.where(r2 > 0, new / r2, 0.0)[:, None, None, None]).add_(res)
            r2 = new
        v[(slice(None),) + core] += x
        del b, x, pv, pc, ap, rr
        vp = v.view(len(i), -1)[:, pe_at]
        es.append((rho * vp).sum(1) * dv)
        grad = []
        for e in range(3):
            dd = sum(w1[k] / dxi[e] * (v.view(len(i), -1)[:, pe_at + k * int(stride[e])] -
                                       v.view(len(i), -1)[:, pe_at - k * int(stride[e])]) for k in (1, 2, 3))
            grad.append((rho * dd) @ torch.tensor(pe, device=dev, dtype=torch.float64))
        acc = torch.stack(grad, 1)                                    # [pair][b][alpha]
        sg.append(torch.einsum("ab,pbl->pal", torch.tensor(jac, device=dev), acc) / torch.tensor(n, device=dev) * dv)
        if dxx is not None:
            vm = torch.cat([vp, vfar], 1)
            dl, de = torch.tensor(dlo, device=dev).long(), torch.tensor(np.asarray(dbox), device=dev).long()
            for o, f in ((i, fj), (j, fi)):
                k, ok = at(o, dl, de)
                val = torch.where(ok, vm * f, 0.0)
                if o is j:
                    val = torch.where((i == j)[:, None], 0.0, val)
                dxx.view(-1).index_add_(0, (o[:, None] * dxx.shape[1] + k).reshape(-1), val.reshape(-1))
    es, sg = torch.cat(es), torch.cat(sg)
    w = torch.where(torch.tensor(ii == jj, device=dev), 1.0, 2.0).double()
    vol = abs(np.linalg.det(lat))
    e_xx = -float((w * es).sum())
    dedh = -2.0 * (w[:, None, None] * sg).sum(0).cpu().numpy()
    stress = -(dedh @ h.T) / vol
    p_int = float(np.trace(stress)) / 3.0
    if c["stress"] == exx.STRESS_CUBIC:
        p_int = e_xx / (3.0 * vol)
        dedh = np.eye(3) * (-e_xx / (3.0 * lat[0, 0]))
    if c["stress"] != exx.STRESS_FULL:
        stress = np.eye(3) * p_int
    out = {"e_xx": e_xx, "dedh": dedh, "stress": stress, "p_int": p_int, "n_pairs": None}
    if dxx is not None:
        out["dxx"] = dxx.reshape([m] + [int(z) for z in dbox])
    if c["pairs_out"]:
        cap = m * (m + 1) // 2
        out["pair_e"], out["pair_sig"] = torch.zeros(cap, dtype=torch.float64), torch.zeros((cap, 3, 3), dtype=torch.float64)
        out["pair_e"][:len(es)] = es.cpu()
        if c["stress"] != exx.STRESS_CUBIC:
            out["pair_sig"][:len(sg)] = sg.cpu()
    return out


def exact(case, seed):
    """Pair list, far field, CG to 1e-13, integrals and D_xx in FP64; None where this takes over about 20 seconds."""
    if case["kind"] == "list":
        return None
    cells = _batch_cells(case) if case["kind"] == "batch" else [case]
    cost = 0.0
    for c in cells:
        stcl = {"cubic": 19, "ortho": 19, "mono": 25}.get(c["shape"], 37)
        lat, n = _cell(c["shape"], c["length"], c["n"])
        dv = abs(np.linalg.det(lat)) / float(np.prod(n.astype(float)))
        edge = (2 * c["r_pe"]) / dv ** (1 / 3)
        cost += c["steps"] * _pairs(c) * edge ** 4 * stcl
    if cost > 4.5e11:
        return None
    out = []
    for k, c in enumerate(cells):
        steps = _steps(c, seed + 1000 * k)
        out += [_exact_step(c, steps[0][0], s) for s in steps]
    return out
