"""The work that is timed: calls of the Stokes layer-potential library as a
boundary-integral flow code makes them, from one short call on a few cells to
whole near-field and FMM evaluations on a million points.

A case is a dict with a "form" (which entry point), its sizes and its options.
Points are red blood cells (Evans-Fung shape, order-p latitude-longitude grid of
2 p (p + 1) points) and vessel walls of 11 x 11 Clenshaw-Curtis patches, in um;
densities are i.i.d. U[-1, 1]^3, as in the benchmark and the tests.

  listed()             the cases
  draw(rng)            another case of the same ranges
  prepare(case, seed)  inputs and plans on the GPU
  run(state)           one pass through the public entry points
  exact(case, seed)    the same outputs by plain torch in 64 bits
  work(case)           the bytes and operations one pass cannot do without
"""
import math

import numpy as np
import torch

import paper_1909_11085_gb300 as S

SL, DL, SLDL = 1, 2, 3
# FP32 or FP64 operations of a target-source pair (FMA = 2, 1/r not counted)
PAIR_FLOPS = {SL: 27, DL: 29, SLDL: 40}
ADJ_FLOPS = 122 + 97  # source-major and target-major pair of the gradient
CELL_RADIUS = 3.91
PATCH_Q = 10
PATCH_POINTS = (PATCH_Q + 1) ** 2


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # one velocity of a small suspension inside a time step: 8 cells (4,352 points) acting on
        # themselves, a plain call with its allocations
        dict(name="sl_8cells", form="direct", kind=SL, cells=8, p=16, box=40.0, off=0,
             precision="mixed"),
        # the smallest call that recurs: three coarse cells seen from a ragged set of tracer
        # points, recorded once in a CUDA graph and replayed
        dict(name="sldl_graph_3cells", form="graph", kind=SLDL, cells=3, p=12, box=26.0, off=1001,
             precision="mixed"),
        # velocity of 256 cells at their own points and at 65,536 points between them
        dict(name="dl_256cells", form="direct", kind=DL, cells=256, p=16, box=120.0, off=65536,
             precision="mixed"),
        # the same kind of sum where 1e-7 is not enough: 64 cells, every operation in FP64
        dict(name="sldl_64cells_fp64", form="direct", kind=SLDL, cells=64, p=16, box=48.0, off=0,
             precision="fp64"),
        # the near field of one matvec: 1,857 cells and 320 wall patches, 1,048,928 points
        dict(name="p2p_1m", form="p2p", kind=SLDL, cells=1857, patches=320, radius=50.0,
             leaf=256, precision="mixed"),
        # a quarter of it in FP64
        dict(name="p2p_262k_fp64", form="p2p", kind=SLDL, cells=464, patches=80, radius=50.0,
             leaf=256, precision="fp64"),
        # a whole FMM velocity (near and far field) of the large suspension, mixed precision
        dict(name="fmm_1m", form="fmm", kind=SLDL, cells=1857, patches=320, radius=50.0, leaf=256,
             precision="mixed", m2l="fft"),
        # a whole FMM velocity with the plan's default far field (FP64, dense translations)
        dict(name="fmm_65k_fp64", form="fmm", kind=SLDL, cells=116, patches=20, radius=25.0,
             leaf=256, precision="fp64", m2l="dense"),
        # independent suspensions of 1 to 64 cells in their own vessels, one call
        dict(name="batched_64", form="batched", susp=64, max_cells=64, sizes=3,
             precision="mixed"),
        # a training or shape-optimisation step: velocity and all its gradients
        dict(name="adjoint_64cells", form="adjoint", cells=64, p=16, box=48.0, precision="mixed"),
        # one application of the boundary-integral operator on a vessel wall
        dict(name="bie_wall_320", form="bie", patches=320, radius=50.0, length=74.0,
             precision="mixed"),
        # which of a million points lie near the wall, and their closest points on it
        dict(name="near_search_1m", form="near", patches=320, radius=50.0, length=74.0,
             targets=1 << 20),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    form = rng.choice(["direct", "graph", "p2p", "fmm", "batched", "adjoint", "bie", "near"])
    precision = rng.choice(["mixed", "fp64"])
    fp64 = precision == "fp64"
    if form in ("direct", "graph"):
        cells = int(_log(rng, 1, 60 if fp64 else 200))
        p = rng.choice([12, 16, 24]) if cells < 24 else 16
        # random orientations need cell centres about 8.2 um apart
        return dict(form=form, kind=rng.choice([SL, DL, SLDL]), cells=cells, p=p,
                    box=round(math.ceil(cells ** (1 / 3)) * rng.uniform(9.0, 18.0), 2),
                    off=rng.choice([0, int(_log(rng, 17, 1500 if fp64 else 60000))]),
                    precision=precision)
    if form in ("p2p", "fmm"):
        leaf = rng.choice([64, 128, 256])  # the FP64 far field costs by the box
        most = (110 * leaf // 256 if form == "fmm" else 500) if fp64 else 1800
        cells = int(_log(rng, 12, most))
        return dict(form=form, kind=rng.choice([SL, DL, SLDL]), cells=cells,
                    patches=4 * max(3, cells // 24), leaf=leaf,
                    radius=round(min(50.0, 6.0 + 2.2 * math.sqrt(cells)), 2), precision=precision,
                    **(dict(m2l=rng.choice(["dense", "fft"])) if form == "fmm" else {}))
    if form == "batched":
        return dict(form=form, susp=rng.randint(2, 3) if fp64 else int(_log(rng, 2, 60)),
                    max_cells=rng.randint(2, 8 if fp64 else 64), sizes=rng.randrange(1 << 20),
                    precision=precision)
    if form == "adjoint":
        cells = int(_log(rng, 1, 16 if fp64 else 60))
        return dict(form=form, cells=cells, p=rng.choice([12, 16]),
                    box=round(math.ceil(cells ** (1 / 3)) * rng.uniform(9.0, 14.0), 2),
                    precision=precision)
    patches = 4 * rng.randint(2, 8 if fp64 else 75)
    radius = round(rng.uniform(2.2, 2.8) * math.sqrt(patches), 2)
    wall = dict(form=form, patches=patches, radius=radius, length=round(1.5 * radius, 2))
    if form == "near":
        return dict(wall, targets=int(_log(rng, 1000, 900000)))
    return dict(wall, precision=precision)


# ----------------------------------------------------------------- geometry

def _cell_grid(p):
    """One cell in its own frame: points, outward normals, weights (numpy)."""
    t, wt = np.polynomial.legendre.leggauss(p + 1)
    ph = np.pi * np.arange(2 * p) / p
    th, ph = [a.ravel() for a in np.meshgrid(np.arccos(t), ph, indexing="ij")]
    wt = np.repeat(wt * np.pi / p, 2 * p)
    st, ct, sp, cp = np.sin(th), np.cos(th), np.sin(ph), np.cos(ph)
    s, R, c = st * st, CELL_RADIUS, (0.2072, 2.0026, -1.1228)
    g = c[0] + c[1] * s + c[2] * s * s
    dz = 0.5 * R * (-st * g + ct * (c[1] + 2.0 * c[2] * s) * 2.0 * st * ct)
    x = np.stack([R * st * cp, R * st * sp, 0.5 * R * ct * g], 1)
    cr = np.cross(np.stack([R * ct * cp, R * ct * sp, dz], 1),
                  np.stack([-R * st * sp, R * st * cp, 0.0 * st], 1))
    jac = np.linalg.norm(cr, axis=1)
    return x, cr / jac[:, None], wt * jac / st


def _rotations(q):
    """Rotation matrices of quaternions q [n, 4]."""
    w, x, y, z = (q / np.linalg.norm(q, axis=1)[:, None]).T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                     2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                     2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)],
                    1).reshape(-1, 3, 3)


def _cells(centres, rots, p):
    """Cells of order p at the centres: points, normals, weights, spacings (numpy)."""
    x, nn, w = _cell_grid(p)
    n = len(centres)
    pts = np.einsum("cij,pj->cpi", rots, x) + centres[:, None, :]
    nrm = np.einsum("cij,pj->cpi", rots, nn)
    h = np.full(n * w.size, np.sqrt(w.sum() / w.size))
    return pts.reshape(-1, 3), nrm.reshape(-1, 3), np.tile(w, n), h


def _cells_in_box(rng, cells, p, box):
    """Randomly turned cells on a jittered lattice of the box, none touching."""
    m = math.ceil(round(cells ** (1 / 3), 9))
    site = np.stack(np.unravel_index(np.sort(rng.choice(m ** 3, cells, replace=False)),
                                     (m, m, m)), 1)
    pitch = box / m
    jitter = max(0.0, 0.5 * (pitch - 2.0 * CELL_RADIUS - 0.3))
    centres = (site + 0.5) * pitch + rng.uniform(-jitter, jitter, (cells, 3))
    return _cells(centres, _rotations(rng.normal(size=(cells, 4))), p)


def _cc(q):
    """Clenshaw-Curtis nodes and weights on [-1, 1], q even."""
    k, j = np.arange(q + 1), np.arange(1, q // 2 + 1)
    b = np.where(j == q // 2, 1.0, 2.0) / (4.0 * j * j - 1.0)
    c = np.where((k == 0) | (k == q), 1.0, 2.0)
    return np.cos(np.pi * k / q), c / q * (1.0 - np.cos(2 * np.pi * np.outer(k, j) / q) @ b)


def _split(radius, length, patches):
    """Patches around and along a cylinder wall, about square, exactly `patches` in all."""
    want = math.sqrt(patches * 2 * np.pi * radius / length)
    around = min((d for d in range(3, patches + 1) if patches % d == 0),
                 key=lambda d: abs(math.log(d / want)))
    return around, patches // around


def _wall(radius, length, around, along, m=1):
    """A cylinder wall of around x along patches (m x m sub-patches each): points,
    outward normals, weights, spacings (numpy)."""
    dth, dz = 2 * np.pi / around, length / along
    x, w = _cc(PATCH_Q)
    sub = (2.0 * np.arange(m)[:, None] + 1.0 + x) / m - 1.0  # [m, q + 1] in [-1, 1]
    iz, it, su, sv, i, j = [a.ravel() for a in np.meshgrid(
        np.arange(along), np.arange(around), np.arange(m), np.arange(m), np.arange(x.size),
        np.arange(x.size), indexing="ij")]
    # shared patch edges coincide exactly, the seam at angle 0 included
    th = np.mod(it + 0.5 * (sub[su, i] + 1.0), around) * dth
    z = (iz + 0.5 * (sub[sv, j] + 1.0)) * dz
    c, s = np.cos(th), np.sin(th)
    area = radius * dth * dz / 4.0 / (m * m)
    pts = np.stack([radius * c, radius * s, z], 1)
    h = np.full(c.size, math.sqrt(4.0 * area / x.size ** 2))
    return pts, np.stack([c, s, 0.0 * c], 1), w[i] * w[j] * area, h


def _vessel(rng, cells, patches, radius):
    """Cells packed on a lattice of a vessel, tilted a little, and the vessel's wall."""
    step, rmax = (8.0, 8.0, 4.0), radius - CELL_RADIUS - 0.2
    a = np.arange(-int(rmax // step[0]), int(rmax // step[0]) + 1) * step[0]
    X, Y = [v.ravel() for v in np.meshgrid(a, a, indexing="ij")]
    keep = X * X + Y * Y <= rmax * rmax
    layer = np.stack([X[keep], Y[keep]], 1)
    layers = math.ceil(cells / len(layer))
    pick = np.sort(rng.choice(layers * len(layer), cells, replace=False))
    centres = np.column_stack([layer[pick % len(layer)],
                               1.0 + (pick // len(layer) + 0.5) * step[2]])
    spin, tilt, axis = (rng.uniform(0, 2 * np.pi, cells), rng.uniform(0, np.deg2rad(5), cells),
                        rng.uniform(0, 2 * np.pi, cells))
    zero = np.zeros(cells)
    turn = _rotations(np.stack([np.cos(tilt / 2), np.sin(tilt / 2) * np.cos(axis),
                                np.sin(tilt / 2) * np.sin(axis), zero], 1))
    turn = turn @ _rotations(np.stack([np.cos(spin / 2), zero, zero, np.sin(spin / 2)], 1))
    body = _cells(centres, turn, 16)
    length = layers * step[2] + 2.0
    wall = _wall(radius, length, *_split(radius, length, patches))
    return [np.concatenate([b, v]) for b, v in zip(body, wall)]


def _suspension(sizes, rng, max_cells):
    """One suspension of 1 to max_cells cells (log-uniform) in its vessel: arrays and the
    number of cell points.  `sizes` draws how much there is, `rng` where it lies."""
    cells = int(round(math.exp(sizes.uniform(0.0, math.log(max_cells)))))
    radius, points = sizes.uniform(10.0, 30.0), int(sizes.integers(2000, 20001))
    order = sizes.choice([12, 16, 24], cells)
    pitch, rmax = 8.3, radius - CELL_RADIUS - 0.2
    a = np.arange(-int(rmax // pitch), int(rmax // pitch) + 1) * pitch
    X, Y = [v.ravel() for v in np.meshgrid(a, a, indexing="ij")]
    keep = X * X + Y * Y <= rmax * rmax
    layer = np.stack([X[keep], Y[keep]], 1)
    length = max(16.0, cells * 94.1 / (0.10 * np.pi * (radius - 4.0) ** 2),
                 math.ceil(cells / len(layer)) * pitch)
    sites = int(length / pitch + 1e-9) * len(layer)
    pick = np.sort(rng.choice(sites, cells, replace=False))
    centres = np.column_stack([layer[pick % len(layer)], (pick // len(layer) + 0.5) * pitch])
    rots = _rotations(rng.normal(size=(cells, 4)))
    parts = [_cells(centres[order == p], rots[order == p], p) for p in (12, 16, 24)]
    body = [np.concatenate(v) for v in zip(*parts)]
    patches = points / PATCH_POINTS
    around = max(3, round(math.sqrt(patches * 2 * np.pi * radius / length)))
    wall = _wall(radius, length, around, max(1, round(patches / around)))
    return [np.concatenate([b, v]) for b, v in zip(body, wall)], len(body[0])


def _gpu(*arrays):
    return [torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
            for a in arrays]


def _densities(seed, n, count):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.rand((n, 3), dtype=torch.float64, device="cuda", generator=g) * 2 - 1
            for _ in range(count)]


def _off_surface(rng, pts, nrm, count):
    """Points 0.05 to 5 um (log-uniform) off the surface points along their normals."""
    i = rng.integers(0, len(pts), count)
    d = np.exp(rng.uniform(math.log(0.05), math.log(5.0), count))
    return pts[i] + d[:, None] * nrm[i]


# ------------------------------------------------------------ prepare and run

def _direct_inputs(case, seed):
    rng = np.random.default_rng(seed)
    pts, nrm, w, h = _cells_in_box(rng, case["cells"], case["p"], case["box"])
    trg = np.concatenate([pts, _off_surface(rng, pts, nrm, case["off"])]) if case["off"] else None
    f, phi = _densities(seed, len(pts), 2)
    src, nrm, w, h = _gpu(pts, nrm, w, h)
    return dict(src=src, f=f, nrm=nrm, phi=phi, w=w, h=h,
                trg=None if trg is None else _gpu(trg)[0], mu=1.0)


def _point_cloud(case, seed):
    """A vessel's points in the leaf order of the library's octree, with densities."""
    rng = np.random.default_rng(seed)
    pts, nrm, w, h = _vessel(rng, case["cells"], case["patches"], case["radius"])
    f, phi = _densities(seed, len(pts), 2)
    return pts, nrm, w, h, f, phi


def _only(kind, f, nrm, phi):
    return dict(f=f if kind & SL else None, nrm=nrm if kind & DL else None,
                phi=phi if kind & DL else None)


def _wall_inputs(case, seed):
    size = case["radius"], case["length"]
    split = _split(*size, case["patches"])
    x, n, w, _ = _wall(*size, *split)
    (phi,) = _densities(seed, len(x), 1)
    return x, n, w, _wall(*size, *split, 4), phi, math.sqrt(w.sum() / w.size)


def _near_inputs(case, seed):
    size = case["radius"], case["length"]
    x, _, w, _ = _wall(*size, *_split(*size, case["patches"]))
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand((case["targets"], 3), dtype=torch.float64, device="cuda", generator=g)
    r, th = case["radius"] * torch.sqrt(u[:, 0]), 2 * math.pi * u[:, 1]
    trg = torch.stack([r * torch.cos(th), r * torch.sin(th), case["length"] * u[:, 2]], 1)
    return _gpu(x)[0], trg, 2.0 * math.sqrt(w.sum() / w.size)


def _direct(s):
    d, prec = s["in"], s["case"]["precision"]
    kind = s["case"]["kind"]
    if kind == SL:
        return S.sl(d["src"], d["f"], d["w"], d["trg"], d["mu"], h=d["h"], precision=prec)
    if kind == DL:
        return S.dl(d["src"], d["nrm"], d["phi"], d["w"], d["trg"], h=d["h"], precision=prec)
    return S.sldl(d["src"], d["f"], d["nrm"], d["phi"], d["w"], d["trg"], d["mu"], h=d["h"],
                  precision=prec)


def _adjoint(s):
    d, g = s["in"], s["g"]
    for k in ("src", "f", "nrm", "phi", "trg"):
        d[k].grad = None
    u = S.StokesLayerFn.apply(d["src"], d["f"], d["nrm"], d["phi"], d["w"], d["trg"], d["mu"],
                              d["h"], s["case"]["precision"])
    u.backward(g)
    return [u.detach()] + [d[k].grad for k in ("src", "f", "nrm", "phi", "trg")]


def prepare(case, seed):
    form = case["form"]
    if form == "direct":
        return dict(case=case, call=_direct, **{"in": _direct_inputs(case, seed)})
    if form == "graph":
        d = _direct_inputs(case, seed)
        trg = d["src"] if d["trg"] is None else d["trg"]
        plan = S.DirectPlan(len(d["src"]), len(trg), case["kind"], case["precision"],
                            device=torch.device("cuda"))
        graph = plan.capture(d["src"], w=d["w"], trg=trg, mu=d["mu"], h=d["h"],
                             **_only(case["kind"], d["f"], d["nrm"], d["phi"]))
        return dict(case=case, graph=graph, plan=plan, call=lambda s: s["graph"].launch())
    if form == "p2p":
        pts, nrm, w, h, f, phi = _point_cloud(case, seed)
        t = S.octree(pts, case["leaf"])
        o = t["perm"]
        pts, nrm, w, h = _gpu(pts[o], nrm[o], w[o], h[o])
        plan = S.P2PPlan(len(pts), t["leaf_ptr"], t["ulist_ptr"], t["ulist_idx"], case["kind"],
                         case["precision"])
        args = dict(pts=pts, w=w, h=h, mu=1.0, **_only(case["kind"], f, nrm, phi))
        return dict(case=case, plan=plan, args=args, tree=t, call=lambda s: s["plan"](**s["args"]))
    if form == "fmm":
        pts, nrm, w, h, f, phi = _point_cloud(case, seed)
        plan = S.FmmPlan(pts, case["leaf"], p=4, kernels=case["kind"],
                         near_precision=case["precision"], far_precision=case["precision"],
                         m2l=case["m2l"])
        o = plan.perm
        pts, nrm, w, h = _gpu(pts[o], nrm[o], w[o], h[o])
        args = dict(pts=pts, w=w, h=h, **_only(case["kind"], f, nrm, phi))
        return dict(case=case, plan=plan, args=args, call=lambda s: s["plan"](**s["args"]))
    if form == "batched":
        sizes, rng = np.random.default_rng(case["sizes"]), np.random.default_rng(seed)
        parts = [_suspension(sizes, rng, case["max_cells"]) for _ in range(case["susp"])]
        pts, nrm, w, h = _gpu(*[np.concatenate(v) for v in zip(*[a for a, _ in parts])])
        ptr = np.concatenate([[0], np.cumsum([len(a[0]) for a, _ in parts])])
        ncell = np.array([n for _, n in parts])
        f, phi = _densities(seed, len(pts), 2)
        plan = S.BatchedPlan(len(pts), ptr, ncell, case["precision"])
        args = dict(pts=pts, f=f, phi=phi, nrm=nrm, w=w, h=h, mu=1.0)
        return dict(case=case, plan=plan, args=args, ptr=ptr, ncell=ncell,
                    call=lambda s: s["plan"](**s["args"]))
    if form == "adjoint":
        d = _direct_inputs(dict(case, off=0), seed)
        d["trg"] = d["src"].clone()
        (g,) = _densities(seed + 1, len(d["src"]), 1)
        for k in ("src", "f", "nrm", "phi", "trg"):
            d[k].requires_grad_(True)
        return dict(case=case, g=g, call=_adjoint, **{"in": d})
    if form == "bie":
        x, n, w, fine, phi, hc = _wall_inputs(case, seed)
        plan = S.BIEPlan(case["patches"], *_gpu(x, n, w), *_gpu(*fine), R=3.0 * hc, r=hc,
                         precision=case["precision"])
        return dict(case=case, plan=plan, phi=phi, call=lambda s: s["plan"].matvec(s["phi"]))
    x, trg, d_eps = _near_inputs(case, seed)
    return dict(case=case, x=x, trg=trg, d_eps=d_eps,
                call=lambda s: list(S.near_patch_search(s["x"], s["case"]["patches"], s["trg"],
                                                        s["d_eps"])))


def run(state):
    return state["call"](state)


# -------------------------------------------------------- 64-bit values, work

_PAIRS = 1 << 21  # pairs in one block of the dense sums below


def _dense(kind, src, f, nrm, phi, w, trg, mu=1.0):
    """The layer potentials at trg, term by term."""
    out = torch.zeros_like(trg)
    q = w[:, None] * f / (8 * math.pi * mu) if kind & SL else None
    psi = w[:, None] * phi * (6 / (8 * math.pi)) if kind & DL else None
    step = max(1, _PAIRS // max(1, len(src)))
    for a in range(0, len(trg), step):
        dx, dy, dz = [trg[a:a + step, k, None] - src[None, :, k] for k in range(3)]
        r2 = dx * dx + dy * dy + dz * dz
        ri = torch.where(r2 > 0, r2, math.inf).rsqrt_()
        c = 0.0
        if kind & SL:
            c = dx * q[:, 0] + dy * q[:, 1] + dz * q[:, 2]
            out[a:a + step] += ri @ q
        if kind & DL:
            dn = dx * nrm[:, 0] + dy * nrm[:, 1] + dz * nrm[:, 2]
            dp = dx * psi[:, 0] + dy * psi[:, 1] + dz * psi[:, 2]
            c = c + dn * dp / torch.where(r2 > 0, r2, math.inf)
        c = c * ri.pow_(3)
        for k, d in enumerate((dx, dy, dz)):
            out[a:a + step, k] += (d * c).sum(1)
    return out


def _dense_grad(src, f, nrm, phi, w, trg, g, mu):
    """Gradients of sum_i g_i . u_i with respect to src, f, nrm, phi, trg, by autograd
    over blocks of the dense sum."""
    leaves = [t.detach().clone().requires_grad_(True) for t in (src, f, nrm, phi, trg)]
    y, f, n, p, x = leaves
    u = torch.zeros_like(trg)
    step = max(1, _PAIRS // len(src))
    for a in range(0, len(trg), step):
        d = x[a:a + step, None, :] - y[None]
        r2 = (d * d).sum(2)
        near = torch.where(r2 > 0, r2, 1.0)
        one = (r2 > 0).double()
        q, psi = w[:, None] * f / (8 * math.pi * mu), w[:, None] * p * (6 / (8 * math.pi))
        dq, dn, dp = [torch.einsum("tsk,sk->ts", d, v) for v in (q, n, psi)]
        b = torch.einsum("ts,sk->tk", one * near ** -0.5, q) \
            + torch.einsum("ts,tsk->tk", one * (dq * near ** -1.5 + dn * dp * near ** -2.5), d)
        b.backward(g[a:a + step])
        u[a:a + step] = b.detach()
    return [u] + [t.grad for t in leaves]


def _leaf_sums(state):
    """The near field leaf by leaf over the U-lists."""
    t, a, kind = state["tree"], state["args"], state["case"]["kind"]
    ptr, up, ui = (np.asarray(t[k], dtype=np.int64) for k in ("leaf_ptr", "ulist_ptr", "ulist_idx"))
    out = torch.zeros_like(a["pts"])
    pick = lambda v, i: None if v is None else v[i]  # noqa: E731
    for b in range(len(ptr) - 1):
        u = ui[up[b]:up[b + 1]]
        i = torch.from_numpy(np.concatenate([np.arange(ptr[k], ptr[k + 1]) for k in u])).cuda()
        out[ptr[b]:ptr[b + 1]] = _dense(kind, a["pts"][i], pick(a["f"], i), pick(a["nrm"], i),
                                        pick(a["phi"], i), a["w"][i], a["pts"][ptr[b]:ptr[b + 1]])
    return out


def exact(case, seed):
    form = case["form"]
    if form == "bie" or form == "fmm":
        # the operator's outputs hold the error of its extrapolation, the FMM's that of its
        # expansions: they have no 64-bit value short of the same steps
        return None
    if form in ("direct", "graph"):
        d = _direct_inputs(case, seed)
        trg = d["src"] if d["trg"] is None else d["trg"]
        return _dense(case["kind"], d["src"], d["f"], d["nrm"], d["phi"], d["w"], trg, d["mu"])
    if form == "adjoint":
        d = _direct_inputs(dict(case, off=0), seed)
        (g,) = _densities(seed + 1, len(d["src"]), 1)
        return _dense_grad(d["src"], d["f"], d["nrm"], d["phi"], d["w"], d["src"], g, d["mu"])
    if form == "p2p":
        s = prepare(case, seed)
        return _leaf_sums(s) if len(s["tree"]["leaf_ptr"]) < 40000 else None
    if form == "batched":
        s = prepare(case, seed)
        a, out = s["args"], []
        for b, n in enumerate(s["ncell"]):
            lo, mid, hi = s["ptr"][b], s["ptr"][b] + n, s["ptr"][b + 1]
            x = a["pts"][lo:hi]
            out.append(_dense(SL, x[:n], a["f"][lo:mid], None, None, a["w"][lo:mid], x)
                       + _dense(DL, x[n:], None, a["nrm"][mid:hi], a["phi"][mid:hi],
                                a["w"][mid:hi], x))
        return torch.cat(out)
    # the wall is a cylinder: its closest point lies on the radius through the target
    _, trg, d_eps = _near_inputs(case, seed)
    rho = torch.hypot(trg[:, 0], trg[:, 1])
    n = torch.stack([trg[:, 0] / rho, trg[:, 1] / rho, torch.zeros_like(rho)], 1)
    dist = case["radius"] - rho
    y = trg + dist[:, None] * n
    far = dist > d_eps
    n[far], y[far], dist[far] = 0.0, 0.0, -1.0
    return [None, None, y, n, dist]


def _sizes(case):
    """(targets or points, sources, pairs) of a case without making its points, where they
    follow from it alone."""
    cells = case.get("cells", 0) * 2 * case.get("p", 16) * (case.get("p", 16) + 1)
    if case["form"] in ("direct", "graph", "adjoint"):
        nt = cells + case.get("off", 0)
        return nt, cells, nt * cells
    if case["form"] in ("p2p", "fmm"):
        n = cells + case["patches"] * PATCH_POINTS
        # a leaf of the benchmark's tree holds a quarter of its limit and meets 25 leaves
        return n, n, n * 6.3 * case["leaf"]
    if case["form"] == "batched":
        mean = (case["max_cells"] - 1) / math.log(case["max_cells"]) * 720 + 11000
        return int(case["susp"] * mean), int(case["susp"] * mean), case["susp"] * 1.3 * mean ** 2
    nc = case["patches"] * PATCH_POINTS
    if case["form"] == "bie":
        return nc, 16 * nc, 5 * nc * 16 * nc
    return case["targets"], nc, 0


def work(case):
    nt, ns, pairs = _sizes(case)
    form = case["form"]
    if form == "near":
        # targets in; patch, parameters, point, normal and distance out; seven evaluations of
        # the 11 x 11 interpolant and its derivatives for the targets near the wall
        near = nt * 4.0 * math.sqrt(2 * math.pi * case["radius"] * case["length"] / ns) \
            / case["radius"]
        return dict(bytes=24 * ns + nt * (24 + 4 + 8 * 9), flops=near * 7 * 2400.0)
    if form == "adjoint":
        return dict(bytes=ns * 8 * (3 * 4 + 2) + nt * 8 * 6 + 8 * 3 * (4 * ns + 2 * nt),
                    flops=pairs * (PAIR_FLOPS[SLDL] + ADJ_FLOPS))
    kind = DL if form == "bie" else SLDL if form == "batched" else case["kind"]
    flops = pairs * (28 if form == "batched" else PAIR_FLOPS[kind])
    if form == "fmm":
        # the far field's translations, per point about what the near field does
        flops *= 1.5
    vecs = 1 + (1 if kind & SL else 0) + (2 if kind & DL else 0)
    return dict(bytes=ns * 8 * (3 * vecs + 2) + nt * 48, flops=flops)
