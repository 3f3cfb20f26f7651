"""Performance cases of the framework: what its users run, over the sizes, expansion orders, layers and precisions in use.

Most cases are single FMM applies (fmm_apply, fmm_apply_pair): the work of one mat-vec on the quadrature points of a
molecular surface, where nearly all the time of a solve goes.  Three more take the whole way: a tree built for new points
and applied, and two solvation energies.  Sizes and parameters are those of bench.py and the tests (15k points: the 5,120
triangles of the Born ion; 240k: an 80,000-triangle protein surface; 3M to 4M: virus-scale surfaces; p = 4 to 10,
n_crit = 64 to 256, eps 4 / 80, kappa 0.125 / A).

The geometry is synthetic: closed star-shaped surfaces with seeded bumps, radial unit vectors as normals.
"""
import math

import numpy as np
import torch

import paper_2103_01048_gb300 as pb

KAPPA = 0.125
EPS_IN, EPS_OUT = 4.0, 80.0
KCAL = 332.0637
EXACT_PAIRS = 6.5e10          # 64-bit direct sums up to this many pairs (about 15 s)

_ctx = None


def _context():
    """One context for the process, on the current (default) stream, as a program keeps it."""
    global _ctx
    if _ctx is None:
        _ctx = pb.pb_create(0, None)
    return _ctx


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one mat-vec's FMM work on a small ion's mesh (5,120 triangles x 3 points): latency and launches count
        dict(name="pair_15k_p6", kind="pair", n=15360, p=6, ncrit=128, layers="SL+DL", shape="smooth"),
        # a user's own Yukawa single layer on a small point set, a ragged count, the leaf size of the tests
        dict(name="yukawa_sl_20k_p5", kind="single", n=20011, p=5, ncrit=64, kernel="yukawa", layers="SL"),
        # the protein surface of the bench (80,000 triangles): the ordinary mat-vec
        dict(name="pair_240k_p6", kind="pair", n=240003, p=6, ncrit=128, layers="SL+DL", shape="lumpy"),
        # the bench workload, the largest
        dict(name="pair_4m_p6", kind="pair", n=4000000, p=6, ncrit=128, layers="SL+DL", shape="smooth"),
        # virus-scale surfaces are solved at p = 4
        dict(name="pair_3m_p4", kind="pair", n=2995377, p=4, ncrit=128, layers="SL+DL", shape="smooth"),
        # high accuracy on a protein surface
        dict(name="pair_500k_p8", kind="pair", n=499999, p=8, ncrit=128, layers="SL+DL", shape="lumpy"),
        # the refinement study's order (131,072 triangles x 6 points are 786k; here the 32,768-triangle mesh)
        dict(name="pair_197k_p10", kind="pair", n=196608, p=10, ncrit=128, layers="SL+DL", shape="smooth"),
        # the backward direction: K' (target-normal derivatives) of the adjoint and of the derivative formulations
        dict(name="adjoint_240k_p6", kind="dn", n=240000, p=6, ncrit=128, shape="lumpy"),
        # charge -> surface coupling: atoms in a shell as sources, surface points as targets
        dict(name="atoms_to_surface_600k_p4", kind="coupling", n_src=80000, n=600001, p=4, ncrit=128),
        # the all-FP64 option on a small mesh's points
        dict(name="pair_fp64_30k_p6", kind="pair64", n=30720, p=6, ncrit=128, layers="SL+DL"),
        # a new surface every call (moving atoms, mesh refinement): the octree, then one apply
        dict(name="build_apply_120k_p6", kind="build", n=120001, p=6, ncrit=128),
        # a whole solvation energy, direct formulation, from charges to kcal/mol
        dict(name="energy_direct_5292", kind="energy", face=21, atoms=200, form="direct", p=6, ncrit=128),
    ]


def draw(rng):
    def size(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["pair", "pair", "pair", "single", "single", "dn", "coupling", "pair64", "build", "energy"])
    ncrit = rng.choice([64, 100, 128, 128, 192, 256])
    p = rng.choice([4, 5, 6, 6, 8, 10])
    layers = rng.choice(["SL", "DL", "SL+DL", "SL+DL"])
    shape = rng.choice(["smooth", "lumpy"])
    if kind == "pair":
        return dict(kind=kind, n=size(6000, 400000 if p >= 8 else 3000000), p=p, ncrit=ncrit, layers=layers, shape=shape)
    if kind == "single":
        return dict(kind=kind, n=size(6000, 400000 if p >= 8 else 2000000), p=p, ncrit=ncrit,
                    kernel=rng.choice(["laplace", "yukawa"]), layers=layers)
    if kind == "dn":
        return dict(kind=kind, n=size(6000, 400000), p=p, ncrit=ncrit, shape=shape)
    if kind == "coupling":
        return dict(kind=kind, n_src=size(2000, 150000), n=size(15000, 800000), p=min(p, 6), ncrit=ncrit)
    if kind == "pair64":
        return dict(kind=kind, n=size(4000, 31000), p=min(p, 6), ncrit=128, layers=layers)
    if kind == "build":
        return dict(kind=kind, n=size(6000, 400000), p=min(p, 6), ncrit=ncrit)
    form = rng.choice(["direct", "direct", "exterior"])
    return dict(kind=kind, face=rng.randint(8, 21 if form == "direct" else 14), atoms=size(1, 400), form=form,
                p=rng.choice([4, 5, 6]), ncrit=128)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
_SHAPES = {"smooth": (1.1, 0.05, 32, 0.3), "lumpy": (24.0, 0.12, 160, 0.15)}     # radius, bump height, bumps, width


def _bumps(u, nb, width, seed):
    """Seeded smooth field on the unit sphere, largest magnitude 1 over the points."""
    r = np.random.RandomState(seed % (1 << 31))
    c = r.standard_normal((nb, 3))
    c /= np.linalg.norm(c, axis=1, keepdims=True)
    w = r.uniform(-1.0, 1.0, nb)
    f = torch.zeros(len(u), dtype=u.dtype, device=u.device)
    for k in range(nb):
        d2 = (u - torch.tensor(c[k], dtype=u.dtype, device=u.device)).square().sum(1)
        f += w[k] * torch.exp(-d2 / (2 * width * width))
    return f / f.abs().max()


def _surface(n, shape, seed):
    """n points of a bumpy closed surface and their (radial) unit normals, float32 on the GPU."""
    radius, amp, nb, width = _SHAPES[shape]
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.randn(n, 3, dtype=torch.float64, device="cuda", generator=g)
    u /= u.norm(dim=1, keepdim=True)
    x = u * (radius * (1.0 + amp * _bumps(u, nb, width, seed)))[:, None]
    return x.float().contiguous(), u.float().contiguous()


def _densities(n, seed, count):
    g = torch.Generator(device="cuda").manual_seed(seed + 77)
    return [torch.rand(n, device="cuda", generator=g) * 2 - 1 for _ in range(count)]


def _atoms_in_shell(n, seed):
    """Atoms spread through a capsid wall around the lumpy surface's radius, charges in [-0.8, 0.8]."""
    g = torch.Generator(device="cuda").manual_seed(seed + 5)
    u = torch.randn(n, 3, dtype=torch.float64, device="cuda", generator=g)
    u /= u.norm(dim=1, keepdim=True)
    r = 17.0 + 3.5 * torch.rand(n, 1, dtype=torch.float64, device="cuda", generator=g)
    q = torch.rand(n, device="cuda", generator=g) * 1.6 - 0.8
    return (u * r).float().contiguous(), q


def _mesh(face, seed):
    """A cube projected to a bumpy sphere: 12 face^2 triangles, outward; (verts, tris) as numpy arrays."""
    g = np.arange(face + 1)
    i, j = [a.ravel() for a in np.meshgrid(g, g, indexing="ij")]
    sides = []
    for axis in range(3):
        for side in (0, face):
            v = np.zeros((len(i), 3), dtype=np.int64)
            a1, a2 = [a for a in range(3) if a != axis]
            v[:, axis], v[:, a1], v[:, a2] = side, i, j
            sides.append(v)
    grid, back = np.unique(np.concatenate(sides), axis=0, return_inverse=True)
    back = back.ravel()
    m, tris = face + 1, []
    for f in range(6):
        k = back[f * m * m:(f + 1) * m * m].reshape(m, m)
        a, b, c, d = (t.ravel() for t in (k[:-1, :-1], k[1:, :-1], k[1:, 1:], k[:-1, 1:]))
        tris += [np.stack([a, b, c], 1), np.stack([a, c, d], 1)]
    tris = np.concatenate(tris)
    u = grid * (2.0 / face) - 1.0
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    f = _bumps(torch.from_numpy(u), 32, 0.3, seed).numpy()
    verts = u * (12.0 * (1.0 + 0.05 * f))[:, None]
    p0, p1, p2 = (verts[tris[:, k]] for k in range(3))
    flip = (np.cross(p1 - p0, p2 - p0) * (p0 + p1 + p2)).sum(1) < 0
    tris[flip] = tris[flip][:, [0, 2, 1]]
    return np.ascontiguousarray(verts), np.ascontiguousarray(tris.astype(np.int32))


def _mesh_atoms(n, seed):
    """Charges well inside the mesh, none nearer than 2 A to the surface."""
    r = np.random.RandomState((seed + 9) % (1 << 31))
    u = r.standard_normal((n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    return u * (9.0 * r.uniform(0, 1, (n, 1)) ** (1 / 3)), r.uniform(-0.8, 0.8, n)


class _State:
    """The buffers and the handle of one case; gives the handle back with the last reference."""

    def __init__(self, case):
        self.case, self.ctx = case, _context()
        self.tree = self.mesh = None

    def __del__(self):
        if self.tree is not None:
            pb.fmm_tree_destroy(self.tree)
        if self.mesh is not None:
            pb.pb_mesh_destroy(self.mesh)


def _inputs(case, seed):
    """The arrays of a point case: xyz, normals, targets (coupling), q_lap, q_yuk, dip (None: no such layer)."""
    kind, n = case["kind"], case["n"]
    d = dict(q=None, qy=None, dip=None, tgt=None)
    if kind == "coupling":
        d["x"], d["q"] = _atoms_in_shell(case["n_src"], seed)
        d["tgt"], _ = _surface(n, "lumpy", seed)
        d["nrm"] = None
        return d
    d["x"], d["nrm"] = _surface(n, case.get("shape", "lumpy"), seed)
    q, qy, dip = _densities(n, seed, 3)
    layers = case.get("layers", "SL" if kind == "dn" else "SL+DL")
    if "SL" in layers:
        d["q"], d["qy"] = q, qy
    if "DL" in layers:
        d["dip"] = dip
    if kind == "pair64":
        for k in ("nrm", "q", "qy", "dip"):
            d[k] = None if d[k] is None else d[k].double()
    return d


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind == "energy":
        verts, tris = _mesh(case["face"], seed)
        s.atoms, s.charges = _mesh_atoms(case["atoms"], seed)
        s.mesh = pb.pb_mesh_setup(s.ctx, verts, tris, 3, case["p"], case["ncrit"],
                                  pb.PB_P0 if case["form"] == "direct" else pb.PB_P1)
        return s
    s.inp = _inputs(case, seed)
    if kind != "build":
        s.tree = pb.fmm_tree_build(s.ctx, s.inp["x"], case["ncrit"], s.inp["tgt"])
    else:
        # the program's earlier surface, whose tree is replaced by the next one's
        s.tree = pb.fmm_tree_build(s.ctx, _surface(case["n"], "lumpy", seed + 1)[0], case["ncrit"])
    dt = torch.float64 if kind == "pair64" else torch.float32
    s.out = [torch.empty(case["n"], dtype=dt, device="cuda") for _ in range(4 if kind == "dn" else 2)]
    return s


def run(state):
    case, ctx = state.case, state.ctx
    kind = case["kind"]
    if kind == "energy":
        form = pb.PB_FORM_DIRECT if case["form"] == "direct" else pb.PB_FORM_EXTERIOR
        res, status = pb.pb_solve(ctx, state.mesh, state.atoms, state.charges, EPS_IN, EPS_OUT, KAPPA, 1e-7,
                                  formulation=form)
        energy, phi = pb.pb_solvation_energy(ctx, res, case["atoms"])          # kcal/mol, reaction potentials
        pb.pb_result_destroy(res)
        return [energy, phi.astype(np.float32)]           # kept in single precision, the solve's own (PB_MIXED)
    i, o, p = state.inp, state.out, case["p"]
    if kind == "coupling":
        pb.fmm_apply(ctx, state.tree, pb.FMM_LAPLACE, 0.0, p, o[0], q=i["q"])
        return o[0]
    if kind == "single":
        lap = case["kernel"] == "laplace"
        pb.fmm_apply(ctx, state.tree, pb.FMM_LAPLACE if lap else pb.FMM_YUKAWA, 0.0 if lap else KAPPA, p, o[0],
                     q=i["q"], dip=i["dip"], src_n=i["nrm"] if i["dip"] is not None else None)
        return o[0]
    if kind == "dn":
        pb.fmm_apply_pair(ctx, state.tree, KAPPA, p, o[0], o[1], q_lap=i["q"], q_yuk=i["qy"], tgt_n=i["nrm"],
                          dn_lap=o[2], dn_yuk=o[3])
        return o
    tree = state.tree
    if kind == "build":
        tree = pb.fmm_tree_build(ctx, i["x"], case["ncrit"])
        pb.fmm_tree_destroy(state.tree)
        state.tree = tree
    pb.fmm_apply_pair(ctx, tree, KAPPA, p, o[0], o[1], q_lap=i["q"], q_yuk=i["qy"], dip=i["dip"],
                      src_n=i["nrm"] if i["dip"] is not None else None,
                      precision=pb.PB_FP64 if kind == "pair64" else pb.PB_MIXED)
    return o


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _apply_flops(n_src, n_tgt, p, ncrit, near, far, kernels):
    """Order of the kernel-independent FMM's work on a surface, whose leaves hold about half of n_crit points
    and are one of about 14 mutually adjacent ones (6 to 9 n_crit near points per target): near-field pairs,
    check and equivalent surfaces (2 n_e per point), and the translations (n_e^2 multiply-adds for each V-list pair,
    about 0.9 pairs a point at n_crit 128)."""
    ne = 6 * (p - 1) ** 2 + 2
    n = max(n_src, n_tgt)
    return n_tgt * 9.0 * ncrit * near + (n_src + n_tgt) * ne * far + kernels * 0.9 * n * (128.0 / ncrit) * 2.0 * ne * ne


def work(case):
    kind, p, ncrit = case["kind"], case["p"], case["ncrit"]
    if kind == "energy":
        nt = 12 * case["face"] ** 2
        n, direct = 3 * nt, case["form"] == "direct"
        passes = 20 if direct else 8 * 10            # mat-vecs times FMM passes each
        return {"bytes": passes * n * 20.0 + 2.0 * n * 32 + case["atoms"] * 32.0,
                "flops": passes * _apply_flops(n, n, p, ncrit, 30, 30, 2) + 2.0 * n * case["atoms"] * 20}
    n = case["n"]
    ns = case.get("n_src", n)
    item = 8 if kind == "pair64" else 4
    layers = case.get("layers", "SL" if kind in ("dn", "coupling") else "SL+DL")
    kernels = 1 if kind in ("single", "coupling") else 2
    outs = 4 if kind == "dn" else kernels
    reals = (kernels if "SL" in layers else 0) + (4 if "DL" in layers else 0)
    move = ns * (12 + item * reals) + n * item * outs + (n * 12 if kind == "coupling" else 0) + (n * 12 if kind == "dn" else 0)
    near = (16 if "DL" not in layers else 30) * (0.6 if kernels == 1 else 1.0) + (14 if kind == "dn" else 0)
    return {"bytes": float(move), "flops": _apply_flops(ns, n, p, ncrit, near, near, kernels)}


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------
def _direct(x, tgt, q, qy, dip, nrm, tn, kappa, laplace, yukawa):
    """Direct sums over all pairs (coincident ones excluded) in 64 bits: {name: [n_tgt]}."""
    x, t = x.double(), (x if tgt is None else tgt).double()
    c4 = 1.0 / (4.0 * math.pi)
    out = {k: [] for k in ("L", "Y", "dL", "dY")}
    q = None if q is None else q.double()
    qy = None if qy is None else qy.double()
    m = None if dip is None else dip.double()[:, None] * nrm.double()
    step = max(1, int(2.5e8 // len(x)))
    for a in range(0, len(t), step):
        ta = t[a:a + step]
        d = [ta[:, k, None] - x[None, :, k] for k in range(3)]
        r2 = d[0] * d[0]
        r2.addcmul_(d[1], d[1]).addcmul_(d[2], d[2])
        ri = r2.rsqrt_().masked_fill_(r2 == math.inf, 0.0)
        dm = None if m is None else d[0] * m[:, 0] + d[1] * m[:, 1] + d[2] * m[:, 2]
        if dm is not None:
            dm *= ri ** 3
        dt = None
        if tn is not None:
            tna = tn[a:a + step].double()
            dt = (d[0] * tna[:, 0, None] + d[1] * tna[:, 1, None] + d[2] * tna[:, 2, None]) * ri ** 3
        del d
        if laplace:
            s = ri @ q if q is not None else 0.0
            out["L"].append((s + dm.sum(1) if dm is not None else s) * c4)
            if dt is not None:
                out["dL"].append(-(dt @ q) * c4)
        if yukawa:
            kr = torch.where(ri > 0, kappa / ri, 0.0)
            e = torch.exp(-kr)
            s = (ri * e) @ qy if qy is not None else 0.0
            kr.add_(1.0).mul_(e)
            out["Y"].append((s + dm.mul_(kr).sum(1) if dm is not None else s) * c4)
            if dt is not None:
                out["dY"].append(-(dt.mul_(kr) @ qy) * c4)
    return {k: torch.cat(v) for k, v in out.items() if v}


def exact(case, seed):
    kind = case["kind"]
    if kind == "energy":
        return _exact_energy(case, seed)
    if float(case["n"]) * case.get("n_src", case["n"]) > EXACT_PAIRS:
        return None
    i = _inputs(case, seed)
    if kind == "coupling":
        return _direct(i["x"], i["tgt"], i["q"], None, None, None, None, 0.0, True, False)["L"]
    if kind == "single":
        lap = case["kernel"] == "laplace"
        r = _direct(i["x"], None, i["q"], i["q"], i["dip"], i["nrm"], None, KAPPA, lap, not lap)
        return r["L" if lap else "Y"]
    r = _direct(i["x"], None, i["q"], i["qy"], i["dip"], i["nrm"], i["nrm"] if kind == "dn" else None, KAPPA, True, True)
    return [r[k] for k in (("L", "Y", "dL", "dY") if kind == "dn" else ("L", "Y"))]


def _gauss01(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1.0), 0.5 * w


def _touching_rule(shared, n):
    """Points and weights on a pair of reference triangles {0 <= v <= u <= 1} with `shared` common vertices, in the
    regularising coordinates of Sauter and Schwab (Boundary Element Methods, sec. 5.2): (u1, v1, u2, v2, w), [m]."""
    g, gw = _gauss01(n)
    s, a, b, c = (t.ravel() for t in np.meshgrid(g, g, g, g, indexing="ij"))
    w = np.einsum("i,j,k,l->ijkl", gw, gw, gw, gw).ravel()
    o = np.ones_like(s)
    if shared == 3:
        j = s ** 3 * a ** 2 * b
        p = [(o, 1 - a + a * b, 1 - a * b * c, 1 - a), (1 - a * b * c, 1 - a, o, 1 - a + a * b),
             (o, a * (1 - b + b * c), 1 - a * b, a * (1 - b)), (1 - a * b, a * (1 - b), o, a * (1 - b + b * c)),
             (1 - a * b * c, a * (1 - b * c), o, a * (1 - b)), (o, a * (1 - b), 1 - a * b * c, a * (1 - b * c))]
        j = [j] * 6
    elif shared == 2:
        j1, j2 = s ** 3 * a ** 2, s ** 3 * a ** 2 * b
        p = [(o, a * c, 1 - a * b, a * (1 - b)), (o, a, 1 - a * b * c, a * b * (1 - c)),
             (1 - a * b, a * (1 - b), o, a * b * c), (1 - a * b * c, a * b * (1 - c), o, a),
             (1 - a * b * c, a * (1 - b * c), o, a * b)]
        j = [j1, j2, j2, j2, j2]
    else:
        j = [s ** 3 * b] * 2
        p = [(o, a, b, b * c), (b, b * c, o, a)]
    pts = [np.stack([s * t for t in q] + [w * jj]) for q, jj in zip(p, j)]
    return np.concatenate(pts, axis=1)


class _Galerkin:
    """The Galerkin system of a closed mesh in 64 bits: point sums with the 3-point rule for separate triangles, the
    touching pairs by the rules above.  Matrix-free mat-vec over dense point matrices."""

    def __init__(self, verts, tris, p1):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.V = torch.tensor(verts, dtype=torch.float64, device=dev)
        self.F = torch.tensor(tris.astype(np.int64), device=dev)
        self.p1 = p1
        T = self.V[self.F]                                        # [nt, 3, 3]
        c = torch.cross(T[:, 1] - T[:, 0], T[:, 2] - T[:, 0], dim=1)
        self.area = 0.5 * c.norm(dim=1)
        self.n = c / (2 * self.area)[:, None]
        self.lam = torch.tensor([[2, .5, .5], [.5, 2, .5], [.5, .5, 2]], dtype=torch.float64, device=dev) / 3
        self.x = (self.lam @ T).reshape(-1, 3)                    # [3 nt, 3]
        self.w = (self.area / 3).repeat_interleave(3)
        self.nx = self.n.repeat_interleave(3, 0)
        self.curl = torch.stack([T[:, (a + 1) % 3] - T[:, (a + 2) % 3] for a in range(3)], 1) / (2 * self.area)[:, None, None]
        self.tri = torch.arange(len(tris), device=dev).repeat_interleave(3)
        self._touching(tris)
        self._points()

    def _touching(self, tris):
        at = {}
        for t, f in enumerate(tris.tolist()):
            for v in f:
                at.setdefault(v, []).append(t)
        pairs = sorted({(a, b) for ts in at.values() for a in ts for b in ts})
        dev = self.V.device
        self.pi, self.pj = (torch.tensor(t, device=dev) for t in np.array(pairs).T)
        fi, fj = tris[[p[0] for p in pairs]], tris[[p[1] for p in pairs]]
        eq = fi[:, :, None] == fj[:, None, :]
        count = eq.any(2).sum(1)
        # vertex orders that bring the common vertices to the front, in the same order on both
        si = np.argsort(~eq.any(2), axis=1, kind="stable")
        fo = np.take_along_axis(fi, si, 1)
        first = np.where(fj[:, None, :] == fo[:, :, None], np.arange(3)[None, None, :], 9).min(2)
        sj = np.empty_like(si)
        for k in range(len(pairs)):
            f = [v for v in first[k] if v < 9]
            sj[k] = f + [v for v in range(3) if v not in f]
        m = len(pairs)
        self.blocks = torch.zeros(m, 4, 3, 3, dtype=torch.float64, device=dev)     # VL KL VY KY
        for shared in (1, 2, 3):
            k = np.nonzero(count == shared)[0]
            rule = torch.tensor(_touching_rule(shared, 7 if shared == 1 else 8), dtype=torch.float64, device=dev)
            for c in range(0, len(k), 1000):
                kk = k[c:c + 1000]
                kt = torch.tensor(kk, device=dev)
                oi, oj = torch.tensor(si[kk], device=dev), torch.tensor(sj[kk], device=dev)
                self.blocks[kt] = self._rule_blocks(self.pi[kt], self.pj[kt], oi, oj, rule)

    def _rule_blocks(self, i, j, oi, oj, rule):
        Ti = self.V[torch.gather(self.F[i], 1, oi)]
        Tj = self.V[torch.gather(self.F[j], 1, oj)]
        u1, v1, u2, v2, w = rule
        li = torch.stack([1 - u1, u1 - v1, v1], 1)                  # [m, 3]
        lj = torch.stack([1 - u2, u2 - v2, v2], 1)
        d = torch.einsum("mv,pvc->pmc", li, Ti) - torch.einsum("mv,pvc->pmc", lj, Tj)
        r = d.norm(dim=2)
        rn = torch.einsum("pmc,pc->pm", d, self.n[j]) * (i != j)[:, None]
        kr = KAPPA * r
        e = torch.exp(-kr)
        f = [1 / r, rn / r ** 3, e / r, e * (1 + kr) * rn / r ** 3]
        jac = 4 * self.area[i] * self.area[j] / (4 * math.pi)
        out = torch.empty(len(i), 4, 3, 3, dtype=torch.float64, device=d.device)
        for o, g in enumerate(f):
            b = torch.einsum("pm,ma,mb->pab", g * w, li, lj) * jac[:, None, None]
            out[:, o] = torch.zeros_like(b).scatter_(1, oi[:, :, None].expand(-1, 3, 3),
                                                     torch.zeros_like(b).scatter_(2, oj[:, None, :].expand(-1, 3, 3), b))
        return out

    def _points(self):
        n, c4 = len(self.x), 1 / (4 * math.pi)
        dev = self.x.device
        self.G = [torch.empty(n, n, dtype=torch.float64, device=dev) for _ in range(4)]      # gL kL gY kY
        for a in range(0, n, 1536):
            d = self.x[a:a + 1536, None] - self.x[None]
            r = d.norm(dim=2)
            r[torch.arange(r.shape[0], device=dev), a + torch.arange(r.shape[0], device=dev)] = math.inf
            rn = torch.einsum("abc,bc->ab", d, self.nx) / r ** 3
            kr = KAPPA * r
            e = torch.exp(-kr)
            for m, v in zip(self.G, (1 / r, rn, e / r, torch.where(r < math.inf, e * (1 + kr) * rn, 0.0))):
                m[a:a + 1536] = v * c4
        # separate triangles only
        for b in range(9):
            pa, pb_ = 3 * self.pi + b // 3, 3 * self.pj + b % 3
            for m in self.G:
                m[pa, pb_] = 0.0

    # values at the points of a coefficient vector, and the test integrals of point values
    def at_points(self, c):
        return (c[self.F] @ self.lam.T).reshape(-1) if self.p1 else c[self.tri]

    def test(self, local):
        """[nt, 3] integrals against the local hat functions -> coefficients' rows."""
        if not self.p1:
            return local.sum(1)
        out = torch.zeros(len(self.V), dtype=torch.float64, device=local.device)
        return out.index_add_(0, self.F.reshape(-1), local.reshape(-1))

    def loc(self, vals):
        return (self.w * vals).reshape(-1, 3) @ self.lam

    def apply(self, op, c, transpose=False):
        """Local test integrals of V_L, K_L, V_Y, K_Y (op 0..3) of the coefficients c (transpose: K')."""
        v = self.w * self.at_points(c)
        r = self.loc((self.G[op].T if transpose else self.G[op]) @ v)
        cj = c[self.F] if self.p1 else c[:, None].expand(-1, 3)
        if transpose:
            add = torch.einsum("pab,pa->pb", self.blocks[:, op], cj[self.pi])
            return r.index_add(0, self.pj, add)
        return r.index_add(0, self.pi, torch.einsum("pab,pb->pa", self.blocks[:, op], cj[self.pj]))

    def mass(self, c):
        """Local test integrals of the P1 function c."""
        f = c[self.F]
        return (self.area / 12)[:, None] * (f.sum(1, keepdim=True) + f)

    def hyper(self, c):
        """Local test integrals of (W_Y - W_L) c in the integrated-by-parts form."""
        g = torch.einsum("ta,tac->tc", c[self.F], self.curl)
        b = (self.blocks[:, 2] - self.blocks[:, 0]).sum((1, 2))
        out = torch.zeros(len(self.F), 3, dtype=torch.float64, device=c.device)
        for k in range(3):
            u = (self.G[2] - self.G[0]) @ (self.w * g[self.tri, k])
            per = (self.w * u).reshape(-1, 3).sum(1).index_add(0, self.pi, b * g[self.pj, k])
            out += per[:, None] * self.curl[:, :, k]
            v = self.w * self.at_points(c) * self.nx[:, k]
            out += KAPPA ** 2 * self.n[:, k, None] * self.loc(self.G[2] @ v)
        nn = (self.n[self.pi] * self.n[self.pj]).sum(1)
        add = torch.einsum("pab,pb->pa", self.blocks[:, 2], c[self.F][self.pj]) * nn[:, None]
        return out.index_add(0, self.pi, KAPPA ** 2 * add)


def _gmres(A, b, tol, most):
    n = torch.linalg.vector_norm(b)
    Q, H = [b / n], torch.zeros(most + 1, most, dtype=torch.float64)
    for j in range(most):
        w = A(Q[j])
        for _ in range(2):
            h = torch.stack(Q) @ w
            w = w - torch.stack(Q).T @ h
            H[:j + 1, j] += h.cpu()
        H[j + 1, j] = torch.linalg.vector_norm(w)
        e = torch.zeros(j + 2, dtype=torch.float64)
        e[0] = n
        y = torch.linalg.lstsq(H[:j + 2, :j + 1], e[:, None]).solution[:, 0]
        if torch.linalg.vector_norm(H[:j + 2, :j + 1] @ y - e) <= tol * n:
            break
        Q.append(w / H[j + 1, j])
    return torch.stack(Q[:j + 1]).T @ y.to(b.device)


def _exact_energy(case, seed):
    """The solvation energy and reaction potentials of the discrete system, solved to 1e-11."""
    verts, tris = _mesh(case["face"], seed)
    xa, qa = _mesh_atoms(case["atoms"], seed)
    return _galerkin_energy(verts, tris, xa, qa, case["form"] == "exterior")


def _galerkin_energy(verts, tris, xa, qa, exterior):
    S = _Galerkin(verts, tris, exterior)
    dev = S.V.device
    xa, qa = torch.tensor(xa, device=dev), torch.tensor(qa, device=dev)
    e12 = EPS_IN / EPS_OUT
    N = len(S.V) if exterior else len(S.F)
    d = S.x[:, None] - xa[None]
    r = d.norm(dim=2)
    f = (qa / r).sum(1) / (4 * math.pi * (EPS_OUT if exterior else EPS_IN))
    if exterior:
        fn = -(qa * (d * S.nx[:, None]).sum(2) / r ** 3).sum(1) / (4 * math.pi * EPS_OUT)
        b = torch.cat([S.test(S.loc(f)), S.test(S.loc(fn))])
        scale = S.test(S.area[:, None].expand(-1, 3) / 3).repeat(2)
        b = b / scale

        def A(v):
            u, s = v[:N], v[N:]
            r0 = 0.5 * (1 + e12) * S.mass(u) - S.apply(3, u) + e12 * S.apply(1, u) + S.apply(2, s) - S.apply(0, s)
            r1 = e12 * S.hyper(u) + 0.5 * (1 + e12) * S.mass(s) + e12 * S.apply(3, s, True) - S.apply(1, s, True)
            return torch.cat([S.test(r0), S.test(r1)]) / scale
    else:
        b = torch.cat([S.test(S.loc(f)), torch.zeros(N, dtype=torch.float64, device=dev)])
        own = torch.full((4, N), 0.0, dtype=torch.float64, device=dev)
        k = S.pi == S.pj
        own[:, S.pi[k]] = S.blocks[k].sum((2, 3)).T
        a11, a12, a21, a22 = 0.5 * S.area + own[1], -own[0], 0.5 * S.area - own[3], e12 * own[2]
        det = a11 * a22 - a12 * a21

        def P(v):
            u, s = v[:N], v[N:]
            return torch.cat([(a22 * u - a12 * s) / det, (a11 * s - a21 * u) / det])

        def A(v):
            u, s = v[:N], v[N:]
            half = 0.5 * S.area * u
            return P(torch.cat([half + S.test(S.apply(1, u) - S.apply(0, s)),
                                half + S.test(e12 * S.apply(2, s) - S.apply(3, u))]))
        b = P(b)
    sol = _gmres(A, b, 1e-11, 150)
    u, s = S.at_points(sol[:N]), S.at_points(sol[N:]) * (EPS_OUT / EPS_IN if exterior else 1.0)
    reac = ((S.w * s)[:, None] / r + (d * S.nx[:, None]).sum(2) / r ** 3 * (S.w * u)[:, None]).sum(0) / (4 * math.pi)
    return [0.5 * float((qa * reac).sum()) * 4 * math.pi * KCAL, reac]
