"""The packed leaf kernel on trees of one leaf (every pair summed directly):
target-normal derivatives, one and both kernels, sources split over CTAs,
odd counts, one point, a window and its neighbours."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layer", ["SL", "DL", "SL+DL", "DN"])
@pytest.mark.parametrize("n", [1, 2, 127, 255, 257, 513, 1023, 1025, 2049])
def test_one_leaf_direct(n, layer):
    """Bound, relative to the sum of the terms' absolute values: a term is off
    by at most 2^-22 for each of the approximate 1/sqrt (three times) and 2^x
    and 2^-24 for each of its about 16 other roundings, (4 * 4 + 16) 2^-24 in
    all, coordinates included (exact differences of the same FP32 numbers to
    2^-24); a thread adds at most n / 8 + 8 terms, each addition 2^-24."""
    import paper_2103_01048_gb300 as pb
    rng = np.random.default_rng(n)
    kappa = 0.7
    x = rng.uniform(-1, 1, (n, 3)).astype(np.float32)
    nrm = rng.standard_normal((n, 3))
    nrm = (nrm / np.linalg.norm(nrm, axis=1, keepdims=True)).astype(np.float32)
    q, d = (rng.uniform(-1, 1, n).astype(np.float32) for _ in range(2))
    X, N = x.astype(np.float64), nrm.astype(np.float64)
    dx = X[:, None] - X[None]
    r = np.linalg.norm(dx, axis=2)
    np.fill_diagonal(r, np.inf)
    e = np.where(np.isfinite(r), np.exp(-kappa * np.where(np.isfinite(r), r, 0.0)), 0.0)
    kr = np.where(np.isfinite(r), kappa * np.where(np.isfinite(r), r, 0.0), 0.0)
    c4 = 1 / (4 * np.pi)
    terms = {}
    for name, ee, one in (("L", 1.0, 1.0), ("Y", e, 1 + kr)):
        t = []
        if layer in ("SL", "SL+DL", "DN"):
            t.append(ee / r * q[None].astype(np.float64))
        if layer in ("DL", "SL+DL"):
            t.append(ee * one * np.einsum("ijk,jk->ij", dx, N) / r ** 3 * d[None].astype(np.float64))
        terms[name] = t
        if layer == "DN":
            terms["d" + name] = [-ee * one * np.einsum("ijk,ik->ij", dx, N) / r ** 3 * q[None].astype(np.float64)]
    # the dot products' terms can cancel: their bound takes |d| |m| / r^3
    absum = {k: sum(np.abs(v).sum(1) for v in t) * c4 for k, t in terms.items()}
    for k in absum:
        if layer in ("DL", "SL+DL") or k.startswith("d"):
            w = np.abs(d if not k.startswith("d") else q).astype(np.float64)
            absum[k] = absum[k] + (2 * w[None] / r ** 2).sum(1) * c4
    tol = (32 + n / 8 + 8) * 2.0 ** -24
    ctx = pb.pb_create(0, None)
    try:
        dev = lambda a: torch.from_numpy(a).cuda()
        tree = pb.fmm_tree_build(ctx, dev(x), 4096)
        out = {k: torch.full((n,), np.nan, device="cuda") for k in ("L", "Y", "dL", "dY")}
        qq = dev(q) if layer != "DL" else None
        dd = dev(d) if layer in ("DL", "SL+DL") else None
        dn = layer == "DN"
        pb.fmm_apply_pair(ctx, tree, kappa, 4, out["L"], out["Y"], q_lap=qq, q_yuk=qq, dip=dd,
                          src_n=dev(nrm) if dd is not None else None, tgt_n=dev(nrm) if dn else None,
                          dn_lap=out["dL"] if dn else None, dn_yuk=out["dY"] if dn else None)
        torch.cuda.synchronize()
        got = {k: out[k].cpu().numpy() for k in terms}
        for kern, name in ((pb.FMM_LAPLACE, "L"), (pb.FMM_YUKAWA, "Y")):
            o, od = (torch.full((n,), np.nan, device="cuda") for _ in range(2))
            pb.fmm_apply(ctx, tree, kern, kappa, 4, o, q=qq, dip=dd, src_n=dev(nrm) if dd is not None else None,
                         tgt_n=dev(nrm) if dn else None, out_dn=od if dn else None)
            torch.cuda.synchronize()
            got["1" + name] = o.cpu().numpy()
            if dn:
                got["1d" + name] = od.cpu().numpy()
        pb.fmm_tree_destroy(tree)
    finally:
        pb.pb_destroy(ctx)
    for k, v in got.items():
        ref = sum(t.sum(1) for t in terms[k.lstrip("1")]) * c4
        assert np.all(np.abs(v - ref) <= tol * absum[k.lstrip("1")] + 1e-30), k


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("separate", [False, True])
def test_long_lists(mode, separate):
    """Clustered points and small leaves: lists of more than 32 entries, ranges
    that join across them, targets without sources; every direct-list mode
    against the direct sum, the scalar kernel beside it.  1e-5, the bound
    of the FMM applies (here p = 8)."""
    import paper_2103_01048_gb300 as pb
    from oracle.kernels import LAPLACE, YUKAWA, direct_sum, rel_l2
    rng = np.random.default_rng(17)
    pts = lambda a, b: np.concatenate([rng.normal(0, 0.02, (a, 3)), rng.uniform(-1, 1, (b, 3))]).astype(np.float32)
    x = pts(2500, 1500)
    t = pts(500, 2500) if separate else None
    n = len(x if t is None else t)
    q, d = (rng.uniform(-1, 1, len(x)).astype(np.float32) for _ in range(2))
    nrm = rng.standard_normal((len(x), 3))
    nrm = (nrm / np.linalg.norm(nrm, axis=1, keepdims=True)).astype(np.float32)
    dev = lambda a: torch.from_numpy(a).cuda()
    ctx = pb.pb_create(0, None)
    try:
        pb.pb_set_option(ctx, pb.PB_OPT_LIST_DIRECT, mode)
        tree = pb.fmm_tree_build(ctx, dev(x), 12, None if t is None else dev(t))
        off, _ = pb.fmm_tree_export(ctx, tree)["U"]
        assert np.diff(off).max() > 32
        got = []
        for packed in (1, 0):
            pb.pb_set_option(ctx, pb.PB_OPT_LEAF_PACKED, packed)
            oL, oY = torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda")
            pb.fmm_apply_pair(ctx, tree, 0.5, 8, oL, oY, q_lap=dev(q), q_yuk=dev(q), dip=dev(d), src_n=dev(nrm))
            torch.cuda.synchronize()
            got.append((oL.cpu().numpy(), oY.cpu().numpy()))
        pb.fmm_tree_destroy(tree)
    finally:
        pb.pb_destroy(ctx)
    ref = [direct_sum(k, kap, x, q=q, dip=d, src_n=nrm, tgt=t) for k, kap in ((LAPLACE, 0.0), (YUKAWA, 0.5))]
    for o in got:
        for v, r in zip(o, ref):
            assert rel_l2(v, r) < 1e-5
