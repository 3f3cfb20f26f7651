"""A tree's first apply inside a stream capture: the operators come from
another tree of the context, the lists the tree keeps are made on the side."""
import numpy as np
import pytest

import synthetic
from oracle.kernels import LAPLACE, YUKAWA, direct_sum, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KAPPA = 0.5


@pytest.mark.parametrize("options", [{}, {"DETERMINISTIC": 1}, {"LIST_DIRECT": 0}, {"LIST_DIRECT": 0, "DETERMINISTIC": 1},
                                     {"OVERLAP": 1}], ids=str)
@pytest.mark.parametrize("dn", [False, True])
def test_first_apply_captured(options, dn):
    """Points without adaptive lists (a lattice with equal leaves; with
    LIST_DIRECT 0 a cluster in a cloud, with them).  The replayed graph takes
    the inputs of the moment: against the direct sum, twice (1e-5, normal
    derivatives 1e-4, at p = 8)."""
    import paper_2103_01048_gb300 as pb
    rng = np.random.default_rng(5)
    if "LIST_DIRECT" in options:
        x = np.concatenate([rng.normal(0.2, 0.02, (2000, 3)), rng.uniform(-1, 1, (2000, 3))]).astype(np.float32)
        ncrit = 24
    else:
        g = (np.arange(16) + 0.5) / 16
        x = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3).astype(np.float32)
        ncrit = 8
    n = len(x)
    nrm = rng.standard_normal((n, 3))
    nrm = (nrm / np.linalg.norm(nrm, axis=1, keepdims=True)).astype(np.float32)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    X, N = dev(x), dev(nrm)
    stream = torch.cuda.Stream()
    ctx = pb.pb_create(0, stream)
    try:
        for k, v in options.items():
            pb.pb_set_option(ctx, getattr(pb, "PB_OPT_" + k), v)
        Q, o = torch.zeros(n, device="cuda"), [torch.zeros(n, device="cuda") for _ in range(4 if dn else 2)]

        def apply(tree):
            pb.fmm_apply_pair(ctx, tree, KAPPA, 8, o[0], o[1], q_lap=Q, q_yuk=Q, dip=None if dn else Q,
                              src_n=None if dn else N, tgt_n=N if dn else None, dn_lap=o[2] if dn else None,
                              dn_yuk=o[3] if dn else None)

        torch.cuda.synchronize()
        first = pb.fmm_tree_build(ctx, X, ncrit)
        apply(first)
        pb.pb_sync(ctx)
        tree = pb.fmm_tree_build(ctx, X, ncrit)
        assert (pb.fmm_tree_info(tree).n_x > 0) == ("LIST_DIRECT" in options)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            apply(tree)
        for seed in (6, 7):
            q = synthetic.uniform_densities(n, seed=seed)
            Q.copy_(dev(q))
            for a in o:
                a.fill_(float("nan"))
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            pb.pb_sync(ctx)
            want = []
            for kern, kap in ((LAPLACE, 0.0), (YUKAWA, KAPPA)):
                r = direct_sum(kern, kap, x, q=q, dip=None if dn else q, src_n=None if dn else nrm,
                               tgt_n=nrm if dn else None, want_dn=dn)
                want.append(r if dn else (r,))
            for k, a in enumerate(o):
                assert rel_l2(a.cpu().numpy(), want[k % 2][k // 2]) < (1e-5 if k < 2 else 1e-4)
        del graph
        pb.fmm_tree_destroy(tree)
        pb.fmm_tree_destroy(first)
    finally:
        pb.pb_destroy(ctx)


def test_replay_after_other_orders():
    """A captured apply at p = 6 on a tree with X lists, replayed after the tree
    has been used at other orders (which take other lists) and memory has
    changed hands."""
    import paper_2103_01048_gb300 as pb
    rng = np.random.default_rng(8)
    x = np.concatenate([rng.normal(0.2, 0.02, (4000, 3)), rng.uniform(-1, 1, (4000, 3))]).astype(np.float32)
    n = len(x)
    q = synthetic.uniform_densities(n, seed=9)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    X, Q = dev(x), dev(q)
    want = [direct_sum(kern, kap, x, q=q) for kern, kap in ((LAPLACE, 0.0), (YUKAWA, KAPPA))]
    stream = torch.cuda.Stream()
    ctx = pb.pb_create(0, stream)
    try:
        o = [torch.zeros(n, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
        tree = pb.fmm_tree_build(ctx, X, 200)        # leaves above and below the thresholds of all three orders
        assert pb.fmm_tree_info(tree).n_x > 0

        def apply(t, p):
            pb.fmm_apply_pair(ctx, t, KAPPA, p, o[0], o[1], q_lap=Q, q_yuk=Q)

        apply(tree, 6)
        pb.pb_sync(ctx)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            apply(tree, 6)
        for p in (8, 4):
            apply(tree, p)
            other = pb.fmm_tree_build(ctx, X, 30)
            apply(other, p)
            pb.pb_sync(ctx)
            pb.fmm_tree_destroy(other)
            for a in o:
                a.fill_(float("nan"))
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            pb.pb_sync(ctx)
            for a, r in zip(o, want):
                assert rel_l2(a.cpu().numpy(), r) < 1e-5
        del graph
        pb.fmm_tree_destroy(tree)
    finally:
        pb.pb_destroy(ctx)
