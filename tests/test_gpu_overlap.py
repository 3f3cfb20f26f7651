"""PB_OPT_OVERLAP (near field on the context's second stream): the first apply
on a fresh tree, which also builds the tree's leaf lists, and a repeated one."""
import numpy as np
import pytest

import synthetic
from oracle.kernels import LAPLACE, YUKAWA, direct_sum, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KAPPA = 0.125


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("layer", ["SL+DL", "DN"])
@pytest.mark.parametrize("n,ncrit,options", [(20001, 64, {}), (20001, 64, {"LIST_DIRECT": 0}), (90000, 40, {}),
                                             (20001, 64, {"LEAF_PACKED": 0})])
def test_first_apply_on_two_streams(n, ncrit, options, layer):
    """Both kernels against the FP64 direct sum at sampled targets (1e-5, the
    bound of the FMM applies; 1e-4 for the normal derivatives, one order less
    accurate in p) and against one stream (1e-6, the bound of the other
    equality tests: the sums differ in order only)."""
    import paper_2103_01048_gb300 as pb
    x, nrm = synthetic.bumpy_sphere_points(n, seed=12)
    q, d = synthetic.uniform_densities(n, seed=13), synthetic.uniform_densities(n, seed=14)
    X, N, Q, D = dev(x), dev(nrm), dev(q), dev(d)
    dn = layer == "DN"
    ctx = pb.pb_create(0, torch.cuda.Stream())
    try:
        for k, v in options.items():
            pb.pb_set_option(ctx, getattr(pb, "PB_OPT_" + k), v)

        def run(overlap):
            pb.pb_set_option(ctx, pb.PB_OPT_OVERLAP, overlap)
            tree = pb.fmm_tree_build(ctx, X, ncrit)
            try:
                res = []
                for _ in range(2):
                    o = [torch.full((n,), float("nan"), device="cuda") for _ in range(4 if dn else 2)]
                    torch.cuda.synchronize()
                    pb.fmm_apply_pair(ctx, tree, KAPPA, 6, o[0], o[1], q_lap=Q, q_yuk=Q, dip=None if dn else D,
                                      src_n=None if dn else N, tgt_n=N if dn else None, dn_lap=o[2] if dn else None,
                                      dn_yuk=o[3] if dn else None)
                    pb.pb_sync(ctx)
                    res.append([a.cpu().numpy() for a in o])
                return res
            finally:
                pb.fmm_tree_destroy(tree)

        both, one = run(1), run(0)
    finally:
        pb.pb_destroy(ctx)
    idx = synthetic.random_subsample(n, 500, seed=15)
    ref = []
    for kern, kap in ((LAPLACE, 0.0), (YUKAWA, KAPPA)):
        ref.append(direct_sum(kern, kap, x, q=q, dip=None if dn else d, src_n=None if dn else nrm, tgt=x[idx],
                              tgt_n=nrm[idx] if dn else None, want_dn=dn))
    want = [ref[0][0], ref[1][0], ref[0][1], ref[1][1]] if dn else ref
    for out in both:
        for k, (o, s, r) in enumerate(zip(out, one[0], want)):
            assert rel_l2(o[idx], r) < (1e-5 if k < 2 else 1e-4), k
            assert rel_l2(o, s) < 1e-6, k


def test_failed_apply_on_two_streams():
    """An allocation that fails while the second stream runs: PB_ENOMEM,
    and the next apply (which takes the returned memory) is right."""
    import paper_2103_01048_gb300 as pb
    rng = np.random.default_rng(41)         # a cluster in a cloud: X lists, hence allocations after the fork
    x = np.concatenate([rng.normal(0.2, 0.02, (6000, 3)), rng.uniform(-1, 1, (6000, 3))]).astype(np.float32)
    n = len(x)
    q = synthetic.uniform_densities(n, seed=13)
    X, Q = dev(x), dev(q)
    idx = synthetic.random_subsample(n, 300, seed=15)
    want = [direct_sum(kern, kap, x, q=q, tgt=x[idx]) for kern, kap in ((LAPLACE, 0.0), (YUKAWA, KAPPA))]
    ctx = pb.pb_create(0, torch.cuda.Stream())
    try:
        pb.pb_set_option(ctx, pb.PB_OPT_OVERLAP, 1)

        def run(tree):
            o = [torch.zeros(n, device="cuda") for _ in range(2)]
            torch.cuda.synchronize()
            pb.fmm_apply_pair(ctx, tree, KAPPA, 6, o[0], o[1], q_lap=Q, q_yuk=Q)
            pb.pb_sync(ctx)
            return [a.cpu().numpy() for a in o]

        keep = pb.fmm_tree_build(ctx, X, 24)     # holds the operators: the fresh trees allocate lists and workspace only
        run(keep)
        failed = 0
        for nth in range(1, 60):
            tree = pb.fmm_tree_build(ctx, X, 24)
            try:
                pb._test_fail_alloc(nth)
                try:
                    out = run(tree)
                except pb.PBError as e:
                    assert e.code == pb.PB_ENOMEM
                    failed += 1
                    out = None
                finally:
                    pb._test_fail_alloc(0)
                done = out is not None
                out = out or run(tree)
                for o, r in zip(out, want):
                    assert rel_l2(o[idx], r) < 1e-5
            finally:
                pb.fmm_tree_destroy(tree)
            if done:
                break
        assert done and failed >= 10
        pb.fmm_tree_destroy(keep)
    finally:
        pb.pb_destroy(ctx)
