"""Whole applies through the tensor-core box operators (reflected split-half
M2L included) against the fixed-order CUDA-core ones, which take one operator
per offset, unreflected and in FP32."""
import numpy as np
import pytest

import synthetic
from oracle.kernels import LAPLACE, YUKAWA, direct_sum, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOUND = {4: 1e-4, 5: 1e-5, 6: 1e-5, 8: 1e-5, 10: 1e-5}      # against the direct sum, by order


@pytest.mark.parametrize("p", [4, 5, 6, 8, 10])
def test_apply_against_fixed_order(p):
    """Adaptive lists through the surfaces only, so that every far pair passes
    the box operators.  Both modes round in FP32 (their distance to FP64
    levels off at 4e-7 with the order): 1e-6 between them, and each within the
    order's bound of the direct sum at sampled targets."""
    import paper_2103_01048_gb300 as pb
    n = 20000
    x, nrm = synthetic.bumpy_sphere_points(n, seed=0)
    q, d = synthetic.uniform_densities(n, seed=1), synthetic.uniform_densities(n, seed=2)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    Q, D, N = dev(q), dev(d), dev(nrm)
    got = []
    ctx = pb.pb_create(0, None)
    try:
        pb.pb_set_option(ctx, pb.PB_OPT_LIST_DIRECT, 0)
        tree = pb.fmm_tree_build(ctx, dev(x), 64)
        for det in (0, 1):
            pb.pb_set_option(ctx, pb.PB_OPT_DETERMINISTIC, det)
            o = [torch.zeros(n, device="cuda") for _ in range(2)]
            pb.fmm_apply_pair(ctx, tree, 0.125, p, o[0], o[1], q_lap=Q, q_yuk=Q, dip=D, src_n=N)
            pb.pb_sync(ctx)
            got.append([a.cpu().numpy() for a in o])
        pb.fmm_tree_destroy(tree)
    finally:
        pb.pb_destroy(ctx)
    idx = synthetic.random_subsample(n, 1000, seed=6)
    for k, (kern, kap) in enumerate(((LAPLACE, 0.0), (YUKAWA, 0.125))):
        ref = direct_sum(kern, kap, x, q=q, dip=d, src_n=nrm, tgt=x[idx])
        for o in got:
            assert rel_l2(o[k][idx], ref) < BOUND[p]
        print(f"p={p}: {rel_l2(got[0][k], got[1][k]):.2e}")
        assert rel_l2(got[0][k], got[1][k]) < 1e-6


@pytest.mark.parametrize("p", [6, 8, 9, 10])
@pytest.mark.parametrize("direct", [0, 1])
def test_fixed_order_bits(p, direct):
    """PB_OPT_DETERMINISTIC: six applies with the same bits (on an adaptive tree
    with X lists, so that both check -> equivalent solves run), within 1e-5
    of the direct sum."""
    import paper_2103_01048_gb300 as pb
    rng = np.random.default_rng(23)
    x = np.concatenate([rng.normal(0.2, 0.02, (5000, 3)), rng.uniform(-1, 1, (5000, 3))]).astype(np.float32)
    n = len(x)
    q = synthetic.uniform_densities(n, seed=4)
    Q = torch.from_numpy(q).cuda()
    ctx = pb.pb_create(0, None)
    try:
        pb.pb_set_option(ctx, pb.PB_OPT_DETERMINISTIC, 1)
        pb.pb_set_option(ctx, pb.PB_OPT_LIST_DIRECT, direct)
        tree = pb.fmm_tree_build(ctx, torch.from_numpy(x).cuda(), 200 if direct else 40)
        assert pb.fmm_tree_info(tree).n_x > 0
        outs = []
        for _ in range(6):
            o = torch.zeros(2, n, device="cuda")
            pb.fmm_apply_pair(ctx, tree, 0.3, p, o[0], o[1], q_lap=Q, q_yuk=Q)
            pb.pb_sync(ctx)
            outs.append(o)
        pb.fmm_tree_destroy(tree)
    finally:
        pb.pb_destroy(ctx)
    assert all(torch.equal(outs[0], o) for o in outs[1:])
    for k, (kern, kap) in enumerate(((LAPLACE, 0.0), (YUKAWA, 0.3))):
        assert rel_l2(outs[0][k].cpu().numpy(), direct_sum(kern, kap, x, q=q)) < 1e-5
