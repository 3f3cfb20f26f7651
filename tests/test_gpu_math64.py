"""FP64 point sums through the table-driven exponential and the refined
reciprocal square root: one far pair at a time against the closed form, over
distances that take exp(-kappa r) from 1 to below the smallest normal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kappa", [1e-6, 0.125, 4.0, 400.0])
def test_single_pair_distances(kappa):
    """Two points in one leaf (an n_crit above the point count): the apply is
    the direct sum.  exp2 and rsqrt are good to 2.2 and 1.3 units of 2^-53, the
    exponent's rounding adds |kappa r| 2^-52, every other operation half a
    unit: 16 + 2 |kappa r| units bound the whole, and no value below 2^-1022 is asked for."""
    import paper_2103_01048_gb300 as pb
    ctx = pb.pb_create(0, None)
    rng = np.random.default_rng(3)
    try:
        for r in np.concatenate([10.0 ** rng.uniform(-3, 2, 24), [700.0 / kappa, 760.0 / kappa]]):
            x = np.array([[0, 0, 0], [r, 0, 0]], np.float32)
            d = float(x[1, 0])
            q = torch.tensor([0.0, 3.0], dtype=torch.float64, device="cuda")
            oL = torch.zeros(2, dtype=torch.float64, device="cuda")
            oY = torch.zeros(2, dtype=torch.float64, device="cuda")
            tree = pb.fmm_tree_build(ctx, torch.from_numpy(x).cuda(), 8)
            pb.fmm_apply_pair(ctx, tree, kappa, 4, oL, oY, q_lap=q, q_yuk=q, precision=pb.PB_FP64)
            torch.cuda.synchronize()
            pb.fmm_tree_destroy(tree)
            lap = 3.0 / (4 * np.pi * d)
            assert abs(oL[0].item() - lap) <= 16 * 2.0 ** -53 * lap
            t = kappa * d
            yuk = lap * np.exp(-t)
            if t < 700:
                assert abs(oY[0].item() - yuk) <= (16 + 2 * t) * 2.0 ** -53 * yuk
            else:
                assert 0.0 <= oY[0].item() <= 1e-290
            assert oL[1].item() == 0.0 and oY[1].item() == 0.0
    finally:
        pb.pb_destroy(ctx)
