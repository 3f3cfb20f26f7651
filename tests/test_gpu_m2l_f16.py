"""The split-half M2L kernel alone, with reflected rows, against the FP64 product."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npad,nrows", [(32, 1), (64, 129), (128, 128), (160, 127), (160, 40000), (320, 1025), (512, 300)])
def test_reflected_rows(npad, nrows):
    """Rows of very different sizes, entries of a row over six decades, every
    reflection; ragged tiles, fewer and more tiles than CTAs, two segments.

    Bound, relative to sum_k |o_k| |q_k| plus the rows' largest products: each
    factor is hi + lo to 2^-23 of itself or, where lo is subnormal, 2^-40 of
    its row's (operator's) largest; lo * lo is dropped (2^-24 |q||o|, each lo
    at most 2^-12); the FP32 accumulator adds 3 npad products, at most
    2^-23 of the absolute sum for each (truncating adds)."""
    import paper_2103_01048_gb300 as pb
    rng = np.random.default_rng(npad + nrows)
    Q = rng.uniform(-1, 1, (nrows, npad)) * 10.0 ** rng.uniform(-6, 0, (nrows, npad))
    Q *= 10.0 ** rng.uniform(-25, 25, (nrows, 1))
    Q[nrows // 2] = 0.0
    Q = Q.astype(np.float32)
    Op = (rng.uniform(-1, 1, (npad, npad)) * 10.0 ** rng.uniform(-3, 1.5, (npad, npad))).astype(np.float32)
    xs = rng.integers(0, 8, nrows)
    D = pb._selftest_m2l_f16(Q, Op, xs)
    col = np.arange(npad)[None, :] ^ xs[:, None]
    q = np.take_along_axis(Q, col, 1).astype(np.float64)
    o = Op.astype(np.float64).T
    ref = np.take_along_axis(q @ o, col, 1)
    absum = np.take_along_axis(np.abs(q) @ np.abs(o), col, 1)
    floor = npad * np.abs(Q).max(1, keepdims=True).astype(np.float64) * np.abs(Op).max() * 2.0 ** -39
    bound = (2 * 2.0 ** -23 + 2.0 ** -24 + 3 * npad * 2.0 ** -23) * absum + floor
    err = np.abs(D - ref)
    print(f"npad {npad} rows {nrows}: max err / bound {np.max(err / np.maximum(bound, 1e-300)):.3f}")
    assert np.all(err <= bound)
    assert not D[nrows // 2].any()
