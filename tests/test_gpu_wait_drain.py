"""Both tensor-core kernels alone with waits of a few cycles: whichever role
gives up (the epilogue included, with every MMA already issued), the kernel
drains what it started and the next launches are right."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("npad,nrows", [(32, 1), (128, 129), (160, 40000), (320, 700), (512, 300)])
def test_short_waits_drain(mode, npad, nrows):
    """Integers below 2^4 in rows and operator: sums of at most 512 * 2^8 are
    exact in FP32 and in the split products, so a launch that reports success
    is right to the bit."""
    import paper_2103_01048_gb300 as pb
    rng = np.random.default_rng(npad + nrows)
    Q = rng.integers(-15, 16, (nrows, npad)).astype(np.float32)
    Op = rng.integers(-15, 16, (npad, npad)).astype(np.float32)
    ref = Q.astype(np.float64) @ Op.astype(np.float64).T
    prev = pb._test_tc_pair(mode)
    gave_up = 0
    try:
        for limit in (1, 300, 1000, 3000, 10000) * 4:
            pb._test_wait_limit(limit)
            try:
                assert np.array_equal(pb._selftest_m2l_tc(Q, Op), ref)
            except pb.PBError as e:
                assert e.code == pb.PB_ETIMEOUT
                gave_up += 1
            pb._test_wait_limit(0)
            assert np.array_equal(pb._selftest_m2l_tc(Q, Op), ref)
    finally:
        pb._test_wait_limit(0)
        pb._test_tc_pair(prev)
    print(f"mode {mode} npad {npad}: {gave_up} of 20 launches gave up")
