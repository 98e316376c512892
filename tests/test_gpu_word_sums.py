"""A word's mean where the sum of its members' magnitudes passes FP32's range:
a sum whose last bit the order of the additions decides, and with it a tie of
the rounding to FP32.  The words are the oracle's (members in ascending order)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def knng():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_08475_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("D,sign", [(1, 1.0), (1, -1.0), (4, 1.0)])
def test_sums_past_fp32_in_the_defined_order(knng, D, sign):
    # 32 members sum to 64 (2^126 + 2^102), a tie of the mean's rounding; two
    # more of half an FP64 unit each vanish one by one and count together
    x = np.zeros(64)
    x[:32] = 2.0 ** 127
    x[31] += 2.0 ** 108
    x[32:34] = 2.0 ** 79
    X = np.repeat((sign * x).astype(np.float32)[:, None], D, axis=1)
    chain, pieces = 0.0, sum(X[:32, 0].astype(np.float64)) + sum(X[32:, 0].astype(np.float64))
    for v in X[:, 0].astype(np.float64):
        chain += v
    assert np.float32(chain / 64) != np.float32(pieces / 64)
    w1, w2 = knng.knng_rvq_train(torch.from_numpy(X).cuda(), 1, 1, 1, seed=3)
    o1, o2 = oracle.rvq_train(X, 1, 1, 1, seed=3)
    assert o1[0, 0] == np.float32(chain / 64)
    assert np.array_equal(w1.cpu().numpy().view(np.uint32), o1.view(np.uint32))
    assert np.array_equal(w2.cpu().numpy().view(np.uint32), o2.view(np.uint32))
