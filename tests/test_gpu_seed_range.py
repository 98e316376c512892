"""Up to 32 seeds per query whose distances span nearly all of FP32's range: a
first word so near that its distance cancels to a negative value, the others
at 1.7e38 and above; every query's seeds equal the oracle's."""
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


@pytest.mark.parametrize("W1,W2,s", [(2, 1, 2), (2, 4, 8), (5, 3, 11)])
def test_distances_over_the_whole_range(knng, W1, W2, s):
    rng = np.random.default_rng(3)
    D, m = 200, 300
    w1 = np.zeros((W1, D), np.float32)
    w2 = np.zeros((W2, D), np.float32)
    w1[0] = np.float32(1.31e18) * rng.uniform(0.95, 1.0, D).astype(np.float32)   # |w1[0]|^2 about 3.3e38
    Q = (w1[0] * (1.0 + 1e-7 * rng.integers(-8, 9, (m, D)))).astype(np.float32)
    n = W1 * W2
    off, ids = np.arange(n + 1, dtype=np.int32), rng.permutation(n).astype(np.int32)
    dev = [torch.from_numpy(a).cuda() for a in (w1, w2, off, ids, Q)]
    S = knng.knng_rvq_seeds(*dev, W1, s)
    want = oracle.rvq_seeds(w1, w2, off, ids, Q, W1, s)
    assert (want >= 0).any(axis=1).all()
    assert np.array_equal(S.cpu().numpy(), want)
