"""Up to 32 seeds per query on both sides of the line between the two routes.
Distances that span nearly all of FP32's range: a first word so near that its
distance cancels to a negative value, the others at 1.7e38 and above.  The
smallest vocabularies, for few queries and for many.  Every query's seeds
equal the oracle's."""
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


@pytest.mark.parametrize("W1,W2,s,m", [(2, 1, 2, 300), (2, 1, 2, 4097), (2, 4, 8, 4097), (5, 3, 11, 4097), (60, 3, 32, 300),
                                       (130, 2, 7, 300)])
def test_distances_over_the_whole_range(knng, W1, W2, s, m):
    rng = np.random.default_rng(3)
    D = 200
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


@pytest.mark.parametrize("m", [4096, 4097])
@pytest.mark.parametrize("W1,W2,probe1,s,D", [(1, 1, 1, 32, 4), (7, 13, 7, 32, 33), (16, 16, 16, 5, 1), (64, 4, 64, 32, 64),
                                              (3, 200, 1, 20, 40)])
def test_small_vocabularies(knng, W1, W2, probe1, s, D, m):
    rng = np.random.default_rng(W1 + D)
    X = rng.standard_normal((900, D)).astype(np.float32)
    o1, o2 = oracle.rvq_train(X, W1, W2, 1, seed=9)
    _, off, ids = oracle.rvq_index(X, o1, o2)
    Q = rng.standard_normal((m, D)).astype(np.float32)
    S = knng.knng_rvq_seeds(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (o1, o2, off, ids, Q)], probe1, s)
    assert np.array_equal(S.cpu().numpy(), oracle.rvq_seeds(o1, o2, off, ids, Q, probe1, s))
