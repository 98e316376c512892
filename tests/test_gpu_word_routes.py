"""Every route of word training and the index gives the oracle's words and
lists: sizes on both sides of the lines between the FP32 and the screened
assignment and between chained and pieced means, rows of few and of many dims
(no multiple of 4 too), vectors with many words equally near (noise of many
dims, equal points, values near the ends of FP32's range), means whose rounding
the pieces cannot prove, of more dims and members than are staged at once."""
import numpy as np
import pytest

import datagen
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


def _points(kind, n, D):
    rng = np.random.default_rng(n + D)
    if kind == "noise":                       # far more spread within a cluster than between them
        return rng.standard_normal((n, D)).astype(np.float32)
    if kind == "spread":                      # magnitudes 2^-40 to 2^40: sums round in FP64
        return (rng.standard_normal((n, D)) * np.exp2(rng.uniform(-40, 40, (n, D)))).astype(np.float32)
    X = datagen.gaussian_mixture(n, D, 12, seed=n + D)
    if kind == "same":
        X[:] = X[0]
    return X * np.float32({"tiny": 1e-22, "huge": 1e17}.get(kind, 1.0))


@pytest.mark.parametrize("kind,n,D,W1,W2", [
    ("mixture", 131, 160, 33, 32), ("mixture", 132, 160, 33, 33), ("mixture", 1024, 70, 32, 31), ("mixture", 1025, 139, 32, 40),
    ("mixture", 1200, 140, 129, 5), ("noise", 1500, 700, 64, 48), ("noise", 1001, 701, 64, 200), ("same", 900, 160, 64, 64),
    ("tiny", 700, 164, 40, 40), ("huge", 700, 165, 40, 40), ("spread", 900, 150, 3, 5), ("spread", 2500, 300, 2, 2),
    ("spread", 33, 20, 1, 1), ("mixture", 20000, 16, 256, 200)])
def test_words_and_lists_equal_oracle(knng, kind, n, D, W1, W2):
    X = _points(kind, n, D)
    Xd = torch.from_numpy(X).cuda()
    w1, w2 = knng.knng_rvq_train(Xd, W1, W2, 2, seed=7)
    o1, o2 = oracle.rvq_train(X, W1, W2, 2, seed=7)
    assert np.array_equal(w1.cpu().numpy().view(np.uint32), o1.view(np.uint32))
    assert np.array_equal(w2.cpu().numpy().view(np.uint32), o2.view(np.uint32))
    for a, b in zip(knng.knng_rvq_index(Xd, w1, w2), oracle.rvq_index(X, o1, o2)):
        assert np.array_equal(a.cpu().numpy(), b)
