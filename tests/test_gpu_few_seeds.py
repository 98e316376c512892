"""Up to 32 seeds per query: second vocabularies that are no multiple of 4,
few and many kept words, fewer lists than seeds, more equal distances than the
sort holds, one query and more than a product tile, rows off the 16-byte grid
(D no multiple of 4), against the oracle."""
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


@pytest.mark.parametrize("W1,W2,probe1,s,D,m,equal", [
    (64, 256, 16, 32, 40, 65, False), (7, 13, 7, 32, 33, 200, False), (256, 32, 256, 31, 64, 1, False),
    (40, 247, 33, 8, 66, 130, False), (256, 32, 32, 32, 128, 64, True), (1, 1, 1, 32, 4, 3, False),
    (20, 256, 32 // 2, 1, 20, 77, True)])
def test_few_seeds_equal_oracle(knng, W1, W2, probe1, s, D, m, equal):
    X = datagen.gaussian_mixture(20000, D, 20, seed=W1 + D)
    o1, o2 = oracle.rvq_train(X[:4000], W1, W2, 1, seed=9)
    if equal:                      # every second-stage word the same: all keys of a kept word tie
        o2[:] = o2[0]
        n = 20000
        off = (np.arange(W1 * W2 + 1, dtype=np.int64) * n // (W1 * W2)).astype(np.int32)
        ids = np.random.default_rng(2).permutation(n).astype(np.int32)
    else:
        _, off, ids = oracle.rvq_index(X, o1, o2)
    Q = datagen.gaussian_mixture(m, D, 20, seed=W1 + D)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (o1, o2, off, ids, Q)]
    S = knng.knng_rvq_seeds(*dev, probe1, s)
    assert np.array_equal(S.cpu().numpy(), oracle.rvq_seeds(o1, o2, off, ids, Q, probe1, s))
