"""Searches that visit more ids than the visited table keeps, so that ids come
up again and again: one warp and four per query, rows staged narrow and wide,
aligned and not, many useless seeds first, against the oracle bit for bit."""
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


@pytest.mark.parametrize("m", [3, 305])
@pytest.mark.parametrize("n,D,k,s,t0,ks", [(9000, 8, 64, 40, 12, 32), (9000, 8, 20, 3500, 8, 20), (5000, 640, 30, 900, 4, 32),
                                           (5000, 641, 30, 900, 4, 7), (5000, 1026, 50, 33, 5, 32)])
def test_more_visits_than_the_table_keeps(knng, m, n, D, k, s, t0, ks):
    X = datagen.gaussian_mixture(n, D, 12, seed=D)
    Q = datagen.gaussian_mixture(m, D, 12, seed=D)
    rng = np.random.default_rng(m + D)
    G = rng.integers(0, n, size=(n, k)).astype(np.int32)         # far neighbours: many visits
    G[:, : k // 2] = (np.arange(n)[:, None] + np.arange(1, k // 2 + 1)) % n   # and the same ones again
    S = rng.integers(-1, n, size=(m, s)).astype(np.int32)
    S[:, s // 2:] = S[:, : s - s // 2]                           # every seed twice
    ids, d = knng.knng_search(*[torch.from_numpy(a).cuda() for a in (X, G, Q, S)], t0, ks)
    o_ids, o_d = oracle.search(X, G, Q, S, t0, ks)
    assert np.array_equal(ids.cpu().numpy(), o_ids)
    assert np.array_equal(d.cpu().numpy().view(np.uint32), o_d.view(np.uint32))
