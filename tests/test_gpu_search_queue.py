"""The search's queue, staging and visited table: one and several warps per
query, rows of part of a stage, of several and of dims no multiple of 4, off
the 16-byte grid, more visits than the table holds, repeated and missing
seeds, long neighbour lists, against the oracle bit for bit."""
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


@pytest.mark.parametrize("m", [1, 304, 305])
@pytest.mark.parametrize("D,k,s,t0,ks,shift", [(8, 5, 3, 4, 32, 0), (33, 40, 300, 6, 32, 0), (132, 12, 40, 9, 20, 0),
                                               (300, 64, 33, 3, 10, 0), (64, 12, 8, 5, 16, 1), (131, 20, 0, 3, 7, 0)])
def test_search_paths(knng, m, D, k, s, t0, ks, shift):
    n = 2500
    X = datagen.gaussian_mixture(n, D, 12, seed=D)
    Q = datagen.gaussian_mixture(m, D, 12, seed=D)
    rng = np.random.default_rng(m + D)
    G = rng.integers(0, n, size=(n, k)).astype(np.int32)         # far neighbours: many visits
    G[:, : k // 2] = (np.arange(n)[:, None] + np.arange(1, k // 2 + 1)) % n
    G[::7, -1] = -1
    S = rng.integers(-1, n + 2, size=(m, s)).astype(np.int32)
    if s > 4:
        S[:, 3] = S[:, 0]
    buf = torch.empty(n * D + 4, device="cuda")
    Xd = buf[shift:shift + n * D].view(n, D)
    Xd.copy_(torch.from_numpy(X))
    ids, d = knng.knng_search(Xd, *[torch.from_numpy(a).cuda() for a in (G, Q, S)], t0, ks)
    o_ids, o_d = oracle.search(X, G, Q, S, t0, ks)
    assert np.array_equal(ids.cpu().numpy(), o_ids)
    assert np.array_equal(d.cpu().numpy().view(np.uint32), o_d.view(np.uint32))


@pytest.mark.parametrize("shift,bad", [(0, 0), (1, 0), (3, 2), (1, 400), (2, 399)])
def test_non_finite_values_are_found_anywhere(knng, shift, bad):
    buf = torch.zeros(420, device="cuda")
    X = buf[shift:shift + 401].view(401, 1)
    X[bad] = float("nan")
    G = torch.zeros((401, 1), dtype=torch.int32, device="cuda")
    ok = torch.zeros((1, 1), device="cuda")
    seeds = torch.zeros((1, 1), dtype=torch.int32, device="cuda")
    with pytest.raises(knng.KnngError):
        knng.knng_search(X, G, ok, seeds, 1, 1)
    with pytest.raises(knng.KnngError):
        knng.knng_search(torch.zeros_like(X), G, X[bad:bad + 1].contiguous(), seeds, 1, 1)
