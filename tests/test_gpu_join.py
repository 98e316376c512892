"""The FP32 local join: builds whose rounds list only the member blocks that can
make an offer (first rounds with members in leaf order, later ones with new
members) equal the oracle's, over slot sizes from one block per node to the
largest, row lengths that are no multiple of 4, rows that are not 16-byte
aligned and more tree passes than leaf ids are kept for."""
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


@pytest.mark.parametrize("k,mode,D,leaf,passes", [
    (1, oracle.FWD_REV, 7, 20, 3), (2, oracle.FWD_REV, 12, 20, 2), (5, oracle.FWD_REV, 33, 40, 5),
    (16, oracle.FWD_REV, 96, 64, 3), (21, oracle.FWD_REV, 20, 64, 4), (31, oracle.FWD_REV, 50, 90, 1),
    (32, oracle.FWD_REV, 131, 128, 3), (16, oracle.FWD, 64, 64, 3), (33, oracle.FWD, 40, 100, 3),
    (63, oracle.FWD, 100, 200, 2), (64, oracle.FWD, 36, 256, 3)])
@pytest.mark.parametrize("shift", [0, 1])
def test_build_equals_oracle(knng, k, mode, D, leaf, passes, shift):
    # integers: the tree's sums and the distances are exact, so every bit is determined
    n = 2300
    X = np.ascontiguousarray(datagen.sift_like(n, D=D, n_centres=25, seed=3 * k + D) - np.float32(40.0))
    store = torch.empty(n * D + shift, dtype=torch.float32, device="cuda")
    dev = store[shift:].view(n, D)
    dev.copy_(torch.from_numpy(X))
    p = knng.default_params(k=k, leaf_max=leaf, tree_passes=passes, refine_rounds=3, seed=11, join_mode=mode,
                            precision=knng.KNNG_FP32)
    ids, d = knng.knng_build_ex(dev, p)
    o_ids, o_d = oracle.build_graph(X, k, leaf, passes=passes, rounds=3, seed=11, mode=mode)
    np.testing.assert_array_equal(ids.cpu().numpy(), o_ids)
    np.testing.assert_array_equal(d.cpu().numpy(), o_d)


@pytest.mark.parametrize("k", [3, 8, 32, 40])
@pytest.mark.parametrize("hubs", [1, 12])
def test_offers_to_a_few_nodes_match_oracle(knng, k, hubs):
    # every list holds the hubs, so these get from a few to hundreds of offers,
    # most of them repeats, and the others a handful
    n, D = 400, 9
    rng = np.random.default_rng(k + hubs)
    X = rng.integers(-50, 51, size=(n, D)).astype(np.float32)
    ids, d = oracle.new_graph(n, k)
    for i in range(n):
        first = [j for j in range(hubs) if j != i][:k]
        rest = rng.permutation(np.setdiff1d(np.arange(n), first + [i]))[:k - len(first)]
        for j in first + rest.tolist():
            oracle.list_insert(ids[i], d[i], oracle.dist_f32(X[i], X[j]), j)
    mode = oracle.FWD_REV if k <= 32 else oracle.FWD
    o = (ids.copy(), d.copy())
    for _ in range(2):
        o = oracle.refine_round(X, *o, mode=mode)
    p = knng.default_params(k=k, refine_rounds=2, join_mode=mode)
    g_ids, g_d = knng.knng_refine(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (X, ids, d)], p)
    np.testing.assert_array_equal(g_ids.cpu().numpy(), o[0])
    np.testing.assert_array_equal(g_d.cpu().numpy(), o[1])
