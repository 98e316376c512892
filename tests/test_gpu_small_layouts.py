"""Calls whose scratch does not fit take a smaller layout and give the same
results: KNNG_FAULT=optional refuses, on the host, the first allocation that a
call can do without, KNNG_FAULT=optionals every one.  Exact lists by the FP32 kernel with its columns split, words
and codes by the FP32 assignment with every word's mean summed in ascending
order, and up to 32 seeds by the general ranking; the statistics say that those
kernels ran."""
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


@pytest.fixture
def kernels(knng, monkeypatch):
    """Runs a call under the fault; its result and the statistics of the kernels that ran."""
    def run(call, mode="optional"):
        monkeypatch.setenv("KNNG_FAULT", mode)
        knng.stats_reset()
        knng.stats_enable(True, False)
        try:
            out = call()
            torch.cuda.synchronize()
            return out, knng.stats()
        finally:
            knng.stats_enable(False)
            monkeypatch.delenv("KNNG_FAULT")
    return run


def _dev(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


@pytest.mark.parametrize("n,D,k,s", [(256, 33, 64, 100), (2049, 40, 10, 65), (30000, 130, 20, 300), (70001, 16, 33, 1),
                                     (5000, 24, 5, None)])
def test_exact_lists(knng, kernels, n, D, k, s):
    X, = _dev(datagen.gaussian_mixture(n, D, 30, seed=n))
    rows = torch.arange(n, dtype=torch.int32, device="cuda") if s is None else _dev(datagen.sample_rows(n, s, seed=4))[0]
    (ids, d), ran = kernels(lambda: knng.knng_exact(X, k, None if s is None else rows))
    ref_ids, ref_d = knng.knng_exact_noalloc(X, k, rows)
    assert torch.equal(ids, ref_ids) and torch.equal(d.view(torch.int32), ref_d.view(torch.int32))
    assert "k7_exact" in ran and "ks_screen" not in ran


def test_exact_lists_without_partial_lists(knng, kernels):
    """The FP32 lists need no scratch beyond the keys when the partial lists of its column splits do not fit."""
    X, rows = _dev(datagen.gaussian_mixture(30000, 60, 30, seed=1), datagen.sample_rows(30000, 200, seed=4))
    (ids, d), ran = kernels(lambda: knng.knng_exact(X, 12, rows), "optional")
    assert ran["k7_exact"]["launches"] == 2          # the splits, then their merge
    (ids1, d1), ran = kernels(lambda: knng.knng_exact(X, 12, rows), "optionals")
    assert ran["k7_exact"]["launches"] == 1
    assert torch.equal(ids, ids1) and torch.equal(d, d1)


@pytest.mark.parametrize("n,D,W1,W2", [(3000, 33, 16, 20), (2500, 128, 200, 129), (40, 5, 40, 3)])
def test_words_and_index(knng, kernels, n, D, W1, W2):
    X = datagen.gaussian_mixture(n, D, 20, seed=n)
    Xd, = _dev(X)
    (w1, w2), ran = kernels(lambda: knng.knng_rvq_train(Xd, W1, W2, 3, seed=5))
    o1, o2 = oracle.rvq_train(X, W1, W2, 3, seed=5)
    assert np.array_equal(w1.cpu().numpy(), o1) and np.array_equal(w2.cpu().numpy(), o2)
    assert "k9_assign" in ran and "ks_assign" not in ran
    got, ran = kernels(lambda: knng.knng_rvq_index(Xd, w1, w2))
    for a, b in zip(got, oracle.rvq_index(X, o1, o2)):
        assert np.array_equal(a.cpu().numpy(), b)
    assert {"k9_assign", "k9_assign_res"} <= set(ran) and "ks_assign" not in ran


@pytest.mark.parametrize("W1,W2,probe1,s,D,m", [(64, 256, 16, 32, 40, 65), (7, 13, 7, 20, 33, 200), (256, 30, 32, 1, 64, 3)])
def test_seeds(knng, kernels, W1, W2, probe1, s, D, m):
    X = datagen.gaussian_mixture(6000, D, 20, seed=D)
    o1, o2 = oracle.rvq_train(X[:3000], W1, W2, 1, seed=9)
    _, off, ids = oracle.rvq_index(X, o1, o2)
    Q = datagen.gaussian_mixture(m, D, 20, seed=D + 1)
    S, ran = kernels(lambda: knng.knng_rvq_seeds(*_dev(o1, o2, off, ids, Q), probe1, s))
    assert np.array_equal(S.cpu().numpy(), oracle.rvq_seeds(o1, o2, off, ids, Q, probe1, s))
    assert "k9_tables" in ran and "k9_dots" not in ran
