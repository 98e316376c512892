"""Exact lists by tensor-core screening equal the FP32 kernel's bit for bit
(knng_exact_noalloc always takes the FP32 kernel): one and several column
sets, ragged row and column tiles, one K chunk and more than stay resident,
dims that are no multiple of 4, k across 32, integer data, data whose bound
serves no row (a large common offset; magnitudes past the bound's range),
duplicate points, points sorted by cluster, and every row without a sample."""
import numpy as np
import pytest

import datagen

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
    if kind == "integer":
        return datagen.sift_like(n, D=D, n_centres=100, seed=5)
    X = datagen.gaussian_mixture(n, D, 100, seed=6)
    if kind == "offset":
        X += np.float32(3000.0)
    if kind == "huge":
        X *= np.float32(1e17)
    if kind == "duplicates":
        X[n // 2:] = X[: n - n // 2]
    if kind == "sorted":
        X = X[np.lexsort(X.T[:2])]
    return np.ascontiguousarray(X)


@pytest.mark.parametrize("kind,n,D,k,s", [
    ("float", 4096, 300, 10, 1700), ("float", 4097, 400, 20, 1300), ("integer", 70001, 128, 20, 257),
    ("float", 65537, 50, 64, 700), ("float", 20011, 257, 33, 400), ("integer", 30000, 67, 16, 1025),
    ("offset", 20000, 96, 10, 1100), ("huge", 20000, 64, 10, 1600), ("duplicates", 40000, 96, 20, 600),
    ("sorted", 150000, 32, 16, 450)])
def test_screened_lists_equal_fp32(knng, kind, n, D, k, s):
    X = torch.from_numpy(_points(kind, n, D)).cuda()
    rows = torch.from_numpy(datagen.sample_rows(n, s, seed=7)).cuda()
    ids, d = knng.knng_exact(X, k, rows)
    ref_ids, ref_d = knng.knng_exact_noalloc(X, k, rows)
    assert torch.equal(ids, ref_ids) and torch.equal(d.view(torch.int32), ref_d.view(torch.int32))


def test_every_row(knng):
    X = torch.from_numpy(_points("float", 9001, 40)).cuda()
    ids, d = knng.knng_exact(X, 12)
    ref_ids, ref_d = knng.knng_exact_noalloc(X, 12, torch.arange(9001, dtype=torch.int32, device="cuda"))
    assert torch.equal(ids, ref_ids) and torch.equal(d, ref_d)


@pytest.mark.parametrize("n,D,k,s", [(129, 5, 3, 1), (255, 33, 64, 65), (256, 33, 64, 129), (257, 4, 1, 1)])
def test_smallest(knng, n, D, k, s):
    X = torch.from_numpy(_points("float", n, D)).cuda()
    rows = torch.from_numpy(datagen.sample_rows(n, s, seed=8)).cuda()
    ids, d = knng.knng_exact(X, k, rows)
    ref_ids, ref_d = knng.knng_exact_noalloc(X, k, rows)
    assert torch.equal(ids, ref_ids) and torch.equal(d, ref_d)


@pytest.mark.parametrize("n,D,W,spread", [(3000, 130, 16, 20), (5000, 64, 3, 3), (2049, 300, 200, 0)])
def test_word_means_in_the_defined_order(knng, n, D, W, spread):
    """Sums whose magnitudes lie 2^(2 spread) apart round in FP64, so the words must come from the defined order."""
    import oracle
    rng = np.random.default_rng(11)
    X = (rng.standard_normal((n, D)) * np.exp2(rng.uniform(-spread, spread, (n, D)))).astype(np.float32)
    w1, w2 = knng.knng_rvq_train(torch.from_numpy(X).cuda(), W, W, 2, seed=3)
    o1, o2 = oracle.rvq_train(X, W, W, 2, seed=3)
    assert np.array_equal(w1.cpu().numpy().view(np.uint32), o1.view(np.uint32))
    assert np.array_equal(w2.cpu().numpy().view(np.uint32), o2.view(np.uint32))
