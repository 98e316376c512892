"""One-launch levels of the two-means tree: partitions whose levels fit the
shared memory of 1, 2, 4 or 8 CTAs equal the oracle's on integer data (byte
rows, FP32 rows of negative integers, rows that are no multiple of 16 bytes or
not 16-byte aligned, segments one above and below the CTA sizes, more equal
projections than one warp ranks, no iterations), and the 16-bit copies' levels
equal the FP32 ones."""
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
    X = datagen.sift_like(n, D=D, n_centres=30, seed=n + D)
    if kind == "signed":
        X -= np.float32(60.0)
    if kind == "few":         # five distinct points
        X = X[np.arange(n) % 5]
    return np.ascontiguousarray(X)


@pytest.mark.parametrize("kind,n,D,leaf,iters", [
    ("bytes", 129, 128, 64, 4), ("bytes", 2000, 131, 100, 4), ("bytes", 5001, 16, 33, 3), ("bytes", 9000, 257, 256, 2),
    ("signed", 300, 7, 20, 4), ("signed", 2049, 96, 64, 4), ("signed", 4097, 130, 128, 1), ("signed", 700, 960, 60, 2),
    ("few", 3000, 40, 70, 3), ("few", 257, 8, 16, 2), ("signed", 1025, 33, 50, 0), ("bytes", 513, 1, 40, 4)])
@pytest.mark.parametrize("shift", [0, 1])
def test_partition_equals_oracle(knng, kind, n, D, leaf, iters, shift):
    X = _points(kind, n, D)
    buf = torch.empty(n * D + 4, device="cuda")
    Xd = buf[shift:shift + n * D].view(n, D)       # shift 1: rows off the 16-byte grid
    Xd.copy_(torch.from_numpy(X))
    perm, off = knng.knng_partition(Xd, leaf, twomeans_iters=iters, seed=9)
    o_perm, o_off = oracle.partition(X, leaf, iters=iters, seed=9)
    assert np.array_equal(perm.cpu().numpy(), o_perm) and np.array_equal(off.cpu().numpy(), o_off)


@pytest.mark.parametrize("n,D", [(1500, 96), (3001, 70)])
def test_16_bit_copies_give_the_same_levels(knng, n, D):
    X = torch.from_numpy(_points("signed", n, D)).cuda()
    ref = None
    for prec in (knng.KNNG_FP32, knng.KNNG_BF16, knng.KNNG_FP16):
        p = knng.default_params(k=8, leaf_max=64, tree_passes=2, precision=prec, seed=4)
        ids, d = knng.knng_build_ex(X, p)
        if ref is not None:
            assert torch.equal(ids, ref[0]) and torch.equal(d, ref[1])
        ref = ids, d


def test_forest_of_uneven_depths(knng):
    datas = [torch.from_numpy(_points("bytes", n, 24)).cuda() for n in (60, 3000, 129, 700)]
    p = knng.default_params(k=6, leaf_max=64, tree_passes=2, seed=6)
    for x, (ids, d) in zip(datas, knng.knng_build_batched(datas, p)):
        one, od = knng.knng_build_ex(x, p)
        assert torch.equal(ids, one) and torch.equal(d, od)


@pytest.mark.parametrize("kind", ["signed", "few"])
@pytest.mark.parametrize("n,D,levels", [(2049, 960, 1), (4100, 960, 2), (16384, 200, 1), (16385, 200, 1), (32769, 100, 2),
                                        (65537, 64, 1), (131072, 64, 1), (131073, 64, 2)])
def test_one_launch_cuts_of_larger_segments(knng, kind, n, D, levels):
    """Rows too many for a cluster's shared memory: sweeps, with the cut of up to 131,072 points in one launch
    (1, 2, 4 and 8 CTAs, one point more than each holds, hundreds of equal projections across CTAs)."""
    X = _points(kind, n, D)
    leaf = -(-n // 2 ** levels)
    perm, off = knng.knng_partition(torch.from_numpy(X).cuda(), leaf, twomeans_iters=2, seed=3)
    o_perm, o_off = oracle.partition(X, leaf, iters=2, seed=3)
    assert np.array_equal(perm.cpu().numpy(), o_perm) and np.array_equal(off.cpu().numpy(), o_off)


def test_cut_of_uneven_forest(knng):
    """A level whose largest segment takes eight CTAs and whose smallest has fewer points than one warp."""
    datas = [torch.from_numpy(_points("signed", n, 200)).cuda() for n in (40000, 30, 5000)]
    p = knng.default_params(k=4, leaf_max=20, tree_passes=1, twomeans_iters=1, seed=6)
    for x, (ids, d) in zip(datas, knng.knng_build_batched(datas, p)):
        one, od = knng.knng_build_ex(x, p)
        assert torch.equal(ids, one) and torch.equal(d, od)
