"""Levels whose largest segment comes up to the shared memory a CTA may have:
the sizes that just fit a cluster of eight and the first that do not, for FP32
and for byte rows, at the root and one level down, equal the oracle's
partition; direct, recorded and batched builds of such a size agree."""
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
    return X - np.float32(60.0) if kind == "signed" else X  # signed: FP32 rows, integers all the same


# a CTA's shared memory, in bytes: 231,104 .. 231,424 for the first sizes of a
# line, 232,448 (the limit) or just below for the next to last, past it for the last
@pytest.mark.parametrize("kind,D,sizes", [
    ("signed", 32, (8728, 8729, 8736, 8744, 8745, 8776, 8777)), ("signed", 96, (3625, 3632, 3644, 3645)),
    ("signed", 128, (2881, 2888, 2896, 2897)), ("signed", 8, (18641, 18672, 18736, 18737)),
    ("bytes", 128, (8641, 8652, 8680, 8681)), ("bytes", 32, (18593, 18624, 18688, 18689)),
    ("signed", 32, (17459, 17472))])
def test_partition_at_the_limit_equals_oracle(knng, kind, D, sizes):
    for n in sizes:
        X = _points(kind, n, D)
        leaf = n // 2 + 1 if n < 17000 or D != 32 or kind == "bytes" else n // 4 + 1
        perm, off = knng.knng_partition(torch.from_numpy(X).cuda(), leaf, twomeans_iters=2, seed=5)
        o_perm, o_off = oracle.partition(X, leaf, iters=2, seed=5)
        assert np.array_equal(perm.cpu().numpy(), o_perm) and np.array_equal(off.cpu().numpy(), o_off), n


@pytest.mark.parametrize("n,D", [(8736, 32), (2884, 128)])
def test_builds_at_the_limit_agree(knng, n, D):
    X = _points("signed", n, D)
    Xd = torch.from_numpy(X).cuda()
    p = knng.default_params(k=8, leaf_max=100, tree_passes=3, refine_rounds=1, twomeans_iters=2, seed=6)
    ids, d = knng.knng_build_ex(Xd, p)
    o_ids, o_d = oracle.build_graph(X, 8, 100, passes=3, rounds=1, iters=2, mode=int(p.join_mode), seed=6)
    assert np.array_equal(ids.cpu().numpy(), o_ids) and np.array_equal(d.cpu().numpy(), o_d)
    plan = knng.BuildPlan(Xd, p)
    for r_ids, r_d in (plan.launch(), knng.knng_build_batched([Xd], p)[0]):
        torch.cuda.synchronize()
        assert torch.equal(r_ids, ids) and torch.equal(r_d, d)
