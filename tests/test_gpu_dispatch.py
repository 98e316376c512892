"""Which kernels served a call, from the statistics: exact lists from the
tensor-core screen, with the FP32 kernel only for rows whose bound cannot
serve; leaves on the tensor cores exactly where the build's 16-bit copy holds
the data, else the FP32 leaf, with the graph of the FP32 build either way."""
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


def _kernels(knng, call):
    knng.stats_reset()
    knng.stats_enable(True, False)
    try:
        out = call()
        torch.cuda.synchronize()
        return out, knng.stats()
    finally:
        knng.stats_enable(False)


# a row is given up when more than 4,096 columns pass its threshold (about 4 k
# do) or a squared norm is past the bound's arithmetic (1e30)
@pytest.mark.parametrize("kind,given_up", [("float", 0), ("integer", 0), ("twice", 0), ("huge", 900), ("same", 900)])
def test_screened_rows(knng, kind, given_up):
    n, D, s = 20000, 64, 900
    X = datagen.sift_like(n, D=D, n_centres=100, seed=5) if kind == "integer" else datagen.gaussian_mixture(n, D, 100, seed=6)
    if kind == "huge":
        X = X * np.float32(1e17)
    if kind == "twice":
        X[n // 2:] = X[: n // 2]
    if kind == "same":
        X[:] = X[0]
    Xd = torch.from_numpy(np.ascontiguousarray(X)).cuda()
    rows = torch.from_numpy(datagen.sample_rows(n, s, seed=7)).cuda()
    (ids, d), ran = _kernels(knng, lambda: knng.knng_exact(Xd, 10, rows))
    assert "ks_screen" in ran and ran["k7_exact"]["items"] == given_up
    ref_ids, ref_d = knng.knng_exact_noalloc(Xd, 10, rows)
    assert torch.equal(ids, ref_ids) and torch.equal(d, ref_d)


@pytest.mark.parametrize("n,D,s,screened", [(255, 300, 200, False), (256, 32, 4, False), (256, 33, 4, True), (256, 32, 5, True),
                                            (8192, 1, 1, False), (8193, 1, 1, True)])
def test_small_exact_lists(knng, n, D, s, screened):
    X = torch.from_numpy(datagen.gaussian_mixture(n, D, 10, seed=n)).cuda()
    rows = torch.arange(s, dtype=torch.int32, device="cuda")
    (ids, d), ran = _kernels(knng, lambda: knng.knng_exact(X, 7, rows))
    assert ("ks_screen" in ran) == screened
    ref_ids, ref_d = knng.knng_exact_noalloc(X, 7, rows)
    assert torch.equal(ids, ref_ids) and torch.equal(d, ref_d)


@pytest.mark.parametrize("leaf", [64, 128, 256])
@pytest.mark.parametrize("data,exact", [("integer", ("bf16", "fp16")), ("wide", ("fp16",)), ("float", ())])
def test_leaf_kernels(knng, data, exact, leaf):
    X = datagen.gaussian_mixture(3000, 40, 20, seed=3)
    if data == "integer":
        X = datagen.sift_like(3000, D=40, n_centres=20, seed=3)
    if data == "wide":                       # integers of 50 to 542: FP16 holds them, BF16 does not
        X = np.round(X * np.float32(1000.0 / np.abs(X).max()) / 4) + np.float32(300.0)
    Xd = torch.from_numpy(np.ascontiguousarray(X, np.float32)).cuda()
    names = {"bf16": knng.KNNG_BF16, "fp16": knng.KNNG_FP16, "fp8": knng.KNNG_FP8}
    args = dict(k=8, leaf_max=leaf, tree_passes=2, refine_rounds=1, seed=4)
    (ref_ids, ref_d), ran = _kernels(knng, lambda: knng.knng_build_ex(Xd, knng.default_params(**args)))
    assert "k2_leaf_fp32" in ran
    for name, prec in names.items():
        (ids, d), ran = _kernels(knng, lambda: knng.knng_build_ex(Xd, knng.default_params(precision=prec, **args)))
        assert torch.equal(ids, ref_ids) and torch.equal(d, ref_d)
        leaves = {k for k in ran if k.startswith("k2_leaf_")}
        assert leaves == ({"k2_leaf_" + name} if name in exact else {"k2_leaf_fp32"}), (name, leaves)
