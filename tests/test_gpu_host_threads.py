"""Host threads that call at once, each on its own stream, with rows and trees
whose kernels take different amounts of shared memory: every call succeeds and
gives what it gives alone."""
import threading

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


def _at_once(calls, repeats):
    """Runs every call `repeats` times, each in a thread of its own; what failed or differed from a call alone."""
    want = [c() for c in calls]
    torch.cuda.synchronize()
    failed, start = [], threading.Barrier(len(calls))

    def work(i):
        stream = torch.cuda.Stream()
        start.wait()
        with torch.cuda.stream(stream):
            for _ in range(repeats):
                try:
                    got = calls[i]()
                except Exception as e:   # KnngError, or what the wrapper makes of it
                    failed.append((i, str(e)))
            stream.synchronize()
            if not failed and not all(torch.equal(a, b) for a, b in zip(got, want[i])):
                failed.append((i, "differs"))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return failed


def test_builds_of_two_sizes(knng):
    p = knng.default_params(k=4, leaf_max=256, tree_passes=4, twomeans_iters=0, seed=2)
    data = [torch.from_numpy(datagen.gaussian_mixture(n, 96, 20, seed=n)).cuda()
            for n in (1300, 3600, 1300, 3600, 2000, 3000)]
    assert _at_once([lambda x=x: knng.knng_build_ex(x, p) for x in data], 300) == []


def test_calls_of_several_dims(knng):
    p = knng.default_params(k=6, leaf_max=64, tree_passes=1, refine_rounds=1, twomeans_iters=0, seed=2)
    data = [torch.from_numpy(datagen.gaussian_mixture(n, D, 20, seed=n)).cuda()
            for n, D in ((1300, 40), (1100, 96), (900, 250))]
    rows = torch.arange(0, 900, 9, dtype=torch.int32, device="cuda")
    calls = [lambda x=x: knng.knng_build_ex(x, p) for x in data]
    calls += [lambda x=x: knng.knng_exact(x, 10, rows) for x in data]
    assert _at_once(calls, 150) == []
