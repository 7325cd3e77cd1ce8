"""Sequences of calls on one forest: what a batched query keeps between calls
(its scratch, the offsets in it, a graph of repeated arguments) must never
show in a result."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kdt():
    from paper_2210_12859_gb300 import build

    build.build_library()
    from paper_2210_12859_gb300 import kdt as k

    return k


def cu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def offsets(*sizes):
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


@pytest.fixture(scope="module")
def forest(kdt):
    g = np.random.default_rng(17)
    off = offsets(300, 1000, 7)
    return kdt.kdt_build_batched(cu(g.random((off[-1], 3), dtype=np.float32)), off)


def outputs(Q, k):
    return torch.full((Q, k), -7, dtype=torch.int32, device="cuda"), torch.full((Q, k), -7.0, device="cuda")


def same(a, b):
    return torch.equal(a[0], b[0]) and torch.equal(a[1].view(torch.int32), b[1].view(torch.int32))


def test_after_a_failed_growth_of_the_scratch(kdt, forest):
    """A query that needs more scratch than the forest holds gives the old one
    up first; when the new allocation fails, the arguments that ran before must
    not be taken as still in place."""
    g = np.random.default_rng(3)
    k, flags = 4, kdt.KDT_MORTON
    small, large = (cu(g.random((n, 3), dtype=np.float32)) for n in (120, 30000))
    q_small, q_large = offsets(50, 50, 20), offsets(9, 24991, 5000)
    want_small = kdt.kdt_knn_batched(forest, small, q_small, k, flags=kdt.KDT_PER_TREE)
    want_large = kdt.kdt_knn_batched(forest, large, q_large, k, flags=kdt.KDT_PER_TREE)
    out_i, out_d = outputs(120, k)

    def run_small():
        out_i.fill_(-7)
        return kdt.kdt_knn_batched(forest, small, q_small, k, flags=flags, out_ids=out_i, out_d2=out_d)

    assert same(run_small(), want_small)
    kdt.kdt_debug_fail_allocs(1)
    try:
        with pytest.raises(kdt.KdtError) as e:
            kdt.kdt_knn_batched(forest, large, q_large, k, flags=flags)
    finally:
        kdt.kdt_debug_fail_allocs(0)
    assert e.value.code == kdt.KDT_ENOMEM
    assert same(run_small(), want_small)  # the very arguments of the first call
    assert same(kdt.kdt_knn_batched(forest, large, q_large, k, flags=flags), want_large)


def test_many_small_clouds_built_behind_other_work(kdt):
    """40000 clouds of 0 to 12 points and one large one, on a stream that is
    still busy when the build enqueues its tables of first blocks (hundreds of
    kilobytes, copied from the host): every tree and every row is right."""
    import oracle

    g = np.random.default_rng(23)
    sizes = g.integers(0, 13, 40001)
    sizes[20000] = 30011
    off = offsets(*sizes)
    pts = np.floor(g.random((off[-1], 3)) * 32).astype(np.float32)  # many ties
    dp = cu(pts)
    nq = g.integers(0, 4, len(sizes))
    qoff = offsets(*nq)
    dq = cu((g.random((qoff[-1], 3)) * 32).astype(np.float32))
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        torch.cuda._sleep(100_000_000)
        forest = kdt.kdt_build_batched(dp, off)
        ids = kdt.kdt_forest_export(forest)[1].cpu().numpy()
        got = kdt.kdt_knn_batched(forest, dq, qoff, 4, flags=kdt.KDT_MORTON)
        want = kdt.kdt_knn_batched(forest, dq, qoff, 4, flags=kdt.KDT_UNORDERED)
        s.synchronize()
    assert same(got, want)
    for i in [20000, *g.choice(len(sizes), 400, replace=False)]:
        if sizes[i]:
            assert np.array_equal(ids[off[i]:off[i + 1]], oracle.build(pts[off[i]:off[i + 1]])), i
