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


def test_repeated_arguments_on_a_stream(kdt, forest):
    """The same buffers again and again on a stream (enqueued, captured,
    replayed), with new queries in them each time; other offsets in between."""
    g = np.random.default_rng(4)
    k, flags = 5, kdt.KDT_MORTON
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        dq = torch.empty((400, 3), device="cuda")
        out_i, out_d = outputs(400, k)
        for step in range(9):
            dq.copy_(cu(g.random((400, 3), dtype=np.float32)))
            qoff = offsets(100, 250, 50) if step not in (4, 7) else offsets(0, 390, 10)
            got = kdt.kdt_knn_batched(forest, dq, qoff, k, flags=flags, out_ids=out_i, out_d2=out_d)
            assert same(got, kdt.kdt_knn_batched(forest, dq, qoff, k, flags=kdt.KDT_PER_TREE)), step
    s.synchronize()


@pytest.mark.parametrize("before", ["none", "default stream", "stream"])
def test_in_a_graph_of_the_caller(kdt, forest, before):
    """A captured query keeps its own offsets: whether its arguments have run
    before, whatever runs between its replays, also once the forest has needed
    a larger scratch and the caller's offsets array is gone; and a replay
    between repeated calls does not change theirs."""
    g = np.random.default_rng(5)
    k, flags = 5, kdt.KDT_MORTON
    a, b = (cu(g.random((400, 3), dtype=np.float32)) for _ in range(2))
    big = cu(g.random((40000, 3), dtype=np.float32))
    qa, qb, qbig = [0, 100, 350, 400], [0, 0, 390, 400], [0, 40000, 40000, 40000]
    want = [kdt.kdt_knn_batched(forest, x, o, k, flags=kdt.KDT_PER_TREE) for x, o in ((a, qa), (b, qb), (big, qbig))]
    out_a, out_b = outputs(400, k), outputs(400, k)

    def call(x, o, out):
        return kdt.kdt_knn_batched(forest, x, o, k, flags=flags, out_ids=out[0], out_d2=out[1])

    s = torch.cuda.Stream()
    call(b, qb, out_b)  # the scratch is there
    if before == "default stream":
        call(a, qa, out_a)
    torch.cuda.synchronize()
    if before == "stream":
        with torch.cuda.stream(s):
            for _ in range(3):
                call(a, qa, out_a)
    s.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        call(a, list(qa), out_a)
    with torch.cuda.stream(s):
        for rep in range(4):
            assert same(call(b, qb, out_b), want[1]), rep  # repeated: by the forest's own graph in the end
            out_a[0].fill_(-7)
            graph.replay()
            assert same(out_a, want[0]), rep
        assert same(call(b, qb, out_b), want[1])
        assert same(kdt.kdt_knn_batched(forest, big, qbig, k, flags=flags), want[2])
        out_a[0].fill_(-7)
        graph.replay()
        assert same(out_a, want[0])
    s.synchronize()


@pytest.mark.parametrize("D", [1, 3, 4, 6])
def test_classes_of_tree_sizes(kdt, D):
    """Trees on both sides of the builder's classes (128, 1024 and 4096 points)
    and of the box build's (32 buckets), in one forest of more than 2^18 points."""
    import oracle

    g = np.random.default_rng(40 + D)
    sizes = [0, 1, 8, 127, 128, 129, 0, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 4096, 4097, 3, 270000, 64, 0]
    sizes += list(g.integers(100, 160, 50))
    off = offsets(*sizes)
    pts = np.floor(g.random((off[-1], D)) * 200).astype(np.float32)
    forest = kdt.kdt_build_batched(cu(pts), off)
    ids = kdt.kdt_forest_export(forest)[1].cpu().numpy()
    for i, n in enumerate(sizes):
        if n:
            assert np.array_equal(ids[off[i]:off[i + 1]], oracle.build(pts[off[i]:off[i + 1]])), i
    qoff = offsets(*g.integers(0, 60, len(sizes)))
    dq = cu((g.random((qoff[-1], D)) * 200).astype(np.float32))
    for k in (1, 9):
        want = kdt.kdt_knn_batched(forest, dq, qoff, k, flags=kdt.KDT_UNORDERED)
        assert same(kdt.kdt_knn_batched(forest, dq, qoff, k), want)


def test_autotune(kdt):
    """Ordered queries take no launch parameter: they are timed and the
    forest's parameters stay.  Unordered ones are timed as they run when their
    arguments repeat, without the capture of the graph: on a tiny forest, where
    that would be most of the time, the reported time is within the time that a
    replay takes with the binding's own overhead, measured here."""
    g = np.random.default_rng(6)
    f = kdt.kdt_build_batched(cu(g.random((400, 3), dtype=np.float32)), offsets(100, 100, 100, 100))
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        dq = cu(g.random((64, 3), dtype=np.float32))
        qoff, out = offsets(16, 16, 16, 16), outputs(64, 8)
        kdt.kdt_forest_set_launch(f, 32, 17, 1, 5)
        assert kdt.kdt_forest_autotune(f, dq, qoff, 8, flags=kdt.KDT_MORTON)[:4] == (32, 17, 1, 5)
        kdt.kdt_forest_set_launch(f, 0, 0)
        flags = kdt.KDT_MORTON | kdt.KDT_UNORDERED
        reported = min(kdt.kdt_forest_autotune(f, dq, qoff, 8, flags=flags)[4] for _ in range(3))
        ms = []
        for _ in range(23):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            kdt.kdt_knn_batched(f, dq, qoff, 8, flags=flags, out_ids=out[0], out_d2=out[1])
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        assert reported <= np.median(ms[3:]), (reported, ms)
        kdt.kdt_forest_set_launch(f, 0, 0)
