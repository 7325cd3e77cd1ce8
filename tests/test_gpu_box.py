"""kNN by box tree (ordered result queries) against the state machine's
unordered form, which walks the level-order tree by the one-coordinate test of
Sec. 3.2: the same ids and the same distance bits, at the sizes where the box
tree's buckets and records begin, end or are ragged, for every node layout,
list size and kind of tie."""
import math

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


def same(a, b):
    return torch.equal(a[0], b[0]) and torch.equal(a[1].view(torch.int32), b[1].view(torch.int32))


def both(kdt, tree, dq, k, r=math.inf, flags=0):
    got = kdt.kdt_knn(tree, dq, k, r, flags)
    want = kdt.kdt_knn(tree, dq, k, r, kdt.KDT_UNORDERED)
    kdt.kdt_status(tree)
    assert same(got, want), (tree.N, tree.D, k, r, flags)


SIZES = [1, 2, 3, 6, 7, 8, 9, 15, 16, 17, 30, 31, 32, 33, 63, 64, 65, 127, 128, 135, 136, 137, 255, 256, 1023, 1024,
         1032, 4095, 4096, 16391, 40000]


@pytest.mark.parametrize("D", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("N", SIZES)
def test_sizes_and_layouts(kdt, N, D):
    g = np.random.default_rng(N * 10 + D)
    pts = g.random((N, D), dtype=np.float32)
    if N % 3 == 0:
        pts = np.floor(pts * 6).astype(np.float32)  # equal coordinates, equal distances
    qs = np.concatenate([g.random((150, D), dtype=np.float32) * 1.6 - 0.3, pts[:50],
                         np.floor(g.random((100, D)) * 7).astype(np.float32)])
    dq = torch.from_numpy(qs).cuda()
    dp = torch.from_numpy(pts).cuda()
    for opts in ([0, kdt.KDT_BUILD_WIDEST] if D <= 3 else [0]):
        tree = kdt.kdt_build(dp, opts)
        for k in (1, 2, 3, 5, 8, 11, 16, 17, 64):
            both(kdt, tree, dq, k)
        both(kdt, tree, dq, 8, 0.2, kdt.KDT_MORTON)
        both(kdt, tree, dq, 4, 0.0)
        both(kdt, tree, dq, 8, math.inf, kdt.KDT_MORTON | kdt.KDT_COST_ORDER)


@pytest.mark.parametrize("k", [1, 4, 8, 16, 40])
def test_values_that_are_not_ordinary(kdt, k):
    """NaN, infinite and huge coordinates in the queries, a query batch longer
    than the launch's lanes, and points of one place."""
    g = np.random.default_rng(k)
    pts = g.random((3001, 3), dtype=np.float32)
    pts[100:400] = pts[100]
    tree = kdt.kdt_build(torch.from_numpy(pts).cuda())
    qs = g.random((64, 3), dtype=np.float32)
    qs[0, 0] = np.nan
    qs[1] = np.nan
    qs[2, 1] = np.inf
    qs[3] = -np.inf
    qs[4, 2] = 3e38
    qs[5] = 1e20
    qs[6] = -0.0
    qs[7:20] = pts[100]
    both(kdt, tree, torch.from_numpy(qs).cuda(), k)
    both(kdt, tree, torch.from_numpy(qs).cuda(), k, 3e19)
    nan_row = kdt.kdt_knn(tree, torch.from_numpy(qs[:2]).cuda(), k)
    assert bool((nan_row[0] == -1).all()) and bool(torch.isinf(nan_row[1]).all())
    many = torch.from_numpy(g.random((400_003, 3), dtype=np.float32)).cuda()
    both(kdt, tree, many, k, 0.05, kdt.KDT_MORTON)


def test_rebuilt_and_loaded_trees(kdt, tmp_path):
    """The box tree follows the level-order tree: after a rebuild on other
    points, and in a tree read from a file."""
    g = np.random.default_rng(5)
    a, b = (torch.from_numpy(g.random((5003, 3), dtype=np.float32)).cuda() for _ in range(2))
    dq = torch.from_numpy(g.random((500, 3), dtype=np.float32)).cuda()
    tree = kdt.kdt_build(a)
    kdt.kdt_rebuild(tree, b)
    both(kdt, tree, dq, 8)
    path = str(tmp_path / "t.kdt")
    kdt.kdt_tree_save(tree, path)
    back = kdt.kdt_tree_load(path)
    both(kdt, back, dq, 8)
    assert same(kdt.kdt_knn(back, dq, 8), kdt.kdt_knn(kdt.kdt_build(b), dq, 8))


@pytest.mark.parametrize("D", [1, 3, 4, 6])
def test_forests(kdt, D):
    """Trees on both sides of the box build's limits (empty, one bucket, 256
    buckets, a second launch of the records) in one call, by path order and
    as given, in one launch and one a tree."""
    sizes = [0, 1, 7, 8, 40, 0, 2047, 2048, 4100, 16384, 33000, 5, 0]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    qs_n = [3, 5, 100, 0, 33, 7, 200, 1, 300, 1000, 2000, 9, 4]
    qoff = np.concatenate([[0], np.cumsum(qs_n)]).astype(np.int64)
    g = np.random.default_rng(D)
    pts = torch.from_numpy(np.floor(g.random((int(off[-1]), D)) * 64).astype(np.float32) / 64).cuda()
    dq = torch.from_numpy((g.random((int(qoff[-1]), D)) * 1.2 - 0.1).astype(np.float32)).cuda()
    forest = kdt.kdt_build_batched(pts, off)
    for k in (1, 8, 10, 24):
        for r in (math.inf, 0.1):
            want = kdt.kdt_knn_batched(forest, dq, qoff, k, r, kdt.KDT_UNORDERED)
            for flags in (0, kdt.KDT_MORTON, kdt.KDT_PER_TREE):
                assert same(kdt.kdt_knn_batched(forest, dq, qoff, k, r, flags), want), (k, r, flags)


@pytest.mark.parametrize("Q", [1, 2, 33, 1023, 1024, 1025, 4097, 16384, 16385, (1 << 19) + 3])
def test_ordered_queries_at_the_edges_of_the_sort(kdt, Q):
    """Queries that run in path or cost order give every row, whatever the
    number of queries: tiles of the radix sort and the numbers of its passes."""
    g = np.random.default_rng(Q)
    tree = kdt.kdt_build(torch.from_numpy(g.random((30011, 3), dtype=np.float32)).cuda())
    dq = torch.from_numpy(g.random((Q, 3), dtype=np.float32) * 1.4 - 0.2).cuda()
    want = kdt.kdt_knn(tree, dq, 4)
    for flags in (kdt.KDT_MORTON, kdt.KDT_MORTON | kdt.KDT_COST_ORDER):
        assert same(kdt.kdt_knn(tree, dq, 4, flags=flags), want)
