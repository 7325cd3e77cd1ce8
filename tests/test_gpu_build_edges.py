"""Builds at the sizes where the builder changes its way: tiles of the radix
sort (1024 and 4096 pairs), of the top levels' partition (2048 elements),
subtrees built by one block (1024 points, 4096 from 2^18 + 1 points on), all
dimensions sorted together or one after the other (2^21 keys), against the
oracle's tree; and forests whose trees lie on both sides of those sizes."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kdt():
    from paper_2210_12859_gb300 import build

    build.build_library()
    from paper_2210_12859_gb300 import kdt as k

    return k


def points(N, D, kind):
    g = np.random.default_rng(N + 31 * D)
    if kind == "grid":  # few values: ties broken by index throughout
        return g.integers(0, 12, size=(N, D)).astype(np.float32)
    p = g.standard_normal((N, D)).astype(np.float32)
    p[: N // 7] = p[0]  # and one place many times
    return p


def check(kdt, tree, pts, want):
    coords, ids = kdt.kdt_tree_export(tree)
    assert np.array_equal(ids.cpu().numpy(), want)
    assert np.array_equal(coords.cpu().numpy().view(np.uint32), pts[want].view(np.uint32))


@pytest.mark.parametrize("N", [1023, 1024, 1025, 2047, 2048, 2049, 4095, 4096, 4097, 6143, 20011, 131072, 262143,
                               262144, 262145, 300007, (1 << 19) + 1])
@pytest.mark.parametrize("D,kind", [(3, "grid"), (3, "cloud"), (2, "cloud")])
def test_sizes(kdt, N, D, kind):
    pts = points(N, D, kind)
    tree = kdt.kdt_build(torch.from_numpy(pts).cuda())
    check(kdt, tree, pts, oracle.build(pts))


@pytest.mark.parametrize("N", [1, 5, 1025, 9001, 270001])
@pytest.mark.parametrize("D", [1, 4, 5, 8])
def test_dimensions(kdt, N, D):
    pts = points(N, D, "cloud" if N % 2 else "grid")
    tree = kdt.kdt_build(torch.from_numpy(pts).cuda())
    check(kdt, tree, pts, oracle.build(pts))
    other = points(N, D, "grid")
    kdt.kdt_rebuild(tree, torch.from_numpy(other).cuda())
    check(kdt, tree, other, oracle.build(other))


@pytest.mark.parametrize("N", [3, 1024, 1030, 8195, 262144, 275003])
@pytest.mark.parametrize("D", [1, 2, 3])
def test_widest(kdt, N, D):
    pts = points(N, D, "cloud")
    tree = kdt.kdt_build(torch.from_numpy(pts).cuda(), kdt.KDT_BUILD_WIDEST)
    want, dims = oracle.build_widest(pts)
    check(kdt, tree, pts, want)
    assert np.array_equal(kdt.kdt_tree_split_dims(tree).cpu().numpy(), dims)


@pytest.mark.parametrize("D", [1, 3, 5])
@pytest.mark.parametrize("sizes", [[0, 1, 1024, 0, 1025, 2048, 5000, 3], [4096, 4097, 1, 270000, 8193, 0]])
def test_forests(kdt, D, sizes):
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pts = points(int(off[-1]), D, "grid")
    forest = kdt.kdt_build_batched(torch.from_numpy(pts).cuda(), off)
    coords, ids = (x.cpu().numpy() for x in kdt.kdt_forest_export(forest))
    for i, n in enumerate(sizes):
        if n:
            a, b = off[i], off[i + 1]
            want = oracle.build(pts[a:b])
            assert np.array_equal(ids[a:b], want)
            assert np.array_equal(coords[a:b], pts[a:b][want])
