"""Range queries by box tree: the hits in the order of the stack-free machine
(node, left subtree, right subtree) at the sizes where buckets, groups and
records begin, end or are ragged, with an even and an odd number of levels
above the buckets, for every node layout: counts, ids, distance bits and
payload sums, whose rounding follows the order, against the oracle's machine."""
import ctypes

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


def cu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def bits(x):
    return np.ascontiguousarray(x, dtype=np.float32).view(np.uint32)


SIZES = [1, 2, 3, 7, 8, 9, 15, 16, 17, 23, 24, 31, 32, 33, 63, 64, 65, 127, 128, 135, 136, 137, 255, 256, 257, 511,
         512, 1023, 1024, 1032, 2055, 4096, 8200, 20001]


def data(N, D):
    g = np.random.default_rng(1000 * D + N)
    pts = g.random((N, D), dtype=np.float32)
    if N % 3 == 0:
        pts = (np.floor(pts * 6) / 6).astype(np.float32)  # equal coordinates
    qs = np.concatenate([g.random((90, D), dtype=np.float32) * 1.4 - 0.2, pts[:30], np.zeros((8, D), np.float32)])
    special = np.float32([np.nan, np.inf, -np.inf, 3e38, -3e38, 1e20, -0.0, 0.5])
    qs[-8:] = 0.5
    qs[-8:, D - 1] = special
    return g, pts, qs.astype(np.float32)


def radii(N, D):
    # a few hits, some dozens, all points of a small tree
    r = (np.float32(8.0) / max(N, 8)) ** (1.0 / D) * 0.5
    return [0.0, float(r), float(2 * r)] + ([float("inf")] if N <= 300 else [])


@pytest.mark.parametrize("D", [1, 2, 3, 4, 6, 8])
@pytest.mark.parametrize("N", SIZES)
def test_hit_order(kdt, N, D):
    g, pts, qs = data(N, D)
    pay = g.standard_normal((N, 3)).astype(np.float32)
    dq = cu(qs)
    for widest in ([False, True] if D <= 3 else [False]):
        tree = kdt.kdt_build(cu(pts), kdt.KDT_BUILD_WIDEST if widest else 0)
        pid, dims = oracle.build_widest(pts) if widest else (oracle.build(pts), None)
        kdt.kdt_tree_set_payload(tree, cu(pay))
        for r in radii(N, D):
            counts, off, ids, d2 = oracle.range_tree(pts, pid, qs, radius=r, node_dim=dims)
            flags = kdt.KDT_MORTON if r else 0
            got = kdt.kdt_radius_search(tree, dq, r, flags)
            assert np.array_equal(got[0].cpu().numpy(), off) and np.array_equal(got[1].cpu().numpy(), ids), r
            assert np.array_equal(bits(got[2].cpu().numpy()), bits(d2)), r
            want, _ = oracle.range_reduce(pts, pid, qs, r, pay, oracle.REDUCE_SUM, node_dim=dims)
            out, n = kdt.kdt_radius_reduce(tree, dq, r, kdt.KDT_REDUCE_SUM, flags, with_counts=True)
            assert np.array_equal(n.cpu().numpy(), counts) and np.array_equal(bits(out.cpu().numpy()), bits(want)), r
            h = np.float32(r)
            with np.errstate(invalid="ignore"):
                lo, hi = qs - h, qs + h
            _, off, ids = oracle.range_tree(pts, pid, lo, hi, node_dim=dims)[:3]
            got = kdt.kdt_box_search(tree, cu(lo), cu(hi), flags)
            assert np.array_equal(got[0].cpu().numpy(), off) and np.array_equal(got[1].cpu().numpy(), ids), r
        kdt.kdt_status(tree)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("N", [136, 1032, 2055])
def test_slices_of_every_alignment(kdt, N, shift):
    """Slices that start anywhere in the output, with room between them that
    stays untouched, in outputs on and off a 16-byte boundary; with and without
    distances."""
    g, pts, qs = data(N, 3)
    tree = kdt.kdt_build(cu(pts))
    r = radii(N, 3)[2]
    counts, woff, wids, wd2 = oracle.range_tree(pts, oracle.build(pts), qs, radius=r)
    # slice q starts after a gap of 0 to 4 words: its count would not match the next offset,
    # so every query is filled by itself
    dq = cu(qs)
    total = int(woff[-1])
    gap = g.integers(0, 5, len(qs))
    start = woff[:-1] + np.cumsum(gap)
    size = total + int(gap.sum()) + 16
    ids = torch.full((size,), -5, dtype=torch.int32, device="cuda")
    d2 = torch.full((size,), -5.0, device="cuda")
    bare = torch.full((size,), -5, dtype=torch.int32, device="cuda")
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    for q in range(len(qs)):
        off = cu(np.array([start[q], start[q] + counts[q]], dtype=np.int64))
        for out, dist in ((ids, d2), (bare, None)):
            rc = kdt._lib.kdt_radius_fill(tree.handle, ctypes.c_void_p(dq.data_ptr() + 12 * q), 1, ctypes.c_float(r), 0,
                                          ctypes.c_void_p(off.data_ptr()), ctypes.c_void_p(out.data_ptr() + 4 * shift),
                                          ctypes.c_void_p(dist.data_ptr() + 4 * shift) if dist is not None else None,
                                          stream)
            assert rc == 0
        torch.cuda.synchronize()
    kdt.kdt_status(tree)
    want_i, want_d = np.full(size, -5, np.int32), np.full(size, -5, np.float32)
    for q in range(len(qs)):
        at = shift + start[q]
        want_i[at:at + counts[q]] = wids[woff[q]:woff[q + 1]]
        want_d[at:at + counts[q]] = wd2[woff[q]:woff[q + 1]]
    assert np.array_equal(ids.cpu().numpy(), want_i) and np.array_equal(bare.cpu().numpy(), want_i)
    assert np.array_equal(bits(d2.cpu().numpy()), bits(want_d))
