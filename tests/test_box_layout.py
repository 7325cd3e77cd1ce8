"""Index identities of the box tree (csrc/kdt_box.cuh), by enumeration on the CPU.

Buckets are the subtrees of the nodes on level LB = max(H - 3, 0); bucket i
holds one group of eight places (two for the first `big` buckets), group
i + min(i, big).  Every node above the buckets is handed down beside its own
splitting plane, one to a bucket.  The record of node v (counted from 1, the
bucket i is 2^LB + i) holds its four grandchildren 4v .. 4v + 3; with LB odd
the record of the root is v = 0 with children 2 and 3.
"""
import numpy as np
import pytest


def shape(n):
    H = n.bit_length() - 1
    M = n - ((1 << H) - 1)
    LB = H - 3 if H > 3 else 0
    return H, LB, 1 << LB, (M + 7) // 8 if H >= 3 else 0


def bucket_places(n, i):
    """(place, node) of the bucket's own nodes, place counted over its groups."""
    _, LB, _, big = shape(n)
    root = (1 << LB) - 1 + i
    for k in range(2 if i < big else 1):
        for m in range(8):
            if k == 0 and m == 7:
                continue  # the one handed down
            up = 3 if k else (0 if m < 1 else (1 if m < 3 else 2))
            node = ((root + 1) << up) - 1 + (m if k else m + 1 - (1 << up))
            if node < n:
                yield 8 * (i + min(i, big) + k) + m, node


@pytest.mark.parametrize("n", list(range(1, 300)) + [511, 512, 513, 1023, 1024, 1031, 1032, 1033, 2047, 4100, 5000])
def test_every_node_has_one_place(n):
    H, LB, buckets, big = shape(n)
    places = 8 * (buckets + big)
    seen, used = [], []
    for i in range(buckets):
        for p, node in bucket_places(n, i):
            assert 0 <= p < places
            used.append(p)
            seen.append(node)
    upper = (1 << LB) - 1
    assert len(set(used)) == len(used)
    assert sorted(seen) == list(range(upper, n))


@pytest.mark.parametrize("n", [16, 17, 40, 64, 200, 1000, 5000])
def test_every_upper_node_is_handed_to_one_bucket(n):
    """The walk of a bucket, with random sides for 'the point from above lies
    right of this node's plane': each upper node reaches exactly one bucket."""
    _, LB, buckets, _ = shape(n)
    g = np.random.default_rng(n)
    side = {}
    got = []
    for i in range(buckets):
        hand = None
        for l in range(LB):
            t = ((buckets + i) >> (LB - l)) - 1
            right = bool(i >> (LB - l - 1) & 1)
            to_right = hand is not None and side.setdefault((hand, t), bool(g.integers(2)))
            if hand is None or to_right != right:
                if hand is not None or not right:
                    hand = t
        if hand is not None:
            got.append(hand)
    assert sorted(got) == list(range(buckets - 1))


@pytest.mark.parametrize("LB", range(0, 13))
def test_records_reach_every_bucket(LB):
    leaf = 1 << LB
    records = leaf // 2 if LB else 0
    odd = LB % 2 == 1
    todo = [(0 if odd else 1, 12 if odd else 15)]
    found = []
    while todo:
        v, mask = todo.pop()
        if v >= leaf:
            found.append(v - leaf)
            continue
        assert v < records
        for c in range(4):
            if mask >> c & 1:
                child = 4 * v + c
                assert child >> 2 == v
                todo.append((child, 15))
    assert sorted(found) == list(range(leaf))


@pytest.mark.parametrize("LB", range(0, 15))
def test_box_build_writes_every_record(LB):
    """Launches of the box build: the leaf kernel over 2^LB nodes, then levels
    LB - 10, LB - 20, ...; each block of 256 writes its nodes' boxes and those
    of the nodes 2, 4, 6 and 8 levels up as far as it holds four of each."""
    written = set()

    def blocks(level):
        n = 1 << level
        for first in range(0, n, 256):
            v, count = n + first, min(256, n - first)
            while True:
                for t in range(count):
                    if v + t > 1:
                        assert (v + t) not in written
                        written.add(v + t)
                if count < 4:
                    break
                count >>= 2
                assert v % 4 == 0
                v //= 4

    if LB:
        blocks(LB)
        level = LB - 10
        while level >= 1:
            for v in range(1 << level, 2 << level):
                assert all(4 * v + c in written for c in range(4))  # its record is complete
            blocks(level)
            level -= 10
    want = set()
    level = LB
    while level >= 1:
        want |= set(range(1 << level, 2 << level))
        level -= 2
    assert written == want
