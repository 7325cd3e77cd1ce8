"""The box tree's shape and places as csrc/kdt_box.cuh computes them (a host
probe compiled from that header), against an enumeration of the tree: every
node on or below the buckets' level has one place, no place has two nodes, and
the counts of buckets, groups and records are those of the enumeration, also at
the size limit."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROBE_SRC = os.path.join(ROOT, "tests", "host", "box_probe.cu")

pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                                reason="needs nvcc")


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path_factory.mktemp("probe") / "box_probe")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe, PROBE_SRC],
                   check=True, capture_output=True)

    def run(lines):
        r = subprocess.run([exe], input="\n".join(lines) + "\n", capture_output=True, text=True, check=True)
        return [[int(x) for x in line.split()] for line in r.stdout.split("\n")[: len(lines)]]

    return run


def shape(n):
    """Levels above the buckets, buckets, buckets with nodes on the last level, records, groups."""
    H = n.bit_length() - 1
    LB = max(H - 3, 0)
    last = n - ((1 << H) - 1)
    big = sum(1 for b in range(1 << LB) if H >= 3 and 8 * b < last) if LB < 12 else -(-last // 8)
    # records: one for every node v >= 1 on the levels LB - 2, LB - 4, ... and v = 0 for odd LB
    top = [v for level in range(LB - 2, -1, -2) for v in ((1 << level), (2 << level) - 1)]
    records = max(top) + 1 if top else (1 if LB == 1 else 0)
    return [LB, 1 << LB, big, records, (1 << LB) + big]


def test_shapes(probe):
    sizes = list(range(1, 3000)) + [2 ** e + d for e in range(12, 30) for d in (-1, 0, 1, 7, 8, 9)] + [2 ** 30 - 1]
    sizes = [n for n in sizes if n < 2 ** 30]
    for n, got in zip(sizes, probe([f"s {n}" for n in sizes])):
        assert got == shape(n), n


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 14, 15, 16, 17, 31, 32, 40, 63, 64, 65, 127, 128, 135, 136, 137, 500,
                               1023, 1024, 1032, 4099, 20000])
def test_every_node_has_one_place(probe, n):
    LB, buckets, _, _, groups = shape(n)
    places = {}
    for i, row in enumerate(probe([f"b {n} {i}" for i in range(buckets)])):
        first, count, nodes = row[0], row[1], row[2:]
        assert len(nodes) == 8 * count
        for p, node in enumerate(nodes):
            if p == 7 or node >= n:  # the point from above; empty
                continue
            at = 8 * first + p
            assert at < 8 * groups and at not in places
            places[at] = node
            up = node + 1
            while up >= 2 * buckets:
                up //= 2
            assert up == buckets + i  # the bucket's own subtree
    assert sorted(places.values()) == list(range(buckets - 1, n))
