"""Calls on different objects from two host threads at once: a launch's
shared-memory limit belongs to the kernel, so a call that sets its own lower
one makes another's launch fail."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2210_12859_gb300 import build

    lib = build.build_library()
    exe = str(tmp_path_factory.mktemp("probe") / "threads_probe")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe,
                    os.path.join(ROOT, "tests", "host", "threads_probe.cu"), lib,
                    "-Xlinker", "-rpath," + os.path.dirname(lib)], check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("what,n,calls", [("builds", 3001, 20000), ("builds", (1 << 18) + 77, 1000),
                                            ("lists", 500, 20000)])
def test_two_threads(probe, what, n, calls):
    """Builds in one and in eight dimensions, of both block sizes; unordered
    queries whose heaps (k = 50 and 64) exceed the default limit."""
    r = subprocess.run([probe, what, str(n), str(calls)], capture_output=True, text=True, timeout=120, check=True)
    assert r.stdout.split(" ", 1)[0] == "0", r.stdout
