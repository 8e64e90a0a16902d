"""The partition of the double-layer sums on the CPU: built on threads (the root's quarters) and on
one thread it is the same, and every node reaches every point once."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("dlp") / "dlp_tree_harness")
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", os.path.join(ROOT, "tests", "dlp_tree_harness.cpp"),
                    "-o", exe], check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("free", [0, 1])
@pytest.mark.parametrize("n,m,nodes", [(64, 64, 100), (100, 60, 64), (160, 144, 1600), (200, 200, 4000),
                                       (256, 512, 777), (600, 300, 600)])
def test_the_same_with_threads(harness, n, m, nodes, free):
    out = subprocess.run([harness, str(n), str(m), str(nodes), str(free)], check=True, capture_output=True).stdout
    same, covered, boxes, leaves, points = (int(v) for v in out.split())
    assert same and covered and leaves >= 1 and points > 0
