"""The order the library stores links in (host build, tests/tree_order_check.cpp)."""
import math
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_small_subtrees_first_bounds_the_stack(tmp_path):
    """A stack entry is held while all children but the largest are walked, so each entry
    halves what is left: at most log2(links) of them."""
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "tree_order_check"
    subprocess.run([cxx, "-O1", "-std=c++17", "-o", str(exe), os.path.join(HERE, "tree_order_check.cpp")], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rows = [[int(x) for x in line.split()] for line in out.strip().splitlines()]
    assert len(rows) == 8 * 25
    for n, depth, ok in rows:
        assert ok == 1
        assert depth <= math.log2(n + 1), (n, depth)
    assert max(depth for _, depth, _ in rows) >= 6
