"""The implicit-form JVP (FP64 kernels of sim_step_jvp) against the link-frame step on dual
numbers, host FP64 build (tests/wjvp_check.cpp)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = tmp_path_factory.mktemp("j") / "wjvp_check"
    subprocess.run([cxx, "-O1", "-std=c++17", "-o", str(exe), os.path.join(HERE, "wjvp_check.cpp")], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [[float(x) for x in line.split()] for line in out.strip().splitlines()]


@pytest.mark.parametrize("floating", [0, 1])
@pytest.mark.parametrize("links", [1, 2, 3, 5, 8, 11])
def test_implicit_jvp_matches_dual_numbers(rows, floating, links):
    """Rounding of 1e-16 amplified by the trees' conditioning (a few hundred) over a few
    thousand operations; three models of each size, both integrators among them."""
    mine = [r for r in rows if r[0] == floating and r[1] == links]
    assert len(mine) == 3
    for r in mine:
        assert max(r[2:4]) < 1e-11, r
        assert r[4] == 1
