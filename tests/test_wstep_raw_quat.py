"""Free-root kernels on quaternions that are not of unit length, host FP64 build against
the link-frame step, its adjoint and the JVP (tests/wstep_raw_quat.cpp)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_raw_quaternions_match_link_frame(tmp_path):
    """Two formulations of the same step: rounding of 1e-16 amplified by the trees'
    conditioning (a few hundred) over a few thousand operations."""
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "raw_quat"
    subprocess.run([cxx, "-O1", "-std=c++17", "-o", str(exe), os.path.join(HERE, "wstep_raw_quat.cpp")], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rows = [[float(x) for x in line.split()] for line in out.strip().splitlines()]
    assert len(rows) == 10
    for r in rows:
        assert max(r[1:]) < 1e-11, r
