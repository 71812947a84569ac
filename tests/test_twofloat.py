"""The float pairs the FP32 + FP64 D-solve mode computes its D-solves in (host build)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_float_pairs_keep_44_bits(tmp_path):
    """Each pair operation within 2^-44 of exact relative to its largest term (the published
    bounds are a few 2^-48); the free root's solve, rounded to float, within one float ulp of
    double's (2^-23); infinities and NaN come out as plain subtraction gives them."""
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "twofloat"
    subprocess.run([cxx, "-O1", "-std=c++17", "-o", str(exe), os.path.join(HERE, "twofloat_check.cpp")], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    res = {line.split()[0]: float(line.split()[1]) for line in out.strip().splitlines()}
    for name in ("reciprocal", "sqrt", "product", "sum", "minus_product"):
        assert res[name] < 2.0 ** -44, (name, res[name])
    assert res["solve"] < 2.0 ** -23
    assert res["special"] == 1
