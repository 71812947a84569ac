"""Simulators of different sizes called from two host threads at once, each on its own
stream: a kernel's shared-memory attribute is shared by all of them, and every call
succeeds and gives what it gives alone."""
import ctypes
import os
import shutil
import subprocess

import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_two_threads(tmp_path, precision):
    from paper_2109_07719_gb300 import Simulator, lib
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    so = tmp_path / "two_threads.so"
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread", "-o", str(so),
                    os.path.join(HERE, "two_threads.cpp")], check=True)
    hammer = ctypes.CDLL(str(so)).two_threads
    args, keep = [], []
    for w in (wl.quadruped(B=1, T=1), wl.humanoid(B=1, T=1)):
        sim = Simulator(w.model, precision=precision)
        x = [torch.tensor(v).to(sim.dtype).to(sim.device) for v in (w.q0, w.qd0)]
        x.append(w.tau(T=1)[0].to(sim.dtype).to(sim.device).contiguous())
        alone = sim.step(*x)
        x += [torch.empty_like(y) for y in alone]
        torch.cuda.synchronize()
        stream = torch.cuda.Stream()
        keep.append((sim, x, alone, stream))
        args.append((ctypes.c_void_p * 7)(sim._h.value if hasattr(sim._h, "value") else sim._h,
                                          *[t.data_ptr() for t in x], stream.cuda_stream))
    failed = hammer(ctypes.cast(lib.sim_step_batch, ctypes.c_void_p), args[0], args[1], 4000)
    torch.cuda.synchronize()
    assert failed == 0
    for _, x, alone, _ in keep:
        assert torch.equal(x[3], alone[0]) and torch.equal(x[4], alone[1])
