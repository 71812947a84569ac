"""Launches whose blocks would take the whole of a block's shared memory, at the sizes where
rings, state and stacks add up to it exactly: they run (with fewer tiles, producers or no
look-ahead) and agree with the kernels that keep nothing there."""
import numpy as np
import pytest
import torch

import workloads as wl
from tests._parity import check

pytestmark = pytest.mark.gpu


def _free_chain(n, B, seed=3):
    """A free base with a serial chain of n - 1 revolute links."""
    w = wl.serial_chains(B=B, n=n, T=1, seed=seed)
    m = w.model
    m.joint_type = m.joint_type.copy()
    m.joint_type[m.sys_link_offset[:-1]] = wl.FREE
    q0, qd0, mask = wl._state_arrays(m)
    q0[6] = 1.0
    q0[7:] = 0.3 * w.q0[1:]
    mask[6:] = 1.0
    return wl.Workload(m, q0, qd0, 1, 1.0, seed, "fp64", mask)


def _run(w, precision, threads, space, k, T=3):
    from paper_2109_07719_gb300 import Simulator
    sim = Simulator(w.model, precision=precision)
    sim.set_tape_space(space)
    sim.set_launch(threads)
    q0, qd0 = [torch.tensor(x).to(sim.dtype).to(sim.device) for x in (w.q0, w.qd0)]
    tau = w.tau(T=T).to(sim.dtype).to(sim.device)
    qT, qdT, ck, _ = sim.rollout(q0, qd0, tau, k=k)
    out = {"qT": qT, "qdT": qdT}
    if space == "auto" and threads == 0 or space != "auto":
        out.update(zip(("gq0", "gqd0", "gtau", "gmass"), sim.backward(ck, tau, torch.ones_like(qT), torch.ones_like(qdT), k=k)))
    return {n: x.cpu().numpy() for n, x in out.items()}


# links, free base, precision, threads (0: the default block), checkpoint interval
@pytest.mark.parametrize("n,free,precision,threads,k", [
    (64, False, "fp32", 256, 1), (97, False, "fp32", 256, 1), (64, False, "fp64", 128, 1), (97, False, "fp64", 128, 1),
    (172, True, "fp32", 128, 1), (176, True, "fp64", 0, 1), (164, True, "fp64", 0, 2)])
def test_whole_shared_memory(n, free, precision, threads, k):
    """Ordinary short rollouts: rounding amplified over the chain's n links and 3 steps."""
    w = _free_chain(n, 40) if free else wl.serial_chains(B=40, n=n, T=1)
    a = _run(w, precision, threads, "auto", k)
    b = _run(w, precision, 0, "global", k)
    for name in a:
        check(name, a[name], b[name], 1e-3 if precision == "fp32" else 1e-9)


@pytest.mark.parametrize("precision", ["fp32", "fp32_d64"])
@pytest.mark.parametrize("threads", [288, 416, 512])
def test_large_blocks_of_floating_bases(precision, threads):
    """Block sizes that the kernel's registers or shared memory do not allow run as smaller
    blocks: the same arithmetic, so the same results up to the look-ahead's storage."""
    w = wl.quadruped(B=600, T=3, precision=precision)
    a = _run(w, precision, threads, "auto", 1)
    b = _run(w, precision, 32, "auto", 1)
    for name in a:
        check(name, a[name], b[name], 1e-6)
