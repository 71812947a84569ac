"""Constrained batches of more tiles than an SM's registers hold at four warps a tile: they
run with two warps or one, give what small batches of the same systems give, and hold only
the contact tapes of the warps they run."""
import numpy as np
import pytest
import torch

import workloads as wl
from tests._parity import check

pytestmark = pytest.mark.gpu


def _run(w, precision, q0):
    from paper_2109_07719_gb300 import Simulator
    sim = Simulator(w.model, precision=precision)
    q = torch.tensor(q0).to(sim.dtype).to(sim.device)
    qd = torch.zeros(sim.nv_max, sim.B, dtype=sim.dtype, device=sim.device)
    qd[5] = -1.0
    tau = torch.zeros(2, sim.nv_max, sim.B, dtype=sim.dtype, device=sim.device)
    qT, qdT, ck, _ = sim.rollout(q, qd, tau, k=1)
    g = sim.backward(ck, tau, torch.ones_like(qT), torch.ones_like(qdT), k=1)
    return [x.cpu().numpy() for x in (qT, qdT) + tuple(g[:3])]


@pytest.mark.parametrize("precision,B", [("fp64", 9760), ("fp64", 19500), ("fp32", 9760)])
def test_fewer_warps_same_results(precision, B):
    """Two steps with all feet in the ground; the partial sums of the test passes' reverse are
    added in another order: a few roundings, amplified by the solve's conditioning."""
    w = wl.quadruped(B=B, T=1, precision=precision, contacts=True)
    w.q0[7:] *= 0.1
    w.q0[2] = 0.415
    big = _run(w, precision, w.q0)
    pick = np.r_[0:40, B - 8:B]
    w.model = w.model.subset(pick)
    small = _run(w, precision, np.ascontiguousarray(w.q0[:, pick]))
    for name, a, b in zip(("qT", "qdT", "gq0", "gqd0", "gtau"), big, small):
        check(name, a[..., pick], b, 1e-10 if precision == "fp64" else 1e-3)


def test_large_batch_holds_one_contact_tape():
    """119 + 71 words of tapes a link, 245 of one contact tape, 36 of constants and maps, 2878
    words of contact record and 4 more a system."""
    from paper_2109_07719_gb300 import Simulator
    B, n = 20000, 13
    sim = Simulator(wl.quadruped(B=B, T=1, contacts=True).model, precision="fp32")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    del sim
    held = torch.cuda.mem_get_info()[0] - before
    assert held < 4 * B * ((119 + 71 + 245 + 36) * n + 2882) + (32 << 20)
