"""The constraint sweeps visit their rows in the model's link order (fixed sweeps from zero
impulses do not converge, so the order is part of the result), whatever order the library
stores the links in: models whose larger subtrees are numbered first, models not numbered
depth-first, and joint limits on unequal limbs, through the C ABI against the FP64 oracle."""
import numpy as np
import pytest
import torch

import workloads as wl
from oracle.contact import contact_points, limit_gaps
from oracle.dynamics import OracleModel
from tests._parity import check, mass_grad_of, oracle_backward, oracle_forward

pytestmark = pytest.mark.gpu


def _legged(front, hind, breadth_first, seed=5, B=34):
    """Quadrupeds whose two front legs have `front` links and whose hind legs have `hind`,
    a foot sphere on each leg's last link; legs numbered front first, leg by leg or (breadth
    first) level by level."""
    rng = np.random.default_rng(seed)
    legs = [(sx, sy, front if sx > 0 else hind) for sx in (1, -1) for sy in (1, -1)]
    place = [(i, j) for i, leg in enumerate(legs) for j in range(leg[2])]
    if breadth_first:
        place.sort(key=lambda ij: (ij[1], ij[0]))
    number = {ij: 1 + n for n, ij in enumerate(place)}
    nl = 1 + len(place)
    par, ax, r, com, foot = [-1], [(0, 0, 0)], [(0, 0, 0)], [(0, 0, 0)], [False]
    for i, j in place:
        sx, sy, n = legs[i]
        par.append(number[(i, j - 1)] if j else 0)
        ax.append((1, 0, 0) if j == 0 else (0, 1, 0))
        r.append((sx * 0.25, sy * 0.15, 0) if j == 0 else (0, 0, 0) if j == 1 else (0, 0, -0.4 / (n - 1)))
        com.append((0, 0, -0.05 * (j > 0)))
        foot.append(j == n - 1)
    mass = rng.uniform(0.5, 1.5, (B, nl))
    mass[:, 0] = 10.0
    Ic = wl._random_inertias(rng, B * nl, 0.001, 0.01).reshape(B, nl, 6)
    Ic[:, 0] = (0.09, 0.23, 0.28, 0, 0, 0)
    m = wl._assemble([nl] * B, par * B, ([wl.FREE] + [wl.REVOLUTE] * (nl - 1)) * B, ax * B, r * B, mass.reshape(-1),
                     com * B, Ic.reshape(-1, 6), 5e-4, (0.0, 0.0, -9.81), "legged")
    ct = np.full((nl, 4), -1.0)
    for l in range(nl):
        if foot[l]:
            n = front if r[l] == (0, 0, -0.4 / (front - 1)) else hind
            ct[l] = (0.0, 0.0, -0.4 / (n - 1), 0.02)
    m.contact = np.tile(ct, (B, 1))
    q0, qd0, _ = wl._state_arrays(m)
    q0[6] = 1.0
    q0[7:] = rng.uniform(-0.05, 0.05, q0[7:].shape)
    om = OracleModel(m, list(range(B)))
    _, phi = contact_points(om, torch.tensor(q0.T))
    q0[2] -= phi.max(1).values.numpy() + 0.002          # every foot in the ground
    qd0[:] = rng.uniform(-0.3, 0.3, qd0.shape)
    qd0[5] = -1.0
    assert bool((contact_points(om, torch.tensor(q0.T))[1] < 0).all())
    return m, q0, qd0


def _limited(m, q0, qd0):
    """Every joint limited so tightly that most are past a limit."""
    m = m.with_limits(-0.02, 0.02)
    assert float((limit_gaps(OracleModel(m, list(range(m.n_systems))), torch.tensor(q0.T))[1] < 0).double().mean()) > 0.3
    return m, q0, qd0


def _limited_humanoid(B=20):
    w = wl.humanoid(B=B, T=1, seed=77)
    m = w.model.with_limits(-0.04, 0.04, every=2)
    rng = np.random.default_rng(3)
    qd0 = rng.uniform(-1, 1, w.qd0.shape)
    _, phi = limit_gaps(OracleModel(m, list(range(B))), torch.tensor(w.q0.T))
    assert float((phi < 0).double().mean()) > 0.3
    return m, w.q0, qd0


CASES = {
    "larger_legs_first": lambda: _legged(4, 3, False),
    "breadth_first": lambda: _limited(*_legged(3, 3, True)),
    "breadth_first_unequal": lambda: _legged(4, 3, True),
    "humanoid_limits": _limited_humanoid,
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_rows_in_link_order_fp64(name):
    from paper_2109_07719_gb300 import Simulator
    m, q0, qd0 = CASES[name]()
    B, T = m.n_systems, 4
    rng = np.random.default_rng(9)
    tau = rng.standard_normal((T, m.nv_max, B))
    tau[:, :6] = 0.0
    sim = Simulator(m, precision="fp64")
    dq, dqd, dtau = [torch.tensor(x).to(sim.device) for x in (q0, qd0, tau)]
    qT, qdT, ck, _ = sim.rollout(dq, dqd, dtau, k=1)
    gq, gqd = rng.standard_normal(q0.shape), rng.standard_normal(qd0.shape)
    g = sim.backward(ck, dtau, torch.tensor(gq).to(sim.device), torch.tensor(gqd).to(sim.device), k=1)
    systems = list(range(B))
    oq, oqd = oracle_forward(m, systems, q0, qd0, tau)
    check("qT", qT.cpu().numpy(), oq, 1e-8)
    check("qdT", qdT.cpu().numpy(), oqd, 1e-8)
    sel = [0, 7, B - 1]
    o = oracle_backward(m, sel, q0, qd0, tau, gq, gqd)
    for key, mine in zip(("gq0", "gqd0", "gtau"), g):
        check(key, mine.cpu().numpy()[..., sel], o[key], 1e-6)
    gm = mass_grad_of(m, g[3].cpu().numpy(), sel)
    check("gmass", np.concatenate([gm[s] for s in sel]), np.concatenate([o["gm"][s] for s in sel]), 1e-6)
