"""Launch variants of the world-aligned kernels that small models do not reach by themselves
(deep stacks on chip and in global memory, one and two producers, replayed segments of free
bases, the FP64 team rollout) against the one-warp link-frame kernels, in FP64."""
import numpy as np
import pytest
import torch

import workloads as wl
from tests._parity import check

pytestmark = pytest.mark.gpu
NAMES = ("qT", "qdT", "traj", "gq0", "gqd0", "gtau", "gmass")


def _trees(shapes, seed=4, precision="fp64"):
    """Revolute trees of the given parent lists with the workloads' random parameters."""
    parents = np.concatenate([np.asarray(s) for s in shapes])
    counts = [len(s) for s in shapes]
    first = np.zeros(len(parents), bool)
    first[np.cumsum([0] + counts[:-1])] = True
    rng = np.random.default_rng(seed)
    axis, r, mass, com, Ic = wl._random_tree_params(rng, parents, first)
    m = wl._assemble(counts, parents, np.zeros(len(parents)), axis, r, mass, com, Ic, 1e-3, (0.0, 0.0, -9.81), "trees")
    q0, qd0, mask = wl._state_arrays(m)
    q0[:] = rng.uniform(-1, 1, q0.shape) * (np.arange(m.nq_max)[:, None] < m.nq_per_system()[None, :])
    mask[:] = np.arange(m.nv_max)[:, None] < m.nv_per_system()[None, :]
    return wl.Workload(m, q0, qd0, 1, 1.0, seed, precision, mask)


def _run(w, space="auto", k=1, T=5, persistent=False, integrator="semi", ahead=2):
    from paper_2109_07719_gb300 import Simulator
    sim = Simulator(w.model, precision="fp64", integrator=integrator)
    sim.set_tape_space(space)
    sim.set_launch(0, persistent)
    sim.set_prefetch(ahead)
    q0, qd0 = [torch.tensor(x).to(sim.device) for x in (w.q0, w.qd0)]
    tau = w.tau(T=max(T, 1)).to(sim.device)[:T].contiguous()
    qT, qdT, ck, traj = sim.rollout(q0, qd0, tau, k=k, traj=True)
    g = torch.Generator().manual_seed(8)
    gx = torch.randn(traj.shape, generator=g, dtype=torch.float64).to(sim.device)
    out = (qT, qdT, traj) + tuple(sim.backward(ck, tau, torch.ones_like(qT), torch.ones_like(qdT), k=k, g_traj=gx))
    assert sim.status().sum() == 0
    return [x.cpu().numpy() for x in out], sim.last_storage()


def _agree(w, k=1, T=5, persistent=False, integrator="semi", ahead=2):
    """Rounding of 1e-16 amplified over the links and steps: 1e-10 for states, 1e-9 for gradients."""
    a, storage = _run(w, "auto", k, T, persistent, integrator, ahead)
    b, _ = _run(w, "one_warp", k, T, False, integrator)
    for name, x, y in zip(NAMES, a, b):
        if x.size:
            check(name, x, y, 1e-10 if name in NAMES[:3] else 1e-9)
    return storage


@pytest.mark.parametrize("levels", [3, 6])   # 3: stacks in shared memory, 6: in global memory (four of 6 entries)
@pytest.mark.parametrize("k", [1, 3])
def test_complete_binary_trees(levels, k):
    n = 2 ** levels - 1
    w = _trees([[(i - 1) // 2 for i in range(n)]] * 40)
    assert _agree(w, k)[1].startswith("aligned_pipelined")


@pytest.mark.parametrize("family", ["quadruped", "humanoid"])
@pytest.mark.parametrize("k", [2, 5])
def test_free_bases_replay(family, k):
    w = getattr(wl, family)(B=37, T=1, precision="fp64")
    assert _agree(w, k, T=7)[1] == "floating_pipelined_global"


@pytest.mark.parametrize("links,storage", [(3, "aligned_pipelined_shared"), (5, "aligned_pipelined_global"),
                                           (0, "floating_pipelined_global")])
@pytest.mark.parametrize("k", [1, 2])
def test_more_tiles_than_sms(links, storage, k):
    """Two producers (on chip while all tiles run at once) and one (global tapes)."""
    w = wl.serial_chains(B=6000, n=links, T=1) if links else wl.quadruped(B=6000, T=1)
    assert _agree(w, k)[1] == storage


@pytest.mark.parametrize("B", [10000, 26000])
def test_many_fp64_trees(B):
    """Stacks in global memory and (26000) no look-ahead, so that four blocks fit an SM."""
    w = _trees([[(i - 1) // 2 for i in range(63)]] * 8)
    w.model = w.model.subset(np.arange(B) % 8)
    w.q0, w.qd0, w.tau_mask = [np.ascontiguousarray(x[:, np.arange(B) % 8]) for x in (w.q0, w.qd0, w.tau_mask)]
    w.tau_sigma = 0.0
    big, _ = _run(w, T=2)
    w8 = _trees([[(i - 1) // 2 for i in range(63)]] * 8)
    w8.tau_sigma = 0.0
    small, _ = _run(w8, T=2)
    check("qT", big[0][:, -8:], small[0][:, (np.arange(B) % 8)[-8:]], 1e-12)
    check("qdT", big[1][:, -8:], small[1][:, (np.arange(B) % 8)[-8:]], 1e-12)


@pytest.mark.parametrize("n", [3, 9, 10, 14])    # 9: the longest whose tile fits a block
@pytest.mark.parametrize("T", [0, 1, 2, 5])
def test_fp64_chain_rollouts(n, T):
    storage = _agree(wl.serial_chains(B=37, n=n, T=1, precision="fp64"), T=T)
    assert storage[0] == ("pipelined_team" if n <= 9 else "global")


def test_three_link_chains_of_many_tiles():
    """The pipelined rollout where the team's blocks would run in turns."""
    assert _agree(wl.serial_chains(B=10000, n=3, T=1, precision="fp64"), T=2)[0] == "pipelined"


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("integrator", ["semi", "explicit"])
def test_fp64_chains_of_mixed_lengths(persistent, integrator):
    w = _trees([list(range(-1, 2 + i % 7)) for i in range(5000)])   # 3 to 9 links
    w.model = w.model.with_damping(3)
    assert _agree(w, 2, 3, persistent, integrator)[0] == "pipelined_team"


@pytest.mark.parametrize("k", [1, 2])
@pytest.mark.parametrize("free", [False, True])
def test_records_staged_without_look_ahead(free, k):
    """One ring slot: every link waits for its own record."""
    w = wl.humanoid(B=37, T=1) if free else _trees([[(i - 1) // 2 for i in range(40)]] * 37)
    _agree(w, k, ahead=0)
