"""The hand-off of the world-aligned pipelined adjoint (one consumer warp, one to three
producers, tapes in turn, segments replayed between two barriers of the producers) and of
the FP64 team rollout, modelled on the CPU: each warp's barrier operations, tape and replay
buffer accesses in the order the kernels issue them, under random interleavings.  Checks:
no deadlock, no second arrival at a barrier before the wait that matches the first, the
consumer finds its step in the tape and nobody writes there meanwhile, and a producer finds
its own segment in the replay buffer.
"""
import random

import pytest


def producer(w, NP, NT, Tn, k, mem):
    j, buf = w - 1, (w - 1) % NT
    for seg in (range((Tn + k - 1) // k - 1, -1, -1) if k > 1 else [0]):
        t0, t1 = (seg * k, min(seg * k + k, Tn)) if k > 1 else (0, Tn)
        mine = False
        if k > 1:
            mine = j == Tn - t1
            if NP > 1:
                yield "all", "producers", NP
            if mine:
                if j >= NT:
                    yield "sync", f"EMPTY{buf}", 2
                assert buf not in mem["reading"]
                mem["tape"][buf] = "scratch"
                assert not mem["at_ring"], "a producer still reads the previous segment"
                mem["ring"] = seg
            if NP > 1:
                yield "all", "producers", NP
        while Tn - 1 - j >= t0:
            if j >= NT and not mine:
                yield "sync", f"EMPTY{buf}", 2
            mine = False
            assert buf not in mem["reading"], "tape overwritten under the consumer"
            if k > 1:
                mem["at_ring"].add(w)
                yield "step", None, 0
                assert mem["ring"] == seg
                mem["at_ring"].discard(w)
            mem["tape"][buf] = j
            yield "arrive", f"FULL{buf}", 2
            buf, j = (buf + NP) % NT, j + NP


def consumer(NT, Tn, mem):
    for j in range(Tn):
        buf = j % NT
        yield "sync", f"FULL{buf}", 2
        assert mem["tape"].get(buf) == j
        mem["reading"].add(buf)
        yield "step", None, 0
        assert mem["tape"][buf] == j
        mem["reading"].discard(buf)
        if j + NT < Tn:
            yield "arrive", f"EMPTY{buf}", 2


def team_inertias(links, steps):
    for _ in range(steps):
        for l in reversed(range(links)):
            yield "arrive", f"LINK{l}", 2
        yield "all", "block", 2


def team_biases(links, steps):
    for _ in range(steps):
        for l in reversed(range(links)):
            yield "sync", f"LINK{l}", 2
        yield "all", "block", 2


def run(warps, seed):
    """A barrier instance completes at its count of warps; `arrive` goes on, `sync` and `all` wait."""
    rnd = random.Random(seed)
    count, waiting, instance = {}, {}, {}
    blocked = {}                                    # warp -> (barrier, instance) it waits for
    pending = dict(enumerate(warps))
    while pending:
        ready = [w for w in pending if w not in blocked or instance.get(blocked[w][0], 0) > blocked[w][1]]
        assert ready, f"deadlock: {blocked}"
        w = rnd.choice(ready)
        blocked.pop(w, None)
        try:
            op, bar, need = next(pending[w])
        except StopIteration:
            del pending[w]
            continue
        if op == "step":
            continue
        if op == "arrive":
            assert (bar, "arrived") not in waiting, f"second arrival at {bar} before the matching wait"
            waiting[(bar, "arrived")] = w
        else:
            blocked[w] = (bar, instance.get(bar, 0))
        count[bar] = count.get(bar, 0) + 1
        if count[bar] == need:
            count[bar] = 0
            waiting.pop((bar, "arrived"), None)
            instance[bar] = instance.get(bar, 0) + 1
    assert not any(count.values()), "an arrival nobody waited for"


@pytest.mark.parametrize("NP", [1, 2, 3])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 7, 40])
def test_adjoint(NP, k):
    NT = NP if NP > 1 else 2
    for Tn in list(range(1, 16)) + [23, 29]:
        for seed in range(40):
            mem = {"tape": {}, "reading": set(), "ring": None, "at_ring": set()}
            run([consumer(NT, Tn, mem)] + [producer(w, NP, NT, Tn, k, mem) for w in range(1, NP + 1)], seed)


@pytest.mark.parametrize("links", [3, 9, 14])
def test_team_rollout(links):
    for steps in (0, 1, 2, 5):
        for seed in range(40):
            run([team_inertias(links, steps), team_biases(links, steps)], seed)


@pytest.mark.parametrize("mistake", ["tapes shared by producers", "no wait before a reused tape"])
def test_the_model_finds_mistakes(mistake):
    def broken(w, mem):
        if mistake == "tapes shared by producers":  # two producers, three tapes
            yield from producer(w, 2, 3, 12, 1, mem)
        else:
            for op in producer(w, 2, 2, 12, 1, mem):
                if op[0] != "sync":
                    yield op
    with pytest.raises((AssertionError, RuntimeError)):
        for seed in range(200):
            mem = {"tape": {}, "reading": set(), "ring": None, "at_ring": set()}
            run([consumer(3 if "shared" in mistake else 2, 12, mem)] + [broken(w, mem) for w in (1, 2)], seed)
