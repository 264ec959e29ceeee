"""The order in which a worker takes the tiles claimed for it (csrc/pick.cuh, compiled for the host).

A tile may be claimed before its predecessors have finished; it then waits for tiles claimed earlier, possibly for one that
its own worker still holds.  A small model of the workers (one held tile and one priority tile each, as in the kernel) shows
that no such wait can become a cycle."""
import ctypes as C
import os
import random
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
WRAP = 1 << 32


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    out = tmp_path_factory.mktemp("order") / "liborder_host.so"
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-x", "c++", os.path.join(HERE, "pick_host_shim.cc"), "-o", str(out)],
                   check=True)
    fn = C.CDLL(str(out)).priority_goes_first_host
    fn.argtypes = [C.c_int, C.c_uint, C.c_uint]
    fn.restype = C.c_int
    return lambda early, head, at: bool(fn(int(early), head % WRAP, at % WRAP))


class Worker:
    def __init__(self, first):
        self.running, self.held, self.prio, self.head, self.tail = None, [], [], first, first


def unfinished(rule, rnd, n_workers, n_tiles):
    """Claims and runs tiles in a random interleaving; returns the tiles that never finish.

    A tile is (index, indexes of earlier-claimed tiles it waits for); without the latter it was queued after its release."""
    ws = [Worker(WRAP - 2) for _ in range(n_workers)]             # (the counters wrap during the run)
    done, claimed = set(), 0
    while True:
        steps = []
        for w in ws:
            if claimed < n_tiles and not w.held:
                steps.append(("held", w))
            if claimed < n_tiles and w.running is not None and not w.prio:
                steps.append(("prio", w))
            if w.running is None and (w.held or w.prio):
                steps.append(("take", w))
            if w.running is not None and w.running[1] <= done:
                steps.append(("end", w))
        if not steps:
            return n_tiles - len(done)
        what, w = rnd.choice(steps)
        if what in ("held", "prio"):
            waits = {rnd.randrange(claimed) for _ in range(rnd.randint(1, 3))} if claimed and rnd.random() < 0.5 else set()
            if what == "held":
                w.held.append((claimed, waits, 0))
                w.tail += 1
            else:
                w.prio.append((claimed, waits, w.tail))
            claimed += 1
        elif what == "take":
            p = w.prio[0] if w.prio else None
            if p and (rule(bool(p[1]), w.head, p[2]) or p[1] <= done):
                w.running = w.prio.pop()
            elif w.held:
                w.running = w.held.pop()
                w.head += 1
            else:
                return n_tiles - len(done)                        # a worker that refuses the only tile it has
        else:
            done.add(w.running[0])
            w.running = None


def test_held_predecessor_goes_before_the_priority_tile_that_waits_for_it(rule):
    assert not rule(True, 7, 8)              # one tile was held when the early tile was claimed, and still is
    assert rule(True, 8, 8)                  # it has been taken since
    assert rule(True, 9, 8)
    assert rule(False, 7, 8)                 # a released tile need not wait for anything
    assert not rule(True, WRAP - 1, 0) and rule(True, 0, WRAP - 1)


@pytest.mark.parametrize("n_workers", [1, 2, 6])
def test_every_claimed_tile_finishes(rule, n_workers):
    for seed in range(200):
        assert unfinished(rule, random.Random(seed), n_workers, 60) == 0, seed


def test_the_model_shows_the_cycle_when_priority_always_wins():
    assert any(unfinished(lambda early, head, at: True, random.Random(seed), 2, 60) for seed in range(200))
