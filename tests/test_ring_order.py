"""The order in which the cluster kernel's producer and its three groups of consumer warps walk their ring of stages (Section 2.1).

A model of the slots' barriers, one parity bit each: copies land in any order, and whenever a consumer's wait passes, its own stage must
have landed and must not have been overwritten.  The walk itself is the kernel's (lqer_ring.h, compiled for the host).
"""
import ctypes as C
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_02446_b200", "csrc")
PHASES = 3
SOURCE = """
#include "lqer_ring.h"
using namespace lqer;
extern "C" void consumer(int phase, int slots, int n, int* slot, int* parity) {
  RingCursor c(phase);
  for (int i = 0; i < n; ++i) { slot[i] = c.slot; parity[i] = c.parity; c.next(3, slots); }
}
extern "C" void producer(int first, int slots, int n, int* slot, int* parity) {
  RingWalk<3> w(first);
  for (int i = 0; i < n; ++i) { slot[i] = w.turn[0].slot; parity[i] = w.turn[0].parity; w.next(slots); }
}
"""


@pytest.fixture(scope="module")
def ring(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    (d / "ring.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "ring.cpp"), "-o", str(d / "ring.so")], check=True)
    return C.CDLL(str(d / "ring.so"))


def _walk(fn, a, slots, n):
    s, q = (C.c_int * n)(), (C.c_int * n)()
    fn(a, slots, n, s, q)
    return list(zip(s, q))


def _kernel_order(ring, slots, stages):
    fill = [(x, 0) for x in range(min(slots, stages))] + _walk(ring.producer, slots, slots, max(stages - slots, 0))
    take = [None] * stages
    for f in range(PHASES):
        for i, at in enumerate(_walk(ring.consumer, f, slots, (stages - f + PHASES - 1) // PHASES)):
            take[f + PHASES * i] = at
    return fill, take


def _shared_order(slots, stages):
    """All phases in one ring: what the model has to find fault with."""
    at = [(x % slots, (x // slots) & 1) for x in range(stages)]
    return at[:slots] + [(s, q ^ 1) for s, q in at[slots:]], at


def _runs(fill, take, slots, stages, rng):
    """One schedule drawn by rng.  True if every consumer met its own stage and all of them were taken."""
    full, empty, holds = [0] * slots, [0] * slots, [None] * slots    # passes completed; the stage that lies in the slot
    issued, flying, at = 0, [], [f for f in range(PHASES)]
    slow = rng.randrange(stages)                                    # this stage lands when nothing else can go on
    while True:
        moves = []
        if issued < stages:
            s, parity = fill[issued]
            if issued < slots or (empty[s] & 1) != parity:
                moves.append(("issue", s))
        moves += [("land", x) for x in flying if x != slow]
        for f in range(PHASES):
            if at[f] < stages and (full[take[at[f]][0]] & 1) != take[at[f]][1]:
                moves.append(("take", f))
        if not moves:
            if slow in flying:
                moves.append(("land", slow))
            else:
                return issued == stages and all(x >= stages for x in at)
        what, v = rng.choice(moves)
        if what == "issue":
            flying.append(issued)
            issued += 1
        elif what == "land":
            flying.remove(v)
            s = fill[v][0]
            holds[s] = v
            full[s] += 1
        else:
            s = take[at[v]][0]
            if holds[s] != at[v]:
                return False
            empty[s] += 1
            at[v] += PHASES


@pytest.mark.parametrize("slots", range(PHASES, 21))
def test_every_consumer_meets_its_own_stage(ring, slots):
    rng = random.Random(slots)
    for stages in (slots, slots + 1, 2 * slots + 2, 5 * slots + 1):
        fill, take = _kernel_order(ring, slots, stages)
        assert [s for s, _ in fill] == [s for s, _ in take]
        for _ in range(60):
            assert _runs(fill, take, slots, stages, rng)


def test_the_model_finds_a_shared_ring_at_fault():
    for slots in (4, 5, 10, 11, 17):
        rng = random.Random(slots)
        assert not all(_runs(*_shared_order(slots, 4 * slots), slots, 4 * slots, rng) for _ in range(400)), slots
    rng = random.Random(1)
    assert all(_runs(*_shared_order(9, 36), 9, 36, rng) for _ in range(200))      # (whole rounds of the phases are in order)
