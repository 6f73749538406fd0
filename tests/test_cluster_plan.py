"""How a launch of the cluster kernel (3 to 16 rows, Section 2.1) is cut, and what a thread remembers of it: the planner is plain C++, compiled here
for the host with the device's answers made up."""
import ctypes as C
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_02446_b200", "csrc")
SOURCE = """
#include "lqer_cluster_plan.h"
using namespace lqer::dcl;
static Shape shape(int n, int M, int w_bits, const int* k, const int* t, const int* r) {
  Shape s = {};
  s.n = n; s.M = M; s.w_bits = w_bits;
  for (int i = 0; i < n; ++i) { s.k_slabs[i] = k[i]; s.tiles[i] = t[i]; s.r_blocks[i] = r[i]; }
  return s;
}
static int index_of(int CS) { return CS == 8 ? 3 : CS == 4 ? 2 : CS == 2 ? 1 : 0; }
extern "C" {
int asked = 0;
// places: for clusters of 1, 2, 4, 8.  out: CS, steps_max, slots, smem, total, then clusters, t_blocks, t_clusters, t_tiles of each layer
int make(int n, int M, int w_bits, const int* k, const int* t, const int* r, const int* places, int* out) {
  Plan q;
  bool sure;
  if (!make_plan(shape(n, M, w_bits, k, t, r), [&](int CS) { return places[index_of(CS)]; }, q, sure)) return 0;
  out[0] = q.CS; out[1] = q.steps_max; out[2] = q.slots; out[3] = (int)q.smem; out[4] = q.total;
  for (int i = 0; i < n; ++i) { int* o = out + 5 + 4 * i; o[0] = q.clusters[i]; o[1] = q.t_blocks[i]; o[2] = q.t_clusters[i]; o[3] = q.t_tiles[i]; }
  return 1;
}
void* cache_new() { return new PlanCache; }
void cache_free(void* c) { delete static_cast<PlanCache*>(c); }
// the cluster size, or 0
int cache_find(void* c, int n, int M, int w_bits, const int* k, const int* t, const int* r, const int* places) {
  Plan q;
  return static_cast<PlanCache*>(c)->find(shape(n, M, w_bits, k, t, r), [&](int CS) { ++asked; return places[index_of(CS)]; }, q) ? q.CS : 0;
}
int limit(int what) { return what == 0 ? kSmemMax : what == 1 ? kMaxSlots : kPhases; }
}
"""
PLACES = (148, 70, 33, 16)


@pytest.fixture(scope="module")
def planner(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "plan.cpp"), "-o", str(d / "plan.so")], check=True)
    lib = C.CDLL(str(d / "plan.so"))
    lib.cache_new.restype = C.c_void_p
    lib.cache_free.argtypes = [C.c_void_p]
    lib.cache_find.argtypes = [C.c_void_p, C.c_int, C.c_int, C.c_int] + 4 * [C.POINTER(C.c_int)]
    return lib


def _ints(v):
    return (C.c_int * len(v))(*v)


def _shapes(count):
    rng = random.Random(11)
    for _ in range(count):
        n = rng.randint(1, 4)
        k = [rng.randint(1, rng.choice((40, 220))) for _ in range(n)]
        if rng.random() < 0.5:
            k = [k[0]] * n
        yield (n, rng.randint(3, 16), rng.choice((4, 4, 2)), k, [rng.randint(1, rng.choice((40, 170))) for _ in range(n)],
               [rng.choice((0, 1, 2, 4, 16, rng.randint(0, 16))) for _ in range(n)])


def _one_by_one(tiles, steps, places):
    """Every layer one cluster; the others one after the other where the time is longest, as long as every cluster keeps a tile."""
    c = [1] * len(tiles)
    while sum(c) < places:
        length = [t / x * s if x < t else 0.0 for t, x, s in zip(tiles, c, steps)]
        if max(length) == 0.0:
            break
        c[length.index(max(length))] += 1
    return c


@pytest.mark.parametrize("places", [PLACES, (132, 66, 30, 14), (148, -1, 4, 0), (20, 9, 4, -1)])
def test_every_tile_has_a_cluster_and_the_ring_its_slots(planner, places):
    smem_max, slots_max, phases = (planner.limit(i) for i in range(3))
    found = 0
    for n, M, w_bits, k, t, r in _shapes(1500):
        out = (C.c_int * 21)()
        if not planner.make(n, M, w_bits, _ints(k), _ints(t), _ints(r), _ints(places), out):
            continue
        found += 1
        CS, steps_max, slots, smem, total = out[:5]
        clusters, t_blocks, t_clusters, t_tiles = (list(out[5 + j:5 + 4 * n:4]) for j in range(4))
        assert total == sum(clusters) <= places[{1: 0, 2: 1, 4: 2, 8: 3}[CS]]
        steps = [((x + CS - 1) // CS + 1) // 2 for x in k]
        assert steps_max == max(steps) and clusters == _one_by_one(t, steps, total)
        for i in range(n):
            rest, others = t[i] - t_clusters[i] * t_tiles[i], clusters[i] - t_clusters[i]
            assert others >= 1 and rest >= others and (t_tiles[i] >= 1 or t_clusters[i] == 0)     # a tile each at least
            assert t_blocks[i] * clusters[i] >= r[i]                                              # the ranks have clusters that form them
        # a slot for each group of consumers, or one for every stage that any CTA has
        assert smem <= smem_max and 1 <= slots <= slots_max
        assert slots >= phases or slots >= max(t) * steps_max
    assert found > 100


def test_what_could_not_be_asked_is_not_remembered(planner):
    args = (1, 4, 4, _ints([64]), _ints([32]), _ints([2]))
    c = planner.cache_new()
    best = planner.cache_find(c, *args, _ints(PLACES))
    planner.cache_free(c)
    c = planner.cache_new()
    assert best == 4
    assert planner.cache_find(c, *args, _ints((-1, -1, -1, -1))) == 0
    assert planner.cache_find(c, *args, _ints((148, 70, -1, 16))) not in (0, best)   # a plan, but not the one to keep
    assert planner.cache_find(c, *args, _ints(PLACES)) == best
    assert planner.cache_find(c, *args, _ints((-1, -1, -1, -1))) == best             # remembered
    planner.cache_free(c)


def test_a_server_with_a_moving_batch_seldom_plans_anew(planner):
    # the four groups of a decoder layer at every number of rows from 3 to 16
    groups = [([64] * 3, [32] * 3), ([64], [32]), ([64] * 2, [86] * 2), ([172], [32])]
    asked = C.c_int.in_dll(planner, "asked")
    c = planner.cache_new()
    counts = []
    for _ in range(2):
        asked.value = 0
        for M in range(3, 17):
            for k, t in groups:
                assert planner.cache_find(c, len(k), M, 4, _ints(k), _ints(t), _ints([2] * len(k)), _ints(PLACES)) > 0
        counts.append(asked.value)
    planner.cache_free(c)
    assert counts[0] == 14 * 4 * 4 and counts[1] <= counts[0] // 2
