// The order in which a producer and several groups of consumers ("phases") walk a ring of slots, each slot guarded by barriers of one
// parity bit (Section 2.1: few tokens per step stream the weights, which is what such a ring carries).  Plain C++: the host's tests run it too.
#pragma once
#if defined(__CUDACC__)
#define LQER_RING_FN __host__ __device__ __forceinline__
#else
#define LQER_RING_FN inline
#endif

namespace lqer {

// Stage x is for phase x % phases.  The slots are dealt out to the phases in turn (slot s to phase s % phases), and a phase goes round its
// own: so what lay in a slot before stage x was an earlier stage of the same phase, which that phase has waited for.  A wait for one
// parity bit needs this: copies may land in any order, and a phase that came to a slot whose former stage, another phase's, is still under way
// would take the pass before that one for its own.
struct RingCursor {
  int phase, slot;
  unsigned parity;               // of the pass over the phase's slots
  LQER_RING_FN explicit RingCursor(int first = 0) : phase(first), slot(first), parity(0) {}
  LQER_RING_FN void next(int phases, int slots) {
    slot += phases;
    if (slot >= slots) { slot = phase; parity ^= 1u; }
  }
};
// The producer's way over all phases' slots, from stage x on, x being the first that is not the first in its slot.
template <int PHASES>
struct RingWalk {
  RingCursor turn[PHASES];       // turn[0]: the next stage's
  LQER_RING_FN explicit RingWalk(int x) {
    for (int i = 0; i < PHASES; ++i) turn[i] = RingCursor((x + i) % PHASES);
  }
  LQER_RING_FN void next(int slots) {
    RingCursor again = turn[0];
    again.next(PHASES, slots);
    for (int i = 0; i + 1 < PHASES; ++i) turn[i] = turn[i + 1];
    turn[PHASES - 1] = again;
  }
};

}  // namespace lqer
