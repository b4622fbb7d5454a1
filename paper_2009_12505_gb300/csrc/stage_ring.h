// Producer's walk over a ring of SLOTS shared-memory stages guarded by mbarriers
// (full: the stage's copies have landed; empty: its reader is done).  Host and
// device code: the walk is checked on the CPU against a model of the barriers.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define RING_FN __host__ __device__ __forceinline__
#else
#define RING_FN inline
#endif

template <int SLOTS>
struct StageRing {
  int step = 0;     // stages armed so far
  int s = 0;        // slot of the next one
  uint32_t ph = 1;  // parity of the release it waits for

  // the first round waits for nothing
  RING_FN bool fresh() const { return step < SLOTS; }
  RING_FN void pass() {
    ++step;
    if (++s == SLOTS) {
      s = 0;
      ph ^= 1;
    }
  }
  // The steps [pending(), step) are the last armed one of each slot.  Only their
  // copies can be in flight; waiting for full[t % SLOTS] with parity (t / SLOTS) & 1
  // of each of them waits for all.
  RING_FN int pending() const { return step > SLOTS ? step - SLOTS : 0; }
};

// The next n stages: turn(q) waits for stage q's slot, arms it and issues its
// copies, or says false; all(ok) is the answer of every thread of the producer.
// After the first false the ring stands still.  It must not move past a stage
// that was not armed: a round later the parity waited for on that slot would be
// that of a release that lies behind, the slot's stage would be overwritten
// while its reader may still need it, and pending() would name phases that are
// over, so that copies outlive the kernel.
template <int SLOTS, class Turn, class All>
RING_FN bool ring_stages(StageRing<SLOTS> &r, int n, Turn turn, All all) {
  for (int q = 0; q < n; ++q) {
    if (!all(turn(q))) return false;
    r.pass();
  }
  return true;
}
