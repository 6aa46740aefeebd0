// Refilling shared-memory buffers by asynchronous copies that complete on mbarriers, when a bounded wait may run
// out.  The rule that both forms keep: a barrier is armed (arrive.expect_tx) only when its previous phase is known to
// be complete, since arming a phase that is still open takes its arrival count below zero.  So after a wait that did
// not end nothing is armed any more, and what is in flight has to land before the block ends.  Plain C++: the barriers
// come in as functions, so that the rule is tested on the host.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define MPM_RING_FN __host__ __device__ __forceinline__
#else
#define MPM_RING_FN inline
#endif

namespace mpmrom {

// Copies 0 .. n - 1 through a ring of SLOTS buffers, copy i in buffer i % SLOTS as use i / SLOTS of it.  Returns the
// number of copies started.
//   wait_empty(slot, parity)   whether the buffer's previous use is over (bounded; false: given up)
//   issue(slot, i)             arms the buffer's full barrier and starts copy i
template <uint32_t SLOTS, class WaitEmpty, class Issue>
MPM_RING_FN uint32_t ring_fill(uint32_t n, WaitEmpty wait_empty, Issue issue) {
  for (uint32_t i = 0; i < n; ++i) {
    const uint32_t slot = i % SLOTS, use = i / SLOTS;
    if (use > 0 && !wait_empty(slot, (use - 1) & 1u)) return i;
    issue(slot, i);
  }
  return n;
}
// After a timeout, when no thread of the block waits on the ring any more: the last of the `started` copies land
// (otherwise the consumers have waited for every one).  wait_full(slot, parity): bounded.
template <uint32_t SLOTS, class WaitFull>
MPM_RING_FN void ring_land(uint32_t started, WaitFull wait_full) {
  for (uint32_t k = started > SLOTS ? started - SLOTS : 0; k < started; ++k) wait_full(k % SLOTS, (k / SLOTS) & 1u);
}

// One buffer that its consumer refills: n copies started, the last one's landing seen or given up.
struct Refill {
  uint32_t n = 0;
  bool live = true;
  MPM_RING_FN uint32_t last_phase() const { return (n - 1) & 1u; }   // parity of the last copy's phase (n > 0)
  MPM_RING_FN void seen(bool landed) { live = live && landed; }
  MPM_RING_FN bool start() {   // whether the next copy may be started (and counts it)
    n += live ? 1 : 0;
    return live;
  }
};

}  // namespace mpmrom
