"""The refill rule of csrc/ring.cuh on the host, against a model of the mbarrier: an arm (arrive.expect_tx, count 1)
while the previous phase is still open would take the arrival count below zero, and no copy may be in flight when the
block ends.  Waits succeed up to a chosen one and time out from there, copies land only when somebody waits for
them."""
import os
import subprocess


CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2109_12390_gb300", "csrc")
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "ring.cuh"
using namespace mpmrom;
static void need(bool ok, const char* what, int a, int b) {
  if (!ok) { std::printf("%s (%d, %d)\n", what, a, b); std::exit(1); }
}
// A buffer's full barrier: phase k closes when copy k's bytes have landed.
struct Bar {
  uint32_t armed = 0, closed = 0;   // phases armed, phases complete
  void arm() { need(armed == closed, "armed while the previous phase is open", (int)armed, (int)closed); ++armed; }
  void land() { closed = armed; }
  // try_wait on a parity: the phase that precedes the current one
  bool done(uint32_t parity) const { return ((closed - 1) & 1u) == parity && closed > 0; }
};

template <uint32_t SLOTS>
void ring(uint32_t n, uint32_t good) {   // the first `good` waits for an empty buffer succeed
  Bar full[SLOTS];
  uint32_t waits = 0, uses[SLOTS] = {};
  bool aborted = false;
  const uint32_t started = ring_fill<SLOTS>(
      n,
      [&](uint32_t slot, uint32_t parity) {
        if (aborted || waits++ >= good) { aborted = true; return false; }
        full[slot].land();   // the consumer has seen the copy and used it
        need(((uses[slot] - 1) & 1u) == parity, "waits for another use than the last", (int)slot, (int)parity);
        return true;
      },
      [&](uint32_t slot, uint32_t) { full[slot].arm(); ++uses[slot]; });
  need(aborted || started == n, "copies left out without a timeout", (int)started, (int)n);
  if (aborted)
    ring_land<SLOTS>(started, [&](uint32_t slot, uint32_t parity) {
      full[slot].land();
      need(full[slot].done(parity), "waits for the wrong phase", (int)slot, (int)parity);
    });
  for (uint32_t s = 0; s < SLOTS && aborted; ++s)
    need(full[s].armed == full[s].closed, "a copy is in flight at the end", (int)s, (int)n);
}

void refill(uint32_t n, uint32_t good) {   // the first `good` waits for the data succeed
  Bar full;
  Refill f;
  for (uint32_t k = 0; k < n; ++k) {
    if (f.start()) full.arm();
    bool landed = false;
    if (f.live && k < good) {
      full.land();
      landed = full.done(f.last_phase());
      need(landed, "waits for the wrong phase", (int)k, (int)good);
    }
    f.seen(landed);
  }
  if (!f.live) {
    full.land();
    need(full.done(f.last_phase()), "waits for the wrong phase at the end", (int)n, (int)good);
  }
  need(full.armed == full.closed, "a copy is in flight at the end", (int)n, (int)good);
}

int main() {
  for (uint32_t n = 0; n < 60; ++n)
    for (uint32_t good = 0; good <= n; ++good) {
      ring<9>(n, good);
      ring<3>(n, good);
      ring<1>(n, good);
      refill(n, good);
    }
  return 0;
}
"""


def test_no_barrier_is_armed_twice_and_nothing_stays_in_flight(tmp_path):
    (tmp_path / "t.cc").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-I", CSRC, str(tmp_path / "t.cc"), "-o", str(tmp_path / "t")],
                   check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
