// The ring of operand slots under the worst schedule: a copy lands as soon as it is issued, the MMAs
// that read a slot run as late as the waits allow.  No copy may land in a slot that an MMA issued
// before has still to read, and every wait ends.  Prints "ring ok" on success.
#include <cstdio>
#include <deque>

#include "../../paper_2207_10701_gb300/csrc/slot_ring.h"

int main() {
  uint32_t completions[RING_SLOTS] = {};  // of each slot's barrier
  int pending[RING_SLOTS] = {};           // uses whose MMAs have not run
  std::deque<uint32_t> mmas;              // in issue order
  for (uint32_t u = 0; u < 10000; ++u) {
    const RingUse r = ring_use(u);
    if (r.slot >= RING_SLOTS) return std::printf("ring FAIL: slot of use %u\n", u), 1;
    if (r.wait) {
      // a wait for parity p ends once the phase of that parity is complete
      while ((completions[r.slot] & 1) == r.parity) {
        if (mmas.empty()) return std::printf("ring FAIL: use %u waits for nothing\n", u), 1;
        const uint32_t s = mmas.front();
        mmas.pop_front();
        --pending[s];
        ++completions[s];
      }
    }
    if (pending[r.slot] != 0) return std::printf("ring FAIL: use %u overwrites an operand\n", u), 1;
    mmas.push_back(r.slot);
    ++pending[r.slot];
  }
  std::printf("ring ok\n");
  return 0;
}
