// The operand slots under the worst schedule: a copy lands as soon as it is issued, the MMAs that read
// a slot run as late as the waits allow.  No copy may land in a slot that an MMA issued before has
// still to read, every wait ends, and some MMAs are left to run behind it.  Prints "ring ok".
#include <cstdio>
#include <deque>

#include "../../paper_2207_10701_gb300/csrc/slot_ring.h"

struct Op {
  int group;  // -1: the MMAs of a use of `slot`, else the commit of a group
  uint32_t slot;
};

int main() {
  uint32_t completions[RING_GROUPS] = {};
  int pending[RING_SLOTS] = {};  // uses whose MMAs have not run
  std::deque<Op> queue;          // in issue order
  for (uint32_t it = 0; it < 2000; ++it) {
    for (int d = 0; d < RING_DIGITS; ++d) {
      const int g = ring_group(d);
      const uint32_t s = ring_slot(d);
      if (s >= RING_SLOTS || g >= RING_GROUPS) return std::printf("ring FAIL: range\n"), 1;
      if (ring_first(d) && ring_waits(g, it)) {
        const int w = ring_wait_group(g);
        // a wait for parity p ends once the phase of that parity is complete
        while ((completions[w] & 1) == ring_parity(g, it)) {
          if (queue.empty()) return std::printf("ring FAIL: stage %u waits for nothing\n", it), 1;
          const Op o = queue.front();
          queue.pop_front();
          if (o.group < 0) --pending[o.slot];
          else ++completions[o.group];
        }
        if (queue.empty()) return std::printf("ring FAIL: stage %u leaves nothing to run\n", it), 1;
      }
      if (pending[s] != 0) return std::printf("ring FAIL: stage %u digit %d overwrites an operand\n", it, d), 1;
      queue.push_back({-1, s});
      ++pending[s];
      if (ring_last(d)) queue.push_back({g, 0});
    }
  }
  std::printf("ring ok\n");
  return 0;
}
