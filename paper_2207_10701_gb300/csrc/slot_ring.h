// The order in which operand slots are reused: use u of a ring takes slot u mod RING_SLOTS.  Every use
// ends with one completion of the slot's barrier (tcgen05.commit behind the MMAs that read the slot),
// and a use from RING_SLOTS on first waits for that of the use before it in the same slot.  A barrier
// is waited for by the parity of its phase, and it is at most one phase ahead of its waiter.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define RING_FN __host__ __device__ __forceinline__
#else
#define RING_FN inline
#endif

constexpr int RING_SLOTS = 4;

struct RingUse {
  uint32_t slot, wait, parity;  // wait: not the slot's first use; parity: of the phase waited for
};

RING_FN RingUse ring_use(uint32_t u) {
  const uint32_t round = u / RING_SLOTS;
  return RingUse{u % RING_SLOTS, round > 0 ? 1u : 0u, (round - 1) & 1u};
}
