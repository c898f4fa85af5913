// The order in which the operand slots of the FP64 digit products are reused.  The seven digits of a
// stage go through four slots in four groups: digits 0 1 | 2 3 | 4 | 5 6 in slots 0 1 | 2 3 | 0 | 2 3.
// Each group ends with one completion of its barrier (tcgen05.commit behind the MMAs that read its
// slots), and each waits for the group two before it, whose slots it takes.  In between lies always
// one group of four digit pairs or more, so the tensor cores have work while the issuing thread waits.
// A new FP64 design of 500 x 160 takes 38.7 ms so; without the waits it took 38.1, with a group per
// digit (seven waits a stage in the thread that issues) 44.6.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define RING_FN __host__ __device__ __forceinline__
#else
#define RING_FN inline
#endif

constexpr int RING_SLOTS = 4, RING_GROUPS = 4, RING_DIGITS = 7;

RING_FN constexpr uint32_t ring_slot(int digit) { return digit == 4 ? 0u : digit > 4 ? digit - 3u : (uint32_t)digit; }
RING_FN constexpr int ring_group(int digit) { return digit < 4 ? digit / 2 : digit == 4 ? 2 : 3; }
RING_FN constexpr bool ring_first(int digit) { return digit == 0 || ring_group(digit) != ring_group(digit - 1); }
RING_FN constexpr bool ring_last(int digit) { return digit == RING_DIGITS - 1 || ring_first(digit + 1); }

// Before group g of stage `it` (counted from the first of the kernel): the barrier to wait for, and the
// parity of its phase; none in the first stage for the groups whose slots are new.
RING_FN constexpr int ring_wait_group(int g) { return (g + 2) % RING_GROUPS; }
RING_FN bool ring_waits(int g, uint32_t it) { return g >= 2 || it > 0; }
RING_FN uint32_t ring_parity(int g, uint32_t it) { return (g >= 2 ? it : it - 1) & 1u; }
