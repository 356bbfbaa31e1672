// Words of k_small's grid barriers (small.cuh), apart from it so that host code can step through the protocol.
//
// Round r's barrier word counts the CTAs that have arrived in its low half and the vertices they leave active in its high
// half, so that the wait also brings the size of the next frontier.  A round has a word of its own, in one of three slots in
// turn: a CTA may still be reading round r's word while the fastest is at round r + 1 already, but none gets to round r + 2
// before the slow one has arrived at r + 1.  One CTA clears the slot of round r + 1 after it has left round r - 1, whose wait
// every CTA that used the slot before (round r - 2) has entered, and before it arrives at round r, which nobody's
// arrival at round r + 1 can precede.  Nothing accumulates over the rounds: no count wraps, however many there are.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define GPOP_HOST_DEVICE __host__ __device__
#else
#define GPOP_HOST_DEVICE
#endif

namespace gpop {

constexpr uint32_t kSmallSlots = 3;

// slot of round r = 0, 1, ...: the barrier before iteration r, whose frontier the slot's counters describe
GPOP_HOST_DEVICE constexpr uint32_t small_slot_of(uint32_t round) { return round % kSmallSlots; }
// slot that is cleared between the rounds r - 1 and r
GPOP_HOST_DEVICE constexpr uint32_t small_slot_to_clear(uint32_t round) { return small_slot_of(round + 1); }

GPOP_HOST_DEVICE constexpr unsigned long long small_arrival(uint32_t active) { return (unsigned long long)active << 32 | 1ull; }
GPOP_HOST_DEVICE constexpr bool small_all_arrived(unsigned long long word, uint32_t ctas) { return (uint32_t)word == ctas; }
GPOP_HOST_DEVICE constexpr uint32_t small_active(unsigned long long word) { return (uint32_t)(word >> 32); }

}  // namespace gpop
