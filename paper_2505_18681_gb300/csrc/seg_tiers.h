// Lengths of the segmented sort's one-CTA tiers (plain C++, host and device).
#pragma once

#include <cstdint>

namespace evosort {

// Segments of at most this many keys are cut and sorted with 32-bit counters
// (cta_sort.cuh).  A counter is advanced past the last key by up to one step
// before it is compared with the length, so the longest length plus the
// largest step must stay below 2^32: at 2^32 - 1 keys the counter would wrap
// below the length and the loop never end.  2^31 - 1 is the largest length of
// a work-list bucket (floor(log2)) that leaves that room.  Longer segments,
// where no device-wide sort took them, go through radix passes with 64-bit
// counters.
constexpr int kSegLongLog2 = 31;
constexpr uint64_t kSegCutKeys = (1ull << kSegLongLog2) - 1;

}  // namespace evosort
