// A radix-sort tile's published state for one digit, in one 32-bit word: nothing yet (0),
// the tile's own count of the digit, or the inclusive prefix of the counts up to it.
// A tile's count is at most a few thousand, so it takes the values 1 .. 2^31 - 1 as
// count + 1, and the top bit marks a prefix, which has the other 31 bits: the sort holds
// for every element count below 2^31. Host code may include this file.
#pragma once
#include <cstdint>

#include "host_device.h"

namespace rl {

constexpr uint32_t kStatePrefix = 1u << 31;

RELEARN_HOST_DEVICE uint32_t state_of_count(uint32_t count) { return count + 1u; }
RELEARN_HOST_DEVICE uint32_t state_of_prefix(uint32_t prefix) { return kStatePrefix | prefix; }
RELEARN_HOST_DEVICE bool state_published(uint32_t s) { return s != 0u; }
RELEARN_HOST_DEVICE bool state_is_prefix(uint32_t s) { return (s & kStatePrefix) != 0u; }
// The sum held by n words read from a tile backwards, n - 1 counts and then a prefix, whose
// sum as words is given (modulo 2^32).
RELEARN_HOST_DEVICE uint32_t state_sum(uint32_t words, uint32_t n)
{
    return words - (n - 1u) - kStatePrefix;
}

} // namespace rl
