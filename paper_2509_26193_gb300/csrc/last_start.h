// The last of nb block starts that lies at or before tgt (0 if none does), by bisection.
//
// The starts are an exclusive scan of non-negative sums in FP64 by shuffles, whose entries
// add the same sums in different orders: a start may lie below the one before it by its
// rounding, at most ten units of 2^-53 (five additions each). After the bisection k, start
// k + 1 lies past tgt, so a later one at or before tgt lies within that of it: the starts
// after k are looked at as long as they come that close to tgt (32 steps of the last
// place), nearly always one.
#pragma once
#include <cstdint>
#include <cstring>

#include "host_device.h"

namespace rl {

RELEARN_HOST_DEVICE int64_t double_bits(double v)
{
    int64_t b;
    memcpy(&b, &v, sizeof(b));
    return b;
}

RELEARN_HOST_DEVICE int last_start(const double *start, int nb, double tgt)
{
    int k = 0;
    for (int hi = nb - 1; k < hi;) {
        const int mid = (k + hi + 1) >> 1;
        if (start[mid] <= tgt)
            k = mid;
        else
            hi = mid - 1;
    }
    // (non-negative doubles order like their bits)
    const int64_t close = double_bits(tgt) + 32;
    for (int j = k + 1; j < nb && double_bits(start[j]) <= close; ++j)
        if (start[j] <= tgt) k = j;
    return k;
}

} // namespace rl
