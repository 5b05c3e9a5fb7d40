// How the adjoint of a compiled shape takes its paths in ranges whose arrays fit the memory it may
// use. Plain C++ with the allocation passed in, so that a failing one can be run on the host.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace cva {

constexpr uint64_t kRangeBlock = 256;   // a range is whole blocks of this many paths

struct RangePlan {
    uint64_t per = 0, ranges = 0;   // paths of a range (the last may be shorter), ranges
    size_t bytes = 0;               // the arrays of the widest
};

// The widest equal ranges whose arrays, bytes(paths), take `limit` at most; one block's where
// even that takes more.
template <class Bytes>
RangePlan plan_ranges(uint64_t M, size_t limit, Bytes bytes)
{
    RangePlan p;
    for (p.ranges = 1;;) {
        p.per = (M + p.ranges - 1) / p.ranges;
        p.per = (p.per + kRangeBlock - 1) / kRangeBlock * kRangeBlock;
        p.bytes = bytes(std::min(p.per, M));
        if (p.bytes <= limit || p.per == kRangeBlock) break;
        p.ranges = std::max<uint64_t>(p.ranges + 1, p.ranges * (p.bytes / std::max<size_t>(limit, 1)));
    }
    p.ranges = (M + p.per - 1) / p.per;
    p.bytes = std::max(p.bytes, bytes(M - (p.ranges - 1) * p.per));   // (fewer paths may be split finer)
    return p;
}

// plan_ranges within `limit`, or within half of it and so on until allocate(plan), which has to
// free what it got when it fails, succeeds. False when one block a range is too much.
template <class Bytes, class Allocate>
bool fit_ranges(uint64_t M, size_t limit, Bytes bytes, Allocate allocate, RangePlan *plan)
{
    for (;; limit /= 2) {
        *plan = plan_ranges(M, limit, bytes);
        if (allocate(*plan)) return true;
        if (plan->per == kRangeBlock) return false;
    }
}

}  // namespace cva
