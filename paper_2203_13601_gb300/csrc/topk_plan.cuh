// topk_plan.cuh -- the arithmetic behind the exact top-k's plan, in functions that compile
// for the host as well (k_bruteforce.cu uses them, a host-compiled test checks them).
#pragma once

#include "nhq_internal.cuh"

namespace nhq {

// A group's place among the groups and its units' place among the units are claimed in one
// addition to (groups << kUnitBits | units), so that group order is unit order.  Both stay
// below 2^32: at most one group and one unit per query (fewer than 2^30 queries) and, where
// a run takes several slices, at most one unit per list row.  (With 24 bits for the groups
// the count wrapped at 2^24 tuples and rows stayed unwritten.)
constexpr int kUnitBits = 32;
__host__ __device__ inline unsigned long long plan_claim(unsigned long long units) {
    return (1ull << kUnitBits) + units;
}
__host__ __device__ inline uint64_t claimed_groups(unsigned long long at) {
    return at >> kUnitBits;
}
__host__ __device__ inline uint64_t claimed_units(unsigned long long at) {
    return at & ((1ull << kUnitBits) - 1);
}

}  // namespace nhq
