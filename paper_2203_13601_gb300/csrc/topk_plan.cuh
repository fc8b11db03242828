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

// A squared distance that every pair with Gamma <= g stays below or equals.  Gamma is at
// least its vector term in these modes, and sqrt, product and square are each rounded once
// (relative 2^-24), which the factors cover; the addend covers squares below the normal
// range.  A subnormal product w_v delta has no such relative bound: below 1e-37 nothing is
// ruled out, unless w_v >= 1e-6, where every nonzero delta (at least 3.7e-23, the root of the
// smallest squared distance) has a normal product and g stands for delta = 0.
__host__ __device__ inline float admitted_dist2(float g, const Fusion &w) {
    float s = __builtin_huge_valf();
    if (w.mode == NHQ_W_PROPORTIONAL || w.mode == NHQ_W_FILTER)
        s = g;
    else if (w.mode == NHQ_W_CONSTANT && w.wv > 1e-30f && (g >= 1e-37f || w.wv >= 1e-6f))
        s = (g / w.wv) * 1.00001f;
    return s * s * 1.00001f + 1e-36f;
}

// The first slot of the group table (tmask + 1 slots, a power of two) for the run that
// starts at position lo.  All bits of lo count: starts that share a stride, as those of
// balanced attributes do, must not share slots (with the low bits of a product, 256 runs of
// 4,096 objects all met in one slot, 127 probes on average: 2,048 queries over them, d = 32,
// took 685 us and take 407).
__host__ __device__ inline uint32_t table_slot(uint32_t lo, uint32_t tmask) {
    return (uint32_t)mix64(lo + kGolden) & tmask;
}

constexpr int MAX_SLICES = 128;

// Objects per slice of a tuple's run.  Few queries hardly share tuples: short slices, so
// that one query's run fills the chip (9,000 objects on average at a million and 600
// tuples: 36 slices of 256).  Larger batches fill it with tiles of 32 queries and pay for
// slices in lists.  A million objects of 600 even tuples, d = 128, k = 10: 8 queries 37 us
// in slices of 128, 44 of 256, 68 of 1,024; 64 queries 56, 54 and 85; 2,000 queries 521 us of
// 256, 500 of 1,024, 538 of 2,048; 10,000 queries 612, 567 and 577.
__host__ __device__ inline int run_slice_length(int64_t nq) {
    return nq <= 64 ? 256 : nq <= 2048 ? 1024 : 2048;
}

__host__ __device__ inline int64_t run_slices(int64_t len, int slice) {
    const int64_t s = (len + slice - 1) / slice;
    return s > MAX_SLICES ? MAX_SLICES : s;
}

// Rows of k records kept for the lists of sliced runs: none where no run can take two
// slices, never more than nq queries on the longest run could use, six for each query
// (10,000 queries over a million objects of 600 tuples use five) or 24 tiles for each SM,
// and at most 128 MB, since the index keeps them: 10,000 queries take 93 MB at k = 100 and
// 134 MB at k = 256.  (While neither N nor the bytes counted: 266 and 680 MB, and 658 MB for
// 5,000 at k = 256 over 1,300 objects, which use none.  64 MB would cost the 10,000 at
// k = 256 half their speed: 8.2 ms instead of 4.2.)
constexpr size_t kRunListBytes = size_t(128) << 20;
inline int64_t run_list_rows(int64_t nq, int64_t N, int k, int sm_count) {
    const int64_t most = run_slices(N, run_slice_length(nq));
    if (most == 1)
        return 0;
    const int64_t fill = 24 * (int64_t)sm_count * 32;
    int64_t rows = 6 * nq > fill ? 6 * nq : fill;
    rows = rows < nq * most ? rows : nq * most;
    const int64_t fit = (int64_t)(kRunListBytes / ((sizeof(uint32_t) + sizeof(float)) * k));
    return rows < fit ? rows : fit;
}

// Slices of a run that would take `want` of them for `tiles` tiles of queries, where the
// queries of all sliced runs ask for `all` list rows and there are `rows`: every run gives
// up the same share, so that none is left with one slice while others have many (whoever
// came first took all before: 2,000 queries over 100,000 objects of two tuples, k = 100,
// 2.5 ms instead of 2.2), and the rows handed out stay within `rows`.  A run of `busy` tiles
// fills the chip by itself and takes one slice: more would only add lists (candidate sets
// of 30,000 objects of one tuple, 938 tiles: 10.8 ms, 13.2 with six slices).
__host__ __device__ inline int64_t granted_slices(int64_t want, int64_t tiles, uint64_t all,
                                                  int64_t rows, int busy) {
    if (tiles >= busy)
        return 1;
    const int64_t s = all > (uint64_t)rows ? (int64_t)((uint64_t)want * rows / all) : want;
    return s > 1 ? s : 1;
}

}  // namespace nhq
