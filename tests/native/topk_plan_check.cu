// Host-side checks of the exact top-k's plan arithmetic (topk_plan.cuh).  The first
// argument picks the check; prints "ok" or the first failing case.
#include <cstdio>
#include <cstring>

#include "topk_plan.cuh"

using namespace nhq;

// the claims of 2^24 + 9 groups of one unit, and of groups of many units
static int check_claims() {
    const uint64_t n = (1u << 24) + 9;
    unsigned long long counter = 0;
    for (uint64_t g = 0; g < n; ++g) {
        const unsigned long long at = counter;
        counter += plan_claim(1);
        if (claimed_groups(at) != g || claimed_units(at) != g)
            return std::printf("FAIL group %llu\n", (unsigned long long)g), 1;
    }
    if (claimed_groups(counter) != n || claimed_units(counter) != n)
        return std::printf("FAIL total\n"), 1;
    // the largest plan: 2^30 groups, 2^30 units and 2^24 more from sliced runs
    counter = (1ull << 30) * plan_claim(1) + (1ull << 24);
    if (claimed_groups(counter) != 1ull << 30 ||
        claimed_units(counter) != (1ull << 30) + (1ull << 24))
        return std::printf("FAIL largest\n"), 1;
    return 0;
}

int main(int argc, char **argv) {
    int bad = 2;
    if (argc > 1 && !std::strcmp(argv[1], "claims"))
        bad = check_claims();
    if (bad == 0)
        std::printf("ok\n");
    return bad;
}
