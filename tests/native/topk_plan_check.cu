// Host-side checks of the exact top-k's plan arithmetic (topk_plan.cuh).  The first
// argument picks the check; prints "ok" or the first failing case.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

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

// the rows kept for sliced runs: bounded in bytes and by what the runs can use, and never
// handed out twice
static int check_rows() {
    for (int64_t nq : {1, 8, 64, 65, 2048, 2049, 5000, 10000, 1000000, 1 << 29})
        for (int64_t N : {1, 256, 257, 1024, 1025, 1300, 2048, 2049, 70000, 1000000, 0x7FFFFFFE})
            for (int k : {1, 10, 64, 100, 256}) {
                const int64_t rows = run_list_rows(nq, N, k, 152);
                const int64_t most = run_slices(N, run_slice_length(nq));
                bool ok = rows >= 0 && rows <= nq * most && rows * 8 * k <= (128 << 20);
                ok = ok && (most > 1 || rows == 0);
                // groups of ever more queries on ever shorter runs, of one query and more
                uint64_t all = 0, out = 0;
                for (int pass = 0; pass < 2; ++pass) {
                    int64_t left = nq, len = N;
                    for (int64_t cnt = 1; left > 0; cnt = cnt * 3 + 1, len = len * 2 / 3 + 1) {
                        const int64_t n = cnt < left ? cnt : left;
                        const int64_t want = run_slices(len, run_slice_length(nq));
                        left -= n;
                        if (want < 2)
                            continue;
                        if (pass == 0) {
                            all += (uint64_t)(n * want);
                            continue;
                        }
                        const int64_t s = granted_slices(want, (n + 31) / 32, all, rows, 912);
                        ok = ok && s >= 1 && s <= want && (all > (uint64_t)rows || s == want ||
                                                           (n + 31) / 32 >= 912);
                        out += s > 1 ? (uint64_t)(n * s) : 0;
                    }
                }
                ok = ok && out <= (uint64_t)rows;
                if (!ok)
                    return std::printf("FAIL nq=%lld N=%lld k=%d rows=%lld\n", (long long)nq,
                                       (long long)N, k, (long long)rows), 1;
            }
    return 0;
}

// Gamma of a matching pair (every other one is larger), each operation rounded once
static float gamma_of(float d2, const Fusion &w) {
    const volatile float delta = std::sqrt(d2);
    const volatile float g = w.mode == NHQ_W_CONSTANT ? w.wv * delta : delta;
    return g;
}

// no pair that may enter is above the admitted squared distance of the k-th record
static int check_admitted() {
    std::mt19937_64 rng(11);
    auto logu = [&](double lo, double hi) {
        return (float)std::exp2(std::uniform_real_distribution<double>(lo, hi)(rng));
    };
    Fusion w{};
    for (int trial = 0; trial < 4000000; ++trial) {
        w.mode = trial % 3 == 0 ? NHQ_W_PROPORTIONAL : trial % 3 == 1 ? NHQ_W_FILTER
                                                                      : NHQ_W_CONSTANT;
        w.wv = trial % 2 ? logu(-148, -90) : logu(-30, 30);
        const float a = trial % 5 == 0 ? 0.f : logu(-149, 100);
        float b = trial % 7 == 0 ? logu(-149, 100) : a * logu(-1, 1);
        if (trial == 5) {  // both round to the same Gamma, 2 x 2^-149
            w.wv = 2e-30f, w.mode = NHQ_W_CONSTANT;
            b = 2.4e-15f * 2.4e-15f;
        }
        const float kth = trial == 5 ? 2.0e-15f * 2.0e-15f : a;
        const float g = gamma_of(kth, w);
        if (gamma_of(b, w) <= g && !(b <= admitted_dist2(g, w)))
            return std::printf("FAIL mode %d w_v %g kth %g other %g\n", w.mode, w.wv, kth, b), 1;
    }
    return 0;
}

// equal runs of `len` objects (and of lengths that multiplicative hashes dislike) spread over
// the table: at half load a random placement probes 1.5 slots on average
static int check_table() {
    for (uint32_t len : {1u, 16u, 256u, 1000u, 4096u, 46368u, 65536u, 1u << 20})
        for (uint32_t slots : {64u, 4096u, 65536u}) {
            const uint32_t tmask = slots - 1, keys = slots / 2;
            std::vector<char> used(slots, 0);
            uint64_t probes = 0, worst = 0, n = 0;
            for (uint32_t i = 0; i < keys && (uint64_t)i * len < 0x7FFFFFFEu; ++i, ++n) {
                uint32_t s = table_slot(i * len, tmask);
                uint64_t p = 1;
                for (; used[s]; s = (s + 1) & tmask)
                    ++p;
                used[s] = 1;
                probes += p;
                worst = p > worst ? p : worst;
            }
            if (probes > 3 * n || worst > 100)
                return std::printf("FAIL len=%u slots=%u probes=%.1f worst=%d\n", len, slots,
                                   (double)probes / n, (int)worst), 1;
        }
    return 0;
}

int main(int argc, char **argv) {
    int bad = 2;
    if (argc > 1 && !std::strcmp(argv[1], "claims"))
        bad = check_claims();
    else if (argc > 1 && !std::strcmp(argv[1], "rows"))
        bad = check_rows();
    else if (argc > 1 && !std::strcmp(argv[1], "admitted"))
        bad = check_admitted();
    else if (argc > 1 && !std::strcmp(argv[1], "table"))
        bad = check_table();
    if (bad == 0)
        std::printf("ok\n");
    return bad;
}
