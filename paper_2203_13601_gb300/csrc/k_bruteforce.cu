// k_bruteforce.cu -- exact top-k by (Gamma, id) over all objects (Def. 2 with the
// fusion distance of Eq. 6), and with exclude_self the exact candidate sets C(u)
// of Sec. 4.1 (every object is a query, itself excluded).
//
// Two ways to the same answer:
//
// Full scan (scan_kernel).  A CTA takes a tile of queries and a slice of the objects
// in tiles of 128.  Squared distances are register-tiled from 32-wide dimension chunks
// that cp.async brings into a two-stage ring in shared memory; a pair whose squared
// distance is above what its query's k-th record admits is dropped by one comparison
// (no square root, no chi, no division), the rest get their exact Gamma and enter the
// query's sorted list in shared memory.  With several slices the lists go to scratch
// and a warp-per-query k-way merge writes the final rows.
//
// Tuple runs (run_kernel).  Under the filter weighting only the objects that carry the
// query's tuple count, and under constant weights they come first as long as omega_l
// exceeds the vector term.  The queries are grouped by tuple, each group scans only its
// tuple's run of the attribute order, and a query whose k-th record there is below
// Gamma(delta = 0, chi = 1) is finished: Gamma does not fall as delta or chi grows, so no
// other object can enter.  The queries for which that fails (constant weights only) go
// through the full scan afterwards, counted on the device; a long run that is going to fail
// is given up early.
//
// What bounds it: 64 % of the issue slots and 56 % of the FMA pipe's cycles are used, by 21
// warps an SM that wait for shared memory, barriers and fixed latencies about equally (80
// registers, 8 bytes spilled, for three CTAs an SM).  Candidate
// sets of 60,000 objects (d = 96, K = 64, proportional weights) take 40.0 ms, half the FP32
// rate of a difference and an fma per dimension; before (no staging ahead, every pair's
// Gamma with its division, records inserted one by one) 55.5 ms.  2,003 queries, k = 100,
// over 300,007 objects: 9.8 ms, before 16.4 ms.  The runs do a hundredth of the pairs: the
// filter truth of 10,000 queries over a million objects (600 tuples) 1.58 ms, before 206 ms;
// eight queries under constant weights 59 us, before 5,560 us.
#include <cmath>
#include <cstdio>
#include <mutex>

#include "topk_plan.cuh"

namespace nhq {

namespace {

constexpr int TN = 128;     // objects per tile
constexpr int DC = 32;      // dimensions per staged chunk
constexpr int DS = DC + 4;  // staged row stride: 16-byte aligned rows, read as float4
constexpr int NT = 256;     // threads per CTA
constexpr uint32_t PROBE = 512;  // objects (k <= 256) after which a long run is judged
constexpr uint32_t GIVEN_UP = 0x80000000u;  // a run's length is below 2^31
constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr float INF = __builtin_huge_valf();
constexpr unsigned long long NO_RECORD = (0x7F800000ull << 32) | kNone;  // (inf, none)

// Shape of a CTA's tile: TY x (256 / TY) threads of QI queries x OJ objects each.
// CTAS of it fit an SM (registers; shared memory may allow fewer).
template <int TY_, int QI_, int CTAS_>
struct Shape {
    static constexpr int TY = TY_, QI = QI_, TX = NT / TY_, TQ = TY_ * QI_, OJ = TN / TX;
    static_assert(TX == 16 || TX == 64, "the masks of a tile's pairs are written per warp");
    static constexpr int CTAS = CTAS_;
    static constexpr int QW = (TQ + 7) / 8;  // queries whose lists a warp keeps
};
using Mid = Shape<16, 2, 3>;    // 32 queries: 2 x 8 pairs per thread
using Narrow = Shape<4, 1, 4>;  // 4 queries

// shared memory of a CTA; the lists [TQ][k] follow (records as Gamma bits << 32 | id)
template <class T>
struct Smem {
    // two stages of Q and X chunks; 74 KB with lists of 100 records: three CTAs an SM (with
    // a buffer of its own for the distances two would fit: 49.5 ms for the candidate sets)
    union Stage {
        struct {
            float Q[T::TQ][DS];
            float X[TN][DS];
        };
        float D2[T::TQ][TN];    // once the tile is summed: the distances flagged in mask
    } st[2];
    unsigned long long cand[NT / 32][32];  // a warp's records to merge
    uint32_t mask[T::TQ][4];    // pairs of the tile that can enter the list
    float tg[T::TQ];            // the k-th record (Gamma, id); (inf, kNone) while not full
    uint32_t ti[T::TQ];
    int cnt[T::TQ];             // records in the list
    float t2[T::TQ];            // no pair with a squared distance above t2 can enter
    uint32_t q[T::TQ], qa[T::TQ], qh[T::TQ];  // query (or kNone), its word and chi mask
    int unit;
};

template <class T>
size_t tile_smem(int k) {
    return sizeof(Smem<T>) + sizeof(unsigned long long) * (size_t)T::TQ * k;
}

__device__ __forceinline__ bool rec_less(float ga, uint32_t ia, float gb, uint32_t ib) {
    return ga < gb || (ga == gb && ia < ib);
}

// Two differences in one instruction, each rounded as a single one is: six issue slots for
// four dimensions of a pair instead of eight (candidate sets of 60,000 objects 44.8 ->
// 41.2 ms, filter truth of 10,000 queries 1.79 -> 1.65 ms).  The sums stay one chain.
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ void add_squares(float &acc, unsigned long long t) {
    const float lo = __uint_as_float((uint32_t)t), hi = __uint_as_float((uint32_t)(t >> 32));
    acc = fmaf(lo, lo, acc);
    acc = fmaf(hi, hi, acc);
}

__device__ __forceinline__ void cp16(uint32_t dst, const void *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp4(uint32_t dst, const void *src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}

// Merges the records c (one per lane, ~0: none) into the sorted list of cnt records
// (capacity k); whole warp.  A record's place is its rank among the new ones plus its rank
// in the list; the places are distinct, so one mask describes a chunk of 32 places, and a
// place that no new record takes receives the old one as many places below it as new
// records precede it (chunks from the top down, each read before it is written).  A batch
// costs about what one insertion did, and the first tiles of a scan bring batches of 32.
__device__ __forceinline__ void list_merge(unsigned long long *L, int &cnt, int k,
                                           unsigned long long c, unsigned long long *cand,
                                           int lane) {
    if (cnt == k && c > L[k - 1])
        c = ~0ull;
    const bool valid = c != ~0ull;
    const unsigned vb = __ballot_sync(FULL, valid);
    if (vb == 0)
        return;
    const int nv = __popc(vb);
    const unsigned lt = (1u << lane) - 1u;
    cand[valid ? __popc(vb & lt) : nv + __popc(~vb & lt)] = c;
    __syncwarp();
    int pos = k;
    if (valid) {
        int lo = 0, hi = cnt;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (L[mid] < c)
                lo = mid + 1;
            else
                hi = mid;
        }
        pos = lo;
        for (int j = 0; j < nv; ++j)
            pos += cand[j] < c ? 1 : 0;
    }
    const int p0 = (int)__reduce_min_sync(FULL, (unsigned)pos);
    const int nn = min(k, cnt + nv);
    for (int b = (nn - 1) & ~31; b >= (p0 & ~31); b -= 32) {
        const int p = b + lane;
        const unsigned rel = (unsigned)(pos - b);
        const unsigned m = __reduce_or_sync(FULL, valid && rel < 32u ? 1u << rel : 0u);
        const int below = __popc(__ballot_sync(FULL, valid && pos < b)) + __popc(m & lt);
        const bool mv = p >= p0 && p < nn && !((m >> lane) & 1u);
        const unsigned long long val = mv ? L[p - below] : 0ull;
        __syncwarp();
        if (mv)
            L[p] = val;
        __syncwarp();
    }
    if (valid && pos < k)
        L[pos] = c;
    __syncwarp();
    cnt = nn;
}

// The k best of objects [begin, end) for the tile's queries (sm.q), into the lists.
// RUN: position p is object perm[p] and matches every query's tuple (chi = 0).  kth, where
// given, holds for each query the smallest k-th Gamma that any slice has reached (as
// bits): a record above it is in no final list, so every slice stops inserting what
// another one already rules out.  Every thread of the CTA calls it with the same arguments.
// until > 0 (RUN): gives up, returning false, where after PROBE objects more than half of the
// tile's queries have no k records below it.
template <class T, bool RUN>
__device__ __forceinline__ bool scan_objects(const TopkArgs &a, Smem<T> &sm,
                                             unsigned long long *lists, uint32_t begin,
                                             uint32_t end,
                                             const uint32_t *__restrict__ perm,
                                             uint32_t *kth, float until) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ty = tid / T::TX, tx = tid % T::TX;
    const int k = a.k;
    const int chunks = (a.d + DC - 1) / DC;
    const bool q16 = (a.qstride & 3) == 0 && (reinterpret_cast<uintptr_t>(a.Q) & 15) == 0;
    for (int r = tid; r < T::TQ; r += NT) {
        sm.cnt[r] = 0;
        sm.tg[r] = INF;
        sm.ti[r] = kNone;
        sm.t2[r] = sm.q[r] == kNone ? -1.f : INF;  // idle rows: no pair passes
#pragma unroll
        for (int j = 0; j < 4; ++j)
            sm.mask[r][j] = 0;
    }
    __syncthreads();

    // this thread stages 16-byte column xc of rows xr + 32 i of every object tile
    const int xr = tid >> 3, xc = (tid & 7) * 4;
    uint32_t row[4], nrow[4];  // objects of the current and the next tile (or kNone)
    auto rows_of = [&](uint32_t n0, uint32_t(&out)[4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t p = n0 + xr + 32 * i;
            out[i] = p < end ? (RUN ? perm[p] : p) : kNone;
        }
    };
    auto stage = [&](int buf, int dk, const uint32_t(&rw)[4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool ok = rw[i] != kNone && dk + xc < a.xstride;
            cp16((uint32_t)__cvta_generic_to_shared(&sm.st[buf].X[xr + 32 * i][xc]),
                 ok ? a.X + (int64_t)rw[i] * a.xstride + dk + xc : a.X, ok ? 16 : 0);
        }
        if (q16) {
            for (int e = tid; e < T::TQ * (DC / 4); e += NT) {
                const int r = e >> 3, c = (e & 7) * 4;
                const uint32_t q = sm.q[r];
                const int left = q == kNone ? 0 : min(max(a.d - dk - c, 0), 4);
                cp16((uint32_t)__cvta_generic_to_shared(&sm.st[buf].Q[r][c]),
                     left ? a.Q + (int64_t)q * a.qstride + dk + c : a.Q, 4 * left);
            }
        } else {
            for (int e = tid; e < T::TQ * DC; e += NT) {
                const int r = e >> 5, c = e & 31;
                const uint32_t q = sm.q[r];
                const bool ok = q != kNone && dk + c < a.d;
                cp4((uint32_t)__cvta_generic_to_shared(&sm.st[buf].Q[r][c]),
                    ok ? a.Q + (int64_t)q * a.qstride + dk + c : a.Q, ok ? 4 : 0);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    rows_of(begin, row);
    stage(0, 0, row);
    // thread r < TQ watches query r's entry of kth, one tile ahead
    const uint32_t *watch =
        kth != nullptr && tid < T::TQ && sm.q[tid] != kNone ? kth + sm.q[tid] : nullptr;
    uint32_t seen = ~0u;
    int buf = 0;
    bool done = true;
    for (uint32_t n0 = begin; n0 < end; n0 += TN) {  // N < 2^31: no overflow
        if (RUN && until > 0.f && n0 == begin + PROBE) {
            const bool mine = tid < T::TQ && sm.q[tid] != kNone;
            const int open = __syncthreads_count(mine && !(sm.tg[tid] < until));
            if (2 * open > __syncthreads_count(mine)) {
                done = false;
                break;
            }
        }
        rows_of(n0 + TN, nrow);
        if (watch != nullptr) {
            if (seen < __float_as_uint(sm.tg[tid])) {
                sm.tg[tid] = __uint_as_float(seen);
                sm.ti[tid] = kNone;
                sm.t2[tid] = admitted_dist2(__uint_as_float(seen), a.w);
            }
            seen = *reinterpret_cast<const volatile uint32_t *>(watch);
        }
        float acc[T::QI][T::OJ];
#pragma unroll
        for (int i = 0; i < T::QI; ++i)
#pragma unroll
            for (int j = 0; j < T::OJ; ++j)
                acc[i][j] = 0.f;
        for (int ch = 0; ch < chunks; ++ch, buf ^= 1) {
            // this chunk has arrived and every thread is done with the other buffer, which
            // takes the next chunk while this one is summed
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            if (ch + 1 < chunks)
                stage(buf ^ 1, (ch + 1) * DC, row);
            else if (n0 + TN < end)
                stage(buf ^ 1, 0, nrow);
            // four dimensions per shared-memory load; each pair still sums its squared
            // differences one dimension at a time, in dimension order
#pragma unroll 2
            for (int c = 0; c < DC; c += 4) {
                ulonglong2 q[T::QI];
#pragma unroll
                for (int i = 0; i < T::QI; ++i)
                    q[i] = *reinterpret_cast<const ulonglong2 *>(
                        &sm.st[buf].Q[ty + T::TY * i][c]);
#pragma unroll
                for (int j = 0; j < T::OJ; ++j) {
                    const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(
                        &sm.st[buf].X[tx + T::TX * j][c]);
#pragma unroll
                    for (int i = 0; i < T::QI; ++i) {
                        add_squares(acc[i][j], sub2(q[i].x, b.x));
                        add_squares(acc[i][j], sub2(q[i].y, b.y));
                    }
                }
            }
        }

        // The pairs that their query's k-th record still admits by distance alone: the
        // buffer summed last takes their distances (the next chunk goes to the other one)
        // and the warp that keeps the query's list finishes them, a lane each.
        bool any = false;
#pragma unroll
        for (int i = 0; i < T::QI; ++i) {
            const float t2 = sm.t2[ty + T::TY * i];
#pragma unroll
            for (int j = 0; j < T::OJ; ++j)
                any = any || acc[i][j] <= t2;
        }
        float(*const D2)[TN] = sm.st[buf ^ 1].D2;
        if (__syncthreads_or(any)) {
            if (__any_sync(FULL, any)) {
#pragma unroll
                for (int i = 0; i < T::QI; ++i) {
                    const int r = ty + T::TY * i;
                    const float t2 = sm.t2[r];
                    unsigned m[T::OJ];
#pragma unroll
                    for (int j = 0; j < T::OJ; ++j) {
                        const bool pass = acc[i][j] <= t2;
                        if (pass)
                            D2[r][tx + T::TX * j] = acc[i][j];
                        m[j] = __ballot_sync(FULL, pass);
                    }
                    if (T::TX == 16) {  // two rows a warp: 16 columns of each in a ballot
                        const int half = lane & 16;
#pragma unroll
                        for (int j = 0; j < T::OJ; j += 2)
                            if ((lane & 15) == j / 2)
                                sm.mask[r][j / 2] = __byte_perm(m[j] >> half, m[j + 1] >> half,
                                                                0x5410);
                    } else {  // half a row a warp
#pragma unroll
                        for (int j = 0; j < T::OJ; ++j)
                            if (lane == j)
                                sm.mask[r][(warp & 1) + 2 * j] = m[j];
                    }
                }
            }
            __syncthreads();
            // warp w keeps the lists of queries QW w .. QW w + QW - 1; a lane finishes column
            // lane of each 32, whose word (or id) it reads once for all of them
            const int r0 = warp * T::QW;
            const uint32_t mine = lane < 4 * T::QW && r0 + lane / 4 < T::TQ
                                      ? sm.mask[r0 + lane / 4][lane & 3]
                                      : 0u;
            const unsigned rows = __ballot_sync(FULL, mine != 0);
            uint32_t col[4];
            if (rows != 0) {
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const uint32_t p = n0 + 32 * w + lane;
                    col[w] = p < end ? (RUN ? perm[p] : a.attr[p]) : 0u;
                }
            }
#pragma unroll 1
            for (int i = 0; i < T::QW; ++i) {
                if (((rows >> (4 * i)) & 15u) == 0)
                    continue;
                const int r = r0 + i;
                const uint32_t q = sm.q[r];
                unsigned long long *L = lists + r * k;
                const float tg = sm.tg[r];
                const uint32_t ti = sm.ti[r];
                int cnt = sm.cnt[r];
#pragma unroll 1
                for (int w = 0; w < 4; ++w) {
                    const unsigned m = __shfl_sync(FULL, mine, 4 * i + w);
                    if (m == 0)
                        continue;
                    const uint32_t p = n0 + 32 * w + lane;
                    const uint32_t cw = w < 2 ? (w == 0 ? col[0] : col[1])
                                              : (w == 2 ? col[2] : col[3]);
                    unsigned long long c = ~0ull;
                    if (((m >> lane) & 1u) && p < end) {
                        const uint32_t id = RUN ? cw : p;
                        if (!(a.exclude_self && id == q)) {
                            const int chi = RUN ? 0 : chi_packed(sm.qa[r], cw, sm.qh[r], a.w.lo);
                            const float g =
                                fusion_gamma(__fsqrt_rn(D2[r][32 * w + lane]), chi, a.w);
                            if (g < INF && rec_less(g, id, tg, ti))
                                c = ((unsigned long long)__float_as_uint(g) << 32) | id;
                        }
                    }
                    list_merge(L, cnt, k, c, sm.cand[warp], lane);
                }
                if (lane == 0)
                    sm.cnt[r] = cnt;
                if (lane == 0 && cnt == k) {
                    const float lg = __uint_as_float((uint32_t)(L[k - 1] >> 32));
                    const uint32_t li = (uint32_t)L[k - 1];
                    if (rec_less(lg, li, tg, ti)) {
                        sm.tg[r] = lg;
                        sm.ti[r] = li;
                        sm.t2[r] = admitted_dist2(lg, a.w);
                        if (kth != nullptr)
                            atomicMin(kth + q, __float_as_uint(lg));
                    }
                }
            }
            if (mine != 0)
                sm.mask[r0 + lane / 4][lane & 3] = 0;
            __syncthreads();
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            row[i] = nrow[i];
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    return done;
}

// the final row of query q: record e is (g, id) for e < k
__device__ __forceinline__ void write_record(const TopkArgs &a, int64_t q, int e, float g,
                                             uint32_t id) {
    a.ids[q * a.k + e] = id;
    if (a.dists)
        a.dists[q * a.k + e] = g;
    if (a.chi)
        a.chi[q * a.k + e] =
            id == kNone ? (uint8_t)255
                        : (uint8_t)chi_packed(a.qattr[q], a.attr[id], a.qhi ? a.qhi[q] : a.w.hi,
                                              a.w.lo);
}

// Slices of a full scan of nq queries: about `ctas` CTAs in all, at least 8 tiles each.
__host__ __device__ inline int scan_slices(int64_t nq, int tq, int64_t N, int ctas, int max_s) {
    const int64_t tiles = (nq + tq - 1) / tq;
    int64_t s = tiles > 0 ? ctas / tiles : 1;  // whole units fit in one wave
    const int64_t by_n = (N + 8 * TN - 1) / (8 * TN);
    s = s < by_n ? s : by_n;
    s = s < max_s ? s : max_s;
    return (int)(s < 1 ? 1 : s);
}

// The queries of a full scan: all of them, or (qlist) the *qcount listed ones.
struct ScanQueries {
    const uint32_t *qlist;
    const unsigned *qcount;
    int ctas, max_s;
    uint32_t *kth;  // [queries] or null (one slice): see scan_objects
};

template <class T>
__global__ void __launch_bounds__(NT, T::CTAS) scan_kernel(TopkArgs a, ScanQueries sq,
                                                  uint32_t *__restrict__ part_id,
                                                  float *__restrict__ part_g) {
    extern __shared__ __align__(16) unsigned char smem[];
    Smem<T> &sm = *reinterpret_cast<Smem<T> *>(smem);
    unsigned long long *lists = reinterpret_cast<unsigned long long *>(smem + sizeof(Smem<T>));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t nq = sq.qlist ? (int64_t)*sq.qcount : a.nq;
    const int S = scan_slices(nq, T::TQ, a.N, sq.ctas, sq.max_s);
    const int64_t tiles = (nq + T::TQ - 1) / T::TQ;
    const int64_t per = ((a.N + S - 1) / S + TN - 1) / TN * TN;
    for (int64_t u = blockIdx.x; u < tiles * S; u += gridDim.x) {
        const int64_t t0 = u % tiles * T::TQ;
        const int split = (int)(u / tiles);
        __syncthreads();  // the previous unit's lists are written
        for (int r = tid; r < T::TQ; r += NT) {
            const int64_t i = t0 + r;
            const uint32_t q = i >= nq ? kNone : sq.qlist ? sq.qlist[i] : (uint32_t)i;
            sm.q[r] = q;
            sm.qa[r] = q != kNone ? a.qattr[q] : 0u;
            sm.qh[r] = q != kNone && a.qhi ? a.qhi[q] : a.w.hi;
        }
        __syncthreads();
        const int64_t begin = split * per;
        const int64_t end = a.N < begin + per ? a.N : begin + per;
        scan_objects<T, false>(a, sm, lists, (uint32_t)(begin < end ? begin : end),
                               (uint32_t)end, nullptr, S > 1 ? sq.kth : nullptr, 0.f);
        for (int r = warp * T::QW; r < min(warp * T::QW + T::QW, T::TQ); ++r) {
            if (sm.q[r] == kNone)
                continue;
            const int cnt = sm.cnt[r];
            for (int e = lane; e < a.k; e += 32) {
                const unsigned long long rec = e < cnt ? lists[r * a.k + e] : NO_RECORD;
                const float g = __uint_as_float((uint32_t)(rec >> 32));
                const uint32_t id = (uint32_t)rec;
                if (S == 1) {
                    write_record(a, sm.q[r], e, g, id);
                } else {
                    const int64_t o = ((t0 + r) * S + split) * (int64_t)a.k + e;
                    part_id[o] = id;
                    part_g[o] = g;
                }
            }
        }
    }
}

// k-way merge of S <= 128 sorted lists of k records (one warp; a lane holds the heads of
// lists lane, lane + 32, ...); put(e, g, id) receives the records in order.
template <class Put>
__device__ __forceinline__ void merge_lists(const uint32_t *__restrict__ id,
                                            const float *__restrict__ g, int S, int k, int lane,
                                            Put put) {
    constexpr int H = MAX_SLICES / 32;
    int head[H];
    unsigned long long cur[H];
    auto load = [&](int l, int h) -> unsigned long long {
        if (l >= S || h >= k)
            return ~0ull;
        const int64_t o = (int64_t)l * k + h;
        return ((unsigned long long)__float_as_uint(g[o]) << 32) | id[o];
    };
#pragma unroll
    for (int i = 0; i < H; ++i) {
        head[i] = 0;
        cur[i] = load(lane + 32 * i, 0);
    }
    for (int e = 0; e < k; ++e) {
        unsigned long long best = cur[0];
#pragma unroll
        for (int i = 1; i < H; ++i)
            best = cur[i] < best ? cur[i] : best;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long o = __shfl_xor_sync(FULL, best, off);
            best = o < best ? o : best;
        }
        put(e, __uint_as_float((uint32_t)(best >> 32)), (uint32_t)best);
#pragma unroll
        for (int i = 0; i < H; ++i)
            if (cur[i] == best && (uint32_t)best != kNone)
                cur[i] = load(lane + 32 * i, ++head[i]);
    }
}

__global__ void scan_merge_kernel(TopkArgs a, ScanQueries sq, int tq,
                                  const uint32_t *__restrict__ part_id,
                                  const float *__restrict__ part_g) {
    const int lane = threadIdx.x & 31;
    const int64_t nq = sq.qlist ? (int64_t)*sq.qcount : a.nq;
    const int S = scan_slices(nq, tq, a.N, sq.ctas, sq.max_s);
    if (S == 1)
        return;
    for (int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < nq;
         i += (int64_t)gridDim.x * (blockDim.x >> 5)) {
        const int64_t q = sq.qlist ? (int64_t)sq.qlist[i] : i;
        merge_lists(part_id + i * S * a.k, part_g + i * S * a.k, S, a.k, lane,
                    [&](int e, float g, uint32_t id) {
                        if (lane == 0)
                            write_record(a, q, e, g, id);
                    });
    }
}

// ---------------------------------------------------------------- tuple runs
// Planning: the queries' words, the run of each, and the queries grouped by run.  A table
// of T >= 2 nq entries, keyed by the run's start, counts each group; one query of each
// group then claims the group's place among the groups, units (query tile x slice of the
// run), query slots and list rows in single additions.
struct RunHeader {
    unsigned long long groups_units;  // see plan_claim
    unsigned long long asked, list_rows;  // of the lists: asked for, handed out
    unsigned slots, left, next;
};
struct RunGroup {
    uint32_t lo, len, base, cnt;  // the run, the group's slots
    unsigned long long ubase, lbase;
    int slices;  // of the run; 1: no lists, the unit writes the final rows
    uint32_t pad;
};
struct RunPlan {
    RunHeader *hdr;
    uint32_t *key, *tcnt, *tgroup;  // [T] run start + 1, queries, group
    uint32_t tmask;
    uint32_t *lo, *len, *home, *rank;  // [nq]; len with GIVEN_UP where the run was given up
    uint32_t *slot;                    // [nq] queries in group order
    RunGroup *group;                   // [nq]
    uint32_t *left;                    // [nq] queries for the full scan
    uint32_t *part_id;                 // [rows][k]
    float *part_g;
    int64_t rows;
    const uint32_t *attr_sorted, *id_sorted;
    const uint8_t *codes;  // query attributes, or null: the words are given
    uint32_t *words;
    int tq, slice;  // queries per unit, objects per slice aimed at
    int busy;       // tiles of queries that fill the chip
    bool scarce;    // the runs may ask for more list rows than there are
};

__device__ __forceinline__ int64_t lower_bound_word(const uint32_t *a, int64_t n, uint32_t x) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (a[mid] < x)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

// returns the list rows that the query's run would take
__device__ __forceinline__ unsigned plan_lookup(const TopkArgs &a, const RunPlan &p, int64_t q) {
    uint32_t word, hi;
    if (p.codes != nullptr) {
        word = pack_query_word(p.codes + q * a.w.m, a.w, &hi);
        p.words[q] = word;
    } else {
        word = a.qattr[q];
    }
    const int64_t l = lower_bound_word(p.attr_sorted, a.N, word);
    const int64_t h =
        word == 0xFFFFFFFFu ? a.N : lower_bound_word(p.attr_sorted, a.N, word + 1u);
    p.lo[q] = (uint32_t)l;
    p.len[q] = (uint32_t)(h - l);
    if (h == l)
        return 0;
    uint32_t s = table_slot((uint32_t)l, p.tmask);
    for (uint32_t probe = 0; probe <= p.tmask; ++probe) {  // half empty: ends
        // a key stays once it is set, so only an empty slot needs the exchange; few queries
        // hardly meet one another's, and save the read's latency
        uint32_t x =
            a.nq <= 64 ? 0u : *reinterpret_cast<const volatile uint32_t *>(&p.key[s]);
        if (x == 0u)
            x = atomicCAS(&p.key[s], 0u, (uint32_t)l + 1u);
        if (x == 0u || x == (uint32_t)l + 1u)
            break;
        s = (s + 1) & p.tmask;
    }
    p.home[q] = s;
    p.rank[q] = atomicAdd(&p.tcnt[s], 1u);
    const unsigned want = (unsigned)run_slices(h - l, p.slice);
    return want > 1 ? want : 0;
}

// adds up what a warp's queries ask for
__device__ __forceinline__ void plan_ask(const RunPlan &p, unsigned mine) {
    if (!p.scarce)
        return;
    const unsigned sum = __reduce_add_sync(FULL, mine);
    if ((threadIdx.x & 31) == 0 && sum > 0)
        atomicAdd(&p.hdr->asked, (unsigned long long)sum);
}

__device__ __forceinline__ void plan_group(const RunPlan &p, int64_t q) {
    if (p.len[q] == 0 || p.rank[q] != 0)
        return;
    RunGroup g;
    g.lo = p.lo[q];
    g.len = p.len[q];
    g.cnt = p.tcnt[p.home[q]];
    g.base = atomicAdd(&p.hdr->slots, g.cnt);
    const int64_t tiles = (g.cnt + p.tq - 1) / p.tq;
    const int64_t s =
        granted_slices(run_slices(g.len, p.slice), tiles,
                       p.scarce ? *reinterpret_cast<const volatile unsigned long long *>(
                                      &p.hdr->asked)
                                : 0ull,
                       p.rows, p.busy);
    g.lbase = s > 1 ? atomicAdd(&p.hdr->list_rows, (unsigned long long)g.cnt * s) : 0;
    g.slices = (int)s;
    const unsigned long long units = (unsigned long long)tiles * s;
    const unsigned long long at = atomicAdd(&p.hdr->groups_units, plan_claim(units));
    g.ubase = claimed_units(at);
    g.pad = 0;
    const uint32_t gi = (uint32_t)claimed_groups(at);
    p.group[gi] = g;
    p.tgroup[p.home[q]] = gi;
}

__device__ __forceinline__ void plan_slot(const RunPlan &p, int64_t q) {
    if (p.len[q] != 0)
        p.slot[p.group[p.tgroup[p.home[q]]].base + p.rank[q]] = (uint32_t)q;
}

__global__ void run_lookup_kernel(TopkArgs a, RunPlan p) {
    unsigned asked = 0;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < a.nq;
         q += (int64_t)gridDim.x * blockDim.x)
        asked += plan_lookup(a, p, q);
    plan_ask(p, asked);
}
__global__ void run_group_kernel(TopkArgs a, RunPlan p) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < a.nq;
         q += (int64_t)gridDim.x * blockDim.x)
        plan_group(p, q);
}
__global__ void run_slot_kernel(TopkArgs a, RunPlan p) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < a.nq;
         q += (int64_t)gridDim.x * blockDim.x)
        plan_slot(p, q);
}
// the whole plan in one block (small batches: one launch instead of four)
__global__ void __launch_bounds__(1024) run_plan_kernel(TopkArgs a, RunPlan p) {
    if (threadIdx.x == 0)
        *p.hdr = RunHeader{};
    for (uint32_t t = threadIdx.x; t <= p.tmask; t += blockDim.x)
        p.key[t] = p.tcnt[t] = 0u;
    __syncthreads();
    unsigned asked = 0;
    for (int64_t q = threadIdx.x; q < a.nq; q += blockDim.x)
        asked += plan_lookup(a, p, q);
    plan_ask(p, asked);
    __syncthreads();
    for (int64_t q = threadIdx.x; q < a.nq; q += blockDim.x)
        plan_group(p, q);
    __syncthreads();
    for (int64_t q = threadIdx.x; q < a.nq; q += blockDim.x)
        plan_slot(p, q);
}

// Units of the plan, taken from a counter (runs differ in length by orders of magnitude).
// Under constant weights a run of more than a quarter of all objects is judged early: where
// omega_l does not exceed the vector term, the scan answers its queries anyway, and the run
// would have cost up to as much again (candidate sets of 30,000 objects of two tuples,
// w_l = 0.01: 18.5 ms, judged 12.9; the scan alone 11.4).  A run of all objects needs no
// scan afterwards (one tuple: 21.6 ms, now 10.5).
template <class T>
__global__ void __launch_bounds__(NT, T::CTAS) run_kernel(TopkArgs a, RunPlan p) {
    extern __shared__ __align__(16) unsigned char smem[];
    Smem<T> &sm = *reinterpret_cast<Smem<T> *>(smem);
    unsigned long long *lists = reinterpret_cast<unsigned long long *>(smem + sizeof(Smem<T>));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned long long gu = p.hdr->groups_units;
    const int64_t groups = (int64_t)claimed_groups(gu);
    const int64_t units = (int64_t)claimed_units(gu);
    for (;;) {
        __syncthreads();  // the previous unit's lists are written
        if (tid == 0)
            sm.unit = (int)atomicAdd(&p.hdr->next, 1u);
        __syncthreads();
        const int64_t u = (int64_t)(unsigned)sm.unit;
        if (u >= units)
            return;
        int64_t l = 0, h = groups;  // the last group with ubase <= u
        while (h - l > 1) {
            const int64_t mid = (l + h) >> 1;
            if ((int64_t)p.group[mid].ubase <= u)
                l = mid;
            else
                h = mid;
        }
        const RunGroup g = p.group[l];
        const int v = (int)(u - (int64_t)g.ubase);
        const int tile = v / g.slices, split = v % g.slices;
        const float until = a.w.mode == NHQ_W_CONSTANT && g.len < a.N && g.len > a.N / 4
                                ? fusion_gamma(0.f, 1, a.w)
                                : 0.f;
        bool wanted = until == 0.f;
        for (int r = tid; r < T::TQ; r += NT) {
            const uint32_t i = (uint32_t)tile * T::TQ + r;
            const uint32_t q = i < g.cnt ? p.slot[g.base + i] : kNone;
            sm.q[r] = q;
            wanted = wanted ||
                     (q != kNone &&
                      (*reinterpret_cast<const volatile uint32_t *>(p.len + q) & GIVEN_UP) == 0u);
        }
        if (!__syncthreads_or(wanted))
            continue;  // another slice has given up for all of them
        const int64_t per = (((int64_t)g.len + g.slices - 1) / g.slices + TN - 1) / TN * TN;
        const int64_t run_end = (int64_t)g.lo + g.len;
        int64_t begin = (int64_t)g.lo + split * per;
        begin = begin < run_end ? begin : run_end;
        const int64_t end = begin + per < run_end ? begin + per : run_end;
        if (!scan_objects<T, true>(a, sm, lists, (uint32_t)begin, (uint32_t)end, p.id_sorted,
                                   nullptr, until)) {
            for (int r = tid; r < T::TQ; r += NT)
                if (sm.q[r] != kNone && (atomicOr(p.len + sm.q[r], GIVEN_UP) & GIVEN_UP) == 0u)
                    p.left[atomicAdd(&p.hdr->left, 1u)] = sm.q[r];
            continue;
        }
        for (int r = warp * T::QW; r < min(warp * T::QW + T::QW, T::TQ); ++r) {
            if (sm.q[r] == kNone)
                continue;
            const int cnt = sm.cnt[r];
            const uint32_t in_group = (uint32_t)tile * T::TQ + r;
            const int64_t o = ((int64_t)g.lbase + (int64_t)in_group * g.slices + split) * a.k;
            for (int e = lane; e < a.k; e += 32) {
                const unsigned long long rec = e < cnt ? lists[r * a.k + e] : NO_RECORD;
                const float gm = __uint_as_float((uint32_t)(rec >> 32));
                if (g.slices > 1) {
                    p.part_id[o + e] = (uint32_t)rec;
                    p.part_g[o + e] = gm;
                } else {
                    write_record(a, sm.q[r], e, gm, (uint32_t)rec);
                }
            }
            if (g.slices > 1)
                continue;
            if (lane == 0 && a.w.mode != NHQ_W_FILTER && g.len < a.N &&
                !(cnt == a.k && __uint_as_float((uint32_t)(lists[r * a.k + a.k - 1] >> 32)) <
                                       fusion_gamma(0.f, 1, a.w)))
                p.left[atomicAdd(&p.hdr->left, 1u)] = sm.q[r];
        }
    }
}

// Final rows of the queries whose run took several slices or is empty.
__global__ void run_merge_kernel(TopkArgs a, RunPlan p) {
    const int lane = threadIdx.x & 31;
    for (int64_t q = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); q < a.nq;
         q += (int64_t)gridDim.x * (blockDim.x >> 5)) {
        float last = INF;
        const uint32_t len = p.len[q];
        if (len & GIVEN_UP)
            continue;
        if (len == 0) {
            for (int e = lane; e < a.k; e += 32)
                write_record(a, q, e, INF, kNone);
        } else {
            const RunGroup &g = p.group[p.tgroup[p.home[q]]];
            const int S = g.slices;
            if (S == 1)
                continue;
            const int64_t o = ((int64_t)g.lbase + (int64_t)p.rank[q] * S) * a.k;
            merge_lists(p.part_id + o, p.part_g + o, S, a.k, lane,
                        [&](int e, float gm, uint32_t id) {
                            if (lane == 0)
                                write_record(a, q, e, gm, id);
                            last = gm;
                        });
        }
        if (lane == 0 && a.w.mode != NHQ_W_FILTER && len < a.N && !(last < fusion_gamma(0.f, 1, a.w)))
            p.left[atomicAdd(&p.hdr->left, 1u)] = (uint32_t)q;
    }
}

// CTAs of shape T that the chip holds at once
template <class T>
int resident_ctas(int k, int sm_count) {
    int n = (int)((size_t)227 * 1024 / (tile_smem<T>(k) + 1024));
    n = n < 1 ? 1 : n > T::CTAS ? T::CTAS : n;
    return n * sm_count;
}

template <class T>
cudaError_t launch_scan(const TopkArgs &a, const ScanQueries &sq, int sm_count, uint32_t *pid,
                        float *pg, cudaStream_t s) {
    const size_t smem = tile_smem<T>(a.k);
    cudaError_t e = cudaFuncSetAttribute(scan_kernel<T>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return e;
    const int S = scan_slices(a.nq, T::TQ, a.N, sq.ctas, sq.max_s);
    if (sq.kth != nullptr &&
        (e = cudaMemsetAsync(sq.kth, 0xFF, sizeof(uint32_t) * (size_t)a.nq, s)) != cudaSuccess)
        return e;
    int64_t units = (a.nq + T::TQ - 1) / T::TQ * S;
    if (sq.qlist != nullptr)  // fewer queries take more slices: as many CTAs in all
        units = units > sq.ctas ? units : sq.ctas;
    scan_kernel<T><<<(unsigned)(units > 0x7FFFFFFF ? 0x7FFFFFFF : units), NT, smem, s>>>(a, sq, pid,
                                                                                       pg);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    if (S > 1 || sq.qlist != nullptr) {
        const int64_t blocks = (a.nq + 7) / 8;
        const int64_t most = sq.qlist != nullptr ? 4 * (int64_t)sm_count : 0x7FFFFFFF;
        scan_merge_kernel<<<(unsigned)(blocks < most ? blocks : most), 256, 0, s>>>(a, sq, T::TQ,
                                                                                  pid, pg);
        e = cudaGetLastError();
    }
    return e;
}

// Which tile a full scan takes, and its slices.  Up to 8 queries the scan is bound by
// reading the objects, and tiles of 4 queries leave the fewest idle pairs; beyond, tiles of
// 32.  300,000 objects, d = 96, k = 10, tiles of 4 | 32: 4 queries 113 | 243 us, 8 121 | 250,
// 16 155 | 259, 32 230 | 268, so the line could lie higher.  (Tiles of 64 queries, 4 x 8 pairs a thread, read shared memory less per pair but fit
// two CTAs an SM: 53.2 ms against 44.8 ms for the candidate sets of 60,000 objects.)
struct ScanPlan {
    int shape;  // queries per tile: 4 or 32
    ScanQueries sq;
};

ScanPlan plan_scan(int64_t nq, int k, int sm_count) {
    ScanPlan p;
    p.sq.qlist = nullptr;
    p.sq.qcount = nullptr;
    p.sq.kth = nullptr;
    p.sq.max_s = MAX_SLICES;
    if (nq <= 8) {
        p.shape = Narrow::TQ;
        p.sq.ctas = resident_ctas<Narrow>(k, sm_count);
    } else {
        p.shape = Mid::TQ;
        p.sq.ctas = resident_ctas<Mid>(k, sm_count);
    }
    return p;
}

// List rows of a scan of nq queries, or (counted) of at most nq: t tiles that take slices
// make at most ctas units of a tile's rows.
int64_t scan_rows(const ScanPlan &p, int64_t nq, int64_t N, bool counted) {
    if (counted)
        return (int64_t)p.sq.ctas * p.shape;
    const int S = scan_slices(nq, p.shape, N, p.sq.ctas, p.sq.max_s);
    return S > 1 ? nq * S : 0;
}

cudaError_t run_scan(const TopkArgs &a, const ScanPlan &p, int sm_count, uint32_t *pid, float *pg,
                     cudaStream_t s) {
    return p.shape == Narrow::TQ ? launch_scan<Narrow>(a, p.sq, sm_count, pid, pg, s)
                                 : launch_scan<Mid>(a, p.sq, sm_count, pid, pg, s);
}

constexpr size_t REC = sizeof(uint32_t) + sizeof(float);

}  // namespace

// scratch of a scan with lists: kth [nq], then the lists' ids and Gammas
size_t kth_bytes(int64_t nq) { return (sizeof(uint32_t) * (size_t)nq + 255) & ~(size_t)255; }

size_t topk_scratch_bytes(const TopkArgs &a, int sm_count) {
    const size_t rows = (size_t)scan_rows(plan_scan(a.nq, a.k, sm_count), a.nq, a.N, false);
    return rows > 0 ? kth_bytes(a.nq) + rows * a.k * REC : 0;
}

// Takes as many slices as the scratch has room for (none: one slice).
cudaError_t launch_topk(const TopkArgs &a, void *scratch, size_t scratch_bytes, int sm_count,
                        cudaStream_t s) {
    if (a.nq <= 0)
        return cudaSuccess;
    ScanPlan p = plan_scan(a.nq, a.k, sm_count);
    const size_t kb = kth_bytes(a.nq);
    const size_t room =
        scratch && scratch_bytes > kb ? (scratch_bytes - kb) / ((size_t)a.nq * a.k * REC) : 0;
    p.sq.max_s = room < 1 ? 1 : room < MAX_SLICES ? (int)room : MAX_SLICES;
    const size_t rows = (size_t)scan_rows(p, a.nq, a.N, false);
    // Short slices under the filter weighting seldom fill a list, so they share nothing, and
    // clearing kth first is a launch (100 queries over 10,000 objects 96 -> 93 us; other
    // weightings gain by sharing: 100 over 100,000 take 218 us, 234 without).
    const int S = scan_slices(a.nq, p.shape, a.N, p.sq.ctas, p.sq.max_s);
    if (rows > 0 && !(a.w.mode == NHQ_W_FILTER && (a.N + S - 1) / S <= 16 * TN))
        p.sq.kth = reinterpret_cast<uint32_t *>(scratch);
    uint32_t *pid = reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(scratch) + kb);
    return run_scan(a, p, sm_count, pid, reinterpret_cast<float *>(pid + rows * a.k), s);
}

// ---- the run path: its scratch is one block, laid out by run_layout ----
namespace {

struct RunLayout {
    size_t table, words, query, slot, group, left, part, kth, scan, bytes;
    uint32_t tmask;
    int64_t rows, srows;
};

RunLayout run_layout(const TopkArgs &a, int sm_count) {
    RunLayout L;
    uint64_t T = 64;
    while (T < 2 * (uint64_t)a.nq)
        T <<= 1;
    L.tmask = (uint32_t)(T - 1);
    L.rows = run_list_rows(a.nq, a.N, a.k, sm_count);
    L.srows = a.w.mode == NHQ_W_FILTER
                  ? 0
                  : scan_rows(plan_scan(a.nq, a.k, sm_count), a.nq, a.N, true);
    size_t off = 256;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off += (bytes + 255) & ~(size_t)255;
        return at;
    };
    L.table = take(3 * sizeof(uint32_t) * (size_t)T);
    L.words = take(sizeof(uint32_t) * (size_t)a.nq);
    L.query = take(4 * sizeof(uint32_t) * (size_t)a.nq);
    L.slot = take(sizeof(uint32_t) * (size_t)a.nq);
    L.group = take(sizeof(RunGroup) * (size_t)a.nq);
    L.left = take(sizeof(uint32_t) * (size_t)a.nq);
    L.part = take(REC * (size_t)L.rows * a.k);
    L.kth = take(kth_bytes(L.srows > 0 ? a.nq : 0));
    L.scan = take(REC * (size_t)L.srows * a.k);
    L.bytes = off;
    return L;
}

template <class T>
cudaError_t launch_runs(const TopkArgs &a, const RunPlan &p, int ctas, cudaStream_t s) {
    const size_t smem = tile_smem<T>(a.k);
    cudaError_t e = cudaFuncSetAttribute(run_kernel<T>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return e;
    run_kernel<T><<<(unsigned)ctas, NT, smem, s>>>(a, p);
    return cudaGetLastError();
}

}  // namespace

bool topk_runs_apply(const TopkArgs &a) {
    return a.nq < (int64_t(1) << 30) && a.qhi == nullptr && a.w.wild == 0 &&
           (a.w.mode == NHQ_W_FILTER || (a.w.mode == NHQ_W_CONSTANT && a.w.wl > 0.f));
}

size_t topk_runs_scratch_bytes(const TopkArgs &a, int sm_count) {
    return run_layout(a, sm_count).bytes;
}

// codes: the queries' attribute codes [nq][m] (packed here), or null when a.qattr holds
// their words already.
cudaError_t launch_topk_runs(const TopkArgs &args, const uint8_t *codes,
                             const uint32_t *attr_sorted, const uint32_t *id_sorted,
                             void *scratch, size_t scratch_bytes, int sm_count, cudaStream_t s) {
    TopkArgs a = args;
    if (a.nq <= 0)
        return cudaSuccess;
    const RunLayout L = run_layout(a, sm_count);
    if (scratch == nullptr || scratch_bytes < L.bytes)
        return cudaErrorInvalidValue;
    char *base = reinterpret_cast<char *>(scratch);
    RunPlan p;
    const size_t T = (size_t)L.tmask + 1;
    p.hdr = reinterpret_cast<RunHeader *>(base);
    p.key = reinterpret_cast<uint32_t *>(base + L.table);
    p.tcnt = p.key + T;
    p.tgroup = p.tcnt + T;
    p.tmask = L.tmask;
    p.words = reinterpret_cast<uint32_t *>(base + L.words);
    p.lo = reinterpret_cast<uint32_t *>(base + L.query);
    p.len = p.lo + a.nq;
    p.home = p.len + a.nq;
    p.rank = p.home + a.nq;
    p.slot = reinterpret_cast<uint32_t *>(base + L.slot);
    p.group = reinterpret_cast<RunGroup *>(base + L.group);
    p.left = reinterpret_cast<uint32_t *>(base + L.left);
    p.rows = L.rows;
    p.part_id = reinterpret_cast<uint32_t *>(base + L.part);
    p.part_g = reinterpret_cast<float *>(p.part_id + (size_t)L.rows * a.k);
    p.attr_sorted = attr_sorted;
    p.id_sorted = id_sorted;
    p.codes = codes;
    if (codes != nullptr)
        a.qattr = p.words;
    // Few queries hardly share tuples: tiles of 4.  A million objects of 600 even tuples, d =
    // 128, k = 10, tiles of 4 | 32: 8 queries 44 | 73 us, 64 54 | 85, 256 115 | 209, so the line
    // could lie higher.
    const bool few = a.nq <= 64;
    p.tq = few ? Narrow::TQ : Mid::TQ;
    p.slice = run_slice_length(a.nq);
    const int ctas = few ? resident_ctas<Narrow>(a.k, sm_count) : resident_ctas<Mid>(a.k, sm_count);
    p.busy = 2 * ctas;
    p.scarce = a.nq * run_slices(a.N, p.slice) > L.rows && L.rows > 0;
    cudaError_t e;
    if (a.nq <= 2048) {
        run_plan_kernel<<<1, a.nq <= 256 ? 256 : 1024, 0, s>>>(a, p);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return e;
    } else {
        if ((e = cudaMemsetAsync(base, 0, L.table + 2 * sizeof(uint32_t) * T, s)) != cudaSuccess)
            return e;
        const int64_t b = (a.nq + 127) / 128;
        const unsigned grid = (unsigned)(b < 65536 ? b : 65536);
        run_lookup_kernel<<<grid, 128, 0, s>>>(a, p);
        run_group_kernel<<<grid, 128, 0, s>>>(a, p);
        run_slot_kernel<<<grid, 128, 0, s>>>(a, p);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return e;
    }
    e = few ? launch_runs<Narrow>(a, p, ctas, s) : launch_runs<Mid>(a, p, ctas, s);
    if (e != cudaSuccess)
        return e;
    const int64_t mb = (a.nq + 7) / 8;
    run_merge_kernel<<<(unsigned)(mb < 65536 ? mb : 65536), 256, 0, s>>>(a, p);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    if (a.w.mode == NHQ_W_FILTER)
        return cudaSuccess;
    ScanPlan sp = plan_scan(a.nq, a.k, sm_count);
    sp.sq.qlist = p.left;
    sp.sq.qcount = &p.hdr->left;
    sp.sq.kth = reinterpret_cast<uint32_t *>(base + L.kth);
    uint32_t *pid = reinterpret_cast<uint32_t *>(base + L.scan);
    return run_scan(a, sp, sm_count, pid, reinterpret_cast<float *>(pid + (size_t)L.srows * a.k),
                    s);
}

}  // namespace nhq

// ---------------------------------------------------------------------------
// Allocation-free variant of the brute-force top-k (nhq_brute_force_noalloc).
//
// Some callers cannot allocate device memory when they call the library: code
// that runs under a memory budget owned by another allocator (a framework's
// caching pool, an embedded or real-time service that reserves all memory at
// start-up), or code that must not touch the allocator on its hot path.  For
// them the split path's only scratch -- the per-slice sorted lists that
// scan_kernel writes and scan_merge_kernel reads -- lives in the
// file-scope array below.  It is kNoAllocScratchBytes (16 MiB) of device memory
// on every GPU where this module is loaded, and stays there until the process
// exits.  Under CUDA's lazy module loading that happens on a device's first use
// of this file's code, possibly the first nhq_brute_force_noalloc call itself
// (its cudaGetSymbolAddress), so callers make a first call (Q = 0 suffices) at
// start-up, before their own allocator reserves the device's memory and before
// any stream capture.  Every call
// on a device shares it: each call fully rewrites the entries it later reads,
// so nothing has to start at zero, but calls whose kernels overlap on the GPU
// (different streams, or different host threads) race on it.
// ---------------------------------------------------------------------------
namespace nhq {

constexpr size_t kNoAllocScratchBytes = size_t(16) << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

namespace {

// The batches this entry point takes: those whose lists fit the array with tiles of 32
// queries, at most 32 slices of at least 1,024 objects, and about two CTAs per SM.  (The
// scan itself takes as many slices as the array has room for.)
size_t noalloc_list_bytes(const TopkArgs &a, int sm_count) {
    const int64_t tiles = (a.nq + 31) / 32;
    int64_t S = (2 * (int64_t)sm_count + tiles - 1) / tiles;
    const int64_t by_n = (a.N + 8 * TN - 1) / (8 * TN);
    S = S < by_n ? S : by_n;
    S = S < 32 ? S : 32;
    return S <= 1 ? 0 : (size_t)a.nq * S * a.k * (sizeof(uint32_t) + sizeof(float));
}

struct NoAllocDevice {
    bool ready = false;
    void *scratch = nullptr;  // device address of g_noalloc_scratch on this device
    int sm_count = 0;
};
constexpr int kNoAllocMaxDevices = 64;
NoAllocDevice g_noalloc_devices[kNoAllocMaxDevices];
std::mutex g_noalloc_mu;

bool is_device_pointer(const void *p) {
    cudaPointerAttributes at;
    if (p == nullptr || cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

// Per-device set-up, done by the first call on the current device.  In host code
// g_noalloc_scratch names a host-side shadow, not device memory, so the device
// address is looked up with cudaGetSymbolAddress while this device is current.
nhq_status noalloc_setup(NoAllocDevice **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return report_error(NHQ_ERR_CUDA, cudaGetErrorString(e));
    if (dev < 0 || dev >= kNoAllocMaxDevices)
        return report_error(NHQ_ERR_ARG, "nhq_brute_force_noalloc: device ordinal above 63");
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    NoAllocDevice &d = g_noalloc_devices[dev];
    if (!d.ready) {
        void *ptr = nullptr;
        if ((e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch)) != cudaSuccess)
            return report_error(NHQ_ERR_CUDA, cudaGetErrorString(e));
        int sms = 0;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) !=
            cudaSuccess)
            return report_error(NHQ_ERR_CUDA, cudaGetErrorString(e));
        d.scratch = ptr;
        d.sm_count = sms;
        d.ready = true;
    }
    *out = &d;
    return NHQ_OK;
}

}  // namespace

}  // namespace nhq

extern "C" nhq_status nhq_brute_force_noalloc(const float *vectors,
                                              const uint32_t *packed_attributes, int64_t N,
                                              int32_t d, int32_t m, const float *queries,
                                              const uint32_t *packed_query_attributes,
                                              int64_t Q, int32_t k, nhq_weights w, uint32_t *ids,
                                              float *dists, uint8_t *chi, void *stream) {
    using namespace nhq;
    if (N < 1 || N > 0x7FFFFFFE || d < 1 || m < 1 || m > 4 || Q < 0 || k < 1 || k > kMaxK)
        return report_error(NHQ_ERR_ARG, "nhq_brute_force_noalloc: need N >= 1, d >= 1, m in "
                                         "1..4, Q >= 0, k in 1..256");
    if (d % 4 != 0)
        return report_error(NHQ_ERR_ARG, "nhq_brute_force_noalloc: d must be a multiple of 4");
    nhq_status st = validate_weights(w, true);  // the rules of nhq_brute_force
    if (st != NHQ_OK)
        return st;
    // the per-device set-up runs first, so that a call with Q = 0 can make it at start-up
    NoAllocDevice *dv = nullptr;
    if ((st = noalloc_setup(&dv)) != NHQ_OK)
        return st;
    if (Q == 0)
        return NHQ_OK;
    if (!is_device_pointer(vectors) || !is_device_pointer(packed_attributes) ||
        !is_device_pointer(queries) || !is_device_pointer(packed_query_attributes) ||
        !is_device_pointer(ids) || (dists && !is_device_pointer(dists)) ||
        (chi && !is_device_pointer(chi)))
        return report_error(NHQ_ERR_ARG, "nhq_brute_force_noalloc: every array must be device "
                                         "memory (NULL allowed for dists and chi)");
    if ((reinterpret_cast<uintptr_t>(vectors) & 15) != 0)
        return report_error(NHQ_ERR_ARG, "nhq_brute_force_noalloc: vectors must be 16-byte "
                                         "aligned");
    TopkArgs a;
    a.X = vectors;
    a.xstride = d;
    a.d = d;
    a.N = N;
    a.attr = packed_attributes;
    a.Q = queries;
    a.qstride = d;
    a.qattr = packed_query_attributes;
    a.qhi = nullptr;
    a.nq = Q;
    a.k = k;
    a.exclude_self = 0;
    a.w = make_fusion(w, m);
    a.ids = ids;
    a.dists = dists;
    a.chi = chi;
    const size_t need = noalloc_list_bytes(a, dv->sm_count);
    if (need > kNoAllocScratchBytes) {
        char msg[256];
        snprintf(msg, sizeof(msg),
                 "nhq_brute_force_noalloc: Q = %lld, k = %d needs %zu scratch bytes, above the "
                 "fixed %zu (use nhq_brute_force, or fewer queries per call)",
                 (long long)Q, k, need, kNoAllocScratchBytes);
        return report_error(NHQ_ERR_ARG, msg);
    }
    cudaError_t e = launch_topk(a, dv->scratch, kNoAllocScratchBytes, dv->sm_count,
                                reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess)
        return report_error(NHQ_ERR_CUDA, cudaGetErrorString(e));
    return NHQ_OK;
}
