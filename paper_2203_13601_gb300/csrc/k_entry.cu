// k_entry.cu -- where a search enters the graph (a project addition: the paper draws
// the seed set B of Alg. 2 at random, and the library's attribute-entry rule takes
// evenly spaced members of the query's tuple, which for a frequent tuple lie all over
// the vector space).
//
// Coarse cells.  E centroids are the objects floor(j N / E); every object belongs to
// the cell of its nearest centroid by (delta, j) (the brute-force top-1 over the E
// centroid rows, plain L2).  The objects are also sorted by (attribute word, cell) with
// ascending ids inside, so the members of a tuple within one cell form one run.
//
// Entry rule for a query whose tuple has members P (closed queries): S = min(ef, 32, |P|);
// B = the first S members of P in the query's chosen cells (best cell first, ascending
// ids within a cell), then, while fewer than S, the evenly spaced P[floor(j |P| / S2)],
// j < S2 = S - |B|; |P| = 0 takes the random stream of NHQ_SEED_RANDOM.  The chosen
// cells are the T nearest centroids (NHQ_SEED_CELL_NEAREST) or the T best-scored cells
// of the entry model (NHQ_SEED_CELL_LEARNED).
//
// Entry model: a 2-layer perceptron, q (d values) -> x = s q -> 64 ReLU units -> E cell
// logits, fp16 weights and f32 accumulation at inference, f32 master weights for
// training (softmax cross-entropy against the cell of each training query's answer,
// Adam).  Parameters, one flat f32 vector: s | W1 [d][64] | b1 [64] | W2 [64][E] | b2 [E].
//
// Both cell rules score every cell of every query of the batch with one register-tiled
// dense kernel (64 x 64 output tiles, k ascending per output in one fma chain, so the
// seed pass and nhq_entry_forward produce the same bits): the learned rule runs the two
// layers, the nearest rule scores q.c - |c|^2 / 2 against the transposed centroids (the
// largest score is the nearest centroid; every product and sum is exact for integer
// components, where the order equals the (delta, cell) order).  A warp per query then
// takes the T best scores (ties to the smaller cell) and assembles the seeds.
#include <cub/cub.cuh>

#include "nhq_internal.cuh"

namespace nhq {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int EH = NHQ_ENTRY_HIDDEN;

struct EntryLayout {
    int64_t oW1, oB1, oW2, oB2, total;
};
__host__ __device__ inline EntryLayout entry_layout(int d, int E) {
    EntryLayout L;
    L.oW1 = 1;
    L.oB1 = L.oW1 + (int64_t)d * EH;
    L.oW2 = L.oB1 + EH;
    L.oB2 = L.oW2 + (int64_t)EH * E;
    L.total = L.oB2 + E;
    return L;
}

__global__ void gather_centroids_kernel(const float *__restrict__ X, int xstride, int64_t N,
                                        int E, const uint32_t *__restrict__ attr,
                                        float *__restrict__ cent, uint32_t *__restrict__ cattr) {
    const int j = blockIdx.x;
    const int64_t src = (int64_t)j * N / E;
    for (int i = threadIdx.x; i < xstride; i += blockDim.x)
        cent[(int64_t)j * xstride + i] = X[src * xstride + i];
    if (threadIdx.x == 0)
        cattr[j] = attr[src];
}

__global__ void cell_key_kernel(const uint32_t *__restrict__ attr, const uint32_t *__restrict__ cell,
                                int64_t N, unsigned long long *__restrict__ key,
                                uint32_t *__restrict__ iota) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < N;
         v += (int64_t)gridDim.x * blockDim.x) {
        key[v] = ((unsigned long long)attr[v] << 16) | cell[v];
        iota[v] = (uint32_t)v;
    }
}

__device__ __forceinline__ int64_t lower_bound_u64(const unsigned long long *a, int64_t n,
                                                   unsigned long long x) {
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

__device__ __forceinline__ int64_t lower_bound_u32(const uint32_t *a, int64_t n, uint32_t x) {
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

// ---- inference: Y[n][M] = act(s A[n][K] B[K][M] + bias[M]), k ascending per output ----
__device__ __forceinline__ float as_f32(float v) { return v; }
__device__ __forceinline__ float as_f32(__half v) { return __half2float(v); }

template <typename BT>
__global__ void __launch_bounds__(256) dense_kernel(const float *__restrict__ A, int64_t n, int K,
                                                    int64_t lda, const BT *__restrict__ B,
                                                    const BT *__restrict__ bias, int M,
                                                    const float *__restrict__ scale_ptr,
                                                    int relu, float *__restrict__ Y) {
    __shared__ float As[32][65];  // [k][row], padded: the tile loads are free of conflicts
    __shared__ float Bs[32][64];  // [k][col]
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t row0 = (int64_t)blockIdx.x * 64;
    const int col0 = blockIdx.y * 64;
    const float sc = scale_ptr != nullptr ? *scale_ptr : 1.f;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            acc[i][j] = 0.f;
    for (int k0 = 0; k0 < K; k0 += 32) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = (tid >> 5) + 8 * i, kk = tid & 31;
            const int64_t gr = row0 + r;
            const int gk = k0 + kk;
            As[kk][r] = (gr < n && gk < K) ? __fmul_rn(sc, A[gr * lda + gk]) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int kk = (tid >> 6) + 4 * i, c = tid & 63;
            const int gk = k0 + kk, gc = col0 + c;
            Bs[kk][c] = (gk < K && gc < M) ? as_f32(B[(int64_t)gk * M + gc]) : 0.f;
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < 32; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[i] = As[kk][ty * 4 + i];
                b[i] = Bs[kk][tx * 4 + i];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t r = row0 + ty * 4 + i;
        if (r >= n)
            continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = col0 + tx * 4 + j;
            if (c >= M)
                continue;
            float v = __fadd_rn(acc[i][j], as_f32(bias[c]));
            if (relu)
                v = fmaxf(v, 0.f);
            Y[r * M + c] = v;
        }
    }
}

template <typename BT>
cudaError_t launch_dense(const float *A, int64_t n, int K, int64_t lda, const BT *B,
                         const BT *bias, int M, const float *scale_ptr, int relu, float *Y,
                         cudaStream_t s) {
    if (n <= 0)
        return cudaSuccess;
    const int64_t gx = (n + 63) / 64;
    if (gx > 0x7FFFFFFF)
        return cudaErrorInvalidValue;
    dense_kernel<BT><<<dim3((unsigned)gx, (unsigned)((M + 63) / 64)), 256, 0, s>>>(
        A, n, K, lda, B, bias, M, scale_ptr, relu, Y);
    return cudaGetLastError();
}

// centroid columns for the nearest rule: cT[i][j] = cent[j][i], nh[j] = -|c_j|^2 / 2
__global__ void centroid_columns_kernel(const float *__restrict__ cent, int xstride, int d, int E,
                                        float *__restrict__ cT, float *__restrict__ nh) {
    const int j = blockIdx.x;
    for (int i = threadIdx.x; i < d; i += blockDim.x)
        cT[(int64_t)i * E + j] = cent[(int64_t)j * xstride + i];
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int i = 0; i < d; ++i)
            s = fmaf(cent[(int64_t)j * xstride + i], cent[(int64_t)j * xstride + i], s);
        nh[j] = -0.5f * s;
    }
}

// a key whose ascending order is descending logit, then ascending cell
__device__ __forceinline__ unsigned long long logit_key(float t, int o) {
    uint32_t u = __float_as_uint(t);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);  // ascending map of the float order
    return ((unsigned long long)(~u) << 32) | (uint32_t)o;
}

__device__ __forceinline__ void topT_insert(unsigned long long *best, int T,
                                            unsigned long long k) {
    if (k >= best[T - 1])
        return;
    int i = T - 1;
    while (i > 0 && best[i - 1] > k) {
        best[i] = best[i - 1];
        --i;
    }
    best[i] = k;
}

struct CellSeedArgs {
    SearchArgs a;
    const uint32_t *attr_sorted, *id_sorted;         // tuple runs
    const unsigned long long *cell_key;              // (attribute word << 16 | cell), sorted
    const uint32_t *cell_id;                         // ids in that order
    int E, T;
    const float *scores;                             // [nq][E], the larger the better
    int32_t *cells_out;                              // [nq][T] or null
    uint32_t *seeds;                                 // [nq][32]
    uint8_t *bucket;                                 // [nq] or null
};

constexpr int kMaxT = 8;

// One warp per query: the T best cells from the query's score row, then its seeds.
__global__ void __launch_bounds__(256) cell_seeds_kernel(CellSeedArgs c) {
    const SearchArgs &a = c.a;
    const int lane = threadIdx.x & 31;
    const int64_t q = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (q >= a.nq)
        return;
    const int T = c.T;
    {
        uint32_t qhi;
        const uint32_t qa = pack_query_word(a.qattr + q * a.w.m, a.w, &qhi);
        const int ef = a.ef_arr ? a.ef_arr[q] : a.ef;
        const int want = ef < 32 ? ef : 32;
        uint32_t *row = c.seeds + q * 32;
        const int64_t lo = lower_bound_u32(c.attr_sorted, a.N, qa);
        const int64_t hi = qa == 0xFFFFFFFFu ? a.N : lower_bound_u32(c.attr_sorted, a.N, qa + 1u);
        const int64_t P = hi - lo;
        if (lane == 0 && c.bucket != nullptr) {
            const int bits = 64 - __clzll((unsigned long long)P + 1ull);
            c.bucket[q] = (uint8_t)(bits >= 32 ? 0 : 32 - bits);
        }
        unsigned long long best[kMaxT];
#pragma unroll
        for (int t = 0; t < kMaxT; ++t)
            best[t] = ~0ull;
        const float *sr = c.scores + q * (int64_t)c.E;
        for (int o = lane; o < c.E; o += 32)
            topT_insert(best, T, logit_key(sr[o], o));
        int chosen[kMaxT];
        for (int t = 0; t < T; ++t) {
            unsigned long long m = best[0];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long other = __shfl_xor_sync(FULL, m, o);
                m = other < m ? other : m;
            }
            chosen[t] = (int)(uint32_t)m;
            if (best[0] == m) {  // keys are unique: one owner pops its head
#pragma unroll
                for (int u = 0; u + 1 < kMaxT; ++u)
                    best[u] = best[u + 1];
                best[kMaxT - 1] = ~0ull;
            }
        }
        if (lane == 0) {
            if (c.cells_out != nullptr)
                for (int t = 0; t < T; ++t)
                    c.cells_out[q * T + t] = chosen[t];
            int j = 0;
            if (P > 0) {
                const int S = (int64_t)want < P ? want : (int)P;
                for (int t = 0; t < T && j < S; ++t) {
                    const unsigned long long key = ((unsigned long long)qa << 16) | (uint32_t)chosen[t];
                    int64_t r = lower_bound_u64(c.cell_key, a.N, key);
                    for (; r < a.N && c.cell_key[r] == key && j < S; ++r)
                        row[j++] = c.cell_id[r];
                }
                const int S2 = S - j;
                for (int jj = 0; jj < S2; ++jj)
                    row[j++] = c.id_sorted[lo + ((int64_t)jj * P) / S2];
            } else {  // the random stream of NHQ_SEED_RANDOM
                const uint64_t s0 = a.seed ^ mix64((uint64_t)q);
                for (int t = 0; t < 64 && j < want; ++t) {
                    const uint32_t v =
                        (uint32_t)(splitmix_at(s0, (uint64_t)t) % (unsigned long long)a.N);
                    bool dup = false;
                    for (int i = 0; i < j; ++i)
                        dup = dup || row[i] == v;
                    if (!dup)
                        row[j++] = v;
                }
            }
            for (; j < 32; ++j)
                row[j] = kNone;
        }
    }
}

__global__ void entry_to_half_kernel(const float *__restrict__ p, __half *__restrict__ h,
                                     int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        h[i] = __float2half_rn(p[i]);
}

// ---- training (f32 master weights) on a chunk of B samples ----
// The five contractions of a step run on one 64 x 64 register-tiled product (4 x 4 values
// per thread, 32-deep chunks staged in shared memory, the next chunk's global loads in
// flight while the current one is multiplied).  At 16,384 samples, d = 128 and E = 256 a
// step is 2.1 GFLOP over 16 MB that stays in L2, so what counts is how many CTAs a
// contraction fills: the outputs over samples give 256 and 1,024 tiles, and the weight
// gradients (4 and 2 tiles of outputs) split the samples into slices of SLICE, each
// writing its own partial sums, which grad_reduce_kernel adds in slice order (no atomics:
// the gradient is the same in every run).  That step took 2,804 us with one thread per
// output walking all samples of a 2,048-sample chunk in eight chunks, and takes 130 us.
constexpr int GT = 64, GK = 32, GP = GT + 1;
constexpr int SLICE = 128;
// Up to FEW samples and FEW_OUT outputs a step takes kernels with a thread to an output, and
// up to FEW_HIDDEN samples that for H.  Steps at d = 128, on them | on the tiles: 32 samples
// 39.6 | 45.7 us (64 and 256 cells) and 57.5 | 66.7 us (4,096), 128 samples 53.9 | 57.9 and
// 84.2 | 83.0, 200 samples 64.4 | 59.0 and 107 | 92 (each with 4 us of clearing that are gone
// now); H alone takes 2 us off at 1,024 and 2,048 samples (14 at d = 960) and adds 2 to 28 at
// 4,096.
constexpr int FEW = 128, FEW_HIDDEN = 2048;
constexpr int64_t FEW_OUT = 1 << 18;  // samples x cells

// acc[i][j] (+)= sum over k in [k0, k1) of a(k, ty * 4 + i) b(k, tx * 4 + j), k ascending.
// AK / BK: the operand is contiguous along k in memory (the staging loop follows it).
// sum (or null): the threads with ty = 0 also add b(k, tx + 16 j) over k into sum[j].
// LEVELS: 0 sums all k as one chain; 1 the products of 8 k as one chain, four of these (a
// chunk) as another and the chunks as a third; 2 also eight chunks apart from the rest.
// One chain over the E cells of a gradient had up to five times the error of 32 strided
// chains and a tree, which summed them before; 1 has it times 1.1 up to E = 256, 2 times 0.5
// from 1,024 on (1 would have 1.25 at 4,096).  At E = 256 a step took 133.6 us with 0 and
// 1, 135.7 us with 2 or with Kahan's compensation per chunk (each 4 us less since the gradient
// and the loss need no clearing).
template <bool AK, bool BK, int LEVELS = 0, class LA, class LB>
__device__ __forceinline__ void tile_product(float acc[4][4], int64_t k0, int64_t k1, LA la, LB lb,
                                             float (*As)[GP], float (*Bs)[GP],
                                             float *sum = nullptr) {
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    float ra[8], rb[8];
    auto fetch = [&](int64_t kb) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int e = tid + 256 * i;
            const int ka = AK ? e & 31 : e >> 6, r = AK ? e >> 5 : e & 63;
            const int kk = BK ? e & 31 : e >> 6, c = BK ? e >> 5 : e & 63;
            ra[i] = kb + ka < k1 ? la(kb + ka, r) : 0.f;
            rb[i] = kb + kk < k1 ? lb(kb + kk, c) : 0.f;
        }
    };
    float total[4][4] = {};  // of every eight chunks
    fetch(k0);
    for (int64_t kb = k0; kb < k1; kb += GK) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int e = tid + 256 * i;
            As[AK ? e & 31 : e >> 6][AK ? e >> 5 : e & 63] = ra[i];
            Bs[BK ? e & 31 : e >> 6][BK ? e >> 5 : e & 63] = rb[i];
        }
        __syncthreads();
        if (kb + GK < k1)
            fetch(kb + GK);
        if (LEVELS > 0) {
            float chunk[4][4] = {};
#pragma unroll 2
            for (int k8 = 0; k8 < GK; k8 += 8) {
                float p[4][4] = {};
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    float a[4], b[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        a[i] = As[k8 + kk][ty * 4 + i];
                        b[i] = Bs[k8 + kk][tx + 16 * i];
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            p[i][j] = fmaf(a[i], b[j], p[i][j]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        chunk[i][j] += p[i][j];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    acc[i][j] += chunk[i][j];
            if (LEVELS > 1 && ((kb - k0) / GK & 7) == 7) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        total[i][j] += acc[i][j];
                        acc[i][j] = 0.f;
                    }
            }
            __syncthreads();
            continue;
        }
#pragma unroll 8
        for (int kk = 0; kk < GK; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[i] = As[kk][ty * 4 + i];
                b[i] = Bs[kk][tx + 16 * i];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
            if (sum != nullptr && ty == 0) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    sum[j] += b[j];
            }
        }
        __syncthreads();
    }
    if (LEVELS > 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                acc[i][j] += total[i][j];
    }
}

// H[b][j] = relu(b1[j] + sum_i W1[i][j] (s X[b][i])), i ascending; grid (ceil(B/64))
__global__ void __launch_bounds__(256) train_hidden_kernel(const float *__restrict__ P,
                                                           const float *__restrict__ X, int B,
                                                           int d, float *__restrict__ H,
                                                           EntryLayout L) {
    __shared__ float As[GK][GP], Bs[GK][GP];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int b0 = blockIdx.x * GT;
    const float s = P[0];
    float acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float bias = P[L.oB1 + tx + 16 * j];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            acc[i][j] = bias;
    }
    tile_product<true, false>(
        acc, 0, d,
        [&](int64_t k, int r) { return b0 + r < B ? s * X[(int64_t)(b0 + r) * d + k] : 0.f; },
        [&](int64_t k, int c) { return P[L.oW1 + k * EH + c]; }, As, Bs);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int b = b0 + ty * 4 + i;
        if (b >= B)
            continue;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            H[(int64_t)b * EH + tx + 16 * j] = fmaxf(acc[i][j], 0.f);
    }
}

// T[b][o] = b2[o] + sum_h W2[h][o] H[b][h], h ascending; grid (ceil(B/64), ceil(E/64))
__global__ void __launch_bounds__(256) train_out_kernel(const float *__restrict__ P,
                                                        const float *__restrict__ H, int B, int E,
                                                        float *__restrict__ T, EntryLayout L) {
    __shared__ float As[GK][GP], Bs[GK][GP];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int b0 = blockIdx.x * GT, o0 = blockIdx.y * GT;
    float acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int o = o0 + tx + 16 * j;
        const float bias = o < E ? P[L.oB2 + o] : 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            acc[i][j] = bias;
    }
    tile_product<true, false>(
        acc, 0, EH,
        [&](int64_t k, int r) { return b0 + r < B ? H[(int64_t)(b0 + r) * EH + k] : 0.f; },
        [&](int64_t k, int c) { return o0 + c < E ? P[L.oW2 + k * E + o0 + c] : 0.f; }, As, Bs);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int b = b0 + ty * 4 + i;
        if (b >= B)
            continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int o = o0 + tx + 16 * j;
            if (o < E)
                T[(int64_t)b * E + o] = acc[i][j];
        }
    }
}

// dT = (softmax(T) - onehot(label)) * inv_n per sample (a warp each); losses[block] = the sum of
// (lse - t_y) * inv_n over the block's eight samples.
// A label outside 0..E-1 contributes nothing.
// T becomes dT in place (a lane reads the elements that it writes).
__global__ void train_softmax_kernel(float *T, const int32_t *__restrict__ y, int B, int E,
                                     float inv_n, float *__restrict__ losses) {
    __shared__ float part[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b = blockIdx.x * 8 + warp;
    const int lab = b < B ? y[b] : -1;
    float *t = T + (int64_t)b * E;
    float mine = 0.f;
    if (lab >= 0 && lab < E) {
        float mx = -INFINITY;
        for (int o = lane; o < E; o += 32)
            mx = fmaxf(mx, t[o]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, o));
        float se = 0.f;
        for (int o = lane; o < E; o += 32)
            se += expf(t[o] - mx);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            se += __shfl_xor_sync(FULL, se, o);
        const float lse = mx + logf(se);
        mine = (lse - t[lab]) * inv_n;
        __syncwarp();  // the label's logit is read before its lane overwrites it
        for (int o = lane; o < E; o += 32)
            t[o] = (expf(t[o] - lse) - (o == lab ? 1.f : 0.f)) * inv_n;
    } else if (b < B) {
        for (int o = lane; o < E; o += 32)
            t[o] = 0.f;
    }
    if (lane == 0)
        part[warp] = mine;
    __syncthreads();
    if (threadIdx.x == 0) {
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w)
            sum += part[w];
        losses[blockIdx.x] = sum;
    }
}
// dZ[b][h] = [H > 0] sum_o dT[b][o] W2[h][o]; grid (ceil(B/64))
template <int LEVELS>
__global__ void __launch_bounds__(256) train_dz_kernel(const float *__restrict__ P,
                                                       const float *__restrict__ H,
                                                       const float *__restrict__ dT, int B, int E,
                                                       float *__restrict__ dZ, EntryLayout L) {
    __shared__ float As[GK][GP], Bs[GK][GP];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int b0 = blockIdx.x * GT;
    float acc[4][4] = {};
    tile_product<true, true, LEVELS>(
        acc, 0, E,
        [&](int64_t k, int r) { return b0 + r < B ? dT[(int64_t)(b0 + r) * E + k] : 0.f; },
        [&](int64_t k, int c) { return P[L.oW2 + (int64_t)c * E + k]; }, As, Bs);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int b = b0 + ty * 4 + i;
        if (b >= B)
            continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t e = (int64_t)b * EH + tx + 16 * j;
            dZ[e] = H[e] > 0.f ? acc[i][j] : 0.f;
        }
    }
}

// Partial sums of one weight gradient over a slice of samples: part[slice][r][c] =
// sum_b A[b][r] D[b][c] for r < rows (times the input scale when scale is set) and row
// r = rows the plain sums of D (the bias), which the first row of tiles adds up on the
// side (as a row of the product it took a tile row of its own).  A has rows values per
// sample, D cols; grid (ceil(cols/64), ceil(rows/64), slices).
__global__ void __launch_bounds__(256) train_gw_kernel(const float *__restrict__ A, int rows,
                                                       const float *__restrict__ scale,
                                                       const float *__restrict__ D, int cols,
                                                       int B, float *__restrict__ part) {
    __shared__ float As[GK][GP], Bs[GK][GP];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int c0 = blockIdx.x * GT, r0 = blockIdx.y * GT;
    const int64_t b0 = (int64_t)blockIdx.z * SLICE;
    const int64_t b1 = b0 + SLICE < B ? b0 + SLICE : B;
    const float s = scale != nullptr ? *scale : 1.f;
    float acc[4][4] = {}, sum[4] = {};
    tile_product<false, false>(
        acc, b0, b1, [&](int64_t k, int r) { return r0 + r < rows ? s * A[k * rows + r0 + r] : 0.f; },
        [&](int64_t k, int c) { return c0 + c < cols ? D[k * cols + c0 + c] : 0.f; }, As, Bs, sum);
    float *out = part + (int64_t)blockIdx.z * (rows + 1) * cols;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int c = c0 + tx + 16 * j;
        if (c >= cols)
            continue;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = r0 + ty * 4 + i;
            if (r < rows)
                out[(int64_t)r * cols + c] = acc[i][j];
        }
        if (ty == 0 && r0 == 0)
            out[(int64_t)rows * cols + c] = sum[j];
    }
}

// G = (add: +=) the slices of both gradients: 32 values per block, eight warps summing every
// eighth slice in order, then the eight sums in order.  W1 | b1 and W2 | b2 are each one
// run of the parameter vector, laid out as train_gw_kernel lays out its rows.  The last
// block adds the softmax's block sums to the loss (as additions to one value, in whatever
// order, they moved it by 3e-7 of itself between runs).
__global__ void __launch_bounds__(256) grad_reduce_kernel(const float *__restrict__ part1,
                                                          int64_t n1,
                                                          const float *__restrict__ part2,
                                                          int64_t n2, int slices,
                                                          float *__restrict__ G,
                                                          const float *__restrict__ losses,
                                                          int nlosses, float *loss, bool add) {
    __shared__ float sums[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (blockIdx.x == gridDim.x - 1) {
        float acc = 0.f;
        for (int i = threadIdx.x; i < nlosses; i += 256)
            acc += losses[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            acc += __shfl_xor_sync(FULL, acc, o);
        if (lane == 0)
            sums[0][warp] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < 8; ++w)
                acc += sums[0][w];
            *loss = add ? *loss + acc : acc;
            if (!add)
                G[0] = 0.f;  // the input scale is not trained
        }
        return;
    }
    for (int64_t i0 = blockIdx.x * (int64_t)32; i0 < n1 + n2;
         i0 += (int64_t)(gridDim.x - 1) * 32) {
        const int64_t i = i0 + lane;
        float acc = 0.f;
        if (i < n1 + n2) {
            const float *p = i < n1 ? part1 + i : part2 + (i - n1);
            const int64_t step = i < n1 ? n1 : n2;
#pragma unroll 8
            for (int z = warp; z < slices; z += 8)
                acc += p[z * step];
        }
        sums[warp][lane] = acc;
        __syncthreads();
        if (warp == 0 && i < n1 + n2) {
#pragma unroll
            for (int w = 1; w < 8; ++w)
                acc += sums[w][lane];
            G[1 + i] = add ? G[1 + i] + acc : acc;
        }
        __syncthreads();
    }
}

// ---- the same step for few samples ----
// A tile of 64 samples leaves most of the chip idle where there are not many of them, and
// walks all of E (or d) in one chain of loads: a step of 32 samples at d = 128, E = 1,024
// took 105 us on tiles alone and takes 42 with an output to a thread (dZ: to a warp).

// H[b][j] as train_hidden_kernel; 4 samples of 64 units per block
__global__ void few_hidden_kernel(const float *__restrict__ P, const float *__restrict__ X, int B,
                                  int d, float *__restrict__ H, EntryLayout L) {
    const int b = blockIdx.x * 4 + (threadIdx.x >> 6), j = threadIdx.x & 63;
    if (b >= B)
        return;
    const float s = P[0];
    float z = P[L.oB1 + j];
    for (int i = 0; i < d; ++i)
        z = fmaf(P[L.oW1 + (int64_t)i * EH + j], s * X[(int64_t)b * d + i], z);
    H[(int64_t)b * EH + j] = fmaxf(z, 0.f);
}

// T[b][o] as train_out_kernel; grid (ceil(E/128), B)
__global__ void few_out_kernel(const float *__restrict__ P, const float *__restrict__ H, int E,
                               float *__restrict__ T, EntryLayout L) {
    __shared__ float h[EH];
    const int b = blockIdx.y;
    if (threadIdx.x < EH)
        h[threadIdx.x] = H[(int64_t)b * EH + threadIdx.x];
    __syncthreads();
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= E)
        return;
    float t = P[L.oB2 + o];
    for (int k = 0; k < EH; ++k)
        t = fmaf(P[L.oW2 + (int64_t)k * E + o], h[k], t);
    T[(int64_t)b * E + o] = t;
}

// dZ[b][h] = [H > 0] sum_o dT[b][o] W2[h][o], a warp per pair (b, h); the first warp also
// puts the softmax's block sums into the loss, where that is given, and 0 into the input
// scale's place G[0] (add: adds them to the loss)
__global__ void few_dz_kernel(const float *__restrict__ P, const float *__restrict__ H,
                              const float *__restrict__ dT, int B, int E,
                              float *__restrict__ dZ, EntryLayout L,
                              const float *__restrict__ losses, int nlosses, float *loss,
                              float *G, bool add) {
    const int lane = threadIdx.x & 31;
    const int64_t pair = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (pair >= (int64_t)B * EH)
        return;
    if (pair == 0 && loss != nullptr) {
        float sum = 0.f;
        for (int i = lane; i < nlosses; i += 32)
            sum += losses[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            sum += __shfl_xor_sync(FULL, sum, o);
        if (lane == 0) {
            *loss = add ? *loss + sum : sum;
            if (!add)
                G[0] = 0.f;
        }
    }
    const int b = (int)(pair / EH), h = (int)(pair % EH);
    float acc = 0.f;
    for (int o = lane; o < E; o += 32)
        acc = fmaf(dT[(int64_t)b * E + o], P[L.oW2 + (int64_t)h * E + o], acc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        acc += __shfl_xor_sync(FULL, acc, o);
    if (lane == 0)
        dZ[pair] = H[pair] > 0.f ? acc : 0.f;
}

// G[r][c] = (add: +=) sum_b A[b][r] D[b][c] for r < rows (times the input scale when scale is set),
// row r = rows the sums of D, b ascending: W1 | b1 or W2 | b2 from G on.
// COLS columns of THREADS / COLS rows a block
template <int COLS, int THREADS>
__global__ void few_gw_kernel(const float *__restrict__ A, int rows,
                              const float *__restrict__ scale, const float *__restrict__ D,
                              int cols, int B, float *__restrict__ G, bool add) {
    const int c = blockIdx.x * COLS + threadIdx.x % COLS;
    const int r = blockIdx.y * (THREADS / COLS) + threadIdx.x / COLS;
    if (c >= cols || r > rows)
        return;
    const float s = scale != nullptr ? *scale : 1.f;
    const float *pd = D + c;
    float acc = 0.f;
    if (r < rows) {
        const float *pa = A + r;
#pragma unroll 8
        for (int b = 0; b < B; ++b)
            acc = fmaf(s * pa[(int64_t)b * rows], pd[(int64_t)b * cols], acc);
    } else {
#pragma unroll 8
        for (int b = 0; b < B; ++b)
            acc += pd[(int64_t)b * cols];
    }
    float *g = G + (int64_t)r * cols + c;
    *g = add ? *g + acc : acc;
}

// Adam (beta1 0.9, beta2 0.999) on every parameter but the input scale (index 0)
__global__ void train_adam_kernel(float *__restrict__ p, const float *__restrict__ g,
                                  float *__restrict__ m, float *__restrict__ v, int64_t n,
                                  float lr, float c1, float c2) {
    for (int64_t i = 1 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
        m[i] = b1 * m[i] + (1.f - b1) * g[i];
        v[i] = b2 * v[i] + (1.f - b2) * g[i] * g[i];
        p[i] -= lr * (m[i] * c1) / (sqrtf(v[i] * c2) + eps);
    }
}

__global__ void entry_labels_kernel(const uint32_t *__restrict__ ids, int k, int64_t n,
                                    const uint32_t *__restrict__ cell, int64_t N,
                                    int32_t *__restrict__ lab) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n;
         q += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t v = ids[q * k];
        lab[q] = (v != kNone && (int64_t)v < N) ? (int32_t)cell[v] : -1;
    }
}

unsigned grid_for(int64_t n, int per) {
    int64_t g = (n + per - 1) / per;
    return (unsigned)(g < 1 ? 1 : (g > 65535 * 4 ? 65535 * 4 : g));
}

}  // namespace

int64_t entry_param_count(int d, int E) { return entry_layout(d, E).total; }

cudaError_t launch_gather_centroids(const float *X, int xstride, int64_t N, int E,
                                    const uint32_t *attr, float *cent, uint32_t *cattr,
                                    cudaStream_t s) {
    gather_centroids_kernel<<<E, 128, 0, s>>>(X, xstride, N, E, attr, cent, cattr);
    return cudaGetLastError();
}

size_t cell_sort_scratch_bytes(int64_t N) {
    size_t cub_bytes = 0;
    cub::DeviceRadixSort::SortPairs(nullptr, cub_bytes, (const unsigned long long *)nullptr,
                                    (unsigned long long *)nullptr, (const uint32_t *)nullptr,
                                    (uint32_t *)nullptr, (int)N);
    return (sizeof(unsigned long long) + sizeof(uint32_t)) * (size_t)N + 512 + cub_bytes;
}

cudaError_t launch_cell_sort(const uint32_t *attr, const uint32_t *cell, int64_t N,
                             unsigned long long *key_sorted, uint32_t *id_sorted, void *scratch,
                             size_t scratch_bytes, cudaStream_t s) {
    unsigned long long *key = reinterpret_cast<unsigned long long *>(scratch);
    uintptr_t t = reinterpret_cast<uintptr_t>(key + N);
    t = (t + 255) & ~(uintptr_t)255;
    uint32_t *iota = reinterpret_cast<uint32_t *>(t);
    t = reinterpret_cast<uintptr_t>(iota + N);
    t = (t + 255) & ~(uintptr_t)255;
    void *tmp = reinterpret_cast<void *>(t);
    size_t cub_bytes = 0;
    cudaError_t e = cub::DeviceRadixSort::SortPairs(nullptr, cub_bytes, key, key_sorted, iota,
                                                    id_sorted, (int)N, 0, 48);
    if (e != cudaSuccess)
        return e;
    if ((char *)tmp + cub_bytes > (char *)scratch + scratch_bytes)
        return cudaErrorInvalidValue;
    cell_key_kernel<<<grid_for(N, 256), 256, 0, s>>>(attr, cell, N, key, iota);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    return cub::DeviceRadixSort::SortPairs(tmp, cub_bytes, key, key_sorted, iota, id_sorted,
                                           (int)N, 0, 48, s);
}

cudaError_t launch_entry_to_half(const float *params, int64_t n, __half *w16, cudaStream_t s) {
    entry_to_half_kernel<<<grid_for(n, 256), 256, 0, s>>>(params, w16, n);
    return cudaGetLastError();
}

cudaError_t launch_cell_seeds(const SearchArgs &a, const uint32_t *attr_sorted,
                              const uint32_t *id_sorted, const unsigned long long *cell_key,
                              const uint32_t *cell_id, int E, int T, const float *scores,
                              int32_t *cells_out, uint32_t *seeds, uint8_t *bucket,
                              cudaStream_t s) {
    if (a.nq <= 0)
        return cudaSuccess;
    if (T < 1 || T > kMaxT || T > E)
        return cudaErrorInvalidValue;
    CellSeedArgs c;
    c.a = a;
    c.attr_sorted = attr_sorted;
    c.id_sorted = id_sorted;
    c.cell_key = cell_key;
    c.cell_id = cell_id;
    c.E = E;
    c.T = T;
    c.scores = scores;
    c.cells_out = cells_out;
    c.seeds = seeds;
    c.bucket = bucket;
    cell_seeds_kernel<<<(unsigned)((a.nq + 7) / 8), 256, 0, s>>>(c);
    return cudaGetLastError();
}

cudaError_t launch_centroid_columns(const float *cent, int xstride, int d, int E, float *cT,
                                    float *nh, cudaStream_t s) {
    centroid_columns_kernel<<<E, 128, 0, s>>>(cent, xstride, d, E, cT, nh);
    return cudaGetLastError();
}

cudaError_t launch_entry_scores_nearest(const float *cT, const float *nh, int d, int E,
                                        const float *Q, int64_t qstride, int64_t n, float *out,
                                        cudaStream_t s) {
    return launch_dense<float>(Q, n, d, qstride, cT, nh, E, nullptr, 0, out, s);
}

cudaError_t launch_entry_scores_learned(const __half *w16, const float *params, int d, int E,
                                        const float *Q, int64_t qstride, int64_t n,
                                        float *hidden, float *out, cudaStream_t s) {
    const EntryLayout L = entry_layout(d, E);
    cudaError_t e = launch_dense<__half>(Q, n, d, qstride, w16 + L.oW1, w16 + L.oB1, EH, params,
                                         1, hidden, s);
    if (e != cudaSuccess)
        return e;
    return launch_dense<__half>(hidden, n, EH, EH, w16 + L.oW2, w16 + L.oB2, E, nullptr, 0, out,
                                s);
}

cudaError_t launch_entry_labels(const uint32_t *ids, int k, int64_t n, const uint32_t *cell,
                                int64_t N, int32_t *labels, cudaStream_t s) {
    if (n <= 0)
        return cudaSuccess;
    entry_labels_kernel<<<grid_for(n, 256), 256, 0, s>>>(ids, k, n, cell, N, labels);
    return cudaGetLastError();
}

// Samples of one gradient pass: as many as keep a chunk's working memory at about 64 MB
// (it then stays in L2 between the kernels), in whole slices and at least 2,048.
int entry_train_chunk(int64_t n, int d, int E) {
    const int64_t per = 2 * EH + E + ((int64_t)(d + 1) * EH + (int64_t)(EH + 1) * E) / SLICE + 1;
    int64_t B = (int64_t(16) << 20) / per / SLICE * SLICE;
    B = B < 2048 ? 2048 : B > 65536 ? 65536 : B;
    return (int)(n < B ? n : B);
}

// Working memory of one chunk of B samples: H, dZ [B][64], T [B][E], the slices' partial
// sums of (W1 | b1) and (W2 | b2), and the losses [ceil(B/8)].
size_t entry_train_chunk_bytes(int B, int d, int E) {
    const size_t slices = ((size_t)B + SLICE - 1) / SLICE;
    return sizeof(float) * ((size_t)B * EH * 2 + (size_t)B * E + ((size_t)B + 7) / 8 +
                            slices * ((size_t)(d + 1) * EH + (size_t)(EH + 1) * E)) +
           1024;
}

// Which kernel takes dZ of nb samples: the warps cost about max(13, 4 + E / 44) ns a sample,
// the tiles 5.6 us + 56 ns a cell whatever the samples (up to a tile for each SM).  Measured,
// warps | tiles: 512 samples of 64 cells 9.0 | 9.2 us, 1,024 of 256 14.9 | 18.8, 2,048 of 256
// 25.9 | 19.4, 2,048 of 1,024 57 | 60.
static bool tiled_dz(int64_t nb, int64_t E) {
    return nb * (184 + E > 576 ? 184 + E : 576) >= 2450 * (100 + E);
}

// The gradient of the loss over samples [0, n), n >= 1 (divided by `total`), into G and the
// loss into *loss, in chunks of B samples; the first chunk sets them (clearing them before
// would be one or two launches more).
cudaError_t entry_grad(const float *P, int d, int E, const float *X, const int32_t *y, int64_t n,
                       int64_t total, int B, float *G, float *loss, void *work, cudaStream_t s) {
    const EntryLayout L = entry_layout(d, E);
    const int64_t n1 = (int64_t)(d + 1) * EH, n2 = (int64_t)(EH + 1) * E;
    float *H = reinterpret_cast<float *>(work);
    float *dZ = H + (size_t)B * EH;
    float *T = dZ + (size_t)B * EH;
    float *part1 = T + (size_t)B * E;
    float *part2 = part1 + (size_t)((B + SLICE - 1) / SLICE) * n1;
    float *losses = part2 + (size_t)((B + SLICE - 1) / SLICE) * n2;
    const float inv = 1.f / (float)total;
    const unsigned et = (unsigned)((E + GT - 1) / GT);
    cudaError_t e = cudaSuccess;
    for (int64_t b0 = 0; b0 < n; b0 += B) {
        const int nb = (int)(n - b0 < B ? n - b0 : B);
        const float *Xb = X + b0 * d;
        const unsigned bt = (unsigned)((nb + GT - 1) / GT);
        const unsigned sl = (unsigned)((nb + SLICE - 1) / SLICE);
        const unsigned pairs = (unsigned)(((int64_t)nb * EH + 7) / 8);
        const bool few = nb <= FEW && (int64_t)nb * E <= FEW_OUT;
        const int nlosses = (nb + 7) / 8;
        const bool add = b0 > 0;
        if (nb <= FEW_HIDDEN)
            few_hidden_kernel<<<(nb + 3) / 4, 256, 0, s>>>(P, Xb, nb, d, H, L);
        else
            train_hidden_kernel<<<bt, 256, 0, s>>>(P, Xb, nb, d, H, L);
        if (few)
            few_out_kernel<<<dim3((E + 127) / 128, nb), 128, 0, s>>>(P, H, E, T, L);
        else
            train_out_kernel<<<dim3(bt, et), 256, 0, s>>>(P, H, nb, E, T, L);
        train_softmax_kernel<<<nlosses, 256, 0, s>>>(T, y + b0, nb, E, inv, losses);
        if (few)
            few_gw_kernel<128, 128><<<dim3((E + 127) / 128, EH + 1), 128, 0, s>>>(
                H, EH, nullptr, T, E, nb, G + L.oW2, add);
        else
            train_gw_kernel<<<dim3(et, EH / GT, sl), 256, 0, s>>>(H, EH, nullptr, T, E, nb, part2);
        if (!tiled_dz(nb, E))
            few_dz_kernel<<<pairs, 256, 0, s>>>(P, H, T, nb, E, dZ, L, losses, nlosses,
                                                few ? loss : nullptr, G, add);
        else if (E <= 256)
            train_dz_kernel<1><<<bt, 256, 0, s>>>(P, H, T, nb, E, dZ, L);
        else
            train_dz_kernel<2><<<bt, 256, 0, s>>>(P, H, T, nb, E, dZ, L);
        if (few) {
            few_gw_kernel<64, 256><<<dim3(1, (unsigned)(d + 4) / 4), 256, 0, s>>>(
                Xb, d, P, dZ, EH, nb, G + L.oW1, add);
        } else {
            train_gw_kernel<<<dim3(1, (unsigned)((d + GT - 1) / GT), sl), 256, 0, s>>>(
                Xb, d, P, dZ, EH, nb, part1);
            grad_reduce_kernel<<<grid_for(n1 + n2, 32) + 1, 256, 0, s>>>(
                part1, n1, part2, n2, (int)sl, G, losses, nlosses, loss, add);
        }
        if ((e = cudaGetLastError()) != cudaSuccess)
            return e;
    }
    return e;
}

cudaError_t launch_entry_adam(float *p, const float *g, float *m, float *v, int64_t n, float lr,
                              float c1, float c2, cudaStream_t s) {
    train_adam_kernel<<<grid_for(n, 256), 256, 0, s>>>(p, g, m, v, n, lr, c1, c2);
    return cudaGetLastError();
}

}  // namespace nhq
