// Seed selection for the search.  The paper takes seeds from NGT's vp-tree
// (Sec. 2, Table 5), which it does not specify, and also reports a random
// variant (Sec. 3.2, Fig. 5(a)).  Two deterministic rules are provided:
//   random: n_seed distinct ids per query from a SplitMix64 stream (Steele,
//           Lea and Flood 2014) that starts at global_seed + q * 2^32; a draw z
//           maps to floor(z * n / 2^64) and repeats are redrawn.
//   pivot:  the n_seed nearest (distance, id) of the P pivots floor(t * n / P).
#include <cooperative_groups.h>

#include <algorithm>
#include <climits>
#include <cmath>

#include "common.cuh"
#include "warp_sort.cuh"

namespace cg = cooperative_groups;

namespace onng {
namespace {

constexpr int kMaxSeed = 64;

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long &state)
{
    unsigned long long z = (state += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void seeds_random_kernel(unsigned long long global_seed, int64_t nq, int64_t n, int n_seed,
                                    int32_t *__restrict__ out)
{
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= nq)
        return;
    int32_t *o = out + q * n_seed;
    const int m = (int64_t)n_seed < n ? n_seed : (int)n;
    for (int t = m; t < n_seed; ++t)
        o[t] = -1;
    if (2 * (int64_t)m > n) {
        for (int t = 0; t < m; ++t)
            o[t] = t;
        return;
    }
    int32_t chosen[kMaxSeed];
    unsigned long long st = global_seed + ((unsigned long long)q << 32);
    int got = 0;
    while (got < m) {
        const unsigned long long z = splitmix64(st);
        const int32_t id = (int32_t)__umul64hi(z, (unsigned long long)n);
        bool dup = false;
        for (int t = 0; t < got; ++t)
            dup |= chosen[t] == id;
        if (!dup)
            chosen[got++] = id;
    }
    for (int t = 0; t < m; ++t)
        o[t] = chosen[t];
}

// Nearest-pivot seeds.  A CTA owns kPivQ queries and a share of the pivots, walked
// in tiles of kPivT; the S CTAs of a cluster share the queries and split the pivots.
//
// Distances: the squared differences are added coordinate by coordinate in float32,
// one chain per (query, pivot) pair.  What bounds the pass is the float32 pipe (a
// subtraction and a multiply-add per pair and coordinate), so a thread keeps 4
// queries x 8 pivots in registers and the two pivots of a pair share each packed
// instruction (add.f32x2, fma.f32x2: the same rounding per half as the scalar
// forms).  The operands come from shared memory in the layout the packed form
// wants: pivots coordinate-major (a 16-byte read is two pairs), queries negated and
// duplicated; per coordinate 4 reads feed 32 packed instructions.  Chunks of kPivD
// coordinates are double-buffered: the next chunk's global loads are issued before
// the arithmetic of the present one and stored to shared memory after it.
//
// Selection: after each tile a warp per query folds its kPivT (distance bits, pivot
// index) keys into the query's sorted list.  Keys below the list's m-th take part;
// when many do (the first tile), the m-th smallest of the 32 lanes' minima bounds
// the tile's own m-th smallest key first, which leaves little more than m keys to
// insert.  At the end the CTAs of the cluster merge their lists over distributed
// shared memory, each for its share of the queries.
//
// Seeds + search together, before (one CTA per 16 queries over all pivots, scalar
// arithmetic) and after: 1 query, 1,024 pivots, d = 128: 195 -> 118 us; 1,000 queries,
// 8,192 pivots, d = 960: 7.57 -> 1.01 ms; 10,000 queries, 1,024 pivots, d = 128:
// 3.37 -> 3.27 ms.  The packed arithmetic alone (37.5 T float32 operations a second,
// packed or not; packing halves the issue slots) would take 70 us of the last.
constexpr int kPivQ = 32;
constexpr int kPivT = 256;
constexpr int kPivD = 16;
constexpr int kPivThreads = 256;
constexpr int kPivMinCta = 2;
constexpr int kPivRow = kPivT + 4;  // 4 rows apart is 16 banks apart: conflict-free transposing stores
constexpr int kPivMaxCluster = 8;
constexpr int kPivInsertMax = 16;  // more qualifying keys than this are thinned out before insertion
constexpr unsigned long long kNoKey = ~0ull;

struct PivSmem {
    float ts[2][kPivD][kPivRow];   // a chunk of the tile's pivots, coordinate-major
    float2 qs[2][kPivD][kPivQ];    // the queries' chunk, negated, each value twice
    float dist[kPivQ][kPivRow];    // the tile's squared distances
    unsigned long long best[kPivQ][kMaxSeed];
};

// Inserts `key` (warp-uniform, absent from the list) into the ascending list
// whose element e = h * 32 + lane is b[h] of lane `lane`; the last element drops.
__device__ __forceinline__ void list_insert(unsigned long long (&b)[2], unsigned long long key, int lane)
{
    const int pos = __popc(__ballot_sync(0xffffffffu, b[0] < key)) + __popc(__ballot_sync(0xffffffffu, b[1] < key));
    const unsigned long long up0 = __shfl_up_sync(0xffffffffu, b[0], 1);
    const unsigned long long up1 = __shfl_up_sync(0xffffffffu, b[1], 1);
    const unsigned long long last0 = __shfl_sync(0xffffffffu, b[0], 31);
    const int e1 = 32 + lane;
    b[0] = lane < pos ? b[0] : (lane == pos ? key : up0);
    b[1] = e1 < pos ? b[1] : (e1 == pos ? key : (lane == 0 ? last0 : up1));
}

// The list's m-th key (kNoKey while it holds fewer).
__device__ __forceinline__ unsigned long long list_mth(const unsigned long long (&b)[2], int m)
{
    return __shfl_sync(0xffffffffu, m > 32 ? b[1] : b[0], (m - 1) & 31);
}

// Inserts the lanes' keys `v` that lie below kth (the list's m-th key), updating both.
__device__ __forceinline__ void list_fold(unsigned long long (&b)[2], unsigned long long v, unsigned long long &kth, int m,
                                          int lane)
{
    unsigned in = __ballot_sync(0xffffffffu, v < kth);
    while (in) {
        const int src = __ffs(in) - 1;
        in &= in - 1;
        const unsigned long long key = __shfl_sync(0xffffffffu, v, src);
        if (key < kth) {
            list_insert(b, key, lane);
            kth = list_mth(b, m);
        }
    }
}

__global__ void __launch_bounds__(kPivThreads, kPivMinCta)
    seeds_pivot_kernel(const float *__restrict__ X, int64_t n, int d, const float *__restrict__ Q, int64_t nq, int P,
                       int n_seed, int32_t *__restrict__ out)
{
    extern __shared__ __align__(16) unsigned char piv_raw[];
    PivSmem &sm = *reinterpret_cast<PivSmem *>(piv_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int S = (int)gridDim.y, rank = (int)blockIdx.y;  // the cluster spans the grid's y
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t q0 = (int64_t)blockIdx.x * kPivQ;
    const int nrow = nq - q0 < kPivQ ? (int)(nq - q0) : kPivQ;
    const int d4 = d >> 2;
    const int m = n_seed < P ? n_seed : P;
    const int tb = (int)((int64_t)P * rank / S), te = (int)((int64_t)P * (rank + 1) / S);  // this CTA's pivots
    for (int e = tid; e < kPivQ * kMaxSeed; e += kPivThreads)
        sm.best[e / kMaxSeed][e % kMaxSeed] = kNoKey;

    // staging: thread -> 4 pivot quads (row and quad of the chunk) and, below 128, one query quad
    const int prow = warp * 16 + (lane >> 1), pc = lane & 1;
    const int qrow = tid & 31, qc = tid >> 5;
    float4 pv[4], qv;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    auto fetch = [&](int t0, int c0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = t0 + prow + 128 * h;
            const float4 *row = reinterpret_cast<const float4 *>(X + (int64_t)t * n / P * d);
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const int c = c0 + 2 * g + pc;
                pv[2 * h + g] = t < te && c < d4 ? __ldg(row + c) : zero4;
            }
        }
        if (tid < 4 * kPivQ) {
            const int c = c0 + qc;
            qv = qrow < nrow && c < d4 ? __ldg(reinterpret_cast<const float4 *>(Q + (q0 + qrow) * d) + c) : zero4;
        }
    };
    auto store = [&](int b) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const float4 v = pv[2 * h + g];
                const int c = (2 * g + pc) * 4, r = prow + 128 * h;
                sm.ts[b][c][r] = v.x;
                sm.ts[b][c + 1][r] = v.y;
                sm.ts[b][c + 2][r] = v.z;
                sm.ts[b][c + 3][r] = v.w;
            }
        if (tid < 4 * kPivQ) {
            sm.qs[b][qc * 4][qrow] = make_float2(-qv.x, -qv.x);
            sm.qs[b][qc * 4 + 1][qrow] = make_float2(-qv.y, -qv.y);
            sm.qs[b][qc * 4 + 2][qrow] = make_float2(-qv.z, -qv.z);
            sm.qs[b][qc * 4 + 3][qrow] = make_float2(-qv.w, -qv.w);
        }
    };
    // arithmetic: warp -> 16 queries x 64 pivots, lane -> 4 queries x (4 + 4) pivots
    const int tq = (warp & 1) * 16 + (lane & 3) * 4, tp = (warp >> 1) * 64 + (lane >> 2) * 4;
    // (a warp whose queries or pivots are all padding skips the arithmetic: one query against
    // 64 pivots at d = 1,024 took 108 us with every warp at it)
    const int pivots = (warp & 1) * 16 < nrow ? te - (warp >> 1) * 64 : 0;  // busy in tiles from below this
    unsigned long long acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            acc[i][j] = 0ull;

    int b = 0;
    if (tb < te) {
        fetch(tb, 0);
        store(0);
    }
    __syncthreads();
    for (int t0 = tb; t0 < te; t0 += kPivT) {
        for (int c0 = 0; c0 < d4; c0 += kPivD / 4) {
            const bool last = c0 + kPivD / 4 >= d4;
            const int nt = last ? t0 + kPivT : t0, nc = last ? 0 : c0 + kPivD / 4;
            if (nt < te)
                fetch(nt, nc);
            if (t0 < pivots) {
#pragma unroll
                for (int c = 0; c < kPivD; ++c) {
                    const ulonglong2 x0 = *reinterpret_cast<const ulonglong2 *>(&sm.ts[b][c][tp]);
                    const ulonglong2 x1 = *reinterpret_cast<const ulonglong2 *>(&sm.ts[b][c][tp + 32]);
                    const ulonglong2 q01 = *reinterpret_cast<const ulonglong2 *>(&sm.qs[b][c][tq]);
                    const ulonglong2 q23 = *reinterpret_cast<const ulonglong2 *>(&sm.qs[b][c][tq + 2]);
                    const unsigned long long qq[4] = {q01.x, q01.y, q23.x, q23.y};
                    const unsigned long long xx[4] = {x0.x, x0.y, x1.x, x1.y};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const unsigned long long u = add_f32x2(xx[j], qq[i]);
                            acc[i][j] = fma_f32x2(u, u, acc[i][j]);
                        }
                }
            }
            if (last) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    *reinterpret_cast<ulonglong2 *>(&sm.dist[tq + i][tp]) = make_ulonglong2(acc[i][0], acc[i][1]);
                    *reinterpret_cast<ulonglong2 *>(&sm.dist[tq + i][tp + 32]) = make_ulonglong2(acc[i][2], acc[i][3]);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        acc[i][j] = 0ull;
                }
            }
            if (nt < te)
                store(b ^ 1);
            __syncthreads();
            b ^= 1;
        }
        // fold the tile into each query's list; keys order as (distance, pivot index)
        // and NaN distances (non-finite input) are never taken
        for (int i = warp; i < nrow; i += kPivThreads / 32) {
            unsigned long long v[8], l[2] = {sm.best[i][lane], sm.best[i][32 + lane]};
            unsigned long long kth = list_mth(l, m);
            int cnt = 0;
#pragma unroll
            for (int h = 0; h < 8; ++h) {
                const int t = t0 + h * 32 + lane;
                const float dv = sm.dist[i][h * 32 + lane];
                v[h] = (t < te && !isnan(dv)) ? pack_key(dv, t) : kNoKey;
                cnt += __popc(__ballot_sync(0xffffffffu, v[h] < kth));
            }
            if (!cnt)
                continue;
            if (cnt > kPivInsertMax && m > 32) {
#pragma unroll
                for (int h = 0; h < 8; h += 2) {
                    unsigned long long s[4] = {l[0], l[1], v[h], v[h + 1]};
                    warp_bitonic_sort<4>(s, lane);
                    l[0] = s[0];
                    l[1] = s[1];
                }
            } else {
                if (cnt > kPivInsertMax) {
                    unsigned long long mn[1] = {v[0]};
#pragma unroll
                    for (int h = 1; h < 8; ++h)
                        mn[0] = v[h] < mn[0] ? v[h] : mn[0];
                    warp_bitonic_sort<1>(mn, lane);
                    const unsigned long long lim = __shfl_sync(0xffffffffu, mn[0], m - 1);
#pragma unroll
                    for (int h = 0; h < 8; ++h)
                        v[h] = v[h] <= lim ? v[h] : kNoKey;
                }
#pragma unroll
                for (int h = 0; h < 8; ++h)
                    list_fold(l, v[h], kth, m, lane);
            }
            sm.best[i][lane] = l[0];
            sm.best[i][32 + lane] = l[1];
        }
        // Rows of one chunk write the next tile's distances before any further barrier;
        // longer ones pass the barrier of their next tile's first chunk first.
        if (d4 <= kPivD / 4)
            __syncthreads();
    }
    if (S > 1)
        cluster.sync();
    else
        __syncthreads();
    // merge the cluster's lists: this CTA takes the queries rank, rank + S, ...
    for (int i = rank + S * warp; i < nrow; i += S * (kPivThreads / 32)) {
        unsigned long long l[2] = {sm.best[i][lane], sm.best[i][32 + lane]};
        if (S > 1) {
            unsigned long long kth = list_mth(l, m);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h * 32 >= m)
                    break;
                unsigned long long o[kPivMaxCluster];  // the other lists' keys, all loads in flight
#pragma unroll
                for (int r = 0; r < kPivMaxCluster; ++r) {
                    o[r] = kNoKey;
                    if (r < S && r != rank)
                        o[r] = cluster.map_shared_rank(&sm.best[0][0], r)[i * kMaxSeed + h * 32 + lane];
                }
#pragma unroll
                for (int r = 0; r < kPivMaxCluster; ++r)
                    list_fold(l, o[r], kth, m, lane);
            }
        }
        const int64_t q = q0 + i;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = h * 32 + lane;
            const unsigned long long key = r < m ? l[h] : kNoKey;
            if (r < n_seed)
                out[q * n_seed + r] = key == kNoKey ? -1 : (int32_t)((int64_t)(unsigned)(key & 0xFFFFFFFFull) * n / P);
        }
    }
    if (S > 1)
        cluster.sync();  // no CTA leaves while another reads its lists
}

// The same rule for few pivots, where the tiles above are mostly padding and a chunk's
// arithmetic does not cover the next one's loads: 16 queries x tiles of 64 pivots, chunks
// of 64 coordinates, a thread per query and four pivots (16 apart), the same float32 chain
// per pair.  A warp keeps the lists of two queries in registers.
//
// Taken for one tile, and for two where its blocks are fewer than the SMs but more than
// one (few_pivots).  1,000 queries, us with the tiled kernel and with this one: 64 pivots
// at d = 128 22 and 11, at d = 1,024 85 and 47; 100 pivots at d = 128 23 and 18, at d = 1,024 89
// and 88; but 100 pivots at d = 128 for one query 14 and 18, for 10,000 49 and 58.
constexpr int kFewQ = 16;
constexpr int kFewT = 64;
constexpr int kFewD = 64;

__global__ void __launch_bounds__(kPivThreads, 5)
    seeds_few_kernel(const float *__restrict__ X, int64_t n, int d, const float *__restrict__ Q, int64_t nq, int P, int n_seed,
                     int32_t *__restrict__ out)
{
    __shared__ __align__(16) float qs[kFewQ][kFewD];
    __shared__ __align__(16) float ts[kFewT][kFewD + 4];  // padded: 16 rows apart in distinct banks
    __shared__ float dist[kFewQ][kFewT];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int qi = tid >> 4, pj = tid & 15;
    const int64_t q0 = (int64_t)blockIdx.x * kFewQ;
    const int d4 = d >> 2;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    unsigned long long best[2][2];  // queries warp and warp + 8 of the block
#pragma unroll
    for (int i = 0; i < 2; ++i)
        best[i][0] = best[i][1] = kNoKey;
    for (int t0 = 0; t0 < P; t0 += kFewT) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        for (int c0 = 0; c0 < d4; c0 += kFewD / 4) {
            __syncthreads();  // the chunk before has been read (and the tile before folded)
            {
                const int r = tid >> 4, c = c0 + (tid & 15);
                reinterpret_cast<float4 *>(qs[r])[tid & 15] =
                    q0 + r < nq && c < d4 ? __ldg(reinterpret_cast<const float4 *>(Q + (q0 + r) * d) + c) : zero4;
            }
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const int r = g * 16 + (tid >> 4), t = t0 + r, c = c0 + (tid & 15);
                reinterpret_cast<float4 *>(ts[r])[tid & 15] =
                    t < P && c < d4 ? __ldg(reinterpret_cast<const float4 *>(X + (int64_t)t * n / P * d) + c) : zero4;
            }
            __syncthreads();
#pragma unroll 4
            for (int c = 0; c < kFewD / 4; ++c) {
                const float4 a = reinterpret_cast<const float4 *>(qs[qi])[c];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 b = reinterpret_cast<const float4 *>(ts[pj + 16 * j])[c];
                    float u = b.x - a.x;
                    acc[j] = fmaf(u, u, acc[j]);
                    u = b.y - a.y;
                    acc[j] = fmaf(u, u, acc[j]);
                    u = b.z - a.z;
                    acc[j] = fmaf(u, u, acc[j]);
                    u = b.w - a.w;
                    acc[j] = fmaf(u, u, acc[j]);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            dist[qi][pj + 16 * j] = acc[j];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            unsigned long long s[4] = {best[i][0], best[i][1], kNoKey, kNoKey};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int t = t0 + 32 * h + lane;
                const float dv = dist[warp + 8 * i][32 * h + lane];
                if (t < P && !isnan(dv))
                    s[2 + h] = pack_key(dv, t);
            }
            if (t0 == 0) {
                best[i][0] = s[2];
                best[i][1] = s[3];
                warp_bitonic_sort<2>(best[i], lane);
            } else {
                warp_bitonic_sort<4>(s, lane);
                best[i][0] = s[0];
                best[i][1] = s[1];
            }
        }
    }
    const int m = n_seed < P ? n_seed : P;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int64_t q = q0 + warp + 8 * i;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = h * 32 + lane;
            if (q < nq && r < n_seed)
                out[q * n_seed + r] = r >= m || best[i][h] == kNoKey
                                          ? -1
                                          : (int32_t)((int64_t)(unsigned)(best[i][h] & 0xFFFFFFFFull) * n / P);
        }
    }
}

bool few_pivots(int64_t nq, int P)
{
    return P <= kFewT || (P <= 2 * kFewT && nq > kFewQ && nq <= (int64_t)kFewQ * num_sms());
}

// CTAs per cluster: how often the pivots of a query block are split.  The grid's time
// is waves x (tiles per CTA + the fixed selection and merge work, about 64
// coordinates' worth of a tile); the smallest split with the least such time is taken.
int pivot_split(int64_t nq, int P, int d, int64_t slots)
{
    const int64_t blocks = (nq + kPivQ - 1) / kPivQ;
    int best = 1;
    int64_t best_cost = INT64_MAX;
    for (int s = 1; s <= kPivMaxCluster; s *= 2) {
        if (s > 1 && P / s < 64)
            break;
        const int64_t share = (P + s - 1) / s;
        const int64_t waves = (blocks * s + slots - 1) / slots;
        const int64_t cost = waves * ((share + kPivT - 1) / kPivT * d + 64) * 256 + share;
        if (cost < best_cost) {
            best_cost = cost;
            best = s;
        }
    }
    return best;
}
}  // namespace
}  // namespace onng

using namespace onng;

extern "C" int onng_seeds_random(uint64_t global_seed, int64_t nq, int64_t n, int32_t n_seed, int32_t *out,
                                 onng_stream_t stream)
{
    ONNG_RANGE("onng_seeds_random");
    ONNG_REQUIRE(nq >= 0 && n > 0 && n <= INT32_MAX, ONNG_E_INVAL, "onng_seeds_random: bad sizes");
    ONNG_REQUIRE(n_seed >= 1 && n_seed <= kMaxSeed, ONNG_E_UNSUPPORTED, "onng_seeds_random: n_seed must be in [1, %d]",
                 kMaxSeed);
    if (nq == 0)
        return ONNG_OK;
    ONNG_REQUIRE(out, ONNG_E_INVAL, "onng_seeds_random: NULL output");
    seeds_random_kernel<<<(unsigned)((nq + 127) / 128), 128, 0, to_cuda(stream)>>>(global_seed, nq, n, n_seed, out);
    return check_launch("onng_seeds_random");
}

extern "C" size_t onng_seeds_pivot_workspace_bytes(int64_t n, int32_t d, int32_t n_pivot)
{
    (void)n;
    (void)d;
    (void)n_pivot;
    return 0;
}

extern "C" int onng_seeds_pivot(const float *X, int64_t n, int32_t d, const float *Q, int64_t nq, int32_t n_pivot,
                                int32_t n_seed, int32_t *out, void *ws, size_t ws_bytes, onng_stream_t stream)
{
    ONNG_RANGE("onng_seeds_pivot");
    (void)ws;
    (void)ws_bytes;
    ONNG_REQUIRE(nq >= 0 && n > 0 && n <= INT32_MAX, ONNG_E_INVAL, "onng_seeds_pivot: bad sizes");
    ONNG_REQUIRE(d > 0 && d % 4 == 0, ONNG_E_UNSUPPORTED, "onng_seeds_pivot: d must be a positive multiple of 4");
    ONNG_REQUIRE(n_pivot >= 1, ONNG_E_UNSUPPORTED, "onng_seeds_pivot: n_pivot must be >= 1");
    ONNG_REQUIRE(n_seed >= 1 && n_seed <= kMaxSeed, ONNG_E_UNSUPPORTED, "onng_seeds_pivot: n_seed in [1, %d]",
                 kMaxSeed);
    if (nq == 0)
        return ONNG_OK;
    ONNG_REQUIRE(X && Q && out, ONNG_E_INVAL, "onng_seeds_pivot: NULL pointer");
    ONNG_REQUIRE(aligned16(X) && aligned16(Q), ONNG_E_INVAL, "onng_seeds_pivot: X and Q must be 16-byte aligned");
    const int P = (int)std::min<int64_t>(n_pivot, n);
    if (few_pivots(nq, P)) {
        seeds_few_kernel<<<(unsigned)((nq + kFewQ - 1) / kFewQ), kPivThreads, 0, to_cuda(stream)>>>(X, n, d, Q, nq, P, n_seed,
                                                                                                    out);
        return check_launch("onng_seeds_pivot");
    }
    const size_t sm = sizeof(PivSmem);
    ONNG_CUDA_TRY(cudaFuncSetAttribute(reinterpret_cast<const void *>(seeds_pivot_kernel),
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                  "onng_seeds_pivot: smem attribute");
    const int S = pivot_split(nq, P, d, (int64_t)num_sms() * kPivMinCta);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((nq + kPivQ - 1) / kPivQ), (unsigned)S);
    cfg.blockDim = dim3(kPivThreads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = to_cuda(stream);
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1;
    attr.val.clusterDim.y = (unsigned)S;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    ONNG_CUDA_TRY(cudaLaunchKernelEx(&cfg, seeds_pivot_kernel, X, n, (int)d, Q, nq, P, (int)n_seed, out),
                  "onng_seeds_pivot");
    return check_launch("onng_seeds_pivot");
}
