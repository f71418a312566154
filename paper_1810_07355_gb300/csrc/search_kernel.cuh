// KnnSearch (Algorithm 1) on the GPU: one warp per query.  Device code of the
// search kernels; search_inst.cu instantiates it once per (vector type, chunks
// per lane) so the instantiations compile in parallel, and search.cu holds the
// host entry points.
//
// Per warp:
//   - the visited set C, in shared memory, as 512 buckets of a count and seven
//     16-bit tags with two bucket choices per id (the paper's Set/IsSet table,
//     Sec. 2.5, chains collisions off one inline id).  The id's bits go through a
//     bijection (a product with an odd constant modulo 2^bits); its top 9 bits name
//     the bucket and the rest, at most 14, are the tag, so the table is exact for n
//     up to 2^23 and a bucket is one 16-byte read.  A new id takes its slot from the
//     bucket's count with one shared-memory atomic.  Larger n use buckets of 8 ids.
//     An id that finds both of its buckets full moves the query to a per-warp bitmap
//     over all n ids in global memory (one atomicOr per new id), cleared when the
//     warp first needs it; the ids set there are logged and cleared when the query
//     ends.
//   - the candidate set S in three levels of (distance, id) keys: a head of up to 32
//     keys in registers (one per lane, in no order: a batch's keys take free lanes
//     together, and the minimum comes from two warp reductions that the prediction
//     of the next node needs anyway), an unsorted overflow in shared memory whose
//     keys are all >= every head key, and a per-warp spill pool in global memory
//     whose keys are all >= tau > every key above it.  So the head's least key is
//     the minimum of S; a level refills the one above only when
//     that one runs empty.  An entry beyond r(1+eps) can never be expanded (r
//     only shrinks, and popping it ends the search), so such entries are
//     dropped whenever a level is rebuilt.  S stays exact.
//   - the result set R, in registers, as a sorted list of at most k keys.
// The up-to-e_s neighbours of the expanded node are tested and the new ones'
// vectors gathered together: their ids go to shared gather slots in lane order, a
// half warp reads each vector (several in flight per lane) and one transposed butterfly reduction serves a round.  R then takes the k
// best of R and the batch, and S takes the batch members within the new
// r(1+eps).  Applying a batch at once yields the same R, the same r after the
// batch and, since S only loses entries that can never be expanded, the same
// expansion order as the one-at-a-time loop of Algorithm 1.
//
// The node expanded next is known as soon as the batch's distances are: it is
// the nearer of S's head and the batch's nearest member if that one will be
// pushed (its distance is within the bound before the batch).  Its adjacency
// row is loaded right then, so the load overlaps the R and S updates, and once
// the row is in, its neighbours' vectors are prefetched into L2 (float32, d <= 256).
//
// Adjacency is read from the CSR lists, or from an optional padded table
// adj [n, width] (-1 padded) that holds each node's first `width` entries, which
// saves the row-pointer indirection per expansion.
//
// Before (whole-warp gathers, a table of ids read as two 32-byte buckets, a sorted head
// with keys inserted one at a time, one copy of the batch per call site, every bitmap
// cleared before each search) and after, seeds included: 10,000 queries on 1M x 128
// bfloat16 3.27 -> 2.83 ms, float32 4.85 -> 4.30 ms; 137 queries for 100 neighbours
// 380 -> 285 us.  A batch of word vectors takes as long as its slowest query's chain of
// expansions: 200,000 x 100, 2,000 queries, 7 to 50 ms over five draws, 3,700 to 22,000
// expansions of 3,900 to 4,600 cycles, refills of the head 9 to 25 % of them.
//
// Distances are squared float32 sums of (q - x)^2; the bound r^2 (1 + eps)^2 is
// formed in double whenever r changes and kept rounded down to float32, which
// for a float32 d^2 decides d^2 <= r^2 (1 + eps)^2 exactly as the double
// comparison does.  For integer-valued inputs with squared distances below 2^24
// every decision then equals the float64 algorithm's.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "warp_sort.cuh"

// 1: float32 at d <= 256: once the adjacency row of the node expanded next has arrived, ask
// L2 for its neighbours' vectors (the next round's gathers then start from L2: 10,000
// queries on 1M x 128 4.8 ms without, 4.4 with).  The shorter vectors of the reduced forms
// are better off without the extra instructions (bfloat16 2.95 ms with, 2.84 without), and
// so are longer ones, of which most neighbours' lines are not needed (100,000 x 960, 2,000
// queries 7.8 ms with, 5.8 without).
#ifndef ONNG_SEARCH_PREFETCH
#define ONNG_SEARCH_PREFETCH 1
#endif
#ifndef ONNG_SEARCH_MAXV
#define ONNG_SEARCH_MAXV 8  // kernels are built for d <= 128 * ONNG_SEARCH_MAXV (1, 2, 4 or 8)
#endif
// Per vector type, for d <= 256 and k <= 32: 32-bit words of the visited table per warp
// (a power of two), shared-memory overflow keys per warp (128 or more, a power of
// two), the most vector pairs gathered per round at d <= 128 (4 or 8) and the resident
// CTAs per SM the registers are sized for.  What bounds the search is the instructions
// of an expansion (about 820 in float32 and 880 in bfloat16, 108 of them branches and
// their kind, each expansion waiting for the one before) more than its bytes, so resident
// warps help only while a whole batch's loads stay in registers: on 1M x 128, 10,000
// queries, bfloat16 ran 2.84 ms at 5 CTAs, 3.49 at 6 (spills), 3.05 at 4, and 2.97 with 4
// pairs a round; float32 4.41 ms at 4 CTAs, 4.59 at 5, 5.21 at 3, and 4.78 with 4 pairs.
#ifndef ONNG_SEARCH_F32_HV
#define ONNG_SEARCH_F32_HV 2048
#endif
#ifndef ONNG_SEARCH_F32_OVF
#define ONNG_SEARCH_F32_OVF 128
#endif
#ifndef ONNG_SEARCH_F32_PAIRS
#define ONNG_SEARCH_F32_PAIRS 8
#endif
#ifndef ONNG_SEARCH_F32_MINB
#define ONNG_SEARCH_F32_MINB 4
#endif
#ifndef ONNG_SEARCH_BF16_HV
#define ONNG_SEARCH_BF16_HV 2048
#endif
#ifndef ONNG_SEARCH_BF16_OVF
#define ONNG_SEARCH_BF16_OVF 128
#endif
#ifndef ONNG_SEARCH_BF16_PAIRS
#define ONNG_SEARCH_BF16_PAIRS 8
#endif
#ifndef ONNG_SEARCH_BF16_MINB
#define ONNG_SEARCH_BF16_MINB 5
#endif
#ifndef ONNG_SEARCH_FP8_HV
#define ONNG_SEARCH_FP8_HV 2048
#endif
#ifndef ONNG_SEARCH_FP8_OVF
#define ONNG_SEARCH_FP8_OVF 128
#endif
#ifndef ONNG_SEARCH_FP8_PAIRS
#define ONNG_SEARCH_FP8_PAIRS 8
#endif
#ifndef ONNG_SEARCH_FP8_MINB
#define ONNG_SEARCH_FP8_MINB 5
#endif

namespace onng {
namespace sk {

typedef unsigned long long u64;

constexpr unsigned FULL = 0xffffffffu;
constexpr int kWarpsPerCta = 4;
constexpr int kMaxK = 128;
constexpr int kMaxSeed = 64;
template <class T> struct Tune {
    static constexpr int hv = ONNG_SEARCH_F32_HV, ovf = ONNG_SEARCH_F32_OVF,
                         minb = ONNG_SEARCH_F32_MINB, pairs = ONNG_SEARCH_F32_PAIRS;
};
template <> struct Tune<__nv_bfloat16> {
    static constexpr int hv = ONNG_SEARCH_BF16_HV, ovf = ONNG_SEARCH_BF16_OVF,
                         minb = ONNG_SEARCH_BF16_MINB, pairs = ONNG_SEARCH_BF16_PAIRS;
};
template <> struct Tune<__nv_fp8_e4m3> {
    static constexpr int hv = ONNG_SEARCH_FP8_HV, ovf = ONNG_SEARCH_FP8_OVF,
                         minb = ONNG_SEARCH_FP8_MINB, pairs = ONNG_SEARCH_FP8_PAIRS;
};
constexpr int kVisitLog = 16384;     // ids logged per warp for clearing its bitmap
constexpr int kGlobalPool = 16384;   // default per-warp candidate spill pool entries
constexpr u64 kMaxKey = ~0ull;
constexpr int kFeat = 16;

struct SearchArgs {
    const int64_t *row_ptr;
    const int32_t *col;
    const int32_t *adj;
    int adj_w;
    const float *X;
    const uint16_t *Xb;
    const uint8_t *X8;     // e4m3 codes, dequantised as scale8[j] * e4m3
    const float *scale8;
    int64_t n;
    int d;
    const float *Q;
    int64_t nq;
    int k;      // results kept by the search (k_rerank for bf16)
    int k_out;  // results written
    int e_s;
    float eps;
    const float *eps_q;
    const int32_t *es_q;
    const int32_t *seeds;
    int n_seed;
    int max_exp;
    int32_t *out_ids;  // may be NULL (probe only)
    float *out_dist;
    int32_t *stats;
    float *feat;       // [nq, kFeat] probe features, or NULL
    float target;      // feature 0 (the recall the prediction is for)
    int *counter;     // next query, or NULL: every warp of the grid takes one query
    int tag_bits;     // visited table of 16-bit tags over ids of this many bits, or 0: table of ids
    unsigned *gbits;  // [slots, bits_words]: visited bitmap past the shared table (not initialised)
    int64_t bits_words;
    int *glog;        // [slots, kVisitLog]: ids set in the bitmap
    u64 *gpool;       // [slots, gpool_cap]
    int gpool_cap;    // spill pool entries per warp
};

template <int HV, int OVF> struct __align__(16) WarpSmem {
    int vis[HV];
    u64 ovf[OVF];
    int slot[32];  // ids of a batch's new nodes in lane order (gather slots)
    // per-query values read rarely, kept out of the registers
    double f2;            // (1 + eps)^2
    u64 seed1, seed2;     // probe features: the two nearest seeds,
    float seed_sum;       // the seeds' distances,
    int seed_cnt, rins;   // seeds evaluated, result insertions
    int es;               // entries scanned per node
    u64 tau;              // every key in the global pool is >= tau (kMaxKey when it is empty)
    int64_t beg, pf_beg;  // CSR row of the node expanded now, and of the one expanded next
    int pf_m;             // entries of the latter to scan
    int nlog;             // ids logged for clearing the bitmap
    unsigned flags;
#ifdef ONNG_CHECK
    unsigned canary[4];  // between this warp's arrays and the next warp's
#endif
};

#ifdef ONNG_CHECK
constexpr unsigned kCanary = 0x0C4A7A10u;
#endif

__host__ __device__ constexpr int log2i(int v) { return v <= 1 ? 0 : 1 + log2i(v >> 1); }

__device__ __forceinline__ unsigned lanemask_lt(int lane) { return (1u << lane) - 1u; }

__device__ __forceinline__ unsigned hash_id(int id) { return static_cast<unsigned>(id) * 0x9E3779B1u; }
__device__ __forceinline__ unsigned hash2_id(int id) { return (static_cast<unsigned>(id) ^ 0x5BD1E995u) * 0x7FEB352Du; }

__device__ __forceinline__ float key_d2(u64 k) { return __uint_as_float((unsigned)(k >> 32)); }
__device__ __forceinline__ int key_id(u64 k) { return (int)(unsigned)(k & 0xFFFFFFFFull); }

// f(0), f(1), ... f(N - 1) with constant indices.  A loop over a register array that
// is unrolled too late leaves the array, and the object around it, in local memory.
template <int N, class F> __device__ __forceinline__ void static_for(F f)
{
    if constexpr (N > 0) {
        static_for<N - 1>(f);
        f(std::integral_constant<int, N - 1>{});
    }
}

// least and greatest key of the warp: two reductions on 32-bit halves
__device__ __forceinline__ u64 warp_min_key(u64 k)
{
    const unsigned hi = (unsigned)(k >> 32), lo = (unsigned)k;
    const unsigned d = __reduce_min_sync(FULL, hi);
    return ((u64)d << 32) | __reduce_min_sync(FULL, hi == d ? lo : 0xFFFFFFFFu);
}
__device__ __forceinline__ u64 warp_max_key(u64 k)
{
    const unsigned hi = (unsigned)(k >> 32), lo = (unsigned)k;
    const unsigned d = __reduce_max_sync(FULL, hi);
    return ((u64)d << 32) | __reduce_max_sync(FULL, hi == d ? lo : 0u);
}

// Ascending list of 32*N keys striped over the warp: element e sits in v[e / 32]
// of lane e % 32.  Empty slots hold kMaxKey.
template <int N> struct RegList {
    u64 v[N];

    __device__ __forceinline__ void clear()
    {
        static_for<N>([&](auto c) {
            constexpr int i = decltype(c)::value;
            v[i] = kMaxKey; });
    }
    // number of elements smaller than key
    __device__ __forceinline__ int rank(u64 key) const
    {
        int r = 0;
        static_for<N>([&](auto c) {
            constexpr int i = decltype(c)::value;
            r += __popc(__ballot_sync(FULL, v[i] < key)); });
        return r;
    }
    // element e (uniform e < 32*N), broadcast to all lanes
    __device__ __forceinline__ u64 get(int e) const
    {
        u64 x = v[0];
        static_for<N>([&](auto c) {
            constexpr int i = decltype(c)::value;
            x = i == (e >> 5) ? v[i] : x; });
        return __shfl_sync(FULL, x, e & 31);
    }
    // inserts key at position pos (uniform); elements at positions >= limit are emptied
    __device__ __forceinline__ void insert_at(int pos, u64 key, int lane, int limit)
    {
        u64 carry = kMaxKey;  // old element i*32 - 1
        static_for<N>([&](auto c) {
            constexpr int i = decltype(c)::value;
           
            const u64 up = __shfl_up_sync(FULL, v[i], 1);
            const u64 last = __shfl_sync(FULL, v[i], 31);
            const u64 before = lane == 0 ? carry : up;
            const int e = i * 32 + lane;
            const u64 nv = e < pos ? v[i] : (e == pos ? key : before);
            v[i] = e < limit ? nv : kMaxKey;
            carry = last;
        });
    }
};

__device__ __forceinline__ u64 pack_f32x2(float lo, float hi)
{
    return ((u64)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}
__device__ __forceinline__ float lo_f32(u64 v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi_f32(u64 v) { return __uint_as_float((unsigned)(v >> 32)); }
static __device__ const float4 g_zero_quad = {0.f, 0.f, 0.f, 0.f};

// A quad is 4 consecutive coordinates of a stored vector: read() its bytes, value()
// the coordinates as float4 (e4m3 codes unscaled).
template <class T> struct Loader;
template <> struct Loader<float> {
    typedef float4 Raw;
    static __device__ __forceinline__ float4 value(float4 u) { return u; }
};
template <> struct Loader<__nv_bfloat16> {
    typedef uint2 Raw;
    static __device__ __forceinline__ float4 value(uint2 u)
    {
        return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                           __uint_as_float(u.y & 0xFFFF0000u));
    }
};
template <> struct Loader<__nv_fp8_e4m3> {
    typedef unsigned Raw;
    static __device__ __forceinline__ float4 value(unsigned u)
    {
        const __half2 lo(__nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(u & 0xFFFFu), __NV_E4M3));
        const __half2 hi(__nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(u >> 16), __NV_E4M3));
        const float2 a = __half22float2(lo), b = __half22float2(hi);
        return make_float4(a.x, a.y, b.x, b.y);
    }
};
template <class L> __device__ __forceinline__ typename L::Raw read_quad(const void *base, int64_t id, int d, int c)
{
    return __ldg(reinterpret_cast<const typename L::Raw *>(base) + (id * d >> 2) + c);
}

__device__ __forceinline__ float sqdiff4(float4 a, float4 b, float acc)
{
    float t = a.x - b.x;
    acc = fmaf(t, t, acc);
    t = a.y - b.y;
    acc = fmaf(t, t, acc);
    t = a.z - b.z;
    acc = fmaf(t, t, acc);
    t = a.w - b.w;
    return fmaf(t, t, acc);
}

// Sums v[g] over the warp for G values at once (G a power of two <= 16): each
// butterfly stage halves the values a lane holds by swapping halves with its
// partner, then plain butterflies finish.  Afterwards every lane holds the full
// sum of one value index: value g sits in the lanes whose bits 4 .. 5 - log2 G
// spell g, lane g << (5 - log2 G) among them.
template <int G, int OFF> __device__ __forceinline__ void tr_stage(float (&v)[G], int lane, int held)
{
    const int half = held >> 1;
    const bool hi = lane & OFF;
#pragma unroll
    for (int i = 0; i < G / 2; ++i) {
        if (i < half) {
            float send = hi ? v[i] : v[i + half];
            float keep = hi ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(FULL, send, OFF);
        }
    }
}

template <int G> __device__ __forceinline__ float transpose_reduce(float (&v)[G], int lane)
{
    static_assert(G == 1 || G == 2 || G == 4 || G == 8 || G == 16, "G");
    constexpr int m = log2i(G);
    if constexpr (m >= 1)
        tr_stage<G, 16>(v, lane, G);
    if constexpr (m >= 2)
        tr_stage<G, 8>(v, lane, G >> 1);
    if constexpr (m >= 3)
        tr_stage<G, 4>(v, lane, G >> 2);
    if constexpr (m >= 4)
        tr_stage<G, 2>(v, lane, G >> 3);
    float s = v[0];
#pragma unroll
    for (int off = 16 >> m; off >= 1; off >>= 1)
        s += __shfl_xor_sync(FULL, s, off);
    return s;
}

// ---------------------------------------------------------------- candidate levels, slow paths
//
// The refills and evictions between the levels of S run out of line, with their
// state passed by value: they are rare (once per some tens of expansions), and their
// sorts would otherwise take registers and code from every expansion.

struct Levels {
    int no, ng, nh;  // keys in the overflow, the global pool and the head
    unsigned flags;
    u64 tau;   // every global key is >= tau
    u64 head;  // this lane's head key (refill only)
};

__device__ __forceinline__ bool key_in_bound(u64 key, float bnd) { return key_d2(key) <= bnd; }

// Drops the overflow's out-of-bound keys; if `need` more still do not fit, sorts it
// and moves the farther half to the global pool (so at most OVF / 2 keys remain).
template <int OVF>
__device__ __noinline__ Levels make_room_slow(Levels s, u64 *ovf, u64 *gpool, int gcap, float bnd, int need, int lane)
{
    int w = 0;
    for (int base = 0; base < s.no; base += 32) {
        const int e = base + lane;
        const u64 kv = e < s.no ? ovf[e] : kMaxKey;
        const bool keep = e < s.no && key_in_bound(kv, bnd);
        const unsigned km = __ballot_sync(FULL, keep);
        __syncwarp();
        if (keep)
            ovf[w + __popc(km & lanemask_lt(lane))] = kv;
        w += __popc(km);
        __syncwarp();
    }
    s.no = w;
    if (s.no + need <= OVF)
        return s;
    // no > OVF - need >= OVF / 2, so the element at OVF / 2 is a real key
    constexpr int N = OVF / 32;
    u64 v[N];
#pragma unroll
    for (int i = 0; i < N; ++i)
        v[i] = i * 32 + lane < s.no ? ovf[i * 32 + lane] : kMaxKey;
    warp_bitonic_sort<N>(v, lane);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < N / 2; ++i)
        ovf[i * 32 + lane] = v[i];
    s.tau = __shfl_sync(FULL, v[N / 2], 0);
#pragma unroll
    for (int i = N / 2; i < N; ++i) {
        const unsigned m = __ballot_sync(FULL, v[i] != kMaxKey);
        const int dst = s.ng + __popc(m & lanemask_lt(lane));
        if (v[i] != kMaxKey && dst < gcap)
            gpool[dst] = v[i];
        if (s.ng + __popc(m) > gcap)
            s.flags |= ONNG_FLAG_S_OVERFLOW;
        s.ng = min(s.ng + __popc(m), gcap);
    }
    __syncwarp();
    s.no = OVF / 2;
    return s;
}

// Refills the empty head with the 32 nearest in-bound overflow keys.  An empty
// overflow first takes the nearest in-bound global keys, at most 96 of them, in two
// passes over the pool.  In the first every lane keeps the 8 least of the keys it reads;
// any key below the least of the lanes' 8th ones is among those kept, so the kept keys up
// to that one (about 110 of a large pool) are its nearest.  The second drops what was
// taken or is out of bound.  Both have several loads in flight, since one warp reads the
// whole pool twice: a query of 22,000 expansions over word vectors came here 202 times
// for a pool of 7,800 keys on average, a quarter of its cycles.
template <int OVF> __device__ __noinline__ Levels refill_slow(Levels s, u64 *ovf, u64 *gpool, float bnd, int lane)
{
    if (s.no == 0) {
        u64 v[8];  // ascending
#pragma unroll
        for (int i = 0; i < 8; ++i)
            v[i] = kMaxKey;
        for (int base = lane; base < s.ng + lane; base += 128) {
            u64 k[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                k[i] = base + 32 * i < s.ng ? gpool[base + 32 * i] : kMaxKey;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                u64 x = key_in_bound(k[i], bnd) ? k[i] : kMaxKey;
                if (!__any_sync(FULL, x < v[7]))
                    continue;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const bool less = x < v[j];
                    const u64 lo = less ? x : v[j];
                    x = less ? v[j] : x;
                    v[j] = lo;
                }
            }
        }
        u64 cut = warp_min_key(v[7]);
        warp_bitonic_sort<8>(v, lane);
        static_assert(OVF >= 128, "a refill of 96 keys leaves the overflow room");
        const u64 last = __shfl_sync(FULL, v[2], 31);
        cut = last < cut ? last : cut;
        s.no = 0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const bool take = v[i] <= cut && v[i] != kMaxKey;
            if (take)
                ovf[i * 32 + lane] = v[i];
            s.no += __popc(__ballot_sync(FULL, take));
        }
        // keep the global entries beyond the cut that are still in bound
        int w = 0;
        u64 mn = kMaxKey;
        for (int base = 0; base < s.ng; base += 256) {
            u64 k[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                k[i] = base + 32 * i + lane < s.ng ? gpool[base + 32 * i + lane] : kMaxKey;
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const bool keep = k[i] > cut && key_in_bound(k[i], bnd);
                const unsigned km = __ballot_sync(FULL, keep);
                if (keep) {
                    gpool[w + __popc(km & lanemask_lt(lane))] = k[i];
                    mn = k[i] < mn ? k[i] : mn;
                }
                w += __popc(km);
            }
            __syncwarp();
        }
        s.ng = w;
        s.tau = warp_min_key(mn);
        __syncwarp();
    }
    constexpr int N = OVF / 32;
    u64 v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int e = i * 32 + lane;
        const u64 kv = e < s.no ? ovf[e] : kMaxKey;
        v[i] = (kv != kMaxKey && key_in_bound(kv, bnd)) ? kv : kMaxKey;
    }
    warp_bitonic_sort<N>(v, lane);
    s.head = v[0];
    s.nh = __popc(__ballot_sync(FULL, v[0] != kMaxKey));
    int m = 0;
#pragma unroll
    for (int i = 1; i < N; ++i)
        m += __popc(__ballot_sync(FULL, v[i] != kMaxKey));
    __syncwarp();
#pragma unroll
    for (int i = 1; i < N; ++i)
        if ((i - 1) * 32 + lane < m)
            ovf[(i - 1) * 32 + lane] = v[i];
    s.no = m;
    __syncwarp();
    return s;
}

// Every member is inlined: one call out of line would move the whole search state
// from registers to local memory (the k > 32 kernels ran that way).
template <int V, class T, int HV, int KR> struct Warp {
    // A half warp reads each vector, so a lane holds two quads of it per 128 coordinates;
    // the whole warp does where the query, its scales and the lists leave no registers for
    // that (FP8 above d = 512 with lists of more than 32).  d = 960, n = 100,000, ms with the
    // whole warp and with halves: float32, one query 4.11, 1.98, 2,000 queries 12.9, 5.8;
    // bfloat16 2.91, 2.46 and 8.45, 6.55; FP8 3.18, 2.72 and 8.15, 7.19, but 6.15, 7.19 with
    // lists of 100.
    static constexpr bool kHalf = V <= 4 || KR == 1 || !std::is_same<T, __nv_fp8_e4m3>::value;
    static constexpr int G = 2;  // vectors per gather round of the whole-warp form
    // Most vector pairs gathered per round by half warps, of stored vectors and of the
    // float32 ones of a reduced form's rerank: a round's loads are in flight together, as
    // far as registers go.
    template <class L>
    static constexpr int kPairs = V == 1 ? Tune<T>::pairs : V == 2 ? 4 : V == 8 && !std::is_same<L, Loader<T>>::value ? 1 : 2;
    static constexpr int kOvf = Tune<T>::ovf;  // shared-memory overflow keys
    static_assert(kOvf >= 64 && (kOvf & (kOvf - 1)) == 0, "the overflow holds a power of two >= 64 keys");
    static_assert(HV % 8 == 0, "the visited table holds whole buckets of 8 ids");
    static constexpr int kTagBuckets = HV / 4, kTagBucketBits = log2i(HV / 4);
    static_assert(kTagBuckets == 1 << kTagBucketBits, "a power of two of tag buckets");
    WarpSmem<HV, kOvf> &sm;
    const SearchArgs &a;
    const void *xs;  // vectors the search reads (float32 or bfloat16)
    int lane;
    int slot;  // this warp's share of the workspace
    // Query coordinates of this lane.  Whole-warp form: quad lane + 32 v (sv: the e4m3
    // scales).  Half-warp form: quads a = l + 32 v and b = a + 16 (l = lane % 16),
    // negated and in pairs: float32 (a.x a.y)(a.z a.w)(b.x b.y)(b.z b.w), whose
    // coordinates arrive in that order, else (a.x b.x)(a.y b.y)(a.z b.z)(a.w b.w)
    // (sp: the e4m3 scales in the same pairs, not negated).
    float4 qv[kHalf ? 1 : V];
    float4 sv[kHalf ? 1 : V];
    u64 qp[kHalf ? V : 1][4];
    u64 sp[kHalf ? V : 1][4];
    u64 head;  // a candidate of the head (kMaxKey: none)
    RegList<KR> res;
    // per-query state, uniform across the warp
    int nh, no, ng, cnt, ndc, nexp, nscan;
    u64 pf_key;  // the least key of S if known (kMaxKey: not known): the node expanded next
    int pf_id;   // its first 32 neighbours, already loaded
#ifdef ONNG_CHECK
    int64_t nnz_chk;  // row_ptr[n]: every row must lie inside col
#endif
    bool in_row;  // padded table: this lane holds one of the first 32 entries scanned
    bool spill, rset, padded, wide, capped;  // wide: rows of more than 32 entries (padded table)
    bool bits_clean;  // the bitmap is all zero between queries (false until this warp first needs it)
    float r2;
    // r^2 (1 + eps)^2 in double rounded down to float32: for a float32 d^2, d^2 <= the
    // double bound exactly when d^2 <= bnd (the double lies in [bnd, next float above
    // bnd), so no float lies strictly between), which keeps the double comparison's
    // decisions in float32
    float bnd;

    __device__ __forceinline__ Warp(WarpSmem<HV, kOvf> &s, const SearchArgs &args, const void *x, int ln, int sl)
        : sm(s), a(args), xs(x), lane(ln), slot(sl), bits_clean(false)
    {
    }

    // this warp's bitmap, log and pool in the workspace
    __device__ __forceinline__ unsigned *gbits() const { return a.gbits + (int64_t)slot * a.bits_words; }
    __device__ __forceinline__ int *glog() const { return a.glog + (int64_t)slot * kVisitLog; }
    __device__ __forceinline__ u64 *gpool() const { return a.gpool + (int64_t)slot * a.gpool_cap; }

    // ---------------------------------------------------------------- visited set

    // The query's first use of the bitmap: from here on new ids go there.  The bitmap
    // is cleared when the warp first comes here (a query leaves it all zero), which
    // few queries do: clearing it for every resident warp before each search cost
    // 65 us of a 3.3 ms batch at n = 1M.
    __device__ __forceinline__ void start_spill()
    {
        spill = true;
        if (!bits_clean) {
            for (int64_t i = lane; i < a.bits_words / 4; i += 32)
                reinterpret_cast<uint4 *>(gbits())[i] = make_uint4(0u, 0u, 0u, 0u);
            bits_clean = true;
            __syncwarp();
            __threadfence();
        }
    }

    // Appends the ids of the lanes with `set` (bits this warp set) to the bitmap's log.
    __device__ __forceinline__ void log_bits(bool set, int id)
    {
        const unsigned m = __ballot_sync(FULL, set);
        if (set) {
            const int pos = sm.nlog + __popc(m & lanemask_lt(lane));
            if (pos < kVisitLog)
                glog()[pos] = id;
        }
        __syncwarp();
        if (lane == 0)
            sm.nlog += __popc(m);
        __syncwarp();
    }

    // A 16-byte bucket of the tag table holds a 16-bit count and seven tags (bit 15
    // set, bit 14 the choice).  Whether one of its halfwords equals the tag replicated
    // in t: bit 15 or 31 of the result is set if so (x - 1 borrows through a zero
    // halfword; a false bit can only appear above a true one).
    static __device__ __forceinline__ unsigned has_tag(const uint4 &w, unsigned t)
    {
        const unsigned x = w.x ^ t, y = w.y ^ t, z = w.z ^ t, u = w.w ^ t;
        return ((x - 0x00010001u) & ~x) | ((y - 0x00010001u) & ~y) | ((z - 0x00010001u) & ~z) |
               ((u - 0x00010001u) & ~u);
    }

    // Test-and-set of a batch (one id per lane, -1 = none) in the tag table.  True if
    // newly visited; an id held by several lanes (repeated seeds) counts once, at its
    // lowest lane.
    __device__ __forceinline__ bool visit_tags(int id)
    {
        const bool has = id >= 0;
        const int rem = a.tag_bits - kTagBucketBits;
        const unsigned idmask = (1u << a.tag_bits) - 1u, tagmask = (1u << rem) - 1u;
        const unsigned h1 = ((unsigned)id * 0x9E3779B1u) & idmask, h2 = ((unsigned)id * 0x7FEB352Du) & idmask;
        const unsigned b1 = h1 >> rem, b2 = h2 >> rem;
        const unsigned t1 = 0x8000u | (h1 & tagmask), t2 = 0xC000u | (h2 & tagmask);
        const uint4 *bk = reinterpret_cast<const uint4 *>(sm.vis);
        const uint4 p = bk[b1], q = bk[b2];
        const bool found = ((has_tag(p, t1 * 0x10001u) | has_tag(q, t2 * 0x10001u)) & 0x80008000u) != 0u;
        bool want = has && !found;
        if (spill) {
            if (__match_any_sync(FULL, id) & lanemask_lt(lane))
                want = false;
            const unsigned bit = 1u << (id & 31);
            const bool isnew = want && (atomicOr(&gbits()[id >> 5], bit) & bit) == 0;
            log_bits(isnew, id);
            return isnew;
        }
        __syncwarp();  // every lane's `used` and tags are from before the batch
        unsigned short *half = reinterpret_cast<unsigned short *>(sm.vis);
        const unsigned used = p.x & 0xFFFFu;
        unsigned pos = 0;
        if (want) {
            pos = atomicAdd(reinterpret_cast<unsigned *>(sm.vis) + 4 * b1, 1u) & 0xFFFFu;
            if (pos < 7u)
                half[8 * b1 + 1 + pos] = (unsigned short)t1;
        }
        // rare: two lanes of the batch in one bucket, or a full first bucket
        if (__any_sync(FULL, want && (pos != used || pos >= 7u))) {
            const unsigned same = __match_any_sync(FULL, id);
            if (same & lanemask_lt(lane))
                want = false;
            __syncwarp();
            bool full = false;
            if (want && pos >= 7u) {
                const unsigned pos2 = atomicAdd(reinterpret_cast<unsigned *>(sm.vis) + 4 * b2, 1u) & 0xFFFFu;
                full = pos2 >= 7u;
                if (!full)
                    half[8 * b2 + 1 + pos2] = (unsigned short)t2;
            }
            if (__any_sync(FULL, full)) {
                // both buckets full: this id and every later new one go to the bitmap
                start_spill();
                if (full)
                    atomicOr(&gbits()[id >> 5], 1u << (id & 31));
                log_bits(full, id);
            }
        }
        __syncwarp();
        return want;
    }

    // The same in the table of ids, for n beyond what the tags can tell apart:
    // HV / 8 buckets of 8 ids, filled in slot order, two bucket choices per id.
    // Every lane first looks its id up in both buckets; new ids then take free
    // slots of their first bucket (lanes aiming at one bucket in lane order),
    // the rest of their second; an id that finds both full goes to the bitmap,
    // and so does every later new id of the query.  True if newly visited.
    __device__ __forceinline__ bool visit_ids(int id)
    {
        constexpr unsigned NB = HV / 8;
        // an id held by several lanes (repeated seeds) counts once, at its lowest lane
        if (__match_any_sync(FULL, id) & lanemask_lt(lane))
            id = -1;
        const bool has = id >= 0;
        const unsigned b1 = has ? __umulhi(hash_id(id), NB) : 0u;
        const unsigned b2 = has ? __umulhi(hash2_id(id), NB) : 0u;
        const int4 *bk = reinterpret_cast<const int4 *>(sm.vis);
        const int4 p0 = bk[2 * b1], p1 = bk[2 * b1 + 1], q0 = bk[2 * b2], q1 = bk[2 * b2 + 1];
        const bool found = has && (p0.x == id || p0.y == id || p0.z == id || p0.w == id || p1.x == id ||
                                   p1.y == id || p1.z == id || p1.w == id || q0.x == id || q0.y == id ||
                                   q0.z == id || q0.w == id || q1.x == id || q1.y == id || q1.z == id || q1.w == id);
        const bool want = has && !found;
        if (spill) {
            const unsigned bit = 1u << (id & 31);
            const bool isnew = want && (atomicOr(&gbits()[id >> 5], bit) & bit) == 0;
            log_bits(isnew, id);
            return isnew;
        }
        const unsigned wm = __ballot_sync(FULL, want);
        __syncwarp();  // the buckets are read before any is written; a batch always orders shared memory
        if (!wm)
            return false;
        const int used1 = (p0.x != -1) + (p0.y != -1) + (p0.z != -1) + (p0.w != -1) + (p1.x != -1) +
                          (p1.y != -1) + (p1.z != -1) + (p1.w != -1);
        const unsigned g1 = __match_any_sync(FULL, want ? b1 : 0xFFFFFFFFu);
        const int r1 = __popc(g1 & wm & lanemask_lt(lane));
        const bool ok1 = want && used1 + r1 < 8;
        if (ok1)
            sm.vis[b1 * 8 + used1 + r1] = id;
        __syncwarp();
        const bool want2 = want && !ok1;
        const unsigned wm2 = __ballot_sync(FULL, want2);
        if (wm2) {
            const int4 s0 = bk[2 * b2], s1 = bk[2 * b2 + 1];  // after the first-choice stores
            const int used2 = (s0.x != -1) + (s0.y != -1) + (s0.z != -1) + (s0.w != -1) + (s1.x != -1) +
                              (s1.y != -1) + (s1.z != -1) + (s1.w != -1);
            const unsigned g2 = __match_any_sync(FULL, want2 ? b2 : 0xFFFFFFFFu);
            const int r2 = __popc(g2 & wm2 & lanemask_lt(lane));
            const bool ok2 = want2 && used2 + r2 < 8;
            if (ok2)
                sm.vis[b2 * 8 + used2 + r2] = id;
            __syncwarp();
            const bool want3 = want2 && !ok2;
            if (__ballot_sync(FULL, want3)) {
                // both buckets full: this id and every later new one go to the bitmap
                start_spill();
                if (want3)
                    atomicOr(&gbits()[id >> 5], 1u << (id & 31));
                log_bits(want3, id);
            }
        }
        return want;
    }

    // Leaves the bitmap all zero for the next query: clears the logged words,
    // or the whole bitmap if the log overflowed.
    __device__ __forceinline__ void clear_bits()
    {
        if (!spill)
            return;
        if (sm.nlog <= kVisitLog) {
            for (int i = lane; i < sm.nlog; i += 32)
                gbits()[glog()[i] >> 5] = 0u;
        } else {
            for (int64_t i = lane; i < a.bits_words; i += 32)
                gbits()[i] = 0u;
        }
        __syncwarp();
    }

    // ---------------------------------------------------------------- distances

    // One vector's part of a lane in the half-warp form: adds quads a and b of chunk v
    // to the two chains in `acc` (low half a, high half b).
    template <class L>
    __device__ __forceinline__ u64 accumulate(u64 acc, const typename L::Raw &ra, const typename L::Raw &rb, int v)
    {
        const float4 xa = L::value(ra), xb = L::value(rb);
        if constexpr (std::is_same<L, Loader<float>>::value) {
            // the coordinates of a quad are neighbouring registers: packed differences,
            // then one chain of multiply-adds per quad
            u64 n0, n1, n2, n3;
            if constexpr (std::is_same<T, float>::value) {
                n0 = qp[v][0], n1 = qp[v][1], n2 = qp[v][2], n3 = qp[v][3];
            } else {
                n0 = pack_f32x2(lo_f32(qp[v][0]), lo_f32(qp[v][1]));
                n1 = pack_f32x2(lo_f32(qp[v][2]), lo_f32(qp[v][3]));
                n2 = pack_f32x2(hi_f32(qp[v][0]), hi_f32(qp[v][1]));
                n3 = pack_f32x2(hi_f32(qp[v][2]), hi_f32(qp[v][3]));
            }
            const u64 u0 = add_f32x2(pack_f32x2(xa.x, xa.y), n0), u1 = add_f32x2(pack_f32x2(xa.z, xa.w), n1);
            const u64 u2 = add_f32x2(pack_f32x2(xb.x, xb.y), n2), u3 = add_f32x2(pack_f32x2(xb.z, xb.w), n3);
            float sa = fmaf(lo_f32(u0), lo_f32(u0), lo_f32(acc)), sb = fmaf(lo_f32(u2), lo_f32(u2), hi_f32(acc));
            sa = fmaf(hi_f32(u0), hi_f32(u0), sa), sb = fmaf(hi_f32(u2), hi_f32(u2), sb);
            sa = fmaf(lo_f32(u1), lo_f32(u1), sa), sb = fmaf(lo_f32(u3), lo_f32(u3), sb);
            return pack_f32x2(fmaf(hi_f32(u1), hi_f32(u1), sa), fmaf(hi_f32(u3), hi_f32(u3), sb));
        } else {
            const float a4[4] = {xa.x, xa.y, xa.z, xa.w}, b4[4] = {xb.x, xb.y, xb.z, xb.w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                u64 x = pack_f32x2(a4[c], b4[c]);
                if constexpr (std::is_same<L, Loader<__nv_fp8_e4m3>>::value)
                    // dequantised with a rounded product: a packed multiply and the packed add
                    // after it came out as one rounding, a multiply-add of zero does not
                    // (10,000 queries on 1M x 128: 3.61 ms with two scalar multiplies, 3.39 so)
                    x = fma_f32x2(sp[v][c], x, 0ull);
                const u64 u = add_f32x2(x, qp[v][c]);
                acc = fma_f32x2(u, u, acc);
            }
            return acc;
        }
    }

    // Gathers slots b0 .. b0 + 2 PG - 1 by half warps (slot b0 + 2 p + h by half h;
    // slots past m repeat the last one) and returns this lane's distance if its slot
    // is among them, else `mine`.  Per vector the sums run as in the whole-warp form:
    // a chain per quad column, then columns 16, 8, 4, 2 and 1 apart.
    template <class L, int PG> __device__ __forceinline__ float gather_pairs(const void *base, int b0, int m, int rank,
                                                                             bool mine_in, float mine)
    {
        constexpr int QB = sizeof(typename L::Raw);
        const int chunks = a.d >> 2, l = lane & 15, h = lane >> 4;
        const unsigned row_bytes = (unsigned)chunks * QB;
        // quads past d read a zero in place of the vector (their query coordinates are 0)
        const char *at[V][2];
        unsigned step[V][2];
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int c = l + 16 * t + 32 * v;
                at[v][t] = c < chunks ? static_cast<const char *>(base) + c * QB : reinterpret_cast<const char *>(&g_zero_quad);
                step[v][t] = c < chunks ? row_bytes : 0u;
            }
        typename L::Raw raw[PG][V][2];
#pragma unroll
        for (int p = 0; p < PG; ++p) {
            const unsigned id = (unsigned)sm.slot[min(b0 + 2 * p + h, m - 1)];
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int t = 0; t < 2; ++t)
                    raw[p][v][t] = __ldg(reinterpret_cast<const typename L::Raw *>(at[v][t] + (u64)id * step[v][t]));
        }
        float s[PG];
#pragma unroll
        for (int p = 0; p < PG; ++p) {
            u64 acc = 0ull;
#pragma unroll
            for (int v = 0; v < V; ++v)
                acc = accumulate<L>(acc, raw[p][v][0], raw[p][v][1], v);
            s[p] = lo_f32(acc) + hi_f32(acc);
        }
        if constexpr (PG >= 2)
            tr_stage<PG, 8>(s, lane, PG);
        if constexpr (PG >= 4)
            tr_stage<PG, 4>(s, lane, PG / 2);
        if constexpr (PG == 8)
            tr_stage<PG, 2>(s, lane, 2);
        float r = s[0];
#pragma unroll
        for (int off = 8 / PG; off >= 1; off >>= 1)
            r += __shfl_xor_sync(FULL, r, off);
        // pair p of half h sits in lane 16 h + (16 / PG) p
        const int w = rank - b0;
        const float x = __shfl_sync(FULL, r, ((w & 1) << 4) | (((w >> 1) * (16 / PG)) & 15));
        return mine_in && w >= 0 && w < 2 * PG ? x : mine;
    }

    // Squared distances of the ids held by the lanes in `mask`; returns this lane's.
    // The ids go to shared slots in lane order.  Half-warp form: a round gathers 16
    // slots (8 when no more are left), two vectors per load instruction, so a batch's
    // loads are in flight together at half the instructions of one vector per load.
    // Whole-warp form: round b takes slots b .. b + G - 1; empty slots read row 0 and
    // are masked.
    template <class L> __device__ __forceinline__ float distances(const void *base, int id, unsigned mask)
    {
        const int chunks = a.d >> 2;
        const int m = __popc(mask);
        const bool mine_in = (mask >> lane) & 1u;
        const int rank = __popc(mask & lanemask_lt(lane));
        if (mine_in)
            sm.slot[rank] = id;
        __syncwarp();
        float mine = 0.0f;
        if constexpr (kHalf) {
            constexpr int PG = kPairs<L>, few = PG < 4 ? PG : 4;
            int b0 = 0;
            while (m - b0 > 8 && PG == 8) {
                mine = gather_pairs<L, PG>(base, b0, m, rank, mine_in, mine);
                b0 += 2 * PG;
            }
            for (; b0 < m; b0 += 2 * few)
                mine = gather_pairs<L, few>(base, b0, m, rank, mine_in, mine);
        } else {
            for (int b0 = 0; b0 < m; b0 += G) {
                int gid[G];
#pragma unroll
                for (int g = 0; g < G; ++g)
                    gid[g] = b0 + g < m ? sm.slot[b0 + g] : 0;
                float4 xv[G][V];
#pragma unroll
                for (int g = 0; g < G; ++g)
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        const int c = lane + 32 * v;
                        xv[g][v] = L::value(read_quad<L>(base, gid[g], a.d, c < chunks ? c : 0));
                        if constexpr (std::is_same<L, Loader<__nv_fp8_e4m3>>::value) {
                            // dequantise with a rounded product (never fused into the difference)
                            xv[g][v] = make_float4(__fmul_rn(sv[v].x, xv[g][v].x), __fmul_rn(sv[v].y, xv[g][v].y),
                                                   __fmul_rn(sv[v].z, xv[g][v].z), __fmul_rn(sv[v].w, xv[g][v].w));
                        }
                    }
                float acc[G];
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    acc[g] = 0.0f;
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        int c = lane + 32 * v;
                        if (b0 + g < m && c < chunks)
                            acc[g] = sqdiff4(qv[v], xv[g][v], acc[g]);
                    }
                }
                const float red = transpose_reduce<G>(acc, lane);
                // value g of the round sits in lane g << (5 - log2 G)
                const int r = rank - b0;
                const float s = __shfl_sync(FULL, red, (r & (G - 1)) << (5 - log2i(G)));
                if (mine_in && r >= 0 && r < G)
                    mine = s;
            }
        }
        __syncwarp();
        return mine;
    }

    // ---------------------------------------------------------------- result list

    // Inserts key into R of kk entries; false if R keeps them (key would be evicted).
    __device__ __forceinline__ bool r_insert(u64 key, int kk)
    {
        const int pos = res.rank(key);
        if (pos >= kk)
            return false;
        res.insert_at(pos, key, lane, kk);
        cnt = min(cnt + 1, kk);
        return true;
    }

    __device__ __forceinline__ void raise(unsigned flag)
    {
        if (lane == 0)
            sm.flags |= flag;
    }

    // Bounds-checked builds (-DONNG_CHECK): an id read from the graph outside
    // [-1, n) becomes -1 (no access) and flags the query ONNG_FLAG_CHECK.  Called
    // by the whole warp.  Other builds trust the graph.
    __device__ __forceinline__ int graph_id(int id)
    {
#ifdef ONNG_CHECK
        const bool bad = id < -1 || id >= a.n;
        if (__any_sync(FULL, bad))
            raise(ONNG_FLAG_CHECK);
        return bad ? -1 : id;
#else
        return id;
#endif
    }

    __device__ __forceinline__ double bound2() const { return (rset && !isinf(sm.f2)) ? (double)r2 * sm.f2 : INFINITY; }

    __device__ __forceinline__ void update_bound()
    {
        bnd = __double2float_rd(bound2());
    }

    // ---------------------------------------------------------------- candidate pool

    // Appends the keys of the lanes with `put` to the global pool.
    __device__ __forceinline__ void gpool_append(bool put, u64 key)
    {
        unsigned m = __ballot_sync(FULL, put);
        if (!m)
            return;
        if (put) {
            int dst = ng + __popc(m & lanemask_lt(lane));
            if (dst < a.gpool_cap)
                gpool()[dst] = key;
        }
        if (ng + __popc(m) > a.gpool_cap)
            raise(ONNG_FLAG_S_OVERFLOW);
        ng = min(ng + __popc(m), a.gpool_cap);
    }

    // Makes room for `need` (<= 32) more keys in the overflow.
    __device__ __forceinline__ void make_room(int need)
    {
        const Levels r = make_room_slow<kOvf>({no, ng, 0, 0u, sm.tau, kMaxKey}, sm.ovf, gpool(), a.gpool_cap, bnd, need, lane);
        no = r.no;
        ng = r.ng;
        if (r.flags)
            raise(r.flags);
        __syncwarp();
        sm.tau = r.tau;
        __syncwarp();
    }

    __device__ __forceinline__ void ovf_append(u64 key)
    {
        if (no == kOvf)
            make_room(1);
        if (key >= sm.tau) {
            gpool_append(lane == 0, key);
            return;
        }
        if (lane == 0)
            sm.ovf[no] = key;
        ++no;
        __syncwarp();
    }

    // Refills the empty head with the 32 nearest in-bound overflow keys.
    __device__ __forceinline__ void refill_head()
    {
        if (no == 0 && ng == 0)
            return;
        __syncwarp();  // keys that other lanes appended to the levels
        const Levels r = refill_slow<kOvf>({no, ng, 0, 0u, sm.tau, kMaxKey}, sm.ovf, gpool(), bnd, lane);
        no = r.no;
        ng = r.ng;
        nh = r.nh;
        head = r.head;
        __syncwarp();
        sm.tau = r.tau;
        __syncwarp();
    }

    // Appends the keys of the lanes with `put` (all < tau) to the shared overflow,
    // making room first if they do not fit; keys that end up >= tau after that
    // go to the global pool.
    __device__ __forceinline__ void ovf_append_many(bool put, u64 key)
    {
        unsigned m = __ballot_sync(FULL, put);
        if (!m)
            return;
        if (no + __popc(m) > kOvf) {
            make_room(__popc(m));  // tau may drop
            const bool far = put && key >= sm.tau;
            gpool_append(far, key);
            put = put && !far;
            m = __ballot_sync(FULL, put);
        }
        if (put)
            sm.ovf[no + __popc(m & lanemask_lt(lane))] = key;
        no += __popc(m);
        __syncwarp();
    }

    // Adds the batch members marked `push` to S.  Keys >= tau go to the global pool and
    // keys >= the head's maximum to the overflow, each in one step; the others take
    // free lanes of the head together (the j-th of them the j-th free lane, named
    // through the gather slots).  Only when they outnumber the free lanes are they
    // placed in turn, each pushing the head's maximum out.  While S is the head alone
    // (no overflow, empty pool) every key goes to the head.
    __device__ __forceinline__ void pool_push(bool push, u64 key)
    {
        unsigned pm = __ballot_sync(FULL, push);
        if (!pm)
            return;
        if (no > 0 || ng > 0) {
            const bool far = push && key >= sm.tau;
            gpool_append(far, key);
            push = push && !far;
            const u64 hmax = nh > 0 ? warp_max_key(head == kMaxKey ? 0ull : head) : kMaxKey;
            const bool to_ovf = push && key >= hmax;
            ovf_append_many(to_ovf, key);
            push = push && !to_ovf;
            pm = __ballot_sync(FULL, push);
        }
        const int c = __popc(pm);
        if (nh + c <= 32) {
            const bool free = head == kMaxKey;
            const unsigned fm = __ballot_sync(FULL, free);
            if (push)
                sm.slot[__popc(pm & lanemask_lt(lane))] = lane;
            __syncwarp();
            const int j = __popc(fm & lanemask_lt(lane));
            const bool take = free && j < c;
            const u64 got = __shfl_sync(FULL, key, take ? sm.slot[j] : 0);
            if (take)
                head = got;
            nh += c;
            return;
        }
        while (pm) {
            const int src = __ffs(pm) - 1;
            pm &= pm - 1;
            const u64 ck = __shfl_sync(FULL, key, src);
            if (ck >= sm.tau) {
                gpool_append(lane == 0, ck);
                continue;
            }
            const u64 hmax = nh > 0 ? warp_max_key(head == kMaxKey ? 0ull : head) : kMaxKey;
            const bool only_head = no == 0 && ng == 0;
            if (ck < hmax || (only_head && nh < 32)) {
                if (nh == 32) {
                    ovf_append(hmax);  // the evicted maximum stays >= the rest of the head
                    if (head == hmax)
                        head = kMaxKey;
                    --nh;
                }
                const unsigned fm = __ballot_sync(FULL, head == kMaxKey);
                if (lane == __ffs(fm) - 1)
                    head = ck;
                ++nh;
            } else {
                ovf_append(ck);
            }
        }
    }

    // ---------------------------------------------------------------- one batch

    // The CSR row of node s: its start, and how many of its entries are scanned.
    __device__ __forceinline__ int csr_row(int s, int64_t &beg)
    {
        beg = a.row_ptr[s];
        int64_t deg = a.row_ptr[s + 1] - beg;
#ifdef ONNG_CHECK
        if (beg < 0 || deg < 0 || beg + deg > nnz_chk) {
            raise(ONNG_FLAG_CHECK);
            deg = 0;
        }
#endif
        return deg < (int64_t)sm.es ? (int)deg : sm.es;
    }

    // Tests a batch of up to 32 ids (one per lane, -1 = none) and applies it.
    // `predict` (the last batch of an expansion): loads the first 32 neighbours of the
    // node expanded next, from the padded table (1) or the CSR lists (2).
    __device__ __forceinline__ void batch(int id, bool init, int predict)
    {
        const bool isnew = a.tag_bits ? visit_tags(id) : visit_ids(id);
        const unsigned mask = __ballot_sync(FULL, isnew);
        if (!mask)
            return;
        const int nnew = __popc(mask);
        ndc += nnew;
        __syncwarp();
        float d2 = distances<Loader<T>>(xs, id, mask);
        u64 key = pack_key(d2, id);
        if (init && a.feat) {
            float sd = isnew ? sqrtf(d2) : 0.f;
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1)
                sd += __shfl_xor_sync(FULL, sd, off);
            if (lane == 0) {
                sm.seed_sum += sd;
                sm.seed_cnt += nnew;
            }
        }
        int64_t nbeg = 0;
        int nm = 0;
        if (predict) {
            // the next pop is the least of the head and the batch members that will be
            // pushed (checked against the bound once R is updated)
            const u64 mine = isnew && d2 <= bnd && key < head ? key : head;
            pf_key = warp_min_key(mine);
            if (pf_key != kMaxKey) {
                if (predict == 1)
                    pf_id = graph_id(in_row ? a.adj[(int64_t)key_id(pf_key) * a.adj_w + lane] : -1);
                else
                    nm = csr_row(key_id(pf_key), nbeg);
            }
        }
        // R <- the best kk of R and the batch
        unsigned cm = __ballot_sync(FULL, isnew && (init || !rset || d2 <= r2));
        bool moved = false;
        while (cm) {
            int src = __ffs(cm) - 1;
            cm &= cm - 1;
            u64 ck = __shfl_sync(FULL, key, src);
            if (init || !rset || key_d2(ck) <= r2) {
                if (r_insert(ck, a.k) && a.feat && !init && lane == 0)
                    ++sm.rins;
                if (!init && cnt == a.k) {
                    rset = moved = true;
                    r2 = key_d2(res.get(a.k - 1));
                }
            }
        }
        if (moved)  // the bound's double product only when r changed
            update_bound();
        // S <- S + batch members within r(1+eps)
        pool_push(isnew && d2 <= bnd, key);
        // a batch member that was not pushed after all is not in S (the same comparison as
        // the push: no key is within a bound that is NaN, from a NaN eps or distance)
        if (predict && !(key_d2(pf_key) <= bnd))
            pf_key = kMaxKey;
        if (predict == 2 && pf_key != kMaxKey) {
            // the row bounds were loading during the updates above
            pf_id = graph_id(lane < nm ? a.col[nbeg + lane] : -1);
            if (lane == 0) {
                sm.pf_beg = nbeg;
                sm.pf_m = nm;
            }
        }
#if ONNG_SEARCH_PREFETCH
        if (sizeof(T) == 4 && V <= 2 && predict && pf_key != kMaxKey && pf_id >= 0) {
            // the row of the next node is in: its neighbours' vectors into L2
            const int bytes = a.d * (int)sizeof(T);  // float32 4, bfloat16 2, e4m3 1 byte per coordinate
            const char *row = static_cast<const char *>(xs) + (int64_t)pf_id * bytes;
            for (int off = 0; off < bytes; off += 128)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(row + off));
        }
#endif
    }

    __device__ __forceinline__ void run(int q)
    {
        const int d = a.d;
        const float *qp_row = a.Q + (int64_t)q * d;
        const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 *q4 = reinterpret_cast<const float4 *>(qp_row), *s4 = reinterpret_cast<const float4 *>(a.scale8);
        const int chunks = d >> 2;
        if constexpr (kHalf) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int ca = (lane & 15) + 32 * v, cb = ca + 16;
                const float4 x = ca < chunks ? __ldg(q4 + ca) : zero4, y = cb < chunks ? __ldg(q4 + cb) : zero4;
                if constexpr (std::is_same<T, float>::value) {
                    qp[v][0] = pack_f32x2(-x.x, -x.y);
                    qp[v][1] = pack_f32x2(-x.z, -x.w);
                    qp[v][2] = pack_f32x2(-y.x, -y.y);
                    qp[v][3] = pack_f32x2(-y.z, -y.w);
                } else {
                    qp[v][0] = pack_f32x2(-x.x, -y.x);
                    qp[v][1] = pack_f32x2(-x.y, -y.y);
                    qp[v][2] = pack_f32x2(-x.z, -y.z);
                    qp[v][3] = pack_f32x2(-x.w, -y.w);
                }
                if constexpr (std::is_same<T, __nv_fp8_e4m3>::value) {
                    const float4 f = ca < chunks ? __ldg(s4 + ca) : zero4, g = cb < chunks ? __ldg(s4 + cb) : zero4;
                    sp[v][0] = pack_f32x2(f.x, g.x);
                    sp[v][1] = pack_f32x2(f.y, g.y);
                    sp[v][2] = pack_f32x2(f.z, g.z);
                    sp[v][3] = pack_f32x2(f.w, g.w);
                }
            }
        } else {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int c = lane + 32 * v;
                qv[v] = c < chunks ? __ldg(q4 + c) : zero4;
                if constexpr (std::is_same<T, __nv_fp8_e4m3>::value)
                    sv[v] = c < chunks ? __ldg(s4 + c) : zero4;
            }
        }
        const float eps = a.eps_q ? a.eps_q[q] : a.eps;
        int es = a.es_q ? a.es_q[q] : a.e_s;
        if (es <= 0)
            es = INT_MAX;
        padded = a.adj != nullptr && es <= a.adj_w;
        wide = es > 32;
        in_row = lane < es;
        if (lane == 0) {
            sm.f2 = isinf(eps) ? INFINITY : (1.0 + (double)eps) * (1.0 + (double)eps);
            sm.seed_sum = 0.f;
            sm.seed_cnt = sm.rins = 0;
            sm.es = es;
            sm.tau = kMaxKey;
            sm.nlog = 0;
            sm.flags = 0;
        }
        const int fill = a.tag_bits ? 0 : -1;
        const int4 empty = make_int4(fill, fill, fill, fill);
        for (int i = lane; i < HV / 4; i += 32)
            reinterpret_cast<int4 *>(sm.vis)[i] = empty;
        head = kMaxKey;
        res.clear();
        nh = no = ng = cnt = ndc = nexp = nscan = 0;
        pf_key = kMaxKey;
#ifdef ONNG_CHECK
        nnz_chk = a.row_ptr[a.n];
#endif
        spill = rset = capped = false;
        r2 = INFINITY;
        bnd = INFINITY;
        __syncwarp();
        // One loop over batches, so that batch() is expanded once: the seeds first
        // (`init`), then each expanded node's row in chunks of 32 entries.  The last
        // chunk of a row loads the next node's: from the padded table (rows of at most
        // 32 entries) or the CSR lists.
        bool init = true;
        int c0 = 0, m = a.n_seed, node = 0;
        int id = lane < m ? seed_id(a.seeds[(int64_t)q * m + lane]) : -1;
        for (;;) {
            batch(id, init, init || c0 + 32 < m ? 0 : !padded ? 2 : wide ? 0 : 1);
            c0 += 32;
            if (c0 < m) {
                const int e = c0 + lane;
                if (init) {
                    id = e < m ? seed_id(a.seeds[(int64_t)q * m + e]) : -1;
                    continue;
                }
                if (!padded) {
                    id = graph_id(e < m ? a.col[sm.beg + e] : -1);
                    continue;
                }
                id = graph_id(e < m ? a.adj[(int64_t)node * a.adj_w + e] : -1);
                const unsigned got = __ballot_sync(FULL, id >= 0);
                nscan += __popc(got);
                if (got)
                    continue;  // else the padded row ended
            }
            if (init) {
                init = false;
                if (a.feat) {
                    const u64 s1 = warp_min_key(head), s2 = warp_min_key(head == s1 ? kMaxKey : head);
                    if (lane == 0) {
                        sm.seed1 = s1;
                        sm.seed2 = s2;
                    }
                }
            }
            // the next node whose row holds any entry
            bool done = false;
            do {
                if (nh == 0) {
                    refill_head();
                    if (nh == 0) {
                        done = true;
                        break;
                    }
                }
                const bool ready = pf_key != kMaxKey;
                const u64 top = ready ? pf_key : warp_min_key(head);
                pf_key = kMaxKey;
                if (a.max_exp > 0 && nexp >= a.max_exp) {
                    // capped with a candidate still to expand (not merely pending termination)
                    capped = key_d2(top) <= bnd;
                    if (capped)
                        raise(ONNG_FLAG_LIMIT);
                    done = true;
                    break;
                }
                if (head == top)
                    head = kMaxKey;
                --nh;
                if (nh == 0)
                    refill_head();
                if (key_d2(top) > bnd) {
                    done = true;
                    break;
                }
                ++nexp;
                node = key_id(top);
                c0 = 0;
                if (padded) {
                    m = wide ? sm.es : 32;
                    if (!ready || wide)
                        pf_id = graph_id(in_row ? a.adj[(int64_t)node * a.adj_w + lane] : -1);
                    id = pf_id;
                    const unsigned got = __ballot_sync(FULL, id >= 0);
                    nscan += __popc(got);
                    if (!got)
                        m = 0;
                } else {
                    int64_t beg;
                    if (ready) {
                        __syncwarp();
                        beg = sm.pf_beg;
                        m = sm.pf_m;
                        id = pf_id;
                    } else {
                        m = csr_row(node, beg);
                        id = graph_id(lane < m ? a.col[beg + lane] : -1);
                    }
                    if (m > 32 && lane == 0)
                        sm.beg = beg;
                    nscan += m;
                }
            } while (m == 0);
            if (done)
                break;
        }
        __syncwarp();
    }

    // a seed id past the index is no seed
    __device__ __forceinline__ int seed_id(int id) const { return id < 0 || id >= a.n ? -1 : id; }

    // Rescores the kept list in float32 against X and keeps the best k_out.
    __device__ __forceinline__ void rerank()
    {
        u64 nk[KR] = {};
#pragma unroll 1
        for (int i = 0; i < KR; ++i) {  // one copy of the gather; the lists stay in registers
            u64 old = res.v[0];
#pragma unroll
            for (int j = 1; j < KR; ++j)
                old = i == j ? res.v[j] : old;
            const int id = old == kMaxKey ? -1 : key_id(old);
            const unsigned mask = __ballot_sync(FULL, id >= 0);
            const float dv = distances<Loader<float>>(a.X, id, mask);
            const u64 key = id >= 0 ? pack_key(dv, id) : kMaxKey;
#pragma unroll
            for (int j = 0; j < KR; ++j)
                nk[j] = i == j ? key : nk[j];
        }
        res.clear();
        cnt = 0;
#pragma unroll
        for (int i = 0; i < KR; ++i) {
            unsigned m = __ballot_sync(FULL, nk[i] != kMaxKey);
            while (m) {
                const int src = __ffs(m) - 1;
                m &= m - 1;
                r_insert(__shfl_sync(FULL, nk[i], src), a.k_out);
            }
        }
    }

    // Probe features after the capped search (all logs natural, distances Euclidean).
    __device__ __forceinline__ void features(int64_t q)
    {
        const u64 rbk = res.get(0);
        const u64 rkk = res.get(cnt > 0 ? cnt - 1 : 0);
        const u64 hk = warp_min_key(head);
        if (lane != 0)
            return;
        const float e6 = 1e-6f;
        const u64 seed1 = sm.seed1, seed2 = sm.seed2;
        const int seed_cnt = sm.seed_cnt, rins = sm.rins;
        const float seed_sum = sm.seed_sum;
        const float ds1 = seed1 == kMaxKey ? 0.f : sqrtf(key_d2(seed1));
        const float ds2 = seed2 == kMaxKey ? ds1 : sqrtf(key_d2(seed2));
        const float dmean = seed_cnt > 0 ? seed_sum / (float)seed_cnt : ds1;
        const float rb = cnt > 0 ? sqrtf(key_d2(rbk)) : ds1;
        const float rk = cnt > 0 ? sqrtf(key_d2(rkk)) : ds1;
        const float bound = (rset && !isinf(sm.f2)) ? (float)sqrt(bound2()) : INFINITY;
        float top = capped ? fminf(sqrtf(key_d2(hk)), bound) : bound;
        if (isinf(top))
            top = rk;
        float *f = a.feat + q * kFeat;
        f[0] = a.target;
        f[1] = logf(ds1 + e6);
        f[2] = logf((ds2 + e6) / (ds1 + e6));
        f[3] = logf((dmean + e6) / (ds1 + e6));
        f[4] = logf((rb + e6) / (ds1 + e6));
        f[5] = logf((rk + e6) / (rb + e6));
        f[6] = logf((top + e6) / (rb + e6));
        f[7] = (float)ndc / (float)max(1, seed_cnt + nscan);
        f[8] = (float)nexp / (float)max(1, a.max_exp);
        f[9] = log1pf((float)ndc);
        f[10] = (float)rins / (float)max(1, ndc);
        f[11] = rset ? 1.f : 0.f;
        f[12] = logf((rk + e6) / (ds1 + e6));
        f[13] = log1pf((float)nscan);
        f[14] = capped ? 1.f : 0.f;
        f[15] = logf((float)a.d) / 8.f;
    }

    __device__ __forceinline__ void write(int64_t q)
    {
        if (a.feat)
            features(q);
        const int k = a.k_out;
#pragma unroll
        for (int i = 0; i < KR; ++i) {
            const int e = i * 32 + lane;
            if (e < k && a.out_ids) {
                a.out_ids[q * k + e] = e < cnt ? key_id(res.v[i]) : -1;
                a.out_dist[q * k + e] = e < cnt ? sqrtf(key_d2(res.v[i])) : INFINITY;
            }
        }
#ifdef ONNG_CHECK
        if (__any_sync(FULL, lane < 4 && sm.canary[lane] != kCanary + lane))
            raise(ONNG_FLAG_CHECK);
        __syncwarp();
#endif
        if (a.stats && lane == 0) {
            a.stats[q * 4 + 0] = ndc;
            a.stats[q * 4 + 1] = nexp;
            a.stats[q * 4 + 2] = nscan;
            a.stats[q * 4 + 3] = (int)sm.flags;
        }
    }
};

// Resident CTAs per SM the register budget is sized for.  Shared memory holds
// 6 CTAs of warps with a 2048-slot table and 128 overflow keys (37 KB a CTA).  Above d =
// 256 a round's loads need more registers than three CTAs leave (100,000 x 960 float32,
// 2,000 queries: 9.8 ms at 3, 7.8 at 2).
template <class T> __host__ __device__ constexpr int min_blocks(int V, int KR)
{
    return V > 2 ? 2 : KR == 1 ? Tune<T>::minb : 3;
}

template <int V, class T, int HV, int KR>
__global__ void __launch_bounds__(kWarpsPerCta * 32, min_blocks<T>(V, KR)) search_kernel(const __grid_constant__ SearchArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    auto *smem = reinterpret_cast<WarpSmem<HV, Tune<T>::ovf> *>(smem_raw);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int slot = (int)blockIdx.x * kWarpsPerCta + warp;
    const void *xs = std::is_same<T, float>::value           ? static_cast<const void *>(a.X)
                     : std::is_same<T, __nv_bfloat16>::value ? static_cast<const void *>(a.Xb)
                                                              : static_cast<const void *>(a.X8);
    Warp<V, T, HV, KR> w(smem[warp], a, xs, lane, slot);
#ifdef ONNG_CHECK
    if (lane < 4)
        smem[warp].canary[lane] = kCanary + lane;
    __syncwarp();
#endif
    for (int64_t next = slot; next < a.nq; next = a.counter ? slot : a.nq) {
        int q = (int)next;
        if (a.counter) {
            int c = 0;
            if (lane == 0)
                c = atomicAdd(a.counter, 1);
            q = __shfl_sync(FULL, c, 0);
            if (q >= a.nq)
                break;
        }
        w.run(q);
        w.clear_bits();
        if constexpr (!std::is_same<T, float>::value)
            w.rerank();
        w.write(q);
        __syncwarp();
    }
}

struct Launch {
    void (*fn)(SearchArgs);
    size_t smem;
    int table;  // 32-bit words of the visited table
};

// The search kernel for vector type T with V float4 chunks per lane (d <= 128 V)
// and a kept list of at most 32 KR keys (KR = 1 or kMaxK / 32); defined in
// search_inst.cu.
template <class T, int V, int KR> Launch pick();
#define ONNG_SEARCH_DECLARE_PICK(T, V)   \
    template <> Launch pick<T, V, 1>(); \
    template <> Launch pick<T, V, kMaxK / 32>();
#define ONNG_SEARCH_DECLARE_PICKS(T)    \
    ONNG_SEARCH_DECLARE_PICK(T, 1)      \
    ONNG_SEARCH_DECLARE_PICK(T, 2)      \
    ONNG_SEARCH_DECLARE_PICK(T, 4)      \
    ONNG_SEARCH_DECLARE_PICK(T, 8)
ONNG_SEARCH_DECLARE_PICKS(float)
ONNG_SEARCH_DECLARE_PICKS(__nv_bfloat16)
ONNG_SEARCH_DECLARE_PICKS(__nv_fp8_e4m3)
#undef ONNG_SEARCH_DECLARE_PICKS
#undef ONNG_SEARCH_DECLARE_PICK

}  // namespace sk
}  // namespace onng
