// Exact k-nearest-neighbour lists (the exact kNN graph that replaces the
// paper's approximate graph, Sec. 2.6) without materialising the n x n matrix.
//
// knn_tile_kernel: a CTA owns 16, 32, 64 or 128 query rows and sweeps its share of the
// base columns in tiles of 128.  The tile of squared distances |q|^2 + |x|^2 - 2 q.x is
// formed in registers (up to 8 x 8 per thread, packed float32 FMA).  Entries below the row's
// running threshold are appended to a per-row candidate buffer in global
// memory (mostly L2); when a buffer may not absorb another tile it is merged
// with the row's best list (merge_row) and the
// threshold drops to the list's last entry.  The best list keeps KC >= k + 16
// entries so that rounding in the expanded form cannot push a true neighbour
// out of it.
//
// knn_final_kernel: rescoring of the KC survivors of each row by direct
// difference sum (q_j - x_j)^2 in float32, ordering by (distance, id) and
// output of the first k as ids and Euclidean lengths.
//
// Integer-valued inputs whose squared norms stay below 2^23 are ranked exactly:
// every product, partial sum and the expanded form are exact in float32.
//
// Which sweep runs (onng_knn): byte-valued inputs at d = 32 .. 128 take the
// tensor cores exactly (knn_tc_kernel); other non-integer inputs at d >= 32 take
// the tensor cores in a split bfloat16 form (knn_tcs_kernel) whose survivors are
// rescored; everything else, and problems smaller than one tile, the SIMT sweep.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "warp_sort.cuh"

namespace onng {
namespace {

constexpr int BN = 128, BK = 16, NT = 256;
constexpr int BUF = 256;  // candidate buffer entries per row (>= 2 * BN)
constexpr unsigned long long EMPTY_KEY = 0x7F800000FFFFFFFFull;  // (+inf, id -1)

__device__ __forceinline__ float key_dist(unsigned long long k) { return __uint_as_float((unsigned)(k >> 32)); }
__device__ __forceinline__ int key_id(unsigned long long k) { return (int)(unsigned)(k & 0xFFFFFFFFull); }

__global__ void norms_kernel(const float *__restrict__ X, int64_t n, int d, float *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (row >= n)
        return;
    const float4 *p = reinterpret_cast<const float4 *>(X + row * d);
    float s = 0.f;
    for (int c = lane; c < (d >> 2); c += 32) {
        float4 v = __ldg(p + c);
        s = fmaf(v.x, v.x, s);
        s = fmaf(v.y, v.y, s);
        s = fmaf(v.z, v.z, s);
        s = fmaf(v.w, v.w, s);
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1)
        s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0)
        out[row] = s;
}

// Compact warp merge of lists (knn_merge_kernel): the stage loop runs at run time, only
// the loop over a lane's registers is unrolled.
// Element e = i * 32 + lane lives in v[i] of lane `lane`.

// compare-exchange of registers i and i ^ JR (partners 32 JR elements apart),
// ascending where bit `size` of the element index is clear
template <int JR, int N>
__device__ __forceinline__ void cas_regs(unsigned long long (&v)[N], int lane, int size)
{
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int ii = i ^ JR;
        if (ii > i) {
            const bool asc = (((i << 5) | lane) & size) == 0;
            const unsigned long long a = v[i], b = v[ii];
            const bool sw = asc ? (a > b) : (a < b);
            v[i] = sw ? b : a;
            v[ii] = sw ? a : b;
        }
    }
}

// one bitonic step at distance j elements for sequences of length `size`
template <int N>
__device__ __forceinline__ void bitonic_step(unsigned long long (&v)[N], int lane, int size, int j)
{
    if (j >= 32) {
        const int jr = j >> 5;
        if constexpr (N >= 2)
            if (jr == 1)
                cas_regs<1>(v, lane, size);
        if constexpr (N >= 4)
            if (jr == 2)
                cas_regs<2>(v, lane, size);
        if constexpr (N >= 8)
            if (jr == 4)
                cas_regs<4>(v, lane, size);
    } else {
        const bool lower = (lane & j) == 0;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const bool asc = (((i << 5) | lane) & size) == 0;
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, v[i], j);
            const bool take_min = lower == asc;
            v[i] = take_min ? (o < v[i] ? o : v[i]) : (o > v[i] ? o : v[i]);
        }
    }
}

// ascending merge of a bitonic sequence of 32 N keys (one bitonic merge pass with
// every element's direction ascending)
template <int N> __device__ void warp_merge_compact(unsigned long long (&v)[N], int lane)
{
#pragma unroll 1
    for (int j = 16 * N; j > 0; j >>= 1)
        bitonic_step<N>(v, lane, 64 * N, j);
}

// One exchange of a bitonic network between lanes: the lower of the two lanes JL apart
// keeps the smaller key where `up`.
template <int JL> __device__ __forceinline__ void lane_cas(unsigned long long &v, bool up, int lane)
{
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, v, JL);
    const bool keep_min = ((lane & JL) == 0) == up;
    v = (o < v) == keep_min ? o : v;
}
__device__ __forceinline__ void reg_cas(unsigned long long &a, unsigned long long &b, bool up)
{
    const unsigned long long x = a, y = b;
    const bool swap = (y < x) == up;
    a = swap ? y : x;
    b = swap ? x : y;
}
// steps of distance 2 JL .. 2 and 1 elements on pairs (element 2 lane + register)
template <int JL> __device__ __forceinline__ void pair_steps(unsigned long long (&v)[2], bool up, int lane)
{
    if constexpr (JL > 0) {
        lane_cas<JL>(v[0], up, lane);
        lane_cas<JL>(v[1], up, lane);
        pair_steps<JL / 2>(v, up, lane);
    } else {
        reg_cas(v[0], v[1], up);
    }
}

// The warp merges row gr's cnt buffered keys into its sorted best list of KC
// keys and returns list entry kth (< KC), whose distance is the new threshold.
//
// A merge holds up its whole CTA (the next tile's accumulators stay taken), so its
// latency counts: element 64 h + 2 lane + r of the list sits in register m[h][r] of
// `lane`, which makes every distance of 1 and of 64 or more an exchange of registers,
// and the buffer goes in 64 keys at a time, sorted descending: the smaller of each pair
// (list's last 64, sorted keys) and the rest of the list are a bitonic sequence holding
// the KC smallest.  The network is unrolled: 15 of its 21 sort and 5 of its 7 merge
// steps cross lanes.  1M x 128 bytes, k = 100 (about 20 merges a row): 344 -> 277 ms
// against loops over the steps with element 32 r + lane (9,800 cycles a merge, now 5,900
// with eight warps at it).
template <int KC>
__device__ __noinline__ unsigned long long merge_row(int64_t gr, int cnt, int kth, unsigned long long *__restrict__ best,
                                                     const unsigned long long *__restrict__ buf, int lane)
{
    static_assert(BUF % 64 == 0 && (KC & (KC - 1)) == 0, "whole chunks and a power-of-two list");
    constexpr int H = KC < 64 ? 1 : KC / 64;
    ulonglong2 *const list = reinterpret_cast<ulonglong2 *>(best + gr * KC) + lane;
    const ulonglong2 *const row = reinterpret_cast<const ulonglong2 *>(buf + gr * BUF) + lane;
    const bool held = KC >= 64 || lane < KC / 2;  // a list of 32 is the first half of one of 64
    unsigned long long m[H][2];
    __syncwarp();  // the row's own thread wrote the buffer
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const ulonglong2 b = held ? list[h * 32] : make_ulonglong2(EMPTY_KEY, EMPTY_KEY);
        m[h][0] = b.x;
        m[h][1] = b.y;
    }
#pragma unroll 1
    for (int o = 0; o < cnt; o += 64) {
        const ulonglong2 b = row[o >> 1];
        unsigned long long a[2] = {o + 2 * lane < cnt ? b.x : EMPTY_KEY, o + 2 * lane + 1 < cnt ? b.y : EMPTY_KEY};
        reg_cas(a[0], a[1], (lane & 1) == 0);
        pair_steps<1>(a, (lane & 2) == 0, lane);
        pair_steps<2>(a, (lane & 4) == 0, lane);
        pair_steps<4>(a, (lane & 8) == 0, lane);
        pair_steps<8>(a, (lane & 16) == 0, lane);
        pair_steps<16>(a, false, lane);
#pragma unroll
        for (int r = 0; r < 2; ++r)
            m[H - 1][r] = a[r] < m[H - 1][r] ? a[r] : m[H - 1][r];
#pragma unroll
        for (int jh = H / 2; jh > 0; jh /= 2)
#pragma unroll
            for (int h = 0; h < H; ++h)
                if (!(h & jh)) {
                    reg_cas(m[h][0], m[h | jh][0], true);
                    reg_cas(m[h][1], m[h | jh][1], true);
                }
#pragma unroll
        for (int h = 0; h < H; ++h)
            pair_steps<16>(m[h], true, lane);
    }
    unsigned long long kv = m[0][0];
#pragma unroll
    for (int h = 0; h < H; ++h) {
        if (held)
            list[h * 32] = make_ulonglong2(m[h][0], m[h][1]);
        if (kth >> 6 == h)
            kv = kth & 1 ? m[h][1] : m[h][0];
    }
    return __shfl_sync(0xffffffffu, kv, (kth >> 1) & 31);
}

// Which share of a sweep a CTA takes.  The row blocks below `main` are swept by gm
// CTAs each (share g of gm), the later ones by gt: these would fill only part of the
// last wave, so more CTAs share each of them.  Every share keeps a best list and a
// candidate buffer of its own: lists g < gm of all rows, then lists gm .. gt - 1 of
// the rows from block `main` on.
struct Shares {
    int64_t main, blocks;  // row blocks swept by gm CTAs each; all row blocks
    int gm, gt;
    __host__ __device__ int64_t ctas() const { return main * gm + (blocks - main) * gt; }
};

struct Share {
    int64_t block;
    int g, G;
};

__device__ __forceinline__ Share my_share(const Shares &sh, int64_t cta)
{
    const int64_t cut = sh.main * sh.gm;
    if (cta < cut)
        return {cta / sh.gm, (int)(cta % sh.gm), sh.gm};
    return {sh.main + (cta - cut) / sh.gt, (int)((cta - cut) % sh.gt), sh.gt};
}

// first key (or buffer entry) of list g of row 0 if it existed: rows are `per` entries
// apart; `rows` is the block size
__host__ __device__ __forceinline__ int64_t list_base(const Shares &sh, int g, int64_t nq, int rows, int64_t per)
{
    if (g < sh.gm)
        return (int64_t)g * nq * per;
    const int64_t first = sh.main * rows, tail = nq - first;
    return ((int64_t)sh.gm * nq + (int64_t)(g - sh.gm) * tail - first) * per;
}

// The shares of a sweep of `tiles` base tiles by `blocks` row blocks on `slots`
// resident CTAs: whole waves unsplit (gm CTAs a block), and the blocks of the last,
// partial wave split so that its CTAs end soonest (ceil(blocks gt / slots) rounds of
// tiles / gt tiles, plus about `warm` tiles' worth for every further list: its
// threshold starts from nothing).  200,000 x 100 floats, k = 100 (782 row blocks, 5.1
// waves): the whole build 67.5 -> 64.2 ms.  Row blocks of `rows` queries; no more than
// `lists` lists in all (at least gm nq).
Shares plan_shares(int64_t nq, int64_t rows, int64_t tiles, int64_t slots, int gm, int64_t warm, int64_t lists)
{
    Shares sh;
    const int64_t blocks = (nq + rows - 1) / rows;
    sh.blocks = blocks;
    sh.gm = sh.gt = gm;
    sh.main = blocks * gm / slots * slots / gm;
    const int64_t rem = blocks - sh.main;
    if (rem == 0)
        return sh;
    const int64_t tail = nq - sh.main * rows;
    int64_t best = INT64_MAX;
    for (int64_t g = gm; g <= std::min<int64_t>(std::max<int64_t>(tiles / 4, gm), std::max<int64_t>(8, slots / rem)); ++g) {
        if (gm * nq + (g - gm) * tail > lists)
            break;
        const int64_t cost = (rem * g + slots - 1) / slots * ((tiles + g - 1) / g + warm);
        if (cost < best) {
            best = cost;
            sh.gt = (int)g;
        }
    }
    if (sh.gt == gm)
        sh.main = blocks;
    return sh;
}

constexpr int kSweepSms = 152;  // SMs the sweeps are planned for

// The float32 sweep.  RM rows x 8 columns per thread, so a row block is BM = 16 RM
// rows: sweeps of fewer than 128 queries take the smallest block that holds them
// (the arithmetic of padding rows is what bounded them).  The products use packed
// multiply-adds (two columns per instruction, the same rounding as the scalar form);
// the queries sit in shared memory duplicated, the base tile coordinate-major, and the
// next slab's global loads are in flight during the arithmetic of the present one.
// With fewer row blocks than the device holds, several CTAs share a block's base tiles
// (Shares) and knn_merge_kernel merges their lists: 50 queries over 1M x 128 ran on
// one CTA before, 147.5 ms; 0.85 ms now (1.02 with the merges as loops).
template <int RM> struct TileSmem {
    float2 As[2][BK][16 * RM];
    float Bs[2][BK][BN + 4];
    float thr[16 * RM];
    int cnt[16 * RM];
    float qn[16 * RM];
};

template <int KC, int RM>
__global__ void __launch_bounds__(NT, 2)
    knn_tile_kernel(const float *__restrict__ X, int64_t n, int d, const float *__restrict__ Q, int64_t nq,
                    int64_t self_offset, const float *__restrict__ xn, const float *__restrict__ qn, const Shares sh,
                    unsigned long long *__restrict__ best, unsigned long long *__restrict__ buf)
{
    constexpr int RB = 16 * RM;                            // rows of a block
    constexpr int QLD = RB * BK / 4 >= NT ? RB * BK / 4 / NT : 1;  // query quads per thread
    extern __shared__ __align__(16) unsigned char tile_raw[];
    TileSmem<RM> &sm = *reinterpret_cast<TileSmem<RM> *>(tile_raw);
    auto &As = sm.As;
    auto &Bs = sm.Bs;
    auto &s_thr = sm.thr;
    auto &s_cnt = sm.cnt;
    auto &s_qn = sm.qn;

    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int lane = tid & 31, warp = tid >> 5;
    const Share me = my_share(sh, blockIdx.x);
    const int64_t row0 = me.block * RB;
    const int64_t tiles = (n + BN - 1) / BN;
    const int64_t t0 = tiles * me.g / me.G, t1 = tiles * (me.g + 1) / me.G;
    best += list_base(sh, me.g, nq, RB, KC);
    buf += list_base(sh, me.g, nq, RB, BUF);

    for (int r = tid; r < RB; r += NT) {
        s_thr[r] = INFINITY;
        s_cnt[r] = 0;
        s_qn[r] = row0 + r < nq ? qn[row0 + r] : 0.f;
    }
    for (int e = tid; e < RB * KC; e += NT) {
        const int64_t gr = row0 + e / KC;
        if (gr < nq)
            best[gr * KC + e % KC] = EMPTY_KEY;
    }

    // staging: quad kq of row m of the slab; rows past the end and coordinates past d read as 0
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 qv[QLD], xv[2];
    auto fetch = [&](int64_t tile, int k0) {
#pragma unroll
        for (int t = 0; t < QLD; ++t) {
            const int f = tid + t * NT, m = f >> 2, kq = (f & 3) << 2;
            qv[t] = m < RB && row0 + m < nq && k0 + kq < d
                        ? __ldg(reinterpret_cast<const float4 *>(Q + (row0 + m) * d + k0 + kq)) : zero4;
        }
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int f = tid + t * NT, m = f >> 2, kq = (f & 3) << 2;
            xv[t] = tile * BN + m < n && k0 + kq < d
                        ? __ldg(reinterpret_cast<const float4 *>(X + (tile * BN + m) * d + k0 + kq)) : zero4;
        }
    };
    auto store = [&](int b) {
#pragma unroll
        for (int t = 0; t < QLD; ++t) {
            const int f = tid + t * NT, m = f >> 2, kq = (f & 3) << 2;
            if (m < RB) {
                As[b][kq][m] = make_float2(qv[t].x, qv[t].x);
                As[b][kq + 1][m] = make_float2(qv[t].y, qv[t].y);
                As[b][kq + 2][m] = make_float2(qv[t].z, qv[t].z);
                As[b][kq + 3][m] = make_float2(qv[t].w, qv[t].w);
            }
        }
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int f = tid + t * NT, m = f >> 2, kq = (f & 3) << 2;
            Bs[b][kq][m] = xv[t].x;
            Bs[b][kq + 1][m] = xv[t].y;
            Bs[b][kq + 2][m] = xv[t].z;
            Bs[b][kq + 3][m] = xv[t].w;
        }
    };

    int b = 0;
    if (t0 < t1) {
        fetch(t0, 0);
        store(0);
    }
    __syncthreads();
    for (int64_t tile = t0; tile < t1; ++tile) {
        const int64_t col0 = tile * BN;
        unsigned long long acc[RM][4];
#pragma unroll
        for (int i = 0; i < RM; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                acc[i][j] = 0ull;
        for (int k0 = 0; k0 < d; k0 += BK) {
            const bool last = k0 + BK >= d;
            const int64_t nt = last ? tile + 1 : tile;
            if (nt < t1)
                fetch(nt, last ? 0 : k0 + BK);
#pragma unroll
            for (int kk = 0; kk < BK; ++kk) {
                const ulonglong2 x0 = *reinterpret_cast<const ulonglong2 *>(&Bs[b][kk][tx * 4]);
                const ulonglong2 x1 = *reinterpret_cast<const ulonglong2 *>(&Bs[b][kk][64 + tx * 4]);
                const unsigned long long xx[4] = {x0.x, x0.y, x1.x, x1.y};
                unsigned long long qq[RM];
                if constexpr (RM == 1) {
                    qq[0] = *reinterpret_cast<const unsigned long long *>(&As[b][kk][ty]);
                } else {
#pragma unroll
                    for (int i = 0; i < RM; i += 2) {
                        const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(&As[b][kk][ty * RM + i]);
                        qq[i] = v.x;
                        qq[i + 1] = v.y;
                    }
                }
#pragma unroll
                for (int i = 0; i < RM; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        acc[i][j] = fma_f32x2(qq[i], xx[j], acc[i][j]);
            }
            if (nt < t1)
                store(b ^ 1);
            __syncthreads();
            b ^= 1;
        }
        // epilogue: squared distances, threshold filter, append to row buffers
#pragma unroll
        for (int i = 0; i < RM; ++i) {
            const int r = ty * RM + i;
            const int64_t grow = row0 + r;
            if (grow >= nq)
                continue;
            const float thr = s_thr[r];
            const int64_t self = self_offset >= 0 ? self_offset + grow : -1;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int cl = (j < 4) ? tx * 4 + j : 64 + tx * 4 + (j - 4);
                const int64_t c = col0 + cl;
                if (c >= n || c == self)
                    continue;
                const unsigned long long pr = acc[i][j >> 1];
                const float dot = __uint_as_float((unsigned)(j & 1 ? pr >> 32 : pr));
                const float d2 = fmaxf(s_qn[r] + __ldg(xn + c) - 2.f * dot, 0.f);
                if (d2 < thr) {
                    const int pos = atomicAdd(&s_cnt[r], 1);
                    buf[grow * BUF + pos] = pack_key(d2, (int)c);
                }
            }
        }
        __syncthreads();
        const bool last_tile = tile + 1 == t1;
        for (int r = warp; r < RB; r += NT / 32) {
            const int64_t grow = row0 + r;
            if (grow >= nq)
                break;
            const int c = s_cnt[r];
            if (c > BUF - BN || (last_tile && c > 0)) {
                const float t = key_dist(merge_row<KC>(grow, c, KC - 1, best, buf, lane));
                if (lane == 0) {
                    s_thr[r] = t;
                    s_cnt[r] = 0;
                }
            }
        }
        __syncthreads();
    }
}

// Merges the sorted lists of each row that several CTAs swept into list 0 (in place).
// A CTA per row: its warps each fold every W-th list (the next list's load is in
// flight), then the first warp folds the others' results from shared memory.  Keys are
// distinct (the shares' columns are), so the KC smallest of the union are what one
// sweep of all columns would have kept.
constexpr int kMergeWarps = 16;
template <int KC>
__global__ void knn_merge_kernel(const Shares sh, int rows, int64_t nq, int64_t first, unsigned long long *__restrict__ best)
{
    constexpr int PB = KC / 32;
    __shared__ unsigned long long part[kMergeWarps][KC];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, W = blockDim.x >> 5;
    const int64_t row = first + blockIdx.x;
    const int L = row / rows < sh.main ? sh.gm : sh.gt;
    unsigned long long m[PB] = {}, nx[PB];
    auto load = [&](int g) {
        const unsigned long long *p = best + list_base(sh, g, nq, rows, KC) + row * KC;
#pragma unroll
        for (int i = 0; i < PB; ++i)
            nx[i] = g < L ? p[i * 32 + lane] : EMPTY_KEY;
    };
    auto fold = [&]() {  // m <- the KC smallest of the sorted lists m and nx
        const unsigned long long least = __shfl_sync(0xffffffffu, nx[0], 0), most = __shfl_sync(0xffffffffu, m[PB - 1], 31);
        if (least >= most)
            return;
        unsigned long long o[PB];
#pragma unroll
        for (int i = 0; i < PB; ++i) {
            const unsigned long long r = __shfl_sync(0xffffffffu, nx[PB - 1 - i], 31 - lane);
            o[i] = m[i] < r ? m[i] : r;
        }
        warp_merge_compact<PB>(o, lane);
#pragma unroll
        for (int i = 0; i < PB; ++i)
            m[i] = o[i];
    };
    load(warp);
#pragma unroll
    for (int i = 0; i < PB; ++i)
        m[i] = nx[i];
    load(warp + W);
    for (int g = warp + W; g < L; g += W) {
        unsigned long long cur[PB];
#pragma unroll
        for (int i = 0; i < PB; ++i)
            cur[i] = nx[i];
        load(g + W);
        unsigned long long ahead[PB];
#pragma unroll
        for (int i = 0; i < PB; ++i) {
            ahead[i] = nx[i];
            nx[i] = cur[i];
        }
        fold();
#pragma unroll
        for (int i = 0; i < PB; ++i)
            nx[i] = ahead[i];
    }
#pragma unroll
    for (int i = 0; i < PB; ++i)
        part[warp][i * 32 + lane] = m[i];
    __syncthreads();
    if (warp)
        return;
    for (int w = 1; w < W; ++w) {
#pragma unroll
        for (int i = 0; i < PB; ++i)
            nx[i] = part[w][i * 32 + lane];
        fold();
    }
#pragma unroll
    for (int i = 0; i < PB; ++i)
        best[row * KC + i * 32 + lane] = m[i];
}

// Merges what the plan split: all rows when gm > 1, else the rows from block `main` on.
template <int KC>
int merge_lists(const Shares &sh, int rows, int64_t nq, unsigned long long *best, cudaStream_t s)
{
    const int64_t first = sh.gm > 1 ? 0 : std::min<int64_t>(sh.main * rows, nq);
    if (first >= nq || std::max(sh.gm, sh.gt) == 1)
        return ONNG_OK;
    const int W = std::min(kMergeWarps, std::max(sh.gm, sh.gt));
    knn_merge_kernel<KC><<<(unsigned)(nq - first), 32 * W, 0, s>>>(sh, rows, nq, first, best);
    return check_launch("onng_knn: list merge");
}

// Rescores the KC survivors of each row by direct difference and writes the best k.
template <int KC>
__global__ void knn_final_kernel(const float *__restrict__ X, int d, const float *__restrict__ Q, int64_t nq,
                                 const unsigned long long *__restrict__ best, int k, int32_t *__restrict__ nbr,
                                 float *__restrict__ len)
{
    constexpr int PER = KC / 32;
    const int lane = threadIdx.x & 31;
    const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (row >= nq)
        return;
    unsigned long long v[PER];
    const float4 *q4 = reinterpret_cast<const float4 *>(Q + row * d);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int e = i * 32 + lane;
        const unsigned long long key = best[row * KC + e];
        const int id = key_id(key);
        // every lane walks the 32 candidates of this slice in turn
        float mine = INFINITY;
        for (int t = 0; t < 32; ++t) {
            const int cid = __shfl_sync(0xffffffffu, id, t);
            if (cid < 0)
                continue;
            const float4 *x4 = reinterpret_cast<const float4 *>(X + (int64_t)cid * d);
            float s = 0.f;
            for (int c = lane; c < (d >> 2); c += 32) {
                float4 a = __ldg(q4 + c), b = __ldg(x4 + c);
                float u = a.x - b.x;
                s = fmaf(u, u, s);
                u = a.y - b.y;
                s = fmaf(u, u, s);
                u = a.z - b.z;
                s = fmaf(u, u, s);
                u = a.w - b.w;
                s = fmaf(u, u, s);
            }
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1)
                s += __shfl_xor_sync(0xffffffffu, s, off);
            if (lane == t)
                mine = s;
        }
        v[i] = id < 0 ? EMPTY_KEY : pack_key(mine, id);
    }
    if constexpr (PER >= 1) {
        if constexpr ((PER & (PER - 1)) == 0)
            warp_bitonic_sort<PER>(v, lane);
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int e = i * 32 + lane;
        if (e < k) {
            const int id = key_id(v[i]);
            nbr[row * k + e] = id;
            len[row * k + e] = id < 0 ? INFINITY : sqrtf(key_dist(v[i]));
        }
    }
}

// The byte-valued tensor-core form ranks exactly: its best lists are already in
// (squared distance, id) order with the exact integer squared distances a float32
// direct-difference rescore would recompute, so the first k entries are written
// as they are.
__global__ void knn_emit_kernel(int64_t nq, const unsigned long long *__restrict__ best, int kc, int k,
                                int32_t *__restrict__ nbr, float *__restrict__ len)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nq * k; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = e / k;
        const unsigned long long key = best[row * kc + e % k];
        const int id = key_id(key);
        nbr[e] = id;
        len[e] = id < 0 ? INFINITY : sqrtf(key_dist(key));
    }
}

// ---------------------------------------------------------------- tensor cores
//
// knn_tc_kernel: the same sweep with the dot products on the 5th-generation
// tensor cores, for byte-valued inputs (integers in [0, 255], e.g. 8-bit image
// descriptors) at d = 32 .. 128: they are exact in bfloat16, every product and
// partial sum is an integer below 2^23, so the float32 accumulation, and with it
// the ranking, is exact.
//
// One CTA owns 256 query rows, two blocks of 128 (the A operands, loaded once by
// TMA), and sweeps the base in tiles of 128 rows (the B operand, a three-stage
// TMA ring) that both row blocks share.  Shared memory holds the operands
// K-major in 128-byte-swizzled atoms (8 rows x 64 bfloat16).  Warp 9 allocates
// the 512 TMEM columns: for each row block two 128 x 128 float32 accumulators
// (tiles alternate between them).  The warp runs converged and an elected lane of it
// issues tcgen05.mma (M = 128,
// N = 128, K = 16 per instruction, both row blocks per K step) and commits to
// mbarriers that free the smem stage and hand the accumulators to the epilogue.
// Warp 8 lane 0 issues the TMA loads.
//
// Epilogue (warps 0-7): thread (w, l) owns query row 128 (w / 4) + 32 (w % 4) + l
// outright, reading it from TMEM lanes 32 (w % 4) .. +31 with tcgen05.ld.  Per
// 32-column chunk it takes the maximum of q.x - |x|^2 / 2; a chunk whose maximum
// passes the threshold of any of the warp's rows appends their hits (tc_chunk) to the
// rows' candidate buffers.  A row whose
// buffer may not absorb another tile is merged into its sorted best list by its
// warp (merge_row).  No barrier
// couples the epilogue warps: each arrives on the accumulator's "empty" barrier
// when its TMEM reads are done and merges afterwards.  Every mbarrier wait gives
// up after 2 s, records an error code and lets all roles reach the teardown,
// where TMEM is freed.
constexpr int TC_M = 128, TC_N = 128, TC_BUF = BUF;
constexpr int TC_RB = 2;                    // 128-row blocks per CTA
// Buffered keys that trigger a merge: with the last tile's hits they mostly still fit one
// chunk of 64 (64: 246, 56: 240, 48: 245, 40: 251 ms at 1M x 128 bytes, k = 100).
constexpr int TC_EAGER = 56;
constexpr int TC_ROWS = TC_M * TC_RB;       // query rows per CTA
constexpr int TC_EPI = 256;                 // epilogue threads (8 warps), one per row
constexpr int TC_THREADS = TC_EPI + 64;     // + TMA warp + MMA warp
constexpr unsigned long long TC_TIMEOUT_NS = 2000000000ull;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok)
                 : "r"(smem_u32(bar)), "r"(parity)
                 : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait on a phase; false (and *err set) after TC_TIMEOUT_NS or when
// another role has already given up.
__device__ bool mbar_wait(uint64_t *bar, uint32_t parity, int *err, int code)
{
    if (mbar_try_wait(bar, parity))
        return true;
    const uint64_t t0 = global_ns();
    for (uint32_t it = 0;; ++it) {
        if (mbar_try_wait(bar, parity))
            return true;
        if ((it & 63) == 0) {
            if (*reinterpret_cast<volatile int *>(err) != 0)
                return false;
            if (global_ns() - t0 > TC_TIMEOUT_NS) {
                atomicCAS(err, 0, code);
                return false;
            }
        }
    }
}
// Bounded wait for a role's own work in flight before teardown: unlike
// mbar_wait it keeps waiting when another role has already given up; on its
// own timeout it records `code` in *err (global memory) and returns.
__device__ void mbar_drain(uint64_t *bar, uint32_t parity, int *err, int code)
{
    const uint64_t t0 = global_ns();
    for (uint32_t it = 0;; ++it) {
        if (mbar_try_wait(bar, parity))
            return;
        if ((it & 63) == 0 && global_ns() - t0 > TC_TIMEOUT_NS) {
            atomicCAS(err, 0, code);
            return;
        }
    }
}
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int c0, int c1, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}
// Shared-memory matrix descriptor: K-major operand in 128-byte-swizzled atoms of
// 8 rows x 128 bytes stacked 1024 bytes apart (start address >> 4, leading
// offset unused, stride offset 1024 >> 4, descriptor version 1, swizzle 128B).
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr)
{
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// Instruction descriptor, kind::f16: float32 accumulator, bfloat16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t umma_idesc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// One lane of a converged warp.
__device__ __forceinline__ uint32_t elect_one()
{
    uint32_t x;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xFFFFFFFF;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(x));
    return x;
}
// The MMA and the commit are issued where `lead` is set, by a warp that runs converged
// with the same operands in every lane: issued by a single diverged lane they came more
// slowly (1M x 128 bytes, k = 100: 354 ms, 344 by the whole warp).
__device__ __forceinline__ void umma_bf16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc,
                                          uint32_t lead)
{
    asm volatile("{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
                 " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(dtmem),
                 "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc), "r"(lead)
                 : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t *bar, uint32_t lead)
{
    asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
                 " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(smem_u32(bar)),
                 "r"(lead)
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// KA atoms per row: KA - 1 of data and the spare atom.  A holds the data atoms of
// both row blocks and one spare atom (1.0 in its first three columns for every
// row) that both blocks share; only its first K = 16 step is non-zero, so the MMA
// takes that step alone.
template <int KA> struct TcSmem {
    static constexpr int A_ATOM = TC_M * 128;   // bytes of one 64-wide K atom of a 128-row block
    static constexpr int B_ATOM = TC_N * 128;
    static constexpr int A_BYTES = (TC_RB * (KA - 1) + 1) * A_ATOM;
    static constexpr int B_STAGE = KA * B_ATOM;
    static constexpr int STAGES = 3;
    // alignment slack, operands, then barriers and the TMEM address
    static constexpr int BYTES = 1024 + A_BYTES + STAGES * B_STAGE + 256;
    static_assert(BYTES <= 232448, "more than 227 KB of shared memory");
};

// tcgen05.ld of 32 columns without the wait; tmem_wait32 completes it (its
// operands tie the registers to the wait, so nothing reads them earlier)
__device__ __forceinline__ void tmem_ld32_async(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                 "%13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, "
                 "[%32];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                   "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]),
                   "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]),
                   "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait32(uint32_t (&v)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]),
                   "+r"(v[15]), "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]),
                   "+r"(v[22]), "+r"(v[23]), "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]),
                   "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
                 :
                 : "memory");
}

// The three forms of a column's value in the accumulators.
//   EPI_BYTE:  v = q.x - floor(|x|^2 / 2), an integer (the spare K atom adds the norm).
//              v >= q.x - |x|^2 / 2, so v >= tr selects a superset of the hits; a hit is
//              corrected by the parity of |x|^2 (one bit per column) to a = q.x - |x|^2 / 2
//              and kept when a >= tr, i.e. d^2 <= thr.  The comparison is not strict
//              because thr is the k-th distance so far here (ranking is exact, so the list
//              needs no slack): a later column at that distance may still win its tie by
//              id.  In a tile whose ids all lie above the k-th entry's none can, and tr is
//              raised by 1/2 (values are multiples of it), which leaves out the ties:
//              100,000 equal rows of 36 bytes, k = 10, ran 162 ms with every tie appended
//              and merged (39 on the float32 sweep).
//   EPI_FOLD:  v = q.x - |x|^2 / 2 of the split form, the half norm added by spare columns
//              of K; kept when v > tr.
//   EPI_NORMS: v = q.x of the split form; the epilogue subtracts the half norms.
enum { EPI_BYTE, EPI_FOLD, EPI_NORMS };

// One 32-column chunk of a row: f[j] is column cb + j.  The maxima of eight groups of
// four columns give each row the groups that hold hits of its own; every row then takes
// its next group at the same time, picking the group's four values out of its registers
// by selects on the bits of the group number, and appends the hits among them.  At 1M x
// 128 bytes, k = 100, two thirds of the chunks hold a hit of some row (1.3 on average),
// so one turn mostly serves all rows, and a turn is 28 selects instead of branches over
// the groups (about 20 cycles each): 277 ms with a branch for every group that any row
// needs, 263 with these by halves, 240 as it is (252 without the vote on the chunk's
// maximum; groups of two or eight columns 245, 255).  Reading hit columns back from TMEM
// one by one is slower by a twentieth than the branches; a jump by group number, or
// anything that writes f, takes twice as long (the next chunk's TMEM load then no longer
// runs ahead).
// sj = the row's own column in the chunk (self-joins), nl = columns of the chunk below n,
// odd = the parity bits (EPI_BYTE).
template <int EPI>
__device__ __forceinline__ void tc_chunk(const float (&f)[32], float tr, float qnr, int cb, int sj, int nl, unsigned odd,
                                         unsigned long long *__restrict__ brow, int &cnt)
{
    constexpr int NG = 8;
    float m[NG];
#pragma unroll
    for (int i = 0; i < NG; ++i)
        m[i] = fmaxf(fmaxf(f[i], f[i + 8]), fmaxf(f[i + 16], f[i + 24]));
    const float mx = fmaxf(fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])), fmaxf(fmaxf(m[4], m[5]), fmaxf(m[6], m[7])));
    if (!__any_sync(0xffffffffu, EPI == EPI_BYTE ? mx >= tr : mx > tr))
        return;
    unsigned groups = 0;  // this row's
#pragma unroll
    for (int i = 0; i < NG; ++i)
        groups |= ((EPI == EPI_BYTE ? m[i] >= tr : m[i] > tr) ? 1u : 0u) << i;
#pragma unroll 1
    do {
        const bool any = groups != 0;
        const int g = any ? __ffs((int)groups) - 1 : 0;
        groups &= groups - 1;
#pragma unroll
        for (int t = 0; t < 32; t += NG) {
            float x[NG];
#pragma unroll
            for (int i = 0; i < NG; ++i)
                x[i] = f[t + i];
#pragma unroll
            for (int b = 1; b < NG; b *= 2) {
                const bool upper = (g & b) != 0;
#pragma unroll
                for (int i = 0; i < NG; i += 2 * b)
                    x[i] = upper ? x[i + b] : x[i];
            }
            const int j = t + g;
            const float a = EPI == EPI_BYTE && (odd >> j & 1u) ? x[0] - 0.5f : x[0];
            if (any && (EPI == EPI_BYTE ? a >= tr : a > tr) && j != sj && j < nl)
                brow[cnt++] = pack_key(fmaxf(qnr - 2.f * a, 0.f), cb + j);
        }
    } while (__any_sync(0xffffffffu, groups != 0));
}

// Which base tiles a CTA sweeps, in order: its u-th tile is (t0 + g + u G) mod
// `all`, for u < count.  G CTAs share a row set and take every G-th tile (g = this
// CTA's share); t0 rotates a self-join's sweep to start at its own rows.
struct TileMap {
    int64_t all, t0, count;
    int G, g;
    __device__ TileMap(int64_t all_, int64_t t0_, int G_, int g_)
        : all(all_), t0(t0_), count((all_ - g_ + G_ - 1) / G_), G(G_), g(g_)
    {
    }
    __device__ __forceinline__ int64_t tile(int64_t u) const { return (t0 + g + u * G) % all; }
};

// The epilogue of the tensor-core kernels (warps 0-7; see knn_tc_kernel): one
// query row per thread, tile by tile from the TMEM accumulators (row block rb =
// warp / 4 at columns (2 rb + b) * TC_N, b = tile & 1).
// `xh` holds the padded half norms (EPI_NORMS), `par` the parity bits (EPI_BYTE).
template <int KC, int EPI>
__device__ void tc_epilogue(uint64_t *accf, uint64_t *acce, uint32_t tmem, int warp, int lane, int64_t row0,
                            int64_t nq, int64_t n, const TileMap tm, int kth, int64_t self_offset,
                            const float *__restrict__ xh,
                            const unsigned *__restrict__ par, const float *__restrict__ qn,
                            unsigned long long *__restrict__ best, unsigned long long *__restrict__ buf, int *err)
{
    const int rb = warp >> 2, qd = warp & 3;
    const int64_t grow = row0 + rb * TC_M + qd * 32 + lane;
    const bool row_ok = grow < nq;
    const float qnr = row_ok ? qn[grow] : 0.f;
    const int64_t self = (self_offset >= 0 && row_ok) ? self_offset + grow : -1;
    float thr = row_ok ? INFINITY : -INFINITY;
    int cnt = 0, kid = -1;  // kid: id of the list entry at thr
    unsigned long long *brow = buf + (row_ok ? grow : 0) * TC_BUF;
    const uint32_t lane_base = tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)(rb * 2 * TC_N);
    for (int64_t t = 0; t < tm.count; ++t) {
        const int b = (int)(t & 1);
        const int64_t col0 = tm.tile(t) * TC_N;
        uint4 odd = make_uint4(0u, 0u, 0u, 0u);
        if constexpr (EPI == EPI_BYTE)
            odd = __ldg(reinterpret_cast<const uint4 *>(par + (col0 >> 5)));
        const bool ok = mbar_wait(&accf[b], (uint32_t)((t >> 1) & 1), err, 5);
        if (!__all_sync(0xffffffffu, ok))
            break;
        tc_fence_after();
        // d^2 = |q|^2 + |x|^2 - 2 q.x < thr  <=>  q.x - |x|^2 / 2 > (|q|^2 - thr) / 2, every
        // term an exact integer or half-integer for byte-valued inputs (approximate in
        // the split float form, whose survivors are rescored)
        float tr = 0.5f * (qnr - thr);
        if (EPI == EPI_BYTE && (int)col0 > kid)
            tr += 0.5f;
        // columns of the tile below n (fewer than 128 in the last; none for rows that are no
        // query, whose accumulators may never have been written)
        const int cb0 = (int)col0, left = row_ok ? (int)min(n - col0, (int64_t)TC_N) : 0;
        const int64_t sd = self - col0;
        const int sj0 = sd >= 0 && sd < TC_N ? (int)sd : -1;
        const float4 *h4 = reinterpret_cast<const float4 *>(xh + (EPI == EPI_NORMS ? col0 : 0));
        const uint32_t tb = lane_base + (uint32_t)(b * TC_N);
        // TMEM loads run one chunk ahead of the filter (chunk pairs: va even, vb odd)
        uint32_t va[32], vb[32];
        auto chunk = [&](uint32_t (&v)[32], int c, unsigned bits) {
            float f[32];
#pragma unroll
            for (int j = 0; j < 32; ++j)
                f[j] = __uint_as_float(v[j]);
            if constexpr (EPI == EPI_NORMS) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 x = __ldg(h4 + c * 8 + i);
                    f[4 * i] -= x.x;
                    f[4 * i + 1] -= x.y;
                    f[4 * i + 2] -= x.z;
                    f[4 * i + 3] -= x.w;
                }
            }
            tc_chunk<EPI>(f, tr, qnr, cb0 + c * 32, sj0 - c * 32, left - c * 32, bits, brow, cnt);
        };
        tmem_ld32_async(tb, va);
        tmem_wait32(va);
#pragma unroll 1
        for (int c = 0; c < TC_N / 32; c += 2) {
            tmem_ld32_async(tb + (uint32_t)((c + 1) * 32), vb);
            chunk(va, c, c ? odd.z : odd.x);
            tmem_wait32(vb);
            if (c + 2 < TC_N / 32) {
                tmem_ld32_async(tb + (uint32_t)((c + 2) * 32), va);
            } else {
                // the accumulators are read: the next tile's MMAs may start meanwhile
                tc_fence_before();
                mbar_arrive(&acce[b]);
            }
            chunk(vb, c + 1, c ? odd.w : odd.y);
            if (c + 2 < TC_N / 32)
                tmem_wait32(va);
        }
        // rows whose buffer may not absorb another tile, or holds TC_EAGER keys (an
        // earlier merge lowers the threshold, which saves later appends: cheaper
        // than the smaller sorts it costs), and all rows after the last tile
        const bool last = t + 1 == tm.count;
        unsigned need = __ballot_sync(0xffffffffu, row_ok && (cnt > TC_BUF - TC_N || cnt >= TC_EAGER ||
                                                              (last && cnt > 0)));
        while (need) {
            const int src = __ffs(need) - 1;
            need &= need - 1;
            const int64_t gr = __shfl_sync(0xffffffffu, grow, src);
            const int c = __shfl_sync(0xffffffffu, cnt, src);
            const unsigned long long kk = merge_row<KC>(gr, c, kth, best, buf, lane);
            if (lane == src) {
                thr = key_dist(kk);
                kid = key_id(kk);
                cnt = 0;
            }
        }
    }
}

template <int KC, int KA>
__global__ void __launch_bounds__(TC_THREADS, 1)
    knn_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int64_t n,
                  int64_t nq, int k, const Shares sh, int64_t self_offset, const unsigned *__restrict__ par,
                  const float *__restrict__ qn, unsigned long long *__restrict__ best,
                  unsigned long long *__restrict__ buf, int *err)
{
    using L = TcSmem<KA>;
    extern __shared__ unsigned char tc_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(tc_raw) + 1023) & ~uintptr_t(1023));
    unsigned char *sA = base;
    unsigned char *sB = base + L::A_BYTES;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sB + L::STAGES * L::B_STAGE);
    uint64_t *full = bars, *empty = bars + L::STAGES, *accf = bars + 2 * L::STAGES, *acce = accf + 2, *abar = acce + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(abar + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Share me = my_share(sh, blockIdx.x);
    const int64_t row0 = me.block * TC_ROWS;
    const int64_t all = (n + TC_N - 1) / TC_N;
    const int nrb = row0 + TC_M < nq ? TC_RB : 1;  // row blocks holding any query row
    // a self-join starts its sweep at the tile of its own rows and wraps around:
    // where nearby rows sit together, the thresholds fall within the first tiles
    const int64_t t0 = self_offset >= 0 ? ((self_offset + row0) / TC_N) % all : 0;
    const TileMap tm(all, t0, me.G, me.g);
    const int64_t tiles = tm.count;
    best += list_base(sh, me.g, nq, TC_ROWS, KC);
    buf += list_base(sh, me.g, nq, TC_ROWS, TC_BUF);

    if (tid == 0) {
        for (int s = 0; s < L::STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&accf[b], 1);
            mbar_init(&acce[b], TC_EPI);
        }
        mbar_init(abar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int e = tid; e < TC_ROWS * KC; e += blockDim.x) {
        const int64_t gr = row0 + e / KC;
        if (gr < nq)
            best[gr * KC + e % KC] = EMPTY_KEY;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 8) {
        // ------------------------------------------------ TMA producer
        if (lane == 0) {
            int64_t issued = 0;
            mbar_expect_tx(abar, (nrb * (KA - 1) + 1) * L::A_ATOM);
            for (int rb = 0; rb < nrb; ++rb)
                for (int a = 0; a < KA - 1; ++a)
                    tma_load_2d(sA + (rb * (KA - 1) + a) * L::A_ATOM, &tmA, a * 64, (int)(row0 + rb * TC_M), abar);
            // the spare atom from block 0's rows: a valid row of block 1 sits 128 rows
            // past a valid row of block 0, and all valid rows carry the same 1.0s
            tma_load_2d(sA + TC_RB * (KA - 1) * L::A_ATOM, &tmA, (KA - 1) * 64, (int)row0, abar);
            for (int64_t t = 0; t < tiles; ++t) {
                const int s = (int)(t % L::STAGES);
                if (t >= L::STAGES && !mbar_wait(&empty[s], (uint32_t)(((t / L::STAGES) & 1) ^ 1), err, 1))
                    break;
                mbar_expect_tx(&full[s], L::B_STAGE);
                for (int a = 0; a < KA; ++a)
                    tma_load_2d(sB + s * L::B_STAGE + a * L::B_ATOM, &tmB, a * 64, (int)(tm.tile(t) * TC_N), &full[s]);
                issued = t + 1;
            }
            // our copies in flight complete before the CTA may exit (bounded)
            mbar_drain(abar, 0, err, 6);
            for (int64_t t = issued > L::STAGES ? issued - L::STAGES : 0; t < issued; ++t)
                mbar_drain(&full[t % L::STAGES], (uint32_t)((t / L::STAGES) & 1), err, 6);
        }
    } else if (warp == 9) {
        // ------------------------------------------------ MMA issuer
        constexpr uint32_t idesc = umma_idesc(TC_M, TC_N);
        const uint32_t lead = elect_one();
        const uint64_t a0 = umma_desc(smem_u32(sA)), b0 = umma_desc(smem_u32(sB));
        int64_t done = 0;
        bool ok = __all_sync(0xffffffffu, mbar_wait(abar, 0, err, 2));
        int s = 0;
        uint32_t sp = 0;  // ring stage and its parity
        for (int64_t t = 0; ok && t < tiles; ++t) {
            const int b = (int)(t & 1);
            if (!__all_sync(0xffffffffu, mbar_wait(&full[s], sp, err, 3)))
                break;
            if (t >= 2 && !__all_sync(0xffffffffu, mbar_wait(&acce[b], (uint32_t)(((t >> 1) & 1) ^ 1), err, 4)))
                break;
            tc_fence_after();
            const uint64_t bt = b0 + (uint32_t)(s * (L::B_STAGE >> 4));
#pragma unroll
            for (int rb = 0; rb < TC_RB; ++rb) {
                if (rb >= nrb)
                    break;
                const uint64_t at = a0 + (uint32_t)(rb * (KA - 1) * (L::A_ATOM >> 4));
                const uint32_t dt = tmem + (uint32_t)((rb * 2 + b) * TC_N);
#pragma unroll
                for (int kk = 0; kk < 4 * (KA - 1); ++kk) {
                    const uint32_t off = (uint32_t)((kk & 3) * 32);  // 16 bf16 = 32 bytes inside the atom
                    umma_bf16(dt, at + (((kk >> 2) * L::A_ATOM + off) >> 4), bt + (((kk >> 2) * L::B_ATOM + off) >> 4),
                              idesc, kk > 0 ? 1u : 0u, lead);
                }
                // the spare atom's first K step adds -floor(|x|^2 / 2)
                umma_bf16(dt, a0 + (uint32_t)(TC_RB * (KA - 1) * (L::A_ATOM >> 4)),
                          bt + (uint32_t)((KA - 1) * (L::B_ATOM >> 4)), idesc, 1u, lead);
            }
            umma_commit(&empty[s], lead);
            umma_commit(&accf[b], lead);
            done = t + 1;
            if (++s == L::STAGES) {
                s = 0;
                sp ^= 1;
            }
        }
        // the MMAs issued so far complete before TMEM is freed (bounded)
        if (done > 0)
            mbar_drain(&accf[(done - 1) & 1], (uint32_t)(((done - 1) >> 1) & 1), err, 7);
    } else {
        // ------------------------------------------------ epilogue (warps 0-7)
        tc_epilogue<KC, EPI_BYTE>(accf, acce, tmem, warp, lane, row0, nq, n, tm, k - 1, self_offset, nullptr, par, qn,
                              best, buf, err);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 9) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// ---------------------------------------------------------------- float inputs
//
// knn_tcs_kernel: the tensor-core sweep for float inputs.  Both vector sets are
// first centred on the mean of the base (distances do not change) and split into
// bfloat16 pairs c = hi + lo with hi = bf16(c), lo = bf16(c - hi); a dot product
// is then qh.xh + qh.xl + ql.xh in float32 (three tcgen05.mma per K step; the
// dropped ql.xl and the rounding of lo are below 2^-16 |q| |x|).  The ranking of
// this expanded form only selects the KC survivors of a row, which
// knn_final_kernel rescores by direct difference in float32 from the original
// vectors, as for the SIMT sweep.  Rows are zero-padded to dp = 64 ceil(d / 64),
// so K runs in chunks of one 64-wide atom: A (both row blocks, hi and lo) and B
// (hi and lo) stream through a two-stage ring of 96 KB, the accumulators stay in
// TMEM across the chunks of a tile, and the epilogue is tc_epilogue.  Where d leaves
// three padding columns (FOLD), they carry 1.0 in the queries and the half norm's three
// bfloat16 pieces (its 24 bits), negated, in the base, so the accumulator arrives with
// the norm subtracted (it cost the epilogue 8 loads and 32 subtractions per chunk).
constexpr int TCS_STAGES = 2;
struct TcsSmem {
    static constexpr int ATOM = TC_M * 128;  // 128 rows x 64 bfloat16 (TC_N == TC_M)
    static constexpr int STAGE = 6 * ATOM;   // A hi (2 blocks), A lo (2 blocks), B hi, B lo
    static constexpr int BYTES = 1024 + TCS_STAGES * STAGE + 256;
};
static_assert(TC_N == TC_M, "the split kernel's atoms are 128 rows for A and B alike");

template <int KC, bool FOLD>
__global__ void __launch_bounds__(TC_THREADS, 1)
    knn_tcs_kernel(const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmAl,
                   const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ CUtensorMap tmBl, int64_t n,
                   int64_t nq, int nk, const Shares sh, int64_t self_offset, const float *__restrict__ xh,
                   const float *__restrict__ qn, unsigned long long *__restrict__ best,
                   unsigned long long *__restrict__ buf, int *err)
{
    using L = TcsSmem;
    extern __shared__ unsigned char tc_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(tc_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *bars = reinterpret_cast<uint64_t *>(base + TCS_STAGES * L::STAGE);
    uint64_t *full = bars, *empty = bars + TCS_STAGES, *accf = bars + 2 * TCS_STAGES, *acce = accf + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acce + 2);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Share me = my_share(sh, blockIdx.x);
    const int64_t row0 = me.block * TC_ROWS;
    const int64_t tiles = (n + TC_N - 1) / TC_N;
    const int nrb = row0 + TC_M < nq ? TC_RB : 1;  // row blocks holding any query row
    // a self-join starts its sweep at the tile of its own rows and wraps around:
    // where nearby rows sit together, the thresholds fall within the first tiles
    const int64_t t0 = self_offset >= 0 ? ((self_offset + row0) / TC_N) % tiles : 0;
    const TileMap tm(tiles, t0, me.G, me.g);
    const int64_t steps = tm.count * nk;
    // this CTA's lists: share g of the row set keeps its own best list and buffers
    best += list_base(sh, me.g, nq, TC_ROWS, KC);
    buf += list_base(sh, me.g, nq, TC_ROWS, TC_BUF);

    if (tid == 0) {
        for (int s = 0; s < TCS_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&accf[b], 1);
            mbar_init(&acce[b], TC_EPI);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int e = tid; e < TC_ROWS * KC; e += blockDim.x) {
        const int64_t gr = row0 + e / KC;
        if (gr < nq)
            best[gr * KC + e % KC] = EMPTY_KEY;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 8) {
        // ------------------------------------------------ TMA producer
        if (lane == 0) {
            const uint32_t bytes = (uint32_t)((2 * nrb + 2) * L::ATOM);
            int64_t issued = 0;
            for (int64_t step = 0; step < steps; ++step) {
                const int s = (int)(step % TCS_STAGES);
                const int64_t t = step / nk;
                const int kc = (int)(step % nk);
                if (step >= TCS_STAGES &&
                    !mbar_wait(&empty[s], (uint32_t)(((step / TCS_STAGES) & 1) ^ 1), err, 1))
                    break;
                unsigned char *st = base + s * L::STAGE;
                mbar_expect_tx(&full[s], bytes);
                for (int rb = 0; rb < nrb; ++rb) {
                    tma_load_2d(st + rb * L::ATOM, &tmAh, kc * 64, (int)(row0 + rb * TC_M), &full[s]);
                    tma_load_2d(st + (2 + rb) * L::ATOM, &tmAl, kc * 64, (int)(row0 + rb * TC_M), &full[s]);
                }
                tma_load_2d(st + 4 * L::ATOM, &tmBh, kc * 64, (int)(tm.tile(t) * TC_N), &full[s]);
                tma_load_2d(st + 5 * L::ATOM, &tmBl, kc * 64, (int)(tm.tile(t) * TC_N), &full[s]);
                issued = step + 1;
            }
            // our copies in flight complete before the CTA may exit (bounded)
            for (int64_t step = issued > TCS_STAGES ? issued - TCS_STAGES : 0; step < issued; ++step)
                mbar_drain(&full[step % TCS_STAGES], (uint32_t)((step / TCS_STAGES) & 1), err, 6);
        }
    } else if (warp == 9) {
        // ------------------------------------------------ MMA issuer
        constexpr uint32_t idesc = umma_idesc(TC_M, TC_N);
        constexpr uint32_t atom = L::ATOM >> 4;
        const uint32_t lead = elect_one();
        const uint64_t r0 = umma_desc(smem_u32(base));
        int64_t last = -1;  // the last step whose MMAs were issued (and committed to empty)
        int kc = 0;
        int64_t t = 0;
        for (int64_t step = 0; step < steps; ++step) {
            const int s = (int)(step % TCS_STAGES);
            const int b = (int)(t & 1);
            if (!__all_sync(0xffffffffu, mbar_wait(&full[s], (uint32_t)((step / TCS_STAGES) & 1), err, 3)))
                break;
            if (kc == 0 && t >= 2 &&
                !__all_sync(0xffffffffu, mbar_wait(&acce[b], (uint32_t)(((t >> 1) & 1) ^ 1), err, 4)))
                break;
            tc_fence_after();
            const uint64_t st = r0 + (uint32_t)(s * (L::STAGE >> 4));
            const uint32_t first = kc > 0 ? 1u : 0u;
#pragma unroll
            for (int rb = 0; rb < TC_RB; ++rb) {
                if (rb >= nrb)
                    break;
                const uint32_t dt = tmem + (uint32_t)((rb * 2 + b) * TC_N);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint32_t off = (uint32_t)(kk * 2);  // 16 bf16 = 32 bytes inside the atom
                    const uint64_t ah = st + rb * atom + off, al = st + (2 + rb) * atom + off;
                    const uint64_t bh = st + 4 * atom + off, bl = st + 5 * atom + off;
                    umma_bf16(dt, ah, bh, idesc, kk > 0 ? 1u : first, lead);
                    umma_bf16(dt, ah, bl, idesc, 1u, lead);
                    umma_bf16(dt, al, bh, idesc, 1u, lead);
                }
            }
            umma_commit(&empty[s], lead);
            if (kc == nk - 1)
                umma_commit(&accf[b], lead);
            last = step;
            if (++kc == nk) {
                kc = 0;
                ++t;
            }
        }
        // the MMAs issued so far complete before TMEM is freed (bounded)
        if (last >= 0)
            mbar_drain(&empty[last % TCS_STAGES], (uint32_t)((last / TCS_STAGES) & 1), err, 7);
    } else {
        // ------------------------------------------------ epilogue (warps 0-7)
        tc_epilogue<KC, FOLD ? EPI_FOLD : EPI_NORMS>(accf, acce, tmem, warp, lane, row0, nq, n, tm, KC - 1, self_offset, xh,
                                                     nullptr, qn, best, buf, err);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 9) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// sums[j] += the base's coordinates j (float64), for the centring mean
__global__ void col_sums_kernel(const float *__restrict__ X, int64_t n, int d, double *__restrict__ sums)
{
    const int64_t per = (n + gridDim.x - 1) / gridDim.x;
    const int64_t r0 = (int64_t)blockIdx.x * per, r1 = r0 + per < n ? r0 + per : n;
    for (int j = threadIdx.x; j < d; j += blockDim.x) {
        double acc = 0.0;
        for (int64_t r = r0; r < r1; ++r)
            acc += (double)X[r * d + j];
        if (r1 > r0)
            atomicAdd(&sums[j], acc);
    }
}

__global__ void mean_kernel(const double *__restrict__ sums, int64_t n, int d, float *__restrict__ mu)
{
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < d; j += gridDim.x * blockDim.x)
        mu[j] = (float)(sums[j] / (double)n);
}

// Row r of M [rows, d] centred on mu, split into bfloat16 hi / lo rows of
// length dp (zeros past d), and its centred squared norm (half of it when
// `half`; +inf for the padded rows rows .. padded_rows of a half-norm array).  With
// `fold` (dp >= d + 3), columns d .. d + 2 of the hi row are 1.0 (queries) or the
// bfloat16 pieces of minus the half norm (base rows).
__global__ void split_rows_kernel(const float *__restrict__ M, int64_t rows, int d, int dp,
                                  const float *__restrict__ mu, __nv_bfloat16 *__restrict__ hi,
                                  __nv_bfloat16 *__restrict__ lo, float *__restrict__ norm, bool half,
                                  int64_t padded_rows, bool fold)
{
    const int lane = threadIdx.x & 31;
    for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; r < padded_rows;
         r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        if (r >= rows) {
            if (lane == 0)
                norm[r] = INFINITY;
            continue;
        }
        float s = 0.f;
        for (int j = lane; j < dp; j += 32) {
            const float c = j < d ? M[r * d + j] - mu[j] : 0.f;
            const __nv_bfloat16 h = __float2bfloat16_rn(c);
            if (!fold || j < d || j >= d + 3)
                hi[r * dp + j] = h;
            lo[r * dp + j] = __float2bfloat16_rn(c - __bfloat162float(h));
            s = fmaf(c, c, s);
        }
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1)
            s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane == 0)
            norm[r] = half ? 0.5f * s : s;
        if (fold && lane < 3) {
            float rest = -0.5f * s;  // the piece of lane p: what the pieces before it left, rounded
            __nv_bfloat16 piece = __float2bfloat16_rn(rest);
            for (int p = 0; p < lane; ++p) {
                rest -= __bfloat162float(piece);
                piece = __float2bfloat16_rn(rest);
            }
            hi[r * dp + d + lane] = half ? piece : __float2bfloat16_rn(1.f);
        }
    }
}

// One pass over the rows of M for what every sweep needs to know of them (one read of
// the base instead of three; the whole call at 30,011 x 100: 2.89 -> 2.62 ms):
// - the squared norms s_r, in norms_kernel's order of sums;
// - bit 0 of *flag if any value is not an integer in [0, 255] (byte-valued
//   descriptors: exact in bfloat16, and at d <= 128 every squared norm, dot product,
//   |x|^2 / 2 and distance of the tensor-core path is an exact float32 below 2^23), and
//   bit 1 if any value is not an integer at all;
// - with `out`, as long as no other value has been seen, the byte-valued form's
//   operands: row r in bfloat16 in columns [0, d) of a row of dpa = dp + 64 (dp = d
//   rounded up to whole K atoms, and a spare one), then in columns dp, dp + 1, dp + 2
//   either 1.0 (queries) or the three pieces of -floor(s_r / 2) (base rows; s_r is an
//   integer below 2^23): its 8-bit fields times 2^16, 2^8 and 1, each exact in
//   bfloat16; zeros elsewhere.  The MMA then accumulates q.x - floor(|x|^2 / 2) exactly.
//   Padding d to whole K atoms takes byte rows of any d = 32 .. 128 here from the float32
//   sweep (30,011 x 100, the whole build: 20.5 -> 9.3 ms by this alone, 5.7 now); below
//   32 a padded row would be mostly zeros, and the float32 sweep serves it.
__global__ void prepare_rows_kernel(const float *__restrict__ M, int64_t rows, int d, int dpa, bool base,
                                    float *__restrict__ norm, __nv_bfloat16 *__restrict__ out, int *flag)
{
    const int lane = threadIdx.x & 31;
    auto kind = [](float v) {
        const bool integer = v == rintf(v);
        return (integer && v >= 0.f && v <= 255.f ? 0u : 1u) | (integer ? 0u : 2u);
    };
    for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; r < rows;
         r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const float4 *p = reinterpret_cast<const float4 *>(M + r * d);
        float s = 0.f;
        unsigned bad = 0;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int c = lane; c < (d >> 2); c += 32) {
            v = __ldg(p + c);
            s = fmaf(v.x, v.x, s);
            s = fmaf(v.y, v.y, s);
            s = fmaf(v.z, v.z, s);
            s = fmaf(v.w, v.w, s);
            bad |= kind(v.x) | kind(v.y) | kind(v.z) | kind(v.w);
        }
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1)
            s += __shfl_xor_sync(0xffffffffu, s, off);
        bad = __reduce_or_sync(0xffffffffu, bad);
        const int seen = *reinterpret_cast<volatile int *>(flag);
        if (lane == 0) {
            norm[r] = s;
            if (bad & ~(unsigned)seen)
                atomicOr(flag, (int)bad);
        }
        if (!out || ((bad | (unsigned)seen) & 1u))
            continue;
        // d <= 128: v is this lane's quad of the row
        auto bits = [](float x, float y) {
            const __nv_bfloat162 b = __floats2bfloat162_rn(x, y);
            return *reinterpret_cast<const unsigned *>(&b);
        };
        uint2 *row = reinterpret_cast<uint2 *>(out + r * dpa);
        const int quads = (dpa - 64) >> 2;
        if (lane < quads)
            row[lane] = make_uint2(bits(v.x, v.y), bits(v.z, v.w));
        if (lane < 16) {
            float a = 0.f, b = 0.f, c = 0.f;
            if (lane == 0) {
                const unsigned h = (unsigned)s >> 1;
                a = base ? -(float)((h >> 16) << 16) : 1.f;
                b = base ? -(float)(((h >> 8) & 255u) << 8) : 1.f;
                c = base ? -(float)(h & 255u) : 1.f;
            }
            row[quads + lane] = make_uint2(bits(a, b), bits(c, 0.f));
        }
    }
}

// Bit i of par = the parity of the integer s_i (0 past n), one word per 32 columns.
__global__ void parity_kernel(const float *__restrict__ s, int64_t n, int64_t words, unsigned *__restrict__ par)
{
    const int lane = threadIdx.x & 31;
    for (int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; w < words;
         w += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int64_t i = w * 32 + lane;
        const unsigned bit = i < n ? ((unsigned)s[i] & 1u) : 0u;
        const unsigned b = __ballot_sync(0xffffffffu, bit != 0);
        if (lane == 0)
            par[w] = b;
    }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// 2-D bf16 tensor map over rows x d (row-major), box 64 x box_rows, 128B swizzle,
// zero fill outside the matrix.
int make_map(CUtensorMap *m, const void *ptr, int64_t rows, int d, int box_rows)
{
    auto fn = encode_fn();
    if (!fn)
        return set_error(ONNG_E_CUDA, "onng_knn: cuTensorMapEncodeTiled unavailable");
    cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)d * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        return set_error(ONNG_E_CUDA, "onng_knn: tensor map encode failed (%d)", (int)r);
    return ONNG_OK;
}

// CTAs sharing one row set in the split sweep: above d = 128 a CTA's A chunks
// (256 rows x dp x 4 bytes) over all resident CTAs would exceed L2, so two CTAs take
// alternate tiles of the same rows (half the A data in flight) and keep a best list
// each, merged before the rescore.
int split_share(int d) { return d > 128 ? 2 : 1; }

int tile_rows(int64_t nq) { return nq <= 16 ? 16 : nq <= 32 ? 32 : nq <= 64 ? 64 : 128; }

// Lists (of one row each: KC keys and a buffer of BUF) a call cannot do without, and
// those its workspace request has room for.  The spare ones let every CTA that the
// device holds keep lists of its own (a wave: two float32 CTAs of 128 rows, or one of 256
// rows, per SM), as far as a sweep of n columns can be split that often; for some tens of
// thousands of queries, whose row blocks fill about half a wave, two more for each (20,000
// integer rows over 100,000 x 100: 28 ms with a wave's lists, 19 with these, 17 with six
// more).  The request grows with nq, so a buffer for the largest batch serves every
// smaller one; a smaller buffer is planned into (fewer shares).
constexpr int64_t kWaveLists = 2 * kSweepSms * 128;
static_assert(kWaveLists == (int64_t)kSweepSms * TC_ROWS, "a wave of either sweep holds as many rows");

int64_t least_lists(int d, int64_t nq) { return nq * split_share(d); }

int64_t asked_lists(int64_t n, int d, int64_t nq)
{
    const int64_t most = std::max<int64_t>(1, std::min<int64_t>((n + BN - 1) / BN / 4, 2 * kSweepSms));
    return least_lists(d, nq) + std::min(nq * (most - 1), std::max(kWaveLists, std::min(2 * nq, kWaveLists * 3 / 2)));
}

// The plans of the two kinds of sweep, for a workspace of `lists` lists.  kSweepSms is
// the GB300's SM count (two resident CTAs per SM in the float32 sweep, one in the
// tensor-core sweeps).
Shares plan_tile(int64_t n, int64_t nq, int64_t lists)
{
    return plan_shares(nq, tile_rows(nq), (n + BN - 1) / BN, 2 * kSweepSms, 1, 8, lists);
}

Shares plan_tc(int64_t n, int d, int64_t nq, int kc, int64_t lists)
{
    return plan_shares(nq, TC_ROWS, (n + TC_N - 1) / TC_N, kSweepSms, split_share(d), 8 * (int64_t)kc, lists);
}

int pick_kc(int k)
{
    for (int kc = 32; kc <= 256; kc <<= 1)
        if (k + 16 <= kc)
            return kc;
    return 0;
}

template <int KC, int RM>
int launch_tile(const float *X, int64_t n, int d, const float *Q, int64_t nq, int64_t self_offset, const Shares &sh,
                const float *xn, const float *qn, unsigned long long *best, unsigned long long *bufp, cudaStream_t s)
{
    ONNG_CUDA_TRY(cudaFuncSetAttribute(reinterpret_cast<const void *>(knn_tile_kernel<KC, RM>),
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TileSmem<RM>)),
                  "onng_knn: tile kernel smem attribute");
    knn_tile_kernel<KC, RM><<<(unsigned)sh.ctas(), NT, sizeof(TileSmem<RM>), s>>>(X, n, d, Q, nq, self_offset, xn, qn, sh,
                                                                                best, bufp);
    return check_launch("onng_knn: tile kernel");
}

template <int KC>
int launch(const float *X, int64_t n, int d, const float *Q, int64_t nq, int k, const Shares &sh, int64_t self_offset,
           int32_t *nbr, float *len, float *xn, float *qn, unsigned long long *best, unsigned long long *bufp,
           cudaStream_t s)
{
    const int rows = tile_rows(nq);
    int st = rows == 16   ? launch_tile<KC, 1>(X, n, d, Q, nq, self_offset, sh, xn, qn, best, bufp, s)
             : rows == 32 ? launch_tile<KC, 2>(X, n, d, Q, nq, self_offset, sh, xn, qn, best, bufp, s)
             : rows == 64 ? launch_tile<KC, 4>(X, n, d, Q, nq, self_offset, sh, xn, qn, best, bufp, s)
                          : launch_tile<KC, 8>(X, n, d, Q, nq, self_offset, sh, xn, qn, best, bufp, s);
    if (st || (st = merge_lists<KC>(sh, rows, nq, best, s)))
        return st;
    knn_final_kernel<KC><<<(unsigned)((nq * 32 + 255) / 256), 256, 0, s>>>(X, d, Q, nq, best, k, nbr, len);
    return check_launch("onng_knn: final kernel");
}

template <int KC, int KA>
int launch_tc_kc(const CUtensorMap &ma, const CUtensorMap &mb, int64_t n, int64_t nq, int k, const Shares &sh,
                 int64_t self_offset, const unsigned *par, const float *qn, unsigned long long *best, unsigned long long *bufp, int *err,
                 cudaStream_t s)
{
    const size_t smem = TcSmem<KA>::BYTES;
    ONNG_CUDA_TRY(cudaFuncSetAttribute(reinterpret_cast<const void *>(knn_tc_kernel<KC, KA>),
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                  "onng_knn: tensor kernel smem attribute");
    knn_tc_kernel<KC, KA><<<(unsigned)sh.ctas(), TC_THREADS, smem, s>>>(ma, mb, n, nq, k, sh, self_offset, par, qn, best,
                                                                        bufp, err);
    int st = check_launch("onng_knn: tensor kernel");
    return st ? st : merge_lists<KC>(sh, TC_ROWS, nq, best, s);
}

int launch_tc(const float *X, int64_t n, int d, const float *Q, int64_t nq, int k, int kc, const Shares &sh,
              int64_t self_offset, int32_t *nbr, float *len, const float *xn, unsigned *par, float *qn, unsigned long long *best,
              unsigned long long *bufp, int *err, __nv_bfloat16 *xb, __nv_bfloat16 *qb, cudaStream_t s)
{
    const int gb = num_sms() * 8;
    const int dpa = (d + 63) / 64 * 64 + 64;  // whole K atoms; the extra one carries -floor(|x|^2 / 2)
    parity_kernel<<<gb, 256, 0, s>>>(xn, n, (n + TC_N - 1) / TC_N * (TC_N / 32), par);
    int st = check_launch("onng_knn: parity");
    if (st)
        return st;
    CUtensorMap ma, mb;
    if ((st = make_map(&ma, qb, nq, dpa, TC_M)) || (st = make_map(&mb, xb, n, dpa, TC_N)))
        return st;
    const int ka = dpa / 64;
    if (kc == 32)
        st = ka == 2 ? launch_tc_kc<32, 2>(ma, mb, n, nq, k, sh, self_offset, par, qn, best, bufp, err, s)
                     : launch_tc_kc<32, 3>(ma, mb, n, nq, k, sh, self_offset, par, qn, best, bufp, err, s);
    else if (kc == 64)
        st = ka == 2 ? launch_tc_kc<64, 2>(ma, mb, n, nq, k, sh, self_offset, par, qn, best, bufp, err, s)
                     : launch_tc_kc<64, 3>(ma, mb, n, nq, k, sh, self_offset, par, qn, best, bufp, err, s);
    else
        st = ka == 2 ? launch_tc_kc<128, 2>(ma, mb, n, nq, k, sh, self_offset, par, qn, best, bufp, err, s)
                     : launch_tc_kc<128, 3>(ma, mb, n, nq, k, sh, self_offset, par, qn, best, bufp, err, s);
    if (st)
        return st;
    int code = 0;
    ONNG_CUDA_TRY(cudaMemcpyAsync(&code, err, sizeof(int), cudaMemcpyDeviceToHost, s), "onng_knn: error flag");
    ONNG_CUDA_TRY(cudaStreamSynchronize(s), "onng_knn: tensor kernel");
    if (code)
        return set_error(ONNG_E_LIMIT, "onng_knn: tensor-core pipeline wait timed out (role %d)", code);
    knn_emit_kernel<<<gb, 256, 0, s>>>(nq, best, kc, k, nbr, len);
    return check_launch("onng_knn: output");
}

template <int KC, bool FOLD>
int launch_tcs_kc(const CUtensorMap *m, int64_t n, int64_t nq, int nk, const Shares &sh, int64_t self_offset,
                  const float *xh,
                  const float *qn, unsigned long long *best, unsigned long long *bufp, int *err, cudaStream_t s)
{
    const size_t smem = TcsSmem::BYTES;
    ONNG_CUDA_TRY(cudaFuncSetAttribute(reinterpret_cast<const void *>(knn_tcs_kernel<KC, FOLD>),
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                  "onng_knn: split tensor kernel smem attribute");
    knn_tcs_kernel<KC, FOLD><<<(unsigned)sh.ctas(), TC_THREADS, smem, s>>>(m[0], m[1], m[2], m[3], n, nq, nk, sh, self_offset,
                                                                     xh, qn, best, bufp, err);
    int st = check_launch("onng_knn: split tensor kernel");
    return st ? st : merge_lists<KC>(sh, TC_ROWS, nq, best, s);
}

// Float inputs on the tensor cores: centre, split into bfloat16 hi / lo, sweep
// (knn_tcs_kernel), rescore the survivors from the original vectors.
int launch_tcs(const float *X, int64_t n, int d, const float *Q, int64_t nq, int k, int kc, const Shares &sh,
               int64_t self_offset, int32_t *nbr, float *len, float *xh, float *qn, unsigned long long *best, unsigned long long *bufp,
               int *err, __nv_bfloat16 *xs, __nv_bfloat16 *qs, double *sums, float *mu, cudaStream_t s)
{
    const int dp = (d + 63) / 64 * 64;
    const int gb = num_sms() * 8;
    __nv_bfloat16 *xhi = xs, *xlo = xs + (size_t)n * dp;
    __nv_bfloat16 *qhi = qs, *qlo = qs + (size_t)nq * dp;
    ONNG_CUDA_TRY(cudaMemsetAsync(sums, 0, sizeof(double) * (size_t)d, s), "onng_knn: clear sums");
    col_sums_kernel<<<(unsigned)std::min<int64_t>(n, 1024), 256, 0, s>>>(X, n, d, sums);
    mean_kernel<<<(d + 255) / 256, 256, 0, s>>>(sums, n, d, mu);
    const bool fold = dp >= d + 3;
    split_rows_kernel<<<gb, 256, 0, s>>>(X, n, d, dp, mu, xhi, xlo, xh, true, (n + TC_N - 1) / TC_N * TC_N, fold);
    split_rows_kernel<<<gb, 256, 0, s>>>(Q, nq, d, dp, mu, qhi, qlo, qn, false, nq, fold);
    int st = check_launch("onng_knn: split copies");
    if (st)
        return st;
    CUtensorMap m[4];
    if ((st = make_map(&m[0], qhi, nq, dp, TC_M)) || (st = make_map(&m[1], qlo, nq, dp, TC_M)) ||
        (st = make_map(&m[2], xhi, n, dp, TC_N)) || (st = make_map(&m[3], xlo, n, dp, TC_N)))
        return st;
    const int nk = dp / 64;
    auto sweep = [&](auto kcc) {
        constexpr int KC = decltype(kcc)::value;
        return fold ? launch_tcs_kc<KC, true>(m, n, nq, nk, sh, self_offset, xh, qn, best, bufp, err, s)
                    : launch_tcs_kc<KC, false>(m, n, nq, nk, sh, self_offset, xh, qn, best, bufp, err, s);
    };
    st = kc == 32 ? sweep(std::integral_constant<int, 32>{})
         : kc == 64 ? sweep(std::integral_constant<int, 64>{})
                    : sweep(std::integral_constant<int, 128>{});
    if (st)
        return st;
    int code = 0;
    ONNG_CUDA_TRY(cudaMemcpyAsync(&code, err, sizeof(int), cudaMemcpyDeviceToHost, s), "onng_knn: error flag");
    ONNG_CUDA_TRY(cudaStreamSynchronize(s), "onng_knn: split tensor kernel");
    if (code)
        return set_error(ONNG_E_LIMIT, "onng_knn: tensor-core pipeline wait timed out (role %d)", code);
    const unsigned grid = (unsigned)((nq * 32 + 255) / 256);
    if (kc == 32)
        knn_final_kernel<32><<<grid, 256, 0, s>>>(X, d, Q, nq, best, k, nbr, len);
    else if (kc == 64)
        knn_final_kernel<64><<<grid, 256, 0, s>>>(X, d, Q, nq, best, k, nbr, len);
    else
        knn_final_kernel<128><<<grid, 256, 0, s>>>(X, d, Q, nq, best, k, nbr, len);
    return check_launch("onng_knn: final kernel");
}

// The workspace of a call with room for `lists` lists; `used` is its size, which grows by
// the same for every list (32-key lists are already whole 256-byte lines).
struct KnnWs {
    float *xn, *qn;
    unsigned long long *best, *buf;
    int *flags;
    __nv_bfloat16 *xb, *qb;  // hi and lo rows of dp = 64 ceil(d / 64) (the byte path's rows of dp + 64 fit)
    float *xh;
    double *sums;
    float *mu;
    unsigned *par;
    size_t used;

    KnnWs(void *ws, int64_t n, int d, int64_t nq, int kc, int64_t lists)
    {
        n = std::max<int64_t>(n, 1);
        nq = std::max<int64_t>(nq, 1);
        const size_t dp = (size_t)(std::max(d, 1) + 63) / 64 * 64, tiles = (size_t)(n + TC_N - 1) / TC_N;
        WsCarver c(ws);
        xn = c.take<float>((size_t)n);
        qn = c.take<float>((size_t)nq);
        best = c.take<unsigned long long>((size_t)lists * kc);
        buf = c.take<unsigned long long>((size_t)lists * BUF);
        flags = c.take<int>(64);
        xb = c.take<__nv_bfloat16>((size_t)n * dp * 2);
        qb = c.take<__nv_bfloat16>((size_t)nq * dp * 2);
        xh = c.take<float>(tiles * TC_N);
        sums = c.take<double>((size_t)std::max(d, 1));
        mu = c.take<float>((size_t)std::max(d, 1));
        par = c.take<unsigned>(tiles * (TC_N / 32));
        used = c.used;
    }
};

}  // namespace
}  // namespace onng

using namespace onng;

extern "C" size_t onng_knn_workspace_bytes(int64_t n, int32_t d, int64_t nq, int32_t k)
{
    const int kc = pick_kc(k) ? pick_kc(k) : 32;
    return KnnWs(nullptr, n, d, nq, kc, asked_lists(std::max<int64_t>(n, 1), d, std::max<int64_t>(nq, 1))).used;
}

extern "C" int onng_knn(const float *X, int64_t n, int32_t d, const float *Q, int64_t nq, int32_t k,
                        int64_t self_offset, int32_t *nbr, float *len, void *ws, size_t ws_bytes, onng_stream_t stream)
{
    ONNG_RANGE("onng_knn");
    ONNG_REQUIRE(n >= 0 && nq >= 0 && n <= INT32_MAX, ONNG_E_INVAL, "onng_knn: bad sizes");
    ONNG_REQUIRE(d > 0 && d % 4 == 0, ONNG_E_UNSUPPORTED, "onng_knn: d must be a positive multiple of 4");
    ONNG_REQUIRE(k >= 1, ONNG_E_INVAL, "onng_knn: k must be >= 1");
    ONNG_REQUIRE(pick_kc(k) > 0, ONNG_E_UNSUPPORTED, "onng_knn: k must be <= 240");
    ONNG_REQUIRE(self_offset < 0 || self_offset + nq <= n, ONNG_E_INVAL, "onng_knn: self rows outside the base");
    if (nq == 0)
        return ONNG_OK;
    ONNG_REQUIRE(X && Q && nbr && len, ONNG_E_INVAL, "onng_knn: NULL pointer");
    ONNG_REQUIRE(aligned16(X) && aligned16(Q), ONNG_E_INVAL, "onng_knn: X and Q must be 16-byte aligned");
    const int kc = pick_kc(k);
    const size_t need = KnnWs(nullptr, n, d, nq, kc, least_lists(d, nq)).used;
    ONNG_REQUIRE(ws && ws_bytes >= need, ONNG_E_WORKSPACE, "onng_knn: workspace %zu < %zu bytes", ws_bytes, need);
    const int64_t lists = std::min(asked_lists(std::max<int64_t>(n, 1), d, nq),
                                   least_lists(d, nq) + (int64_t)((ws_bytes - need) / ((kc + BUF) * sizeof(unsigned long long))));
    const KnnWs w(ws, n, d, nq, kc, lists);
    float *const xn = w.xn, *const qn = w.qn;
    int *const flags = w.flags;
    cudaStream_t s = to_cuda(stream);
    // tensor-core paths (k + 16 <= 128, from one row block of queries): byte-valued inputs
    // at d = 32 .. 128 exactly; other non-integer inputs at d >= 32 by the split bfloat16
    // form.  Integer-valued inputs otherwise take the SIMT sweep, which ranks them exactly.
    const bool tc = nq >= TC_M && n >= TC_N && kc <= 128 && n <= INT32_MAX - TC_N;
    int st;
    if (tc) {
        ONNG_CUDA_TRY(cudaMemsetAsync(flags, 0, 64 * sizeof(int), s), "onng_knn: clear flags");
        const int gb = num_sms() * 8;
        const bool byte_d = d >= 32 && d <= 128;
        const int dpa = (d + 63) / 64 * 64 + 64;
        prepare_rows_kernel<<<gb, 256, 0, s>>>(Q, nq, d, dpa, false, qn, byte_d ? w.qb : nullptr, flags);
        prepare_rows_kernel<<<gb, 256, 0, s>>>(X, n, d, dpa, true, xn, byte_d ? w.xb : nullptr, flags);
        st = check_launch("onng_knn: rows");
        if (st)
            return st;
        int kind = 3;
        ONNG_CUDA_TRY(cudaMemcpyAsync(&kind, flags, sizeof(int), cudaMemcpyDeviceToHost, s), "onng_knn: flag");
        ONNG_CUDA_TRY(cudaStreamSynchronize(s), "onng_knn: value check");
        if (!(kind & 1) && byte_d)
            return launch_tc(X, n, d, Q, nq, k, kc, plan_tc(n, d, nq, kc, lists), self_offset, nbr, len, xn, w.par, qn,
                             w.best, w.buf, flags + 1, w.xb, w.qb, s);
        if ((kind & 2) && d >= 32)
            return launch_tcs(X, n, d, Q, nq, k, kc, plan_tc(n, d, nq, kc, lists), self_offset, nbr, len, w.xh, qn, w.best,
                              w.buf, flags + 1, w.xb, w.qb, w.sums, w.mu, s);
    } else {
        if (n > 0)
            norms_kernel<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(X, n, d, xn);
        norms_kernel<<<(unsigned)((nq * 32 + 255) / 256), 256, 0, s>>>(Q, nq, d, qn);
        st = check_launch("onng_knn: norms");
        if (st)
            return st;
    }
    const Shares sh = plan_tile(n, nq, lists);
    switch (kc) {
    case 32: return launch<32>(X, n, d, Q, nq, k, sh, self_offset, nbr, len, xn, qn, w.best, w.buf, s);
    case 64: return launch<64>(X, n, d, Q, nq, k, sh, self_offset, nbr, len, xn, qn, w.best, w.buf, s);
    case 128: return launch<128>(X, n, d, Q, nq, k, sh, self_offset, nbr, len, xn, qn, w.best, w.buf, s);
    default: return launch<256>(X, n, d, Q, nq, k, sh, self_offset, nbr, len, xn, qn, w.best, w.buf, s);
    }
}

extern "C" int onng_build_knng(const float *X, int64_t n, int32_t d, int32_t k, int32_t *nbr, float *len, void *ws,
                               size_t ws_bytes, onng_stream_t stream)
{
    ONNG_RANGE("onng_build_knng");
    ONNG_REQUIRE(k <= n - 1 || n == 0, ONNG_E_INVAL, "onng_build_knng: k must be <= n - 1");
    return onng_knn(X, n, d, X, n, k, 0, nbr, len, ws, ws_bytes, stream);
}
