// Graph adjustment on the GPU.
//
// Static degree adjustment (Algorithm 2, set form):
//   N_e(y) = first_{e_o}(N_k(y))  united with  { o : y in first_{e_i}(N_k(o)) }.
// The reversed edge y->o carries the length stored for o->y; it is skipped when
// y->o is already one of y's forward edges (the forward length wins).  The
// count pass computes every row's exact size (forward edges plus non-duplicate
// reversed edges), a device scan turns the sizes into row_ptr, the fill pass
// writes (length, id) keys, and each row is sorted by (length, id): a warp
// register bitonic sort for rows up to 512 edges, an in-place CTA sort for
// longer rows (hubs).
//
// Degree adjustment with constraints (Algorithm 3, "SAC"): its greedy pass reads
// in a closed form.  N(G_t, o) = { n : o in first_{e_i}(N_k(n)) } (Algorithm 2
// with (0, e_i)), so a node n is considered only by the nodes of its own first
// e_i kNN entries, at most e_i of them: the in-degree test |N(G_i, n)| < e_i
// always holds when n is met.  Taking the nodes o in increasing
// (|N(G_t, o)|, o) and each list in increasing (length, id), o therefore adds
// its first e_o members unconditionally and a later member n exactly when no
// earlier node has added n, i.e. when o is the first of n's considerers in that
// order (that one always adds n).  Both rules are per-edge, so the pass runs in
// parallel and equals the sequential one edge for edge.  The last loop then
// gives every node with fewer than e_o edges its nearest kNN neighbours not yet
// in its list.
//
// Algorithm 4 taken literally (rounds over the partial output; a variant beside
// the order-free rule below): in round p every node s with more than p input
// edges decides its p-th edge (s, t) (input rows are in (length, id) order), in
// ascending s, and keeps it unless HasPath (Algorithm 5) finds, in the partial
// output G_p, a kept edge (s, m) and a kept edge (m, t) shorter than (s, t).
// (s, m) was decided in an earlier round; (m, t) sits at m's position r of t:
// decided when r < p, or earlier in this round when r = p and m < s.  A round
// first decides every edge whose answer needs no same-round edge, then repeats
// a resolution pass: an edge waiting on same-round edges of smaller nodes is
// removed once one of them is kept and kept once all are removed; the smallest
// waiting node can always be decided, so each pass makes progress.  Positions
// of t in m's row come from a per-row copy sorted by id (binary search).
//
// Path adjustment (Algorithms 4/5, order-free reading): edge (i, j) is dropped
// if the input graph holds i->m and m->j with len(i,m) < len(i,j) and
// len(m,j) < len(i,j).  A warp owns a node i at a time (persistent warps stride
// over the nodes): N(i) goes into a shared-memory hash (id -> position); for
// every m in N(i) shorter than i's longest edge, the prefix of m's list shorter
// than that edge (a binary search: rows are sorted by length) is tested against
// it, and every hit j that satisfies both strict comparisons records the smallest
// witness position.  Nodes with more than 256 edges use a CTA in the same way, and
// those with more than 1,024 several.  A count / scan / compact sequence then writes
// the kept edges in their input order.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "scan.cuh"
#include "warp_sort.cuh"

namespace onng {
namespace {

constexpr unsigned long long EMPTY_KEY = 0x7F800000FFFFFFFFull;

// How often `id` stands in the first f entries of row `row`, and how many of them are
// valid.  Rows that start on 16 bytes are read four ids at a time: the row is a random
// gather, and it is all the count and fill passes read besides their own rows.
__device__ __forceinline__ bool in_first(const int32_t *__restrict__ nbr, int64_t row, int k, int f, int32_t id, bool vec,
                                         int *valid)
{
    const int32_t *p = nbr + row * k;
    bool found = false;
    int c = 0, t = 0;
    if (vec) {
#pragma unroll 5
        for (; t + 4 <= f; t += 4) {
            const int4 v = __ldg(reinterpret_cast<const int4 *>(p + t));
            found = found || v.x == id || v.y == id || v.z == id || v.w == id;
            c += (v.x >= 0) + (v.y >= 0) + (v.z >= 0) + (v.w >= 0);
        }
    }
    for (; t < f; ++t) {
        const int32_t v = __ldg(p + t);
        found = found || v == id;
        c += v >= 0;
    }
    *valid = c;
    return found;
}

// Count and fill take a warp per node, a lane per kNN entry (the entries of a node are
// read together; a thread per node read 400 bytes apart and tested 60 entries in turn:
// 1M x 100, (20, 60): count 8.1 ms, fill 7.3 ms).
//
// fwd[y] = valid forward edges of y; incnt[y] += non-duplicate reversed edges.
__global__ void degree_count_kernel(const int32_t *__restrict__ nbr, int64_t n, int k, int fo, int fi, bool vec,
                                    int64_t *__restrict__ fwd, int *__restrict__ incnt)
{
    const int lane = threadIdx.x & 31;
    for (int64_t o = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; o < n;
         o += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        int w = 0;
        for (int p0 = 0; p0 < max(fo, fi); p0 += 32) {
            const int p = p0 + lane;
            const int32_t y = p < max(fo, fi) ? nbr[o * k + p] : -1;
            w += __popc(__ballot_sync(0xffffffffu, p < fo && y >= 0));
            int valid;
            if (p < fi && y >= 0 && y < n && !in_first(nbr, y, k, fo, (int32_t)o, vec, &valid))
                atomicAdd(&incnt[y], 1);
        }
        if (lane == 0)
            fwd[o] = w;
    }
}

// deg[y] = fwd[y] + incnt[y], in place
__global__ void degree_total_kernel(int64_t n, const int *__restrict__ incnt, int64_t *__restrict__ deg)
{
    for (int64_t y = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; y < n; y += (int64_t)gridDim.x * blockDim.x)
        deg[y] += incnt[y];
}

__global__ void degree_fill_kernel(const int32_t *__restrict__ nbr, const float *__restrict__ len, int64_t n, int k,
                                   int fo, int fi, bool vec, const int64_t *__restrict__ row_ptr,
                                   int *__restrict__ cursor, unsigned long long *__restrict__ keys)
{
    const int lane = threadIdx.x & 31;
    for (int64_t o = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; o < n;
         o += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int64_t row = row_ptr[o];
        int w = 0;
        for (int p0 = 0; p0 < max(fo, fi); p0 += 32) {
            const int p = p0 + lane;
            const int32_t y = p < max(fo, fi) ? nbr[o * k + p] : -1;
            const float l = p < max(fo, fi) ? len[o * k + p] : 0.f;
            // forward edges of o occupy the head of its row
            const unsigned fm = __ballot_sync(0xffffffffu, p < fo && y >= 0);
            if (p < fo && y >= 0)
                keys[row + w + __popc(fm & ((1u << lane) - 1u))] = pack_key(l, y);
            w += __popc(fm);
            // reversed edges y->o go after y's forward edges
            int valid;
            if (p < fi && y >= 0 && y < n && !in_first(nbr, y, k, fo, (int32_t)o, vec, &valid)) {
                const int pos = atomicAdd(&cursor[y], 1);
                keys[row_ptr[y] + valid + pos] = pack_key(l, (int32_t)o);
            }
        }
    }
}

// Sorts a row of m <= 32 N keys in registers and writes it back, or, with `col`, as ids
// and lengths.
template <int N>
__device__ __forceinline__ void sort_row(unsigned long long *__restrict__ keys, int64_t beg, int m, int lane,
                                         int32_t *__restrict__ col, float *__restrict__ len)
{
    unsigned long long v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int e = i * 32 + lane;
        v[i] = e < m ? keys[beg + e] : EMPTY_KEY;
    }
    warp_bitonic_sort<N>(v, lane);
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int e = i * 32 + lane;
        if (e < m) {
            if (col) {
                col[beg + e] = (int32_t)(unsigned)(v[i] & 0xFFFFFFFFull);
                len[beg + e] = __uint_as_float((unsigned)(v[i] >> 32));
            } else {
                keys[beg + e] = v[i];
            }
        }
    }
}

// Sorts rows of up to 512 keys, one warp per row, by the smallest network that holds the
// row (rows of 69 keys on average were sorted as 512: 9.2 ms of 1M rows); with `col`
// the sorted row is written as ids and lengths.  Longer rows are listed for the CTA sort.
__global__ void sort_small_rows(const int64_t *__restrict__ row_ptr, int64_t n, unsigned long long *__restrict__ keys,
                                int64_t *__restrict__ big_rows, int *__restrict__ n_big, int32_t *__restrict__ col,
                                float *__restrict__ len)
{
    const int lane = threadIdx.x & 31;
    const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (row >= n)
        return;
    const int64_t beg = row_ptr[row], m = row_ptr[row + 1] - beg;
    if (m < 1 || (m == 1 && !col))
        return;
    if (m > 512) {
        if (lane == 0)
            big_rows[atomicAdd(n_big, 1)] = row;
    } else if (m <= 32) {
        sort_row<1>(keys, beg, (int)m, lane, col, len);
    } else if (m <= 64) {
        sort_row<2>(keys, beg, (int)m, lane, col, len);
    } else if (m <= 128) {
        sort_row<4>(keys, beg, (int)m, lane, col, len);
    } else if (m <= 256) {
        sort_row<8>(keys, beg, (int)m, lane, col, len);
    } else {
        sort_row<16>(keys, beg, (int)m, lane, col, len);
    }
}

// In-place ascending sort of a[0..m) by one CTA: bitonic network in the form
// whose comparators all point upward (first stage of each merge compares
// mirrored positions), so positions >= m act as +inf and are never touched.
__device__ void cta_sort(unsigned long long *a, int64_t m)
{
    int64_t P = 1;
    while (P < m)
        P <<= 1;
    for (int64_t size = 2; size <= P; size <<= 1) {
        for (int64_t t = threadIdx.x; t < P / 2; t += blockDim.x) {
            const int64_t blk = t / (size / 2), off = t % (size / 2);
            const int64_t i = blk * size + off, j = blk * size + size - 1 - off;
            if (j < m && a[j] < a[i]) {
                unsigned long long x = a[i];
                a[i] = a[j];
                a[j] = x;
            }
        }
        __syncthreads();
        for (int64_t h = size / 4; h >= 1; h >>= 1) {
            for (int64_t t = threadIdx.x; t < P / 2; t += blockDim.x) {
                const int64_t blk = t / h, off = t % h;
                const int64_t i = blk * 2 * h + off, j = i + h;
                if (j < m && a[j] < a[i]) {
                    unsigned long long x = a[i];
                    a[i] = a[j];
                    a[j] = x;
                }
            }
            __syncthreads();
        }
    }
}

__global__ void sort_big_rows(const int64_t *__restrict__ row_ptr, unsigned long long *__restrict__ keys,
                              const int64_t *__restrict__ big_rows, const int *__restrict__ n_big,
                              int32_t *__restrict__ col, float *__restrict__ len)
{
    for (int b = blockIdx.x; b < *n_big; b += gridDim.x) {
        const int64_t row = big_rows[b], beg = row_ptr[row], m = row_ptr[row + 1] - beg;
        cta_sort(keys + beg, m);
        __syncthreads();
        if (col) {
            for (int64_t e = threadIdx.x; e < m; e += blockDim.x) {
                const unsigned long long k = keys[beg + e];
                col[beg + e] = (int32_t)(unsigned)(k & 0xFFFFFFFFull);
                len[beg + e] = __uint_as_float((unsigned)(k >> 32));
            }
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ path

constexpr int kPathSmall = 256;  // rows up to this many edges: one warp
constexpr int kPathMid = 1024;   // up to this many: a CTA of 256 threads; longer rows: several CTAs of 1,024
constexpr int kPathBlock = 8192; // targets of a long row in shared memory at a time
constexpr int kPathWarps = 4;
constexpr int kPathUnroll = 4;   // lists walked together, an entry of each per lane

// N(i) in shared memory: ids and lengths by position, and a chained hash from id to
// position (heads by hash, the next position by position), so that an entry that is
// not in N(i) mostly costs one look at an empty head.
template <int CAP, int HEADS> struct PathRow {
    int head[HEADS];
    int ids[CAP];
    float li[CAP];
    int wit[CAP];
    short nxt[CAP];
    static_assert(CAP <= 32767, "positions are 16-bit");
};

__device__ __forceinline__ unsigned phash(int id) { return static_cast<unsigned>(id) * 0x9E3779B1u; }

// Fills the row structure with node i's deg edges (threads first, first + step, ...).
template <int CAP, int HEADS>
__device__ __forceinline__ void path_row_clear(PathRow<CAP, HEADS> &sm, int first, int step)
{
    for (int t = first; t < HEADS; t += step)
        sm.head[t] = -1;
}
template <int CAP, int HEADS>
__device__ __forceinline__ void path_row_load(PathRow<CAP, HEADS> &sm, int64_t beg, int deg, const int32_t *__restrict__ col,
                                              const float *__restrict__ len, int first, int step)
{
    constexpr int shift = 32 - (HEADS == 512 ? 9 : HEADS == 2048 ? 11 : 13);
    static_assert(HEADS == 512 || HEADS == 2048 || HEADS == 8192, "HEADS");
    for (int t = first; t < deg; t += step) {
        const int j = col[beg + t];
        sm.ids[t] = j;
        sm.li[t] = len[beg + t];
        sm.wit[t] = INT_MAX;
        sm.nxt[t] = (short)atomicExch(&sm.head[phash(j) >> shift], t);
    }
}

// One warp tests the paths over the 32 neighbours u0 .. u0 + 31 of the row at `beg` of
// deg edges, to the targets in `sm` (the row's positions from j0 on): of every neighbour
// m closer than lmax (the row's longest edge) only the prefix of its list shorter than
// lmax can witness (rows are sorted by length), found by binary search, a lane per
// neighbour.  Four lists are walked at a time, 32 entries of each per step.
//
// The gathers' latency bounds this, so a step's ids are loaded a step ahead, and only
// the ids: a length is needed just for entries that are targets, farther than m, and not
// yet removed by a nearer witness.  Those few wait in `queue` until 32 of them fetch
// their lengths together.  1M rows, 68.8M edges, the whole pass: 67 ms when every entry
// looked its list up by binary search over prefix sums, loaded its length and probed an
// open table; 58 with whole lists per step and the chained hash; 46 as it is.
struct PathQueue {
    int64_t at[64];      // list entry whose length decides
    int tgt[64], u[64];  // target (position in sm), witness position
};
template <int CAP, int HEADS>
__device__ __forceinline__ void path_flush(PathRow<CAP, HEADS> &sm, PathQueue &queue, int first, int count,
                                           const float *__restrict__ len, int lane)
{
    if (lane < count) {
        const int p = queue.tgt[first + lane];
        if (__ldg(len + queue.at[first + lane]) < sm.li[p])
            atomicMin(&sm.wit[p], queue.u[first + lane]);
    }
    __syncwarp();
}
template <int CAP, int HEADS>
__device__ __forceinline__ void path_scan(PathRow<CAP, HEADS> &sm, PathQueue &queue, int64_t beg, int u0, int deg, float lmax,
                                          const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
                                          const float *__restrict__ len, int lane)
{
    constexpr int shift = 32 - (HEADS == 512 ? 9 : HEADS == 2048 ? 11 : 13);
    const int u = u0 + lane;
    int64_t mb = 0;
    int cnt = 0;
    const float lu = u < deg ? len[beg + u] : INFINITY;
    if (lu < lmax) {
        const int m = col[beg + u];
        mb = rp[m];
        int lo = 0, hi = (int)(rp[m + 1] - mb);
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (len[mb + mid] < lmax)
                lo = mid + 1;
            else
                hi = mid;
        }
        cnt = lo;
    }
    __syncwarp();
    const volatile int *wit = sm.wit;
    int pending = 0;  // queued entries
    // the lists of the step in hand (g, e) and of the one being loaded
    int64_t b[kPathUnroll];
    int c[kPathUnroll], j[kPathUnroll], most = 0;
    auto lists = [&](int g) {
        most = 0;
#pragma unroll
        for (int r = 0; r < kPathUnroll; ++r) {
            b[r] = __shfl_sync(0xffffffffu, mb, g + r) + lane;
            c[r] = __shfl_sync(0xffffffffu, cnt, g + r);
            most = max(most, c[r]);
        }
    };
    auto load = [&](int e) {
#pragma unroll
        for (int r = 0; r < kPathUnroll; ++r)
            j[r] = e + lane < c[r] ? __ldg(col + b[r] + e) : -1;
    };
    const int gend = min(32, deg - u0);
    int g = 0, e = 0;
    lists(0);
    load(0);
    while (g < gend) {
        int64_t cb[kPathUnroll];
        int cj[kPathUnroll];
#pragma unroll
        for (int r = 0; r < kPathUnroll; ++r) {
            cb[r] = b[r] + e;
            cj[r] = j[r];
        }
        const int cg = g;
        e += 32;
        if (e >= most) {
            e = 0;
            g += kPathUnroll;
            if (g < gend)
                lists(g);
        }
        if (g < gend)
            load(e);
#pragma unroll
        for (int r = 0; r < kPathUnroll; ++r) {
            const float l = __shfl_sync(0xffffffffu, lu, cg + r);
            int p = cj[r] >= 0 ? sm.head[phash(cj[r]) >> shift] : -1;
            while (p >= 0 && sm.ids[p] != cj[r])
                p = sm.nxt[p];
            const bool need = p >= 0 && l < sm.li[p] && wit[p] > u0 + cg + r;
            const unsigned nm = __ballot_sync(0xffffffffu, need);
            if (!nm)
                continue;
            if (need) {
                const int at = pending + __popc(nm & ((1u << lane) - 1u));
                queue.at[at] = cb[r];
                queue.tgt[at] = p;
                queue.u[at] = u0 + cg + r;
            }
            pending += __popc(nm);
            __syncwarp();
            if (pending >= 32) {
                pending -= 32;
                path_flush(sm, queue, pending, 32, len, lane);
            }
        }
    }
    path_flush(sm, queue, 0, pending, len, lane);
}

// Marks removals of the edges of node i (deg <= kPathSmall) by one warp.
__device__ void path_row_warp(int64_t i, const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
                              const float *__restrict__ len, PathRow<kPathSmall, 512> &sm, PathQueue &queue,
                              int *__restrict__ wit_out, int lane)
{
    const int64_t beg = rp[i];
    const int deg = (int)(rp[i + 1] - beg);
    path_row_clear(sm, lane, 32);
    __syncwarp();
    path_row_load(sm, beg, deg, col, len, lane, 32);
    __syncwarp();
    // the longest edge, wherever it stands: a row that is nobody's neighbour need not be sorted
    float lmax = 0.f;
    for (int t = lane; t < deg; t += 32)
        lmax = fmaxf(lmax, sm.li[t]);
    lmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(lmax)));
    for (int u0 = 0; u0 < deg; u0 += 32)
        path_scan(sm, queue, beg, u0, deg, lmax, rp, col, len, lane);
    __syncwarp();
    for (int t = lane; t < deg; t += 32)
        wit_out[beg + t] = sm.wit[t] == INT_MAX ? -1 : sm.wit[t];
    __syncwarp();
}

// Warps stride over the rows (the grid is what stays resident), so a warp whose
// row ends early takes the next one instead of idling until the slowest row of
// its CTA is done.
__global__ void __launch_bounds__(kPathWarps * 32)
    path_small_kernel(const int64_t *__restrict__ rp, const int32_t *__restrict__ col, const float *__restrict__ len,
                      int64_t n, int *__restrict__ wit, int64_t *__restrict__ big_rows, int *__restrict__ n_big)
{
    __shared__ PathRow<kPathSmall, 512> sm[kPathWarps];
    __shared__ PathQueue queue[kPathWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * kPathWarps;
    for (int64_t i = (int64_t)blockIdx.x * kPathWarps + warp; i < n; i += stride) {
        const int64_t deg = rp[i + 1] - rp[i];
        if (deg > kPathSmall) {
            // rows of several CTAs are listed from the end; their marks are combined in place
            const bool several = deg > kPathMid;
            if (lane == 0)
                big_rows[several ? n - 1 - atomicAdd(n_big + 1, 1) : atomicAdd(n_big, 1)] = i;
            if (several)
                for (int64_t t = lane; t < deg; t += 32)
                    wit[rp[i] + t] = INT_MAX;
            continue;
        }
        if (deg >= 2)
            path_row_warp(i, rp, col, len, sm[warp], queue[warp], wit, lane);
        else if (deg == 1 && lane == 0)
            wit[rp[i]] = -1;
    }
}

// Listed rows of kPathSmall < edges <= kPathMid: a CTA per row, its warps taking 32
// neighbours at a time, everything but the graph in shared memory.
__global__ void __launch_bounds__(256)
    path_mid_kernel(const int64_t *__restrict__ rp, const int32_t *__restrict__ col, const float *__restrict__ len,
                    int *__restrict__ wit, const int64_t *__restrict__ big_rows, const int *__restrict__ n_big)
{
    __shared__ PathRow<kPathMid, 2048> sm;
    __shared__ PathQueue queue[256 / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int b = blockIdx.x; b < n_big[0]; b += gridDim.x) {
        const int64_t beg = rp[big_rows[b]];
        const int deg = (int)(rp[big_rows[b] + 1] - beg);
        path_row_clear(sm, threadIdx.x, blockDim.x);
        __syncthreads();
        path_row_load(sm, beg, deg, col, len, threadIdx.x, blockDim.x);
        __syncthreads();
        const float lmax = sm.li[deg - 1];
        for (int u0 = warp * 32; u0 < deg; u0 += blockDim.x)
            path_scan(sm, queue[warp], beg, u0, deg, lmax, rp, col, len, lane);
        __syncthreads();
        for (int t = threadIdx.x; t < deg; t += blockDim.x)
            wit[beg + t] = sm.wit[t] == INT_MAX ? -1 : sm.wit[t];
        __syncthreads();
    }
}

// Rows of more than kPathMid edges, as tasks of 1,024 neighbours by kPathBlock targets
// dealt out over the CTAs (one CTA per row left a hub of 9,679 edges alone on its SM for
// 7 ms of a 60 ms pass).  A task's marks go to the row by atomicMin; marks that stay
// INT_MAX count as kept.
struct PathLong {
    PathRow<kPathBlock, 8192> row;
    PathQueue queue[32];
};
__global__ void __launch_bounds__(1024)
    path_long_kernel(const int64_t *__restrict__ rp, const int32_t *__restrict__ col, const float *__restrict__ len, int64_t n,
                     int *__restrict__ wit, const int64_t *__restrict__ big_rows, const int *__restrict__ n_big)
{
    extern __shared__ __align__(16) unsigned char path_raw[];
    PathLong &sm = *reinterpret_cast<PathLong *>(path_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t task = 0;
    for (int b = 0; b < n_big[1]; ++b) {
        const int64_t i = big_rows[n - 1 - b], beg = rp[i];
        const int deg = (int)(rp[i + 1] - beg);
        const int segs = (deg + 1023) / 1024, blocks = (deg + kPathBlock - 1) / kPathBlock;
        const float lmax = len[beg + deg - 1];
        for (int t = 0; t < segs * blocks; ++t, ++task) {
            if (task % gridDim.x != blockIdx.x)
                continue;
            const int j0 = t % blocks * kPathBlock, targets = min(kPathBlock, deg - j0);
            path_row_clear(sm.row, threadIdx.x, 1024);
            __syncthreads();
            path_row_load(sm.row, beg + j0, targets, col, len, threadIdx.x, 1024);
            __syncthreads();
            const int u0 = t / blocks * 1024 + warp * 32;
            if (u0 < deg)
                path_scan(sm.row, sm.queue[warp], beg, u0, deg, lmax, rp, col, len, lane);
            __syncthreads();
            for (int e = threadIdx.x; e < targets; e += 1024)
                if (sm.row.wit[e] != INT_MAX)
                    atomicMin(&wit[beg + j0 + e], sm.row.wit[e]);
            __syncthreads();
        }
    }
}

// a witness position, or none: -1, or INT_MAX in the rows of several CTAs
__device__ __forceinline__ bool path_kept(int w) { return (unsigned)w >= (unsigned)INT_MAX; }

__global__ void path_count_kernel(const int64_t *__restrict__ rp, int64_t n, const int *__restrict__ wit,
                                  int64_t *__restrict__ kept)
{
    const int lane = threadIdx.x & 31;
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (i >= n)
        return;
    int64_t c = 0;
    for (int64_t e = rp[i] + lane; e < rp[i + 1]; e += 32)
        c += path_kept(wit[e]);
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1)
        c += __shfl_xor_sync(0xffffffffu, c, off);
    if (lane == 0)
        kept[i] = c;
}

__global__ void path_compact_kernel(const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
                                    const float *__restrict__ len, int64_t n, const int *__restrict__ wit,
                                    const int64_t *__restrict__ rp_out, int32_t *__restrict__ col_out,
                                    float *__restrict__ len_out, int32_t *__restrict__ removed_by)
{
    const int lane = threadIdx.x & 31;
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (i >= n)
        return;
    const int64_t beg = rp[i], end = rp[i + 1];
    int64_t w = rp_out[i];
    for (int64_t e0 = beg; e0 < end; e0 += 32) {
        const int64_t e = e0 + lane;
        const bool keep = e < end && path_kept(wit[e]);
        const unsigned km = __ballot_sync(0xffffffffu, keep);
        if (keep) {
            const int64_t dst = w + __popc(km & ((1u << lane) - 1u));
            col_out[dst] = col[e];
            len_out[dst] = len[e];
        }
        if (removed_by && e < end)
            removed_by[e] = path_kept(wit[e]) ? -1 : col[beg + wit[e]];
        w += __popc(km);
    }
}

// ------------------------------------------------------------------ Algorithm 4, literal

// byid[e] = (id << 32 | position) of every edge, per row; sorted per row afterwards
__global__ void alg4_byid_kernel(const int64_t *__restrict__ rp, const int32_t *__restrict__ col, int64_t n,
                                 unsigned long long *__restrict__ byid)
{
    const int lane = threadIdx.x & 31;
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (i >= n)
        return;
    for (int64_t e = rp[i] + lane; e < rp[i + 1]; e += 32)
        byid[e] = ((unsigned long long)(unsigned)col[e] << 32) | (unsigned)(e - rp[i]);
}

// position of t in row m (its id-sorted copy), or -1
__device__ __forceinline__ int alg4_find(const int64_t *__restrict__ rp, const unsigned long long *__restrict__ byid,
                                         int32_t m, int32_t t)
{
    int64_t lo = rp[m], hi = rp[m + 1];
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        const int32_t id = (int32_t)(byid[mid] >> 32);
        if (id < t)
            lo = mid + 1;
        else
            hi = mid;
    }
    if (lo < rp[m + 1] && (int32_t)(byid[lo] >> 32) == t)
        return (int)(unsigned)(byid[lo] & 0xFFFFFFFFull);
    return -1;
}

// Edge states: 0 undecided, 1 kept, 2 removed.
// One warp per node s = order[w] (nodes by degree, descending: the nodes with
// more than p edges are a prefix).  Decides s's p-th edge if it can; counts the
// edges still waiting in *waiting.
__global__ void alg4_round_kernel(const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
                                  const float *__restrict__ len, const unsigned long long *__restrict__ byid,
                                  const int32_t *__restrict__ order, int64_t active, int p,
                                  unsigned char *__restrict__ state, int *__restrict__ waiting)
{
    const int lane = threadIdx.x & 31;
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (w >= active)
        return;
    const int32_t s = order[w];
    const int64_t beg = rp[s];
    if (state[beg + p] != 0)
        return;
    const int32_t t = col[beg + p];
    const float lst = len[beg + p];
    bool path = false, wait = false;
    for (int q0 = 0; q0 < p; q0 += 32) {
        const int q = q0 + lane;
        if (q < p && state[beg + q] == 1) {
            const int32_t m = col[beg + q];
            const int r = alg4_find(rp, byid, m, t);
            if (r >= 0 && len[rp[m] + r] < lst) {
                if (r < p) {
                    path |= state[rp[m] + r] == 1;
                } else if (r == p && m < s) {
                    const unsigned char sm = state[rp[m] + r];
                    path |= sm == 1;
                    wait |= sm == 0;
                }
            }
        }
    }
    path = __any_sync(0xffffffffu, path);
    wait = __any_sync(0xffffffffu, wait);
    if (lane == 0) {
        if (path)
            state[beg + p] = 2;
        else if (!wait)
            state[beg + p] = 1;
        else
            atomicAdd(waiting, 1);
    }
}

__global__ void alg4_hist_kernel(const int64_t *__restrict__ rp, int64_t n, int *__restrict__ hist)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&hist[rp[i + 1] - rp[i]], 1);
}

// order[] = nodes grouped by degree, largest first (offset[d] = nodes of degree > d)
__global__ void alg4_order_kernel(const int64_t *__restrict__ rp, int64_t n, const int64_t *__restrict__ offset,
                                  int *__restrict__ cursor, int32_t *__restrict__ order)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t d = rp[i + 1] - rp[i];
        order[offset[d] + atomicAdd(&cursor[d], 1)] = (int32_t)i;
    }
}

__global__ void alg4_wit_kernel(const unsigned char *__restrict__ state, int64_t nnz, int *__restrict__ wit)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x)
        wit[e] = state[e] == 2 ? 0 : -1;
}

// ------------------------------------------------------------------ SAC

// first[n] = the first node, in the order (|N(G_t, o)|, o), among the valid ids
// of first_{fi}(N_k(n)) (-1 if none): the node of Algorithm 3 that meets n first.
__global__ void sac_first_kernel(const int32_t *__restrict__ nbr, int64_t n, int k, int fi,
                                 const int64_t *__restrict__ gt_ptr, int32_t *__restrict__ first)
{
    for (int64_t y = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; y < n; y += (int64_t)gridDim.x * blockDim.x) {
        int64_t best_deg = INT64_MAX;
        int32_t best = -1;
        for (int p = 0; p < fi; ++p) {
            const int32_t o = nbr[y * k + p];
            if (o < 0 || o >= n)
                continue;
            const int64_t dg = gt_ptr[o + 1] - gt_ptr[o];
            if (dg < best_deg || (dg == best_deg && o < best)) {
                best_deg = dg;
                best = o;
            }
        }
        first[y] = best;
    }
}

// One warp per node o.  Row = the members of N(G_t, o) (keys sorted by (length,
// id)) at positions < e_o or first-met at o, then, if fewer than e_o, o's kNN
// neighbours in order that are not in N(G_t, o), up to e_o in all.  Count mode
// (keys == NULL) writes the row sizes; fill mode writes the keys at row_ptr[o].
__global__ void sac_row_kernel(const int32_t *__restrict__ nbr, const float *__restrict__ len, int64_t n, int k,
                               int e_o, const int64_t *__restrict__ gt_ptr,
                               const unsigned long long *__restrict__ gt_keys, const int32_t *__restrict__ first,
                               int64_t *__restrict__ cnt, const int64_t *__restrict__ row_ptr,
                               unsigned long long *__restrict__ keys)
{
    const int lane = threadIdx.x & 31;
    const int64_t o = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (o >= n)
        return;
    const int64_t beg = gt_ptr[o];
    const int64_t m = gt_ptr[o + 1] - beg;
    const int64_t out = keys ? row_ptr[o] : 0;
    int64_t w = 0;
    for (int64_t c0 = 0; c0 < m; c0 += 32) {
        const int64_t p = c0 + lane;
        unsigned long long key = 0;
        bool take = false;
        if (p < m) {
            key = gt_keys[beg + p];
            take = p < e_o || first[(int32_t)(unsigned)(key & 0xFFFFFFFFull)] == (int32_t)o;
        }
        const unsigned tm = __ballot_sync(0xffffffffu, take);
        if (keys && take)
            keys[out + w + __popc(tm & ((1u << lane) - 1u))] = key;
        w += __popc(tm);
    }
    if (m < e_o) {
        // every member was taken; the nearest kNN neighbours not among them follow
        for (int p0 = 0; p0 < k && w < e_o; p0 += 32) {
            const int p = p0 + lane;
            const int32_t x = p < k ? nbr[o * k + p] : -1;
            bool cand = x >= 0 && x < n;
            for (int64_t t = 0; cand && t < m; ++t)
                cand = (int32_t)(unsigned)(gt_keys[beg + t] & 0xFFFFFFFFull) != x;
            const unsigned cm = __ballot_sync(0xffffffffu, cand);
            const int rank = __popc(cm & ((1u << lane) - 1u));
            if (keys && cand && w + rank < e_o)
                keys[out + w + rank] = pack_key(len[o * k + p], x);
            w = min((int64_t)e_o, w + __popc(cm));
            // kNN rows are padded with -1 at their end: the list stops there
            if (__ballot_sync(0xffffffffu, p < k && x < 0))
                break;
        }
    }
    if (!keys && lane == 0)
        cnt[o] = w;
}

// whether every row of k ids starts on 16 bytes
bool rows16(const int32_t *nbr, int k) { return aligned16(nbr) && k % 4 == 0; }

int grid1d(int64_t work, int threads)
{
    return (int)std::max<int64_t>(1, std::min<int64_t>((work + threads - 1) / threads, (int64_t)num_sms() * 16));
}

}  // namespace
}  // namespace onng

using namespace onng;

// ------------------------------------------------------------------ degree ABI

extern "C" size_t onng_adjust_degree_workspace_bytes(int64_t n, int32_t k)
{
    WsCarver c(nullptr);
    c.take<int>((size_t)std::max<int64_t>(n, 1));  // in-counts / cursors
    c.take<int64_t>((size_t)std::max<int64_t>(n, 1));  // row sizes
    c.take<int64_t>((size_t)std::max<int64_t>(n, 1));  // long rows
    c.take<int>(64);
    c.take<char>(scan_workspace_bytes(std::max<int64_t>(n, 1)));
    c.take<unsigned long long>((size_t)std::max<int64_t>(n, 1) * (size_t)std::max(k, 1) * 2);  // keys
    return c.used;
}

static int degree_args(const int32_t *nbr, const float *len, int64_t n, int32_t k, int32_t e_o, int32_t e_i,
                       void *ws, size_t ws_bytes, const char *who)
{
    ONNG_REQUIRE(n >= 0 && n <= INT32_MAX && k >= 1 && e_o >= 0 && e_i >= 0, ONNG_E_INVAL, "%s: bad sizes", who);
    ONNG_REQUIRE(n == 0 || (nbr && len), ONNG_E_INVAL, "%s: NULL input", who);
    const size_t need = onng_adjust_degree_workspace_bytes(n, k);
    ONNG_REQUIRE(ws && ws_bytes >= need, ONNG_E_WORKSPACE, "%s: workspace %zu < %zu bytes", who, ws_bytes, need);
    return ONNG_OK;
}

extern "C" int onng_adjust_degree_count(const int32_t *nbr, const float *len, int64_t n, int32_t k, int32_t e_o,
                                        int32_t e_i, int64_t *row_ptr, int64_t *nnz_host, void *ws, size_t ws_bytes,
                                        onng_stream_t stream)
{
    ONNG_RANGE("onng_adjust_degree_count");
    int st = degree_args(nbr, len, n, k, e_o, e_i, ws, ws_bytes, "onng_adjust_degree_count");
    if (st)
        return st;
    ONNG_REQUIRE(row_ptr, ONNG_E_INVAL, "onng_adjust_degree_count: NULL row_ptr");
    cudaStream_t s = to_cuda(stream);
    const int fo = std::min(e_o, k), fi = std::min(e_i, k);
    WsCarver c(ws);
    int *incnt = c.take<int>((size_t)std::max<int64_t>(n, 1));
    int64_t *deg = c.take<int64_t>((size_t)std::max<int64_t>(n, 1));
    c.take<int64_t>((size_t)std::max<int64_t>(n, 1));
    c.take<int>(64);
    char *scan_ws = c.take<char>(scan_workspace_bytes(std::max<int64_t>(n, 1)));
    if (n > 0) {
        ONNG_CUDA_TRY(cudaMemsetAsync(incnt, 0, sizeof(int) * n, s), "adjust_degree: clear");
        degree_count_kernel<<<grid1d(n * 32, 256), 256, 0, s>>>(nbr, n, k, fo, fi, rows16(nbr, k), deg, incnt);
        degree_total_kernel<<<grid1d(n, 256), 256, 0, s>>>(n, incnt, deg);
        st = check_launch("onng_adjust_degree_count");
        if (st)
            return st;
    }
    st = exclusive_scan(deg, row_ptr, n, scan_ws, scan_workspace_bytes(std::max<int64_t>(n, 1)), s);
    if (st)
        return st;
    if (nnz_host) {
        ONNG_CUDA_TRY(cudaMemcpyAsync(nnz_host, row_ptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s),
                      "adjust_degree: nnz");
        ONNG_CUDA_TRY(cudaStreamSynchronize(s), "adjust_degree: sync");
    }
    return ONNG_OK;
}

extern "C" int onng_adjust_degree(const int32_t *nbr, const float *len, int64_t n, int32_t k, int32_t e_o, int32_t e_i,
                                  const int64_t *row_ptr, int32_t *col, float *len_out, void *ws, size_t ws_bytes,
                                  onng_stream_t stream)
{
    ONNG_RANGE("onng_adjust_degree");
    int st = degree_args(nbr, len, n, k, e_o, e_i, ws, ws_bytes, "onng_adjust_degree");
    if (st)
        return st;
    if (n == 0)
        return ONNG_OK;
    ONNG_REQUIRE(row_ptr && col && len_out, ONNG_E_INVAL, "onng_adjust_degree: NULL output");
    cudaStream_t s = to_cuda(stream);
    const int fo = std::min(e_o, k), fi = std::min(e_i, k);
    WsCarver c(ws);
    int *cursor = c.take<int>((size_t)n);
    c.take<int64_t>((size_t)n);
    int64_t *big = c.take<int64_t>((size_t)n);
    int *n_big = c.take<int>(64);
    c.take<char>(scan_workspace_bytes(n));
    unsigned long long *keys = c.take<unsigned long long>((size_t)n * k * 2);
    ONNG_CUDA_TRY(cudaMemsetAsync(cursor, 0, sizeof(int) * n, s), "adjust_degree: clear");
    ONNG_CUDA_TRY(cudaMemsetAsync(n_big, 0, sizeof(int), s), "adjust_degree: clear");
    degree_fill_kernel<<<grid1d(n * 32, 256), 256, 0, s>>>(nbr, len, n, k, fo, fi, rows16(nbr, k), row_ptr, cursor, keys);
    sort_small_rows<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(row_ptr, n, keys, big, n_big, col, len_out);
    sort_big_rows<<<num_sms() * 2, 1024, 0, s>>>(row_ptr, keys, big, n_big, col, len_out);
    return check_launch("onng_adjust_degree: fill/sort");
}

// ------------------------------------------------------------------ SAC ABI

namespace onng {
namespace {

struct SacWs {
    int *incnt;
    int64_t *cnt, *big, *gt_ptr;
    int *n_big;
    char *scan_ws;
    size_t scan_bytes;
    unsigned long long *gt_keys, *keys;
    int32_t *first;
    size_t used;
};

SacWs sac_carve(void *ws, int64_t n, int k)
{
    const int64_t nn = std::max<int64_t>(n, 1);
    WsCarver c(ws);
    SacWs w;
    w.incnt = c.take<int>((size_t)nn);
    w.cnt = c.take<int64_t>((size_t)nn);
    w.big = c.take<int64_t>((size_t)nn);
    w.n_big = c.take<int>(64);
    w.scan_bytes = scan_workspace_bytes(nn + 1);
    w.scan_ws = c.take<char>(w.scan_bytes);
    w.gt_ptr = c.take<int64_t>((size_t)nn + 1);
    w.gt_keys = c.take<unsigned long long>((size_t)nn * std::max(k, 1));
    w.first = c.take<int32_t>((size_t)nn);
    w.keys = c.take<unsigned long long>((size_t)nn * std::max(k, 1) * 2);  // rows hold <= n k + n k edges
    w.used = c.used;
    return w;
}

// G_t of Algorithm 3 (Algorithm 2 with (0, e_i)) as sorted (length, id) keys,
// then every node's first considerer.
int sac_prepare(const int32_t *nbr, const float *len, int64_t n, int k, int fi, const SacWs &w, cudaStream_t s)
{
    ONNG_CUDA_TRY(cudaMemsetAsync(w.incnt, 0, sizeof(int) * n, s), "adjust_degree_sac: clear");
    ONNG_CUDA_TRY(cudaMemsetAsync(w.n_big, 0, sizeof(int), s), "adjust_degree_sac: clear");
    degree_count_kernel<<<grid1d(n * 32, 256), 256, 0, s>>>(nbr, n, k, 0, fi, rows16(nbr, k), w.cnt, w.incnt);
    degree_total_kernel<<<grid1d(n, 256), 256, 0, s>>>(n, w.incnt, w.cnt);
    int st = check_launch("onng_adjust_degree_sac: G_t count");
    if (st)
        return st;
    st = exclusive_scan(w.cnt, w.gt_ptr, n, w.scan_ws, w.scan_bytes, s);
    if (st)
        return st;
    ONNG_CUDA_TRY(cudaMemsetAsync(w.incnt, 0, sizeof(int) * n, s), "adjust_degree_sac: clear");
    degree_fill_kernel<<<grid1d(n * 32, 256), 256, 0, s>>>(nbr, len, n, k, 0, fi, rows16(nbr, k), w.gt_ptr, w.incnt,
                                                           w.gt_keys);
    sort_small_rows<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(w.gt_ptr, n, w.gt_keys, w.big, w.n_big, nullptr,
                                                                    nullptr);
    sort_big_rows<<<num_sms() * 2, 1024, 0, s>>>(w.gt_ptr, w.gt_keys, w.big, w.n_big, nullptr, nullptr);
    sac_first_kernel<<<grid1d(n, 256), 256, 0, s>>>(nbr, n, k, fi, w.gt_ptr, w.first);
    return check_launch("onng_adjust_degree_sac: G_t");
}

}  // namespace
}  // namespace onng

extern "C" size_t onng_adjust_degree_sac_workspace_bytes(int64_t n, int32_t k)
{
    return sac_carve(nullptr, n, k).used;
}

extern "C" int onng_adjust_degree_sac_count(const int32_t *nbr, const float *len, int64_t n, int32_t k, int32_t e_o,
                                            int32_t e_i, int64_t *row_ptr, int64_t *nnz_host, void *ws,
                                            size_t ws_bytes, onng_stream_t stream)
{
    ONNG_RANGE("onng_adjust_degree_sac_count");
    ONNG_REQUIRE(n >= 0 && n <= INT32_MAX && k >= 1 && e_o >= 0 && e_i >= 0, ONNG_E_INVAL,
                 "onng_adjust_degree_sac_count: bad sizes");
    ONNG_REQUIRE(n == 0 || (nbr && len), ONNG_E_INVAL, "onng_adjust_degree_sac_count: NULL input");
    ONNG_REQUIRE(row_ptr, ONNG_E_INVAL, "onng_adjust_degree_sac_count: NULL row_ptr");
    const size_t need = onng_adjust_degree_sac_workspace_bytes(n, k);
    ONNG_REQUIRE(ws && ws_bytes >= need, ONNG_E_WORKSPACE, "onng_adjust_degree_sac_count: workspace %zu < %zu bytes",
                 ws_bytes, need);
    cudaStream_t s = to_cuda(stream);
    const SacWs w = sac_carve(ws, n, k);
    int st;
    if (n > 0) {
        st = sac_prepare(nbr, len, n, k, std::min(e_i, k), w, s);
        if (st)
            return st;
        sac_row_kernel<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(nbr, len, n, k, e_o, w.gt_ptr, w.gt_keys,
                                                                       w.first, w.cnt, nullptr, nullptr);
        st = check_launch("onng_adjust_degree_sac_count: rows");
        if (st)
            return st;
    }
    st = exclusive_scan(w.cnt, row_ptr, n, w.scan_ws, w.scan_bytes, s);
    if (st)
        return st;
    if (nnz_host) {
        ONNG_CUDA_TRY(cudaMemcpyAsync(nnz_host, row_ptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s),
                      "adjust_degree_sac: nnz");
        ONNG_CUDA_TRY(cudaStreamSynchronize(s), "adjust_degree_sac: sync");
    }
    return ONNG_OK;
}

extern "C" int onng_adjust_degree_sac(const int32_t *nbr, const float *len, int64_t n, int32_t k, int32_t e_o,
                                      int32_t e_i, const int64_t *row_ptr, int32_t *col, float *len_out, void *ws,
                                      size_t ws_bytes, onng_stream_t stream)
{
    ONNG_RANGE("onng_adjust_degree_sac");
    ONNG_REQUIRE(n >= 0 && n <= INT32_MAX && k >= 1 && e_o >= 0 && e_i >= 0, ONNG_E_INVAL,
                 "onng_adjust_degree_sac: bad sizes");
    ONNG_REQUIRE(n == 0 || (nbr && len), ONNG_E_INVAL, "onng_adjust_degree_sac: NULL input");
    const size_t need = onng_adjust_degree_sac_workspace_bytes(n, k);
    ONNG_REQUIRE(ws && ws_bytes >= need, ONNG_E_WORKSPACE, "onng_adjust_degree_sac: workspace %zu < %zu bytes",
                 ws_bytes, need);
    if (n == 0)
        return ONNG_OK;
    ONNG_REQUIRE(row_ptr && col && len_out, ONNG_E_INVAL, "onng_adjust_degree_sac: NULL output");
    cudaStream_t s = to_cuda(stream);
    const SacWs w = sac_carve(ws, n, k);
    int st = sac_prepare(nbr, len, n, k, std::min(e_i, k), w, s);
    if (st)
        return st;
    sac_row_kernel<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(nbr, len, n, k, e_o, w.gt_ptr, w.gt_keys, w.first,
                                                                   nullptr, row_ptr, w.keys);
    ONNG_CUDA_TRY(cudaMemsetAsync(w.n_big, 0, sizeof(int), s), "adjust_degree_sac: clear");
    sort_small_rows<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(row_ptr, n, w.keys, w.big, w.n_big, col, len_out);
    sort_big_rows<<<num_sms() * 2, 1024, 0, s>>>(row_ptr, w.keys, w.big, w.n_big, col, len_out);
    return check_launch("onng_adjust_degree_sac: fill/sort");
}

// ------------------------------------------------------------------ literal Algorithm 4 ABI

extern "C" size_t onng_adjust_path_literal_workspace_bytes(int64_t n, int64_t nnz)
{
    const int64_t nn = std::max<int64_t>(n, 1), mm = std::max<int64_t>(nnz, 1);
    WsCarver c(nullptr);
    c.take<unsigned long long>((size_t)mm);  // id-sorted rows
    c.take<unsigned char>((size_t)mm);       // edge states
    c.take<int>((size_t)mm);                 // removal marks
    c.take<int64_t>((size_t)nn);             // kept counts / long rows
    c.take<int64_t>((size_t)nn + 1);         // degree offsets
    c.take<int>((size_t)nn + 1);             // degree histogram / cursors
    c.take<int32_t>((size_t)nn);             // nodes by degree
    c.take<int>(64);
    c.take<char>(scan_workspace_bytes(nn + 1));
    return c.used;
}

extern "C" int onng_adjust_path_literal(const int64_t *row_ptr, const int32_t *col, const float *len, int64_t n,
                                        int64_t *row_ptr_out, int32_t *col_out, float *len_out, int64_t *nnz_host,
                                        void *ws, size_t ws_bytes, onng_stream_t stream)
{
    ONNG_RANGE("onng_adjust_path_literal");
    // ids are sorted as (id << 32 | position) keys below the sorters' padding key
    ONNG_REQUIRE(n >= 0 && n < 0x7F800000LL, ONNG_E_INVAL, "onng_adjust_path_literal: bad n");
    ONNG_REQUIRE(row_ptr && row_ptr_out, ONNG_E_INVAL, "onng_adjust_path_literal: NULL row_ptr");
    cudaStream_t s = to_cuda(stream);
    int64_t nnz = 0;
    ONNG_CUDA_TRY(cudaMemcpyAsync(&nnz, row_ptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s),
                  "adjust_path_literal: nnz");
    ONNG_CUDA_TRY(cudaStreamSynchronize(s), "adjust_path_literal: sync");
    const size_t need = onng_adjust_path_literal_workspace_bytes(n, nnz);
    ONNG_REQUIRE(ws && ws_bytes >= need, ONNG_E_WORKSPACE, "onng_adjust_path_literal: workspace %zu < %zu bytes",
                 ws_bytes, need);
    ONNG_REQUIRE(nnz == 0 || (col && len && col_out && len_out), ONNG_E_INVAL,
                 "onng_adjust_path_literal: NULL arrays");
    const int64_t nn = std::max<int64_t>(n, 1), mm = std::max<int64_t>(nnz, 1);
    WsCarver c(ws);
    unsigned long long *byid = c.take<unsigned long long>((size_t)mm);
    unsigned char *state = c.take<unsigned char>((size_t)mm);
    int *wit = c.take<int>((size_t)mm);
    int64_t *kept = c.take<int64_t>((size_t)nn);
    int64_t *offset = c.take<int64_t>((size_t)nn + 1);
    int *hist = c.take<int>((size_t)nn + 1);
    int32_t *order = c.take<int32_t>((size_t)nn);
    int *flags = c.take<int>(64);
    char *scan_ws = c.take<char>(scan_workspace_bytes(nn + 1));
    int st;
    if (n > 0 && nnz > 0) {
        // rows by id for the position lookups of Algorithm 5
        ONNG_CUDA_TRY(cudaMemsetAsync(flags, 0, sizeof(int) * 64, s), "adjust_path_literal: clear");
        alg4_byid_kernel<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(row_ptr, col, n, byid);
        sort_small_rows<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(row_ptr, n, byid, kept, flags, nullptr, nullptr);
        sort_big_rows<<<num_sms() * 2, 1024, 0, s>>>(row_ptr, byid, kept, flags, nullptr, nullptr);
        // nodes by degree, largest first
        ONNG_CUDA_TRY(cudaMemsetAsync(hist, 0, sizeof(int) * (n + 1), s), "adjust_path_literal: clear");
        alg4_hist_kernel<<<grid1d(n, 256), 256, 0, s>>>(row_ptr, n, hist);
        ONNG_CUDA_TRY(cudaMemsetAsync(state, 0, (size_t)nnz, s), "adjust_path_literal: clear");
        st = check_launch("onng_adjust_path_literal: prepare");
        if (st)
            return st;
        std::vector<int> h((size_t)n + 1);
        ONNG_CUDA_TRY(cudaMemcpyAsync(h.data(), hist, sizeof(int) * (n + 1), cudaMemcpyDeviceToHost, s),
                      "adjust_path_literal: histogram");
        ONNG_CUDA_TRY(cudaStreamSynchronize(s), "adjust_path_literal: sync");
        int64_t maxdeg = 0;
        for (int64_t d = n; d >= 0; --d)
            if (h[d]) {
                maxdeg = d;
                break;
            }
        std::vector<int64_t> off((size_t)n + 1, 0), active((size_t)maxdeg + 1, 0);
        int64_t acc = 0;
        for (int64_t d = maxdeg; d >= 0; --d) {
            off[d] = acc;  // nodes of degree > d come first
            acc += h[d];
        }
        for (int64_t p = 0; p <= maxdeg; ++p)
            active[p] = off[p];  // nodes with more than p edges
        ONNG_CUDA_TRY(cudaMemcpyAsync(offset, off.data(), sizeof(int64_t) * (n + 1), cudaMemcpyHostToDevice, s),
                      "adjust_path_literal: offsets");
        ONNG_CUDA_TRY(cudaMemsetAsync(hist, 0, sizeof(int) * (n + 1), s), "adjust_path_literal: clear");
        alg4_order_kernel<<<grid1d(n, 256), 256, 0, s>>>(row_ptr, n, offset, hist, order);
        st = check_launch("onng_adjust_path_literal: order");
        if (st)
            return st;
        int *waiting = flags + 32;
        for (int64_t p = 0; p < maxdeg; ++p) {
            const int64_t act = active[p];
            // every pass decides at least the smallest waiting node, so act + 1 passes suffice
            for (int64_t pass = 0;; ++pass) {
                ONNG_REQUIRE(pass <= act, ONNG_E_LIMIT, "onng_adjust_path_literal: round %lld did not settle",
                             (long long)p);
                ONNG_CUDA_TRY(cudaMemsetAsync(waiting, 0, sizeof(int), s), "adjust_path_literal: clear");
                alg4_round_kernel<<<(unsigned)((act * 32 + 255) / 256), 256, 0, s>>>(row_ptr, col, len, byid, order,
                                                                                  act, (int)p, state, waiting);
                st = check_launch("onng_adjust_path_literal: round");
                if (st)
                    return st;
                int left = 0;
                ONNG_CUDA_TRY(cudaMemcpyAsync(&left, waiting, sizeof(int), cudaMemcpyDeviceToHost, s),
                              "adjust_path_literal: waiting");
                ONNG_CUDA_TRY(cudaStreamSynchronize(s), "adjust_path_literal: sync");
                if (left == 0)
                    break;
            }
        }
        alg4_wit_kernel<<<grid1d(nnz, 256), 256, 0, s>>>(state, nnz, wit);
        path_count_kernel<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(row_ptr, n, wit, kept);
        st = check_launch("onng_adjust_path_literal: count");
        if (st)
            return st;
    } else if (n > 0) {
        ONNG_CUDA_TRY(cudaMemsetAsync(kept, 0, sizeof(int64_t) * n, s), "adjust_path_literal: clear");
    }
    st = exclusive_scan(kept, row_ptr_out, n, scan_ws, scan_workspace_bytes(nn + 1), s);
    if (st)
        return st;
    if (n > 0 && nnz > 0) {
        path_compact_kernel<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(row_ptr, col, len, n, wit, row_ptr_out,
                                                                           col_out, len_out, nullptr);
        st = check_launch("onng_adjust_path_literal: compact");
        if (st)
            return st;
    }
    if (nnz_host) {
        ONNG_CUDA_TRY(cudaMemcpyAsync(nnz_host, row_ptr_out + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s),
                      "adjust_path_literal: nnz");
        ONNG_CUDA_TRY(cudaStreamSynchronize(s), "adjust_path_literal: sync");
    }
    return ONNG_OK;
}

// ------------------------------------------------------------------ path ABI

extern "C" size_t onng_adjust_path_workspace_bytes(int64_t n, int64_t nnz)
{
    WsCarver c(nullptr);
    c.take<int>((size_t)std::max<int64_t>(nnz, 1));        // witness positions
    c.take<int64_t>((size_t)std::max<int64_t>(n, 1));      // kept counts / long rows
    c.take<int64_t>((size_t)std::max<int64_t>(n, 1));
    c.take<int>(64);
    c.take<char>(scan_workspace_bytes(std::max<int64_t>(n, 1)));
    return c.used;
}

extern "C" int onng_adjust_path(const int64_t *row_ptr, const int32_t *col, const float *len, int64_t n,
                                int64_t *row_ptr_out, int32_t *col_out, float *len_out, int64_t *nnz_host,
                                int32_t *removed_by, void *ws, size_t ws_bytes, onng_stream_t stream)
{
    ONNG_RANGE("onng_adjust_path");
    ONNG_REQUIRE(n >= 0 && n <= INT32_MAX, ONNG_E_INVAL, "onng_adjust_path: bad n");
    ONNG_REQUIRE(row_ptr && row_ptr_out, ONNG_E_INVAL, "onng_adjust_path: NULL row_ptr");
    cudaStream_t s = to_cuda(stream);
    int64_t nnz = 0;
    ONNG_CUDA_TRY(cudaMemcpyAsync(&nnz, row_ptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s), "adjust_path: nnz");
    ONNG_CUDA_TRY(cudaStreamSynchronize(s), "adjust_path: sync");
    const size_t need = onng_adjust_path_workspace_bytes(n, nnz);
    ONNG_REQUIRE(ws && ws_bytes >= need, ONNG_E_WORKSPACE, "onng_adjust_path: workspace %zu < %zu bytes", ws_bytes,
                 need);
    ONNG_REQUIRE(nnz == 0 || (col && len && col_out && len_out), ONNG_E_INVAL, "onng_adjust_path: NULL arrays");
    WsCarver c(ws);
    int *wit = c.take<int>((size_t)std::max<int64_t>(nnz, 1));
    int64_t *kept = c.take<int64_t>((size_t)std::max<int64_t>(n, 1));
    int64_t *big = c.take<int64_t>((size_t)std::max<int64_t>(n, 1));
    int *n_big = c.take<int>(64);
    char *scan_ws = c.take<char>(scan_workspace_bytes(std::max<int64_t>(n, 1)));
    int st;
    if (n > 0) {
        ONNG_CUDA_TRY(cudaMemsetAsync(n_big, 0, 2 * sizeof(int), s), "adjust_path: clear");
        int per_sm = 0;
        ONNG_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, path_small_kernel, kPathWarps * 32, 0),
                      "adjust_path: occupancy");
        const int64_t resident = (int64_t)num_sms() * std::max(per_sm, 1);
        const int64_t ctas = std::min<int64_t>((n + kPathWarps - 1) / kPathWarps, resident);
        path_small_kernel<<<(unsigned)ctas, kPathWarps * 32, 0, s>>>(row_ptr, col, len, n, wit, big, n_big);
        // longer rows, of which nnz edges hold only so many: the kernels read the counts of
        // listed rows on the device (two launches that find none cost a small graph 9 us)
        if (nnz > kPathSmall)
            path_mid_kernel<<<(unsigned)std::min<int64_t>(num_sms() * 8, nnz / (kPathSmall + 1)), 256, 0, s>>>(
                row_ptr, col, len, wit, big, n_big);
        if (nnz > kPathMid) {
            ONNG_CUDA_TRY(cudaFuncSetAttribute(reinterpret_cast<const void *>(path_long_kernel),
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PathLong)),
                          "adjust_path: smem attribute");
            path_long_kernel<<<num_sms(), 1024, sizeof(PathLong), s>>>(row_ptr, col, len, n, wit, big, n_big);
        }
        st = check_launch("onng_adjust_path: mark");
        if (st)
            return st;
        path_count_kernel<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(row_ptr, n, wit, kept);
        st = check_launch("onng_adjust_path: count");
        if (st)
            return st;
    }
    st = exclusive_scan(kept, row_ptr_out, n, scan_ws, scan_workspace_bytes(std::max<int64_t>(n, 1)), s);
    if (st)
        return st;
    if (n > 0) {
        path_compact_kernel<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(row_ptr, col, len, n, wit, row_ptr_out,
                                                                           col_out, len_out, removed_by);
        st = check_launch("onng_adjust_path: compact");
        if (st)
            return st;
    }
    if (nnz_host) {
        ONNG_CUDA_TRY(cudaMemcpyAsync(nnz_host, row_ptr_out + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s),
                      "adjust_path: nnz");
        ONNG_CUDA_TRY(cudaStreamSynchronize(s), "adjust_path: sync");
    }
    return ONNG_OK;
}
