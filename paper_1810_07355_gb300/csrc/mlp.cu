// The per-query parameter predictor: a 16 -> 64 -> 64 -> 2 network with ReLU
// after both hidden layers, trained on the GPU in float32 and evaluated in
// bfloat16.  The paper's counterpart is the fixed policy of Eq. 1 (e_p as a
// function of eps); here the network maps features of a query's first hops to
// (log(eps + 0.01), log e_s).
//
// Parameters are one flat float32 vector: W1[64][16], b1[64], W2[64][64],
// b2[64], W3[2][64], b3[2] (5,378 values).  Loss: batch mean of
// 0.5 * sum_o (y_o - t_o)^2.
//
// One warp evaluates one sample: lane j owns hidden units j and j + 32.  The
// weights sit in shared memory transposed (input-major), so the 32 lanes read
// 32 consecutive words.  Gradients are accumulated in shared memory with
// atomics and written (or added) to global memory once per CTA.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace onng {
namespace {

constexpr int I = 16, H = 64, O = 2;
constexpr int NP = H * I + H + H * H + H + O * H + O;  // 5378
constexpr int kMlpWarps = 8;
constexpr unsigned FULL = 0xffffffffu;

// offsets in the flat (row-major, output-major) parameter vector
constexpr int oW1 = 0, ob1 = oW1 + H * I, oW2 = ob1 + H, ob2 = oW2 + H * H, oW3 = ob2 + H, ob3 = oW3 + O * H;

// Shared-memory image of the parameters, input-major for the weight matrices.
struct MlpShared {
    float w1t[I * H];  // [i][u]
    float b1[H];
    float w2t[H * H];  // [i][u]
    float w2[H * H];   // [u][i], read by the backward pass
    float b2[H];
    float w3[O * H];   // [o][u]
    float b3[O];
};

__device__ void load_params(MlpShared &s, const float *__restrict__ P)
{
    for (int e = threadIdx.x; e < H * I; e += blockDim.x) {
        const int u = e / I, i = e % I;
        s.w1t[i * H + u] = P[oW1 + e];
    }
    for (int e = threadIdx.x; e < H * H; e += blockDim.x) {
        const int u = e / H, i = e % H;
        s.w2t[i * H + u] = P[oW2 + e];
        s.w2[e] = P[oW2 + e];
    }
    for (int e = threadIdx.x; e < H; e += blockDim.x) {
        s.b1[e] = P[ob1 + e];
        s.b2[e] = P[ob2 + e];
    }
    for (int e = threadIdx.x; e < O * H; e += blockDim.x)
        s.w3[e] = P[oW3 + e];
    if (threadIdx.x < O)
        s.b3[threadIdx.x] = P[ob3 + threadIdx.x];
}

// Writes (or adds) a shared gradient image back to the flat layout.
__device__ void store_grad(const MlpShared &g, float *__restrict__ G, bool add)
{
    for (int e = threadIdx.x; e < NP; e += blockDim.x) {
        float v;
        if (e < ob1) {
            const int u = e / I, i = e % I;
            v = g.w1t[i * H + u];
        } else if (e < oW2) {
            v = g.b1[e - ob1];
        } else if (e < ob2) {
            const int u = (e - oW2) / H, i = (e - oW2) % H;
            v = g.w2t[i * H + u];
        } else if (e < oW3) {
            v = g.b2[e - ob2];
        } else if (e < ob3) {
            v = g.w3[e - oW3];
        } else {
            v = g.b3[e - ob3];
        }
        if (add)
            atomicAdd(&G[e], v);
        else
            G[e] = v;
    }
}

__device__ void zero_shared(MlpShared &g)
{
    float *f = reinterpret_cast<float *>(&g);
    for (int e = threadIdx.x; e < (int)(sizeof(MlpShared) / sizeof(float)); e += blockDim.x)
        f[e] = 0.f;
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1)
        v += __shfl_xor_sync(FULL, v, off);
    return v;
}

// Forward pass of one sample by one warp; returns y in every lane.  h1 (64
// floats of per-warp scratch) receives the first hidden layer.
__device__ void forward_warp(const MlpShared &s, const float *x, float *h1, int lane, float (&a1)[2], float (&a2)[2],
                             float (&h2)[2], float (&y)[O])
{
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int u = lane + 32 * r;
        float acc = s.b1[u];
#pragma unroll
        for (int i = 0; i < I; ++i)
            acc = fmaf(s.w1t[i * H + u], x[i], acc);
        a1[r] = acc;
        h1[u] = fmaxf(acc, 0.f);
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int u = lane + 32 * r;
        float acc = s.b2[u];
#pragma unroll 8
        for (int i = 0; i < H; ++i)
            acc = fmaf(s.w2t[i * H + u], h1[i], acc);
        a2[r] = acc;
        h2[r] = fmaxf(acc, 0.f);
    }
#pragma unroll
    for (int o = 0; o < O; ++o) {
        float p = s.w3[o * H + lane] * h2[0] + s.w3[o * H + lane + 32] * h2[1];
        y[o] = warp_sum(p) + s.b3[o];
    }
}

// Forward and backward of one sample; adds scale * dLoss/dParams into g (shared).
__device__ float fwd_bwd_warp(const MlpShared &s, MlpShared &g, const float *x, const float *t, float scale, float *h1,
                              float *da2s, int lane)
{
    float a1[2], a2[2], h2[2], y[O];
    forward_warp(s, x, h1, lane, a1, a2, h2, y);
    float dy[O], loss = 0.f;
#pragma unroll
    for (int o = 0; o < O; ++o) {
        const float e = y[o] - t[o];
        loss += 0.5f * e * e;
        dy[o] = e * scale;
    }
    if (lane < O)
        atomicAdd(&g.b3[lane], dy[lane]);
    float da2[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int u = lane + 32 * r;
        float dh2 = 0.f;
#pragma unroll
        for (int o = 0; o < O; ++o) {
            atomicAdd(&g.w3[o * H + u], dy[o] * h2[r]);
            dh2 = fmaf(s.w3[o * H + u], dy[o], dh2);
        }
        da2[r] = a2[r] > 0.f ? dh2 : 0.f;
        atomicAdd(&g.b2[u], da2[r]);
        da2s[u] = da2[r];
    }
    // gW2[u][i] += da2[u] * h1[i]  (input-major image: w2t[i][u])
#pragma unroll 8
    for (int i = 0; i < H; ++i) {
        const float hi = h1[i];
        atomicAdd(&g.w2t[i * H + lane], da2[0] * hi);
        atomicAdd(&g.w2t[i * H + lane + 32], da2[1] * hi);
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int u = lane + 32 * r;  // first-layer unit
        float dh1 = 0.f;
#pragma unroll 8
        for (int j = 0; j < H; ++j)
            dh1 = fmaf(s.w2[j * H + u], da2s[j], dh1);
        const float da1 = a1[r] > 0.f ? dh1 : 0.f;
        atomicAdd(&g.b1[u], da1);
#pragma unroll
        for (int i = 0; i < I; ++i)
            atomicAdd(&g.w1t[i * H + u], da1 * x[i]);
    }
    __syncwarp();
    return loss;
}

// Loss and gradient over a batch: every CTA accumulates its samples in shared
// memory and adds them to G (which the host zeroes first).
__global__ void __launch_bounds__(kMlpWarps * 32)
    mlp_loss_grad_kernel(const float *__restrict__ P, const float *__restrict__ X, const float *__restrict__ T,
                         int64_t B, float *__restrict__ G, float *__restrict__ loss_out)
{
    extern __shared__ __align__(16) unsigned char raw[];
    MlpShared &s = *reinterpret_cast<MlpShared *>(raw);
    MlpShared &g = *reinterpret_cast<MlpShared *>(raw + sizeof(MlpShared));
    float *scratch = reinterpret_cast<float *>(raw + 2 * sizeof(MlpShared));
    __shared__ float s_loss;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    load_params(s, P);
    zero_shared(g);
    if (threadIdx.x == 0)
        s_loss = 0.f;
    __syncthreads();
    float *h1 = scratch + warp * 2 * H;
    float *da2s = h1 + H;
    const float scale = 1.f / (float)B;
    float lsum = 0.f;
    for (int64_t b = (int64_t)blockIdx.x * kMlpWarps + warp; b < B; b += (int64_t)gridDim.x * kMlpWarps) {
        float x[I], t[O];
#pragma unroll
        for (int i = 0; i < I; ++i)
            x[i] = X[b * I + i];
        t[0] = T[b * O];
        t[1] = T[b * O + 1];
        lsum += fwd_bwd_warp(s, g, x, t, scale, h1, da2s, lane);
    }
    if (lane == 0)
        atomicAdd(&s_loss, lsum);
    __syncthreads();
    store_grad(g, G, true);
    if (threadIdx.x == 0)
        atomicAdd(loss_out, s_loss * scale);
}

__global__ void __launch_bounds__(kMlpWarps * 32)
    mlp_forward_kernel(const float *__restrict__ P, const float *__restrict__ X, int64_t B, float *__restrict__ Y)
{
    extern __shared__ __align__(16) unsigned char raw[];
    MlpShared &s = *reinterpret_cast<MlpShared *>(raw);
    float *scratch = reinterpret_cast<float *>(raw + sizeof(MlpShared));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    load_params(s, P);
    __syncthreads();
    float *h1 = scratch + warp * H;
    for (int64_t b = (int64_t)blockIdx.x * kMlpWarps + warp; b < B; b += (int64_t)gridDim.x * kMlpWarps) {
        float x[I];
#pragma unroll
        for (int i = 0; i < I; ++i)
            x[i] = X[b * I + i];
        float a1[2], a2[2], h2[2], y[O];
        forward_warp(s, x, h1, lane, a1, a2, h2, y);
        if (lane < O)
            Y[b * O + lane] = y[lane];
        __syncwarp();
    }
}

// Adam (Kingma & Ba 2015) on the flat vectors, step count t >= 1.  The roundings are
// written out (the decayed moment enters with a fused multiply-add), so that the one
// step and the training run, which both call this, take the same ones.
__device__ __forceinline__ void adam1(float &p, float g, float &m, float &v, float lr, float b1, float b2, float eps,
                                      float c1, float c2)
{
    m = fmaf(b1, m, __fmul_rn(1.f - b1, g));
    v = fmaf(b2, v, __fmul_rn(__fmul_rn(1.f - b2, g), g));
    p -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

__global__ void mlp_adam_kernel(float *__restrict__ P, const float *__restrict__ G, float *__restrict__ M,
                                float *__restrict__ Vv, int64_t t, float lr, float b1, float b2, float eps)
{
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < NP; e += gridDim.x * blockDim.x)
        adam1(P[e], G[e], M[e], Vv[e], lr, b1, b2, eps, c1, c2);
}

// Whole training run in one CTA, as batched small matrix products in shared
// memory (no atomics but the loss): per step, for a mini-batch of B <= 128 consecutive
// rows (wrapping around the set) the forward pass keeps h1 = relu(A1) and h2 = relu(A2)
// (their signs decide relu' as well); the backward pass forms dA2, the gradients of W3
// and W2, then dA1 and the gradients of W1; Adam updates the parameters.
//
// The steps depend on each other, so one SM works alone; what bounds it is its float32
// pipe (1.9 M multiply-adds a step, 7.4 us at 128 per cycle) and the chains between its
// barriers.  One result per thread read two shared values per multiply-add, and a
// shared-memory float atomic per sample for the loss queued: 78.5 us a step of 128 rows;
// 19.8 us as it is now.  Every
// product is a register tile of 4 x 4 results per thread with 16-byte reads, over
// arrays that hold a feature's samples in a row: the forward products and dA1 read 4
// weights and 4 samples per term, the weight gradients 4 samples of 4 + 4 features per
// 4 terms.  Rows are 132 floats, so 8 neighbouring rows (or a row's 8 quads) lie in
// distinct banks, and a warp's tiles are laid out along them.  Each result is still one
// chain of multiply-adds in the order of its sum.  The parameters and their moments
// stay in registers for the whole run.
constexpr int kTrainMaxB = 128;
constexpr int kTrainThreads = 512;
constexpr int kTrainPer = (NP + kTrainThreads - 1) / kTrainThreads;  // parameters per thread
constexpr int kTrainX = kTrainMaxB * I / kTrainThreads;              // inputs fetched per thread
constexpr int kTrainRow = kTrainMaxB + 4;

struct __align__(16) TrainShared {
    float G[NP + 2];
    float w1t[I * H];          // [i][u]
    float w2t[H * H];          // [i][u]
    float w2[H * H];           // [u][i]
    float xt[I][kTrainRow];    // [i][b]; samples past the batch are zero
    float h1[H][kTrainRow];    // [i][b]: relu(A1)
    float h2[H][kTrainRow];    // [u][b]: relu(A2)
    float da2[H][kTrainRow];   // [u][b]
    float da1[H][kTrainRow];   // [i][b]
    float dy[O][kTrainRow];    // [o][b]
    float t[kTrainMaxB * O];
    float b1[H], b2[H], w3[O * H], b3[O];
    float loss;
};

__device__ __forceinline__ float4 lds4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// acc[i][j] += sum over k = 0 .. K-1, in order, of a[k][i] b[k][j]: 4 + 4 values of rows
// lda and ldb apart
__device__ __forceinline__ void tile_rows(float (&acc)[4][4], const float *a, int lda, const float *b, int ldb, int K)
{
#pragma unroll 8
    for (int k = 0; k < K; ++k) {
        const float4 x = lds4(a + k * lda), y = lds4(b + k * ldb);
        const float xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                acc[i][j] = fmaf(xs[i], ys[j], acc[i][j]);
    }
}

// acc[i][j] += sum over b = 0 .. B-1, in order, of rows a + i sa and c + j sc
template <int NI, int NJ>
__device__ __forceinline__ void tile_dots(float (&acc)[NI][NJ], const float *a, int sa, const float *c, int sc, int B)
{
    int b = 0;
#pragma unroll 2
    for (; b + 4 <= B; b += 4) {
        float4 x[NI], y[NJ];
#pragma unroll
        for (int i = 0; i < NI; ++i)
            x[i] = lds4(a + i * sa + b);
#pragma unroll
        for (int j = 0; j < NJ; ++j)
            y[j] = lds4(c + j * sc + b);
#pragma unroll
        for (int i = 0; i < NI; ++i)
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                acc[i][j] = fmaf(x[i].x, y[j].x, acc[i][j]);
                acc[i][j] = fmaf(x[i].y, y[j].y, acc[i][j]);
                acc[i][j] = fmaf(x[i].z, y[j].z, acc[i][j]);
                acc[i][j] = fmaf(x[i].w, y[j].w, acc[i][j]);
            }
    }
    for (; b < B; ++b)
#pragma unroll
        for (int i = 0; i < NI; ++i)
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                acc[i][j] = fmaf(a[i * sa + b], c[j * sc + b], acc[i][j]);
}

// sum over b = 0 .. B-1, in order, of a row
__device__ __forceinline__ float row_sum(const float *a, int B)
{
    float acc = 0.f;
    int b = 0;
#pragma unroll 4
    for (; b + 4 <= B; b += 4) {
        const float4 x = lds4(a + b);
        acc += x.x;
        acc += x.y;
        acc += x.z;
        acc += x.w;
    }
    for (; b < B; ++b)
        acc += a[b];
    return acc;
}

// where the forward and backward products read parameter e
__device__ __forceinline__ void train_store(TrainShared &s, int e, float p)
{
    if (e < ob1) {
        s.w1t[(e % I) * H + e / I] = p;
    } else if (e < oW2) {
        s.b1[e - ob1] = p;
    } else if (e < ob2) {
        const int w = e - oW2;
        s.w2t[(w % H) * H + w / H] = p;
        s.w2[w] = p;
    } else if (e < oW3) {
        s.b2[e - ob2] = p;
    } else if (e < ob3) {
        s.w3[e - oW3] = p;
    } else {
        s.b3[e - ob3] = p;
    }
}

__global__ void __launch_bounds__(kTrainThreads, 1)
    mlp_train_kernel(float *__restrict__ Pg, float *__restrict__ M, float *__restrict__ Vv,
                     const float *__restrict__ X, const float *__restrict__ T, int64_t N, int B, int64_t steps,
                     int64_t t0, float lr, float b1, float b2, float eps, float *__restrict__ loss_out)
{
    extern __shared__ __align__(16) unsigned char raw[];
    TrainShared &s = *reinterpret_cast<TrainShared *>(raw);
    const int tid = threadIdx.x;
    // 4 x 4 tiles of the products over features x samples: a warp takes 4 feature quads
    // x 8 sample quads; tiles wholly past the batch are skipped
    const int tu = (((tid >> 3) & 3) | (tid >> 7) << 2) * 4, tb = ((tid & 7) | ((tid >> 5) & 3) << 3) * 4;
    const bool tile = tb < B;
    float p[kTrainPer], m[kTrainPer], v[kTrainPer], xn[kTrainX], tn = 0.f;
#pragma unroll
    for (int r = 0; r < kTrainPer; ++r) {
        const int e = tid + r * kTrainThreads;
        p[r] = e < NP ? Pg[e] : 0.f;
        m[r] = e < NP ? M[e] : 0.f;
        v[r] = e < NP ? Vv[e] : 0.f;
        if (e < NP)
            train_store(s, e, p[r]);
    }
    // the next step's rows are in flight during the present one
    auto fetch = [&](int64_t st) {
        const int64_t first = (st * B) % N;
#pragma unroll
        for (int r = 0; r < kTrainX; ++r) {
            const int e = tid + r * kTrainThreads;
            xn[r] = e < B * I ? X[((first + e / I) % N) * I + e % I] : 0.f;
        }
        if (tid < B * O)
            tn = T[((first + tid / O) % N) * O + tid % O];
    };
    const float invB = 1.f / (float)B;
    fetch(0);
    for (int64_t st = 0; st < steps; ++st) {
#pragma unroll
        for (int r = 0; r < kTrainX; ++r) {
            const int e = tid + r * kTrainThreads;
            s.xt[e % I][e / I] = xn[r];
        }
        if (tid < B * O)
            s.t[tid] = tn;
        if (tid == 0)
            s.loss = 0.f;
        if (st + 1 < steps)
            fetch(st + 1);
        __syncthreads();
        // A1[u][b] = b1[u] + sum_i W1[u][i] x[b][i], then A2 from h1 in the same way
        if (tile) {
            float acc[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    acc[i][j] = s.b1[tu + i];
            tile_rows(acc, s.w1t + tu, H, &s.xt[0][tb], kTrainRow, I);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                *reinterpret_cast<float4 *>(&s.h1[tu + i][tb]) = make_float4(
                    fmaxf(acc[i][0], 0.f), fmaxf(acc[i][1], 0.f), fmaxf(acc[i][2], 0.f), fmaxf(acc[i][3], 0.f));
        }
        __syncthreads();
        if (tile) {
            float acc[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    acc[i][j] = s.b2[tu + i];
            tile_rows(acc, s.w2t + tu, H, &s.h1[0][tb], kTrainRow, H);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                *reinterpret_cast<float4 *>(&s.h2[tu + i][tb]) = make_float4(
                    fmaxf(acc[i][0], 0.f), fmaxf(acc[i][1], 0.f), fmaxf(acc[i][2], 0.f), fmaxf(acc[i][3], 0.f));
        }
        __syncthreads();
        // y[b][o] (each lane starts its sum at its own unit), dY = (y - t) / B, loss
        float loss = 0.f;
        if (tid < B * O) {
            const int b = tid / O, o = tid % O;
            float acc = s.b3[o];
#pragma unroll 16
            for (int j = 0; j < H; ++j) {
                const int u = (j + (tid & 31)) & (H - 1);
                acc = fmaf(s.w3[o * H + u], s.h2[u][b], acc);
            }
            const float err = acc - s.t[tid];
            s.dy[o][b] = err * invB;
            loss = 0.5f * err * err * invB;
        }
        if (loss_out && tid < 2 * kTrainMaxB) {
            loss = warp_sum(loss);  // (a shared-memory float atomic per sample queued 256 deep)
            if ((tid & 31) == 0)
                atomicAdd(&s.loss, loss);
        }
        __syncthreads();
        // dA2[u][b]
        if (tile) {
            const float4 d0 = lds4(&s.dy[0][tb]), d1 = lds4(&s.dy[1][tb]);
            const float dy0[4] = {d0.x, d0.y, d0.z, d0.w}, dy1[4] = {d1.x, d1.y, d1.z, d1.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int u = tu + i;
                const float4 h = lds4(&s.h2[u][tb]);
                const float hs[4] = {h.x, h.y, h.z, h.w};
                float d[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float g = s.w3[u] * dy0[j] + s.w3[H + u] * dy1[j];
                    d[j] = hs[j] > 0.f ? g : 0.f;
                }
                *reinterpret_cast<float4 *>(&s.da2[u][tb]) = make_float4(d[0], d[1], d[2], d[3]);
            }
        }
        __syncthreads();
        // the first half of the threads: gW2[u][i] = sum_b dA2[u][b] h1[i][b]; the other
        // half: dA1[i][b] = relu'(A1) sum_u W2[u][i] dA2[u][b], then gW3, gb2 and gb3
        if (tid < 256) {
            // rows u, u + 8, u + 16, u + 24 of dA2 and i, i + 8, ... of h1
            const int u = ((tid >> 3) & 7) | (tid >> 6 & 1) << 5, i0 = (tid & 7) | (tid >> 7) << 5;
            float acc[4][4] = {};
            tile_dots<4, 4>(acc, s.da2[u], 8 * kTrainRow, s.h1[i0], 8 * kTrainRow, B);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    s.G[oW2 + (u + 8 * i) * H + i0 + 8 * j] = acc[i][j];
        } else {
            for (int e = tid - 256; e < 512; e += 256) {
                const int i0 = (((e >> 3) & 3) | (e >> 7) << 2) * 4, b = ((e & 7) | ((e >> 5) & 3) << 3) * 4;
                if (b >= B)
                    continue;
                float acc[4][4] = {};
                tile_rows(acc, s.w2 + i0, H, &s.da2[0][b], kTrainRow, H);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 h = lds4(&s.h1[i0 + i][b]);
                    *reinterpret_cast<float4 *>(&s.da1[i0 + i][b]) =
                        make_float4(h.x > 0.f ? acc[i][0] : 0.f, h.y > 0.f ? acc[i][1] : 0.f,
                                    h.z > 0.f ? acc[i][2] : 0.f, h.w > 0.f ? acc[i][3] : 0.f);
                }
            }
            const int w = tid - 256;
            if (w < O * H) {
                float acc[1][1] = {};
                tile_dots<1, 1>(acc, s.dy[w / H], 0, s.h2[w % H], 0, B);
                s.G[oW3 + w] = acc[0][0];
            } else if (w < O * H + H) {
                s.G[ob2 + w - O * H] = row_sum(s.da2[w - O * H], B);
            } else if (w < O * H + H + O) {
                s.G[ob3 + w - O * H - H] = row_sum(s.dy[w - O * H - H], B);
            }
        }
        __syncthreads();
        // gW1[u][i] = sum_b dA1[u][b] x[i][b]; gb1[u]
        if (tid < H * I / 4) {
            const int u = ((tid >> 3) & 7) | (tid >> 6 & 1) << 5 | (tid >> 7) << 3, i = tid & 7;
            // rows u, u + 16 of dA1 and i, i + 8 of x
            float acc[2][2] = {};
            tile_dots<2, 2>(acc, s.da1[u], 16 * kTrainRow, s.xt[i], 8 * kTrainRow, B);
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    s.G[oW1 + (u + 16 * a) * I + i + 8 * c] = acc[a][c];
        } else if (tid < H * I / 4 + H) {
            s.G[ob1 + tid - H * I / 4] = row_sum(s.da1[tid - H * I / 4], B);
        }
        __syncthreads();
        const int64_t t = t0 + st + 1;
        const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
#pragma unroll
        for (int r = 0; r < kTrainPer; ++r) {
            const int e = tid + r * kTrainThreads;
            if (e < NP) {
                adam1(p[r], s.G[e], m[r], v[r], lr, b1, b2, eps, c1, c2);
                train_store(s, e, p[r]);
            }
        }
        if (tid == 0 && loss_out)
            loss_out[st] = s.loss;
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < kTrainPer; ++r) {
        const int e = tid + r * kTrainThreads;
        if (e < NP) {
            Pg[e] = p[r];
            M[e] = m[r];
            Vv[e] = v[r];
        }
    }
}

// bfloat16 evaluation: weights and inputs rounded to bfloat16, float32
// accumulation; outputs mapped to eps = max(0, exp(y0) - 0.01) * alpha and
// e_s = clamp(round(exp(y1)), es_min, es_max).
__global__ void __launch_bounds__(kMlpWarps * 32)
    mlp_predict_kernel(const float *__restrict__ P, const float *__restrict__ X, int64_t B, float alpha, int es_min,
                       int es_max, float *__restrict__ eps_out, int32_t *__restrict__ es_out)
{
    extern __shared__ __align__(16) unsigned char raw[];
    MlpShared &s = *reinterpret_cast<MlpShared *>(raw);
    float *scratch = reinterpret_cast<float *>(raw + sizeof(MlpShared));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    load_params(s, P);
    __syncthreads();
    float *f = reinterpret_cast<float *>(&s);
    for (int e = threadIdx.x; e < (int)(sizeof(MlpShared) / sizeof(float)); e += blockDim.x)
        f[e] = __bfloat162float(__float2bfloat16_rn(f[e]));
    __syncthreads();
    float *h1 = scratch + warp * H;
    for (int64_t b = (int64_t)blockIdx.x * kMlpWarps + warp; b < B; b += (int64_t)gridDim.x * kMlpWarps) {
        float x[I];
#pragma unroll
        for (int i = 0; i < I; ++i)
            x[i] = __bfloat162float(__float2bfloat16_rn(X[b * I + i]));
        float a1[2], a2[2], h2[2], y[O];
        forward_warp(s, x, h1, lane, a1, a2, h2, y);
        if (lane == 0) {
            eps_out[b] = fmaxf(0.f, expf(y[0]) - 0.01f) * alpha;
            const float e = rintf(expf(fminf(y[1], 20.f)));
            es_out[b] = (int32_t)fminf(fmaxf(e, (float)es_min), (float)es_max);
        }
        __syncwarp();
    }
}

size_t shared_bytes(int copies, int scratch_per_warp) { return copies * sizeof(MlpShared) + kMlpWarps * scratch_per_warp * sizeof(float); }

int set_smem(const void *fn, size_t bytes)
{
    ONNG_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes), "mlp: smem attribute");
    return ONNG_OK;
}

int grid_for(int64_t B) { return (int)std::max<int64_t>(1, std::min<int64_t>((B + kMlpWarps - 1) / kMlpWarps, num_sms() * 2)); }

}  // namespace
}  // namespace onng

using namespace onng;

extern "C" int onng_mlp_nparam(void) { return NP; }

extern "C" int onng_mlp_forward(const float *P, const float *X, int64_t B, float *Y, onng_stream_t stream)
{
    ONNG_RANGE("onng_mlp_forward");
    ONNG_REQUIRE(B >= 0, ONNG_E_INVAL, "onng_mlp_forward: negative batch");
    if (B == 0)
        return ONNG_OK;
    ONNG_REQUIRE(P && X && Y, ONNG_E_INVAL, "onng_mlp_forward: NULL pointer");
    const size_t sm = shared_bytes(1, H);
    int st = set_smem(reinterpret_cast<const void *>(mlp_forward_kernel), sm);
    if (st)
        return st;
    mlp_forward_kernel<<<grid_for(B), kMlpWarps * 32, sm, to_cuda(stream)>>>(P, X, B, Y);
    return check_launch("onng_mlp_forward");
}

extern "C" int onng_mlp_loss_grad(const float *P, const float *X, const float *T, int64_t B, float *G, float *loss,
                                  onng_stream_t stream)
{
    ONNG_RANGE("onng_mlp_loss_grad");
    ONNG_REQUIRE(B >= 1, ONNG_E_INVAL, "onng_mlp_loss_grad: empty batch");
    ONNG_REQUIRE(P && X && T && G && loss, ONNG_E_INVAL, "onng_mlp_loss_grad: NULL pointer");
    cudaStream_t s = to_cuda(stream);
    ONNG_CUDA_TRY(cudaMemsetAsync(G, 0, sizeof(float) * NP, s), "onng_mlp_loss_grad: clear");
    ONNG_CUDA_TRY(cudaMemsetAsync(loss, 0, sizeof(float), s), "onng_mlp_loss_grad: clear");
    const size_t sm = shared_bytes(2, 2 * H);
    int st = set_smem(reinterpret_cast<const void *>(mlp_loss_grad_kernel), sm);
    if (st)
        return st;
    mlp_loss_grad_kernel<<<grid_for(B), kMlpWarps * 32, sm, s>>>(P, X, T, B, G, loss);
    return check_launch("onng_mlp_loss_grad");
}

extern "C" int onng_mlp_adam(float *P, const float *G, float *M, float *V, int64_t t, float lr, float beta1,
                             float beta2, float eps, onng_stream_t stream)
{
    ONNG_RANGE("onng_mlp_adam");
    ONNG_REQUIRE(t >= 1 && lr > 0.f, ONNG_E_INVAL, "onng_mlp_adam: bad step or rate");
    ONNG_REQUIRE(P && G && M && V, ONNG_E_INVAL, "onng_mlp_adam: NULL pointer");
    mlp_adam_kernel<<<(NP + 255) / 256, 256, 0, to_cuda(stream)>>>(P, G, M, V, t, lr, beta1, beta2, eps);
    return check_launch("onng_mlp_adam");
}

extern "C" int onng_mlp_train(float *P, float *M, float *V, const float *X, const float *T, int64_t N, int32_t batch,
                              int64_t steps, int64_t t0, float lr, float *G, float *losses, onng_stream_t stream)
{
    ONNG_RANGE("onng_mlp_train");
    (void)G;
    ONNG_REQUIRE(N >= 1 && batch >= 1 && steps >= 0 && t0 >= 0 && lr > 0.f, ONNG_E_INVAL, "onng_mlp_train: bad sizes");
    ONNG_REQUIRE(batch <= kTrainMaxB, ONNG_E_UNSUPPORTED, "onng_mlp_train: batch must be <= %d", kTrainMaxB);
    ONNG_REQUIRE(P && M && V && X && T, ONNG_E_INVAL, "onng_mlp_train: NULL pointer");
    if (steps == 0)
        return ONNG_OK;
    const size_t sm = sizeof(TrainShared);
    int st = set_smem(reinterpret_cast<const void *>(mlp_train_kernel), sm);
    if (st)
        return st;
    mlp_train_kernel<<<1, kTrainThreads, sm, to_cuda(stream)>>>(P, M, V, X, T, N, batch, steps, t0, lr, 0.9f, 0.999f,
                                                                1e-8f, losses);
    return check_launch("onng_mlp_train");
}

extern "C" int onng_mlp_predict(const float *P, const float *X, int64_t B, float alpha, int32_t es_min, int32_t es_max,
                                float *eps_out, int32_t *es_out, onng_stream_t stream)
{
    ONNG_RANGE("onng_mlp_predict");
    ONNG_REQUIRE(B >= 0 && es_min >= 1 && es_max >= es_min && alpha >= 0.f, ONNG_E_INVAL, "onng_mlp_predict: bad args");
    if (B == 0)
        return ONNG_OK;
    ONNG_REQUIRE(P && X && eps_out && es_out, ONNG_E_INVAL, "onng_mlp_predict: NULL pointer");
    const size_t sm = shared_bytes(1, H);
    int st = set_smem(reinterpret_cast<const void *>(mlp_predict_kernel), sm);
    if (st)
        return st;
    mlp_predict_kernel<<<grid_for(B), kMlpWarps * 32, sm, to_cuda(stream)>>>(P, X, B, alpha, es_min, es_max, eps_out,
                                                                            es_out);
    return check_launch("onng_mlp_predict");
}
