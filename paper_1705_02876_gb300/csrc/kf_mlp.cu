// Training and batched inference of the learned hit proposal (kf_mlp.cuh).
//
// Training runs in FP32 (master weights, gradients and Adam moments): each
// block takes tiles of 32 samples through the forward pass, the binary
// cross-entropy on the logits and the backward pass, and writes its part of
// the weight gradients; a second kernel sums the parts and applies Adam.
// Inference copies the weights to BF16 and scores on the tensor cores.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "kf.h"
#include "kf_api_internal.h"
#include "kf_mlp.cuh"

namespace kf {

constexpr uint32_t kTcWaitLimit = 1u << 24;  // mbarrier polls before a tcgen05 scoring wait gives up

struct MlpState {
    float *m = nullptr, *v = nullptr;                   // [kMlpParams] each: Adam's moments
    float *partial = nullptr;                           // [2 per SM][kPartLd]: the training blocks' gradients
    float *loss = nullptr;                              // one accumulator
    float *w32 = nullptr;                               // loaded weights, FP32
    __nv_bfloat16 *W1 = nullptr, *W2 = nullptr;         // loaded weights, BF16, transposed and padded
    unsigned *status = nullptr;                         // set by a tcgen05 scoring wait that expired
    uint32_t wait_limit = kTcWaitLimit;                 // polls of such a wait
    bool loaded = false;
};

void destroy_mlp_state(MlpState *s)
{
    if (!s) return;
    cudaFree(s->partial);
    cudaFree(s->m);
    cudaFree(s->v);
    cudaFree(s->loss);
    cudaFree(s->w32);
    cudaFree(s->W1);
    cudaFree(s->W2);
    cudaFree(s->status);
    delete s;
}

bool proposal_loaded(kf_context *ctx)
{
    MlpState *s = context_mlp_state(ctx);
    return s && s->loaded;
}

void proposal_weights(kf_context *ctx, const __nv_bfloat16 **W1, const __nv_bfloat16 **W2, const float **w32)
{
    MlpState *s = context_mlp_state(ctx);
    *W1 = s->W1;
    *W2 = s->W2;
    *w32 = s->w32;
}

namespace {

// Training step: mlp_grad_kernel (forward, loss, backward over tiles of 32
// rows, one partial gradient per block) and mlp_reduce_kernel (sums the
// partials, then Adam).  The step is a serial chain of two short launches:
// what bounds it is one tile's way through a block, and there shared-memory
// bandwidth (4,096 rows are 0.12 GFLOP, 1.5 us of the chip's FP32 rate).  A
// warp therefore owns 4 rows and a lane 2 units: per four inputs that is four
// 8-byte loads of W2, each word read once per warp, and four broadcast loads
// of the rows for 32 FMAs (12 shared-memory cycles; 1 row x 4 units with 16
// lanes across needs 20 for 16).  dW2 keeps 8 x 2 entries per thread.  Rows are
// padded to 68 floats so that the transposed reads of W2 are free of bank
// conflicts; H2, the logit and dH2's factors never leave registers; the
// partials go to memory as plain stores, so that the sum over blocks has a
// fixed order and the result is reproducible.  Both kernels are launched with
// programmatic dependent launch: a block gathers its rows while the previous
// step's Adam still runs.  One step of 4,096 rows: 60 us before (64-row tiles,
// two shared loads per FMA, 5,057 global atomics per block), 10 us now (an
// epoch of 262,147 rows: 3.88 ms before, 0.70 ms now).
constexpr int kTrainThreads = 256, kTrainRows = 32;
constexpr int kTrainLd = 68;                             // padded row of 64 floats
constexpr int kPartLd = (kMlpParams + 1 + 7) / 8 * 8;    // one block's partial: the gradient, then the loss

struct TrainSmem {
    float W2[kMlpHid][kTrainLd];
    float H1[kTrainRows][kTrainLd], dH2[kTrainRows][kTrainLd], dH1[kTrainRows][kTrainLd];
    float W1[kMlpIn][kMlpHid];
    float b1[kMlpHid], b2[kMlpHid], W3[kMlpHid];
    float X[kTrainRows][kMlpIn];
    float y[kTrainRows];
    float b3;
};

__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Samples [start, start + count) of the epoch's order, sample = (j P + off) mod n
// (P < n).
__global__ void __launch_bounds__(kTrainThreads) mlp_grad_kernel(const float *w, const float *X, const float *y, int64_t n,
                                                                 int64_t start, int64_t count, int64_t P, int64_t off,
                                                                 float inv_batch, float *partial)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TrainSmem &s = *reinterpret_cast<TrainSmem *>(smem_raw);
    constexpr int W = kTrainThreads / 32, Q = kTrainRows / W;  // warps; rows per warp
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t tiles = (count + kTrainRows - 1) / kTrainRows;
    auto f2 = [](const float *p) { return *reinterpret_cast<const float2 *>(p); };
    auto f4 = [](const float *p) { return *reinterpret_cast<const float4 *>(p); };
    // row r of a tile: its sample is (the tile's first + r P) mod n
    auto gather = [&](int64_t tile) {
        const int64_t first = ((start + tile * kTrainRows) % n * P + off) % n;
        for (int i = tid; i < kTrainRows * kMlpIn; i += kTrainThreads) {
            const int r = i / kMlpIn, f = i - r * kMlpIn;
            const bool in = tile * kTrainRows + r < count;
            const int64_t row = (first + r * P) % n;
            s.X[r][f] = in ? X[row * kMlpIn + f] : 0.0f;
            if (f == 0) s.y[r] = in ? y[row] : 0.0f;
        }
    };
    gather(blockIdx.x);
    pdl_wait();  // the weights are the previous step's
    pdl_launch_dependents();
    {
        float t2[16], t1[3];  // all loads in flight together
#pragma unroll
        for (int i = 0; i < 16; ++i) t2[i] = w[kOffW2 + i * kTrainThreads + tid];
#pragma unroll
        for (int i = 0; i < 3; ++i) t1[i] = w[kOffW1 + i * kTrainThreads + tid];
        if (tid < kMlpHid) {
            s.b1[tid] = w[kOffB1 + tid];
            s.b2[tid] = w[kOffB2 + tid];
            s.W3[tid] = w[kOffW3 + tid];
        }
        if (tid == 0) s.b3 = w[kOffB3];
#pragma unroll
        for (int i = 0; i < 16; ++i) s.W2[(i * kTrainThreads + tid) >> 6][tid & 63] = t2[i];
#pragma unroll
        for (int i = 0; i < 3; ++i) s.W1[(i * kTrainThreads + tid) >> 6][tid & 63] = t1[i];
    }
    __syncthreads();
    const int r0 = warp * Q;
    float gW2[8][2] = {}, gW1[kMlpIn][2] = {}, gb1[2] = {}, gb2[2] = {}, gW3[2] = {}, gb3 = 0.0f, loss = 0.0f;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        if (tile != blockIdx.x) {
            __syncthreads();  // the previous tile is consumed
            gather(tile);
            __syncthreads();
        }
        {  // H1 = relu(X W1 + b1): rows r0.., units 2 lane, 2 lane + 1
            float a[Q][2];
            const float2 b = f2(&s.b1[2 * lane]);
#pragma unroll
            for (int q = 0; q < Q; ++q) a[q][0] = b.x, a[q][1] = b.y;
#pragma unroll
            for (int f = 0; f < kMlpIn; f += 4) {
                float4 x[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q) x[q] = f4(&s.X[r0 + q][f]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 ww = f2(&s.W1[f + i][2 * lane]);
#pragma unroll
                    for (int q = 0; q < Q; ++q) {
                        const float v = i == 0 ? x[q].x : i == 1 ? x[q].y : i == 2 ? x[q].z : x[q].w;
                        a[q][0] = fmaf(v, ww.x, a[q][0]);
                        a[q][1] = fmaf(v, ww.y, a[q][1]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < Q; ++q)
                *reinterpret_cast<float2 *>(&s.H1[r0 + q][2 * lane]) = make_float2(fmaxf(a[q][0], 0.0f), fmaxf(a[q][1], 0.0f));
        }
        __syncwarp();  // a warp reads only its own rows until dW2
        {  // H2 = relu(H1 W2 + b2), the logit, dL/dz and dH2 = dz W3^T on active units
            float a[Q][2];
            const float2 b = f2(&s.b2[2 * lane]), w3 = f2(&s.W3[2 * lane]);
#pragma unroll
            for (int q = 0; q < Q; ++q) a[q][0] = b.x, a[q][1] = b.y;
#pragma unroll 4
            for (int k = 0; k < kMlpHid; k += 4) {
                float4 h[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q) h[q] = f4(&s.H1[r0 + q][k]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 ww = f2(&s.W2[k + i][2 * lane]);
#pragma unroll
                    for (int q = 0; q < Q; ++q) {
                        const float v = i == 0 ? h[q].x : i == 1 ? h[q].y : i == 2 ? h[q].z : h[q].w;
                        a[q][0] = fmaf(v, ww.x, a[q][0]);
                        a[q][1] = fmaf(v, ww.y, a[q][1]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const float h0 = fmaxf(a[q][0], 0.0f), h1 = fmaxf(a[q][1], 0.0f);
                float z = fmaf(h0, w3.x, h1 * w3.y);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
                z += s.b3;
                float d = 0.0f;
                if (tile * kTrainRows + r0 + q < count) {
                    const float t = s.y[r0 + q];
                    if (lane == 0) loss += fmaxf(z, 0.0f) - z * t + log1pf(expf(-fabsf(z)));
                    d = (1.0f / (1.0f + expf(-z)) - t) * inv_batch;
                }
                const float d0 = h0 > 0.0f ? d * w3.x : 0.0f, d1 = h1 > 0.0f ? d * w3.y : 0.0f;
                gb2[0] += d0;
                gb2[1] += d1;
                gW3[0] = fmaf(h0, d, gW3[0]);
                gW3[1] = fmaf(h1, d, gW3[1]);
                if (lane == 0) gb3 += d;
                *reinterpret_cast<float2 *>(&s.dH2[r0 + q][2 * lane]) = make_float2(d0, d1);
            }
        }
        __syncwarp();
        {  // dH1 = dH2 W2^T on active units: inputs lane, lane + 32
            float a[Q][2] = {};
#pragma unroll 4
            for (int u = 0; u < kMlpHid; u += 4) {
                const float4 w0 = f4(&s.W2[lane][u]), w1 = f4(&s.W2[lane + 32][u]);
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const float4 d = f4(&s.dH2[r0 + q][u]);
                    a[q][0] = fmaf(d.x, w0.x, fmaf(d.y, w0.y, fmaf(d.z, w0.z, fmaf(d.w, w0.w, a[q][0]))));
                    a[q][1] = fmaf(d.x, w1.x, fmaf(d.y, w1.y, fmaf(d.z, w1.z, fmaf(d.w, w1.w, a[q][1]))));
                }
            }
#pragma unroll
            for (int q = 0; q < Q; ++q)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float v = s.H1[r0 + q][lane + 32 * j] > 0.0f ? a[q][j] : 0.0f;
                    s.dH1[r0 + q][lane + 32 * j] = v;
                    gb1[j] += v;
                }
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < Q; ++q) {  // dW1 += X^T dH1 over the warp's rows
            const float2 d = f2(&s.dH1[r0 + q][2 * lane]);
#pragma unroll
            for (int f = 0; f < kMlpIn; f += 4) {
                const float4 x = f4(&s.X[r0 + q][f]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float v = i == 0 ? x.x : i == 1 ? x.y : i == 2 ? x.z : x.w;
                    gW1[f + i][0] = fmaf(v, d.x, gW1[f + i][0]);
                    gW1[f + i][1] = fmaf(v, d.y, gW1[f + i][1]);
                }
            }
        }
        __syncthreads();
#pragma unroll 4
        for (int r = 0; r < kTrainRows; ++r) {  // dW2 += H1^T dH2: rows 8 warp.. of W2, columns 2 lane, 2 lane + 1
            const float4 ha = f4(&s.H1[r][8 * warp]), hb = f4(&s.H1[r][8 * warp + 4]);
            const float2 d = f2(&s.dH2[r][2 * lane]);
            const float h[8] = {ha.x, ha.y, ha.z, ha.w, hb.x, hb.y, hb.z, hb.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                gW2[i][0] = fmaf(h[i], d.x, gW2[i][0]);
                gW2[i][1] = fmaf(h[i], d.y, gW2[i][1]);
            }
        }
    }
    // the block's partial, every entry written once; what the warps hold for
    // their own rows is summed over the warps through shared memory
    float *out = partial + (int64_t)blockIdx.x * kPartLd;
#pragma unroll
    for (int i = 0; i < 8; ++i)
        *reinterpret_cast<float2 *>(out + kOffW2 + (8 * warp + i) * kMlpHid + 2 * lane) = make_float2(gW2[i][0], gW2[i][1]);
    __syncthreads();
    float *rW1 = &s.H1[0][0];  // [W][768]
    float *rb = &s.W2[0][0];   // [3][W][64]: b1, b2, W3; then [2][W]: b3, the loss
    static_assert(3 * sizeof(s.H1) >= W * kMlpIn * kMlpHid * sizeof(float) &&
                      sizeof(s.W2) >= (3 * W * kMlpHid + 2 * W) * sizeof(float),
                  "the reductions fit in the tile's shared memory");
#pragma unroll
    for (int f = 0; f < kMlpIn; ++f)
        *reinterpret_cast<float2 *>(rW1 + (warp * kMlpIn + f) * kMlpHid + 2 * lane) = make_float2(gW1[f][0], gW1[f][1]);
    rb[warp * kMlpHid + lane] = gb1[0];
    rb[warp * kMlpHid + lane + 32] = gb1[1];
    *reinterpret_cast<float2 *>(rb + (W + warp) * kMlpHid + 2 * lane) = make_float2(gb2[0], gb2[1]);
    *reinterpret_cast<float2 *>(rb + (2 * W + warp) * kMlpHid + 2 * lane) = make_float2(gW3[0], gW3[1]);
    if (lane == 0) {
        rb[3 * W * kMlpHid + warp] = gb3;
        rb[3 * W * kMlpHid + W + warp] = loss;
    }
    __syncthreads();
    for (int i = tid; i < kMlpIn * kMlpHid; i += kTrainThreads) {
        float a = 0.0f;
#pragma unroll
        for (int k = 0; k < W; ++k) a += rW1[k * kMlpIn * kMlpHid + i];
        out[kOffW1 + i] = a;
    }
    if (tid < 3 * kMlpHid + 2) {
        const int which = tid >> 6, u = tid & 63;  // which = 3: b3 (u = 0) and the loss (u = 1)
        const float *p = which < 3 ? rb + which * W * kMlpHid + u : rb + 3 * W * kMlpHid + u * W;
        const int ld = which < 3 ? kMlpHid : 1;
        float a = 0.0f;
#pragma unroll
        for (int k = 0; k < W; ++k) a += p[k * ld];
        out[which == 0 ? kOffB1 + u : which == 1 ? kOffB2 + u : which == 2 ? kOffW3 + u : u == 0 ? kOffB3 : kMlpParams] = a;
    }
}

// Sum the blocks' partials (32 entries per block, the partials spread over its
// 8 warps: 128-byte rows, up to 16 loads in flight per thread).  ADAM: update
// the weights (Kingma and Ba) and add the loss to *loss; else write the
// gradient and set *loss.
struct AdamArgs {
    float *w, *m, *v;
    int t;
    float lr, b1, b2, eps;
};
template <bool ADAM>
__global__ void __launch_bounds__(256) mlp_reduce_kernel(const float *partial, int blocks, float *grad, float *loss,
                                                         AdamArgs ad)
{
    __shared__ float part[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    pdl_wait();
    pdl_launch_dependents();
    float g = 0.0f;
    if (i <= kMlpParams) {
#pragma unroll 16
        for (int b = warp; b < blocks; b += 8) g += __ldcg(partial + (int64_t)b * kPartLd + i);
    }
    part[warp][lane] = g;
    __syncthreads();
    if (warp != 0 || i > kMlpParams) return;
#pragma unroll
    for (int k = 1; k < 8; ++k) g += part[k][lane];
    if (i == kMlpParams) {
        *loss = ADAM ? *loss + g : g;
        return;
    }
    if (!ADAM) {
        grad[i] = g;
        return;
    }
    const float mi = ad.b1 * ad.m[i] + (1.0f - ad.b1) * g;
    const float vi = ad.b2 * ad.v[i] + (1.0f - ad.b2) * g * g;
    ad.m[i] = mi;
    ad.v[i] = vi;
    const float mh = mi / (1.0f - powf(ad.b1, (float)ad.t)), vh = vi / (1.0f - powf(ad.b2, (float)ad.t));
    ad.w[i] -= ad.lr * mh / (sqrtf(vh) + ad.eps);
}

// FP32 master weights -> the network inference uses: W1 and W2 as the
// transposed, padded BF16 copies the tensor cores read, W3 rounded to BF16 in
// place in the FP32 copy (w32), the biases left in FP32.
__global__ void to_bf16_kernel(float *w32, __nv_bfloat16 *W1t, __nv_bfloat16 *W2t)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kW1Elems; i += gridDim.x * blockDim.x) {
        const int n = i / kW1Ld, k = i % kW1Ld;
        W1t[i] = __float2bfloat16(k < kMlpIn ? w32[kOffW1 + k * kMlpHid + n] : 0.0f);
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kW2Elems; i += gridDim.x * blockDim.x) {
        const int n = i / kW2Ld, k = i % kW2Ld;
        W2t[i] = __float2bfloat16(k < kMlpHid ? w32[kOffW2 + k * kMlpHid + n] : 0.0f);
    }
    __syncthreads();  // every W1/W2 read above precedes this block's W3 writes (disjoint ranges anyway)
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < kMlpHid; i += blockDim.x)
            w32[kOffW3 + i] = __bfloat162float(__float2bfloat16(w32[kOffW3 + i]));
}

constexpr int kScoreWarps = 4, kScoreLd = 12;
// kf_proposal_score's engine (KF_SCORE_AUTO), chosen by measurement on one
// GB300: mma.sync below this many rows (65,536 rows 9.3 against 10.6 us; the two
// meet near 80,000), tcgen05 from it on (131,072 rows 12.1 against 13.3 us,
// 163,840 12.3 and 16.4, 262,144 16.5 and 24.2, 2^24 512 and 1,145)
constexpr int64_t kScoreTcMinRows = 131072;

struct ScoreSmem {
    MlpSmemWeights w;
    float X[kScoreWarps][32 * kScoreLd];
};

// Each warp scores 32 rows at a time on the tensor cores (mma.sync, split
// activations).
__global__ void __launch_bounds__(32 * kScoreWarps) mlp_score_kernel(const __nv_bfloat16 *W1, const __nv_bfloat16 *W2,
                                                                     const float *w32, const float *X, int64_t n,
                                                                     float *logits)
{
    extern __shared__ __align__(128) unsigned char score_smem_raw[];
    ScoreSmem &s = *reinterpret_cast<ScoreSmem *>(score_smem_raw);
    mlp_load_weights(&s.w, W1, W2, w32);
    __syncthreads();
    const MlpWeightsRef mw{reinterpret_cast<const uint32_t *>(s.w.W1t), reinterpret_cast<const uint32_t *>(s.w.W2t),
                           s.w.b1, s.w.b2, s.w.W3, s.w.b3};
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *xs = s.X[warp];
    const int64_t n_chunks = (n + 31) / 32;
    for (int64_t ch = (int64_t)blockIdx.x * kScoreWarps + warp; ch < n_chunks; ch += (int64_t)gridDim.x * kScoreWarps) {
        const int64_t row = ch * 32 + lane;
#pragma unroll
        for (int i = 0; i < kMlpIn; ++i) xs[lane * kScoreLd + i] = row < n ? X[row * kMlpIn + i] : 0.0f;
        const float z = mlp_score_warp_split(mw, xs, kScoreLd);
        if (row < n) logits[row] = z;
    }
}

// ---------------------------------------------------------------------------
// The same scoring on the fifth-generation tensor cores (tcgen05): a CTA of
// kTcGroups groups of 128 threads, each with a 128-row tile of its own in hand.
// The weights are staged once per CTA in shared memory; per tile the rows'
// split inputs go to shared memory, one thread issues the layer-1 products (hi
// and lo parts into one TMEM accumulator, M = 128, N = 64, K = 16), the four
// warps read the accumulator back from TMEM (warp w owns TMEM lanes
// 32w..32w+31, thread t row t; the bias is in it), apply the ReLU, split the
// result and write it as the layer-2 A operand over the inputs; the layer-2
// products (4 K-steps x hi/lo) accumulate over the layer-1 columns, which the
// warps read back for the 64 -> 1 dot product.
//
// What bounds it is one tile's serial way (load, split, product, read, split,
// product, read: the issue slots are half idle), so tiles in flight count: with
// one set of columns and of operands per tile, and the weights shared by three
// tiles, an SM holds six (before: four, each with its own weights and two
// sets).  4,194,301 rows: 137 us, 158 with four (52 B a row would take 32 us at
// the copy bandwidth).  Of that time the tensor pipe works 29%, the load-store
// data pipe 55%, the ALU pipe (the splits) 54%, and 59% of the issue slots are used.
//
// Operands are K-major without swizzle, in core matrices of 8 rows x 16 bytes
// (8 BF16 values): element (r, k) of a tile with K columns is at byte
// ((r / 8) (K / 8) + k / 8) 128 + (r % 8) 16 + (k % 8) 2.  In the shared
// memory descriptor the leading-dimension offset is the distance between core
// matrices adjacent in K (128 B) and the stride-dimension offset the distance
// between 8-row groups ((K / 8) 128 B).

constexpr int kTcRows = 128, kTcGroups = 3;        // rows per tile; tiles of a CTA
constexpr int kTcThreads = kTcRows * kTcGroups;
constexpr int kTcCols = 256;                       // TMEM columns of a CTA (a power of two): 64 per tile
constexpr int kTcCtasPerSm = 2;                    // 2 x 256 = the SM's 512 TMEM columns

struct __align__(128) TcSmem {
    // per tile, the A operand's hi and lo parts: the first hidden layer (K =
    // 64), and before it, at the start, the inputs (K = 16: 12 used, 3 bias columns)
    uint8_t Ah[kTcGroups][kTcRows * 128], Al[kTcGroups][kTcRows * 128];
    uint8_t ones[kTcRows * 32];                       // (1, 1, 1, 0, ...) per row: K = 16
    uint8_t B1[kMlpHid * 32];                         // W1^T and b1's parts: N = 64 x K = 16
    uint8_t B2[kMlpHid * 128];                        // W2^T: N = 64 x K = 64
    uint8_t B2b[kMlpHid * 32];                        // b2's parts: N = 64 x K = 16 (3 used)
    float W3[kMlpHid], b3;
    unsigned long long mbar[kTcGroups];
    uint32_t taddr;
};

// A bias b as three BF16 parts whose sum is b exactly (8 significant bits
// each: FP32's 24), so that a product with 1.0 on the tensor cores adds b.
__device__ __forceinline__ void bf16_parts3(float b, __nv_bfloat16 p[3])
{
    p[0] = __float2bfloat16(b);
    const float r1 = b - __bfloat162float(p[0]);
    p[1] = __float2bfloat16(r1);
    p[2] = __float2bfloat16(r1 - __bfloat162float(p[1]));
}

__device__ __forceinline__ uint32_t core_offset(int r, int k, int K)
{
    return (uint32_t)(((r >> 3) * (K >> 3) + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// Shared memory matrix descriptor (tcgen05): start address, leading- and
// stride-dimension byte offsets (all >> 4), the fixed version bits 46..48 =
// 0b001, base offset 0, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(const void *p, uint32_t lbo, uint32_t sbo)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    return (uint64_t)((a >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), A
// and B BF16 (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at
// bits 17-22, M >> 4 at bits 24-28.
constexpr uint32_t kTcIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kMlpHid >> 3) << 17) |
                              ((uint32_t)(kTcRows >> 4) << 24);

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(kTcIdesc), "r"(accumulate));
}

__device__ __forceinline__ void tc_commit(unsigned long long *mbar)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(mbar);
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(a) : "memory");
}

// Wait for the mbarrier's phase `parity` to complete, polling at most `limit`
// times; false if it did not.
__device__ __forceinline__ bool mbar_wait(unsigned long long *mbar, uint32_t parity, uint32_t limit)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(mbar);
    for (uint32_t i = 0; i < limit; ++i) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// 16 consecutive FP32 columns of this thread's TMEM lane, without the wait
// (tmem_wait() before the values are used).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t r[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
// Barrier `id` of the group's 128 threads; whether `p` held for any of them.
__device__ __forceinline__ bool group_or(int id, bool p)
{
    uint32_t r;
    asm volatile(
        "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.or.pred q, %2, 128, p;\nselp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"((uint32_t)p), "r"(id)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void st_shared_v4(uint8_t *p, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    *reinterpret_cast<uint4 *>(p) = make_uint4(a, b, c, d);
}

// VEC: the rows start on 16-byte boundaries and are read as three float4.
// A warp one of whose waits for a product expires (`limit` polls) touches
// neither the operands, which the product may still read, nor the accumulator:
// it votes at the group's next barrier (if there is one) to end the group, and
// before the CTA gives its TMEM back it waits on that same phase, with
// kTcWaitLimit polls, for what is in flight.
template <bool VEC>
__global__ void __launch_bounds__(kTcThreads, kTcCtasPerSm) mlp_score_tc_kernel(const float *w32, const float *X,
                                                                                 int64_t n, float *logits,
                                                                                 unsigned *status, uint32_t limit)
{
    extern __shared__ __align__(1024) unsigned char tc_smem_raw[];
    TcSmem &s = *reinterpret_cast<TcSmem *>(tc_smem_raw);
    const int tid = threadIdx.x % kTcRows, group = threadIdx.x / kTcRows, warp = tid >> 5;
    // weights: W1^T with b1's parts as its K rows 12..14, W2^T, and b2's parts
    // (K rows 0..2 of B2b), in BF16, K-major core matrices
    for (int nn = threadIdx.x; nn < kMlpHid; nn += kTcThreads) {
        __nv_bfloat16 p1[3], p2[3];
        bf16_parts3(w32[kOffB1 + nn], p1);
        bf16_parts3(w32[kOffB2 + nn], p2);
        for (int k = 0; k < 16; ++k) {
            const __nv_bfloat16 v = k < kMlpIn ? __float2bfloat16(w32[kOffW1 + k * kMlpHid + nn])
                                    : k < kMlpIn + 3 ? p1[k - kMlpIn]
                                                     : __float2bfloat16(0.0f);
            *reinterpret_cast<__nv_bfloat16 *>(s.B1 + core_offset(nn, k, 16)) = v;
            *reinterpret_cast<__nv_bfloat16 *>(s.B2b + core_offset(nn, k, 16)) = k < 3 ? p2[k] : __float2bfloat16(0.0f);
        }
        s.W3[nn] = w32[kOffW3 + nn];
    }
    for (int i = threadIdx.x; i < kMlpHid * kMlpHid; i += kTcThreads) {
        const int nn = i & 63, k = i >> 6;
        *reinterpret_cast<__nv_bfloat16 *>(s.B2 + core_offset(nn, k, 64)) =
            __float2bfloat16(w32[kOffW2 + k * kMlpHid + nn]);
    }
    if (group == 0) {
        st_shared_v4(s.ones + core_offset(tid, 0, 16), 0x3F803F80u, 0x00003F80u, 0u, 0u);
        st_shared_v4(s.ones + core_offset(tid, 8, 16), 0u, 0u, 0u, 0u);
    }
    if (threadIdx.x == 0) {
        s.b3 = w32[kOffB3];
        for (int g = 0; g < kTcGroups; ++g) {
            const uint32_t mb = (uint32_t)__cvta_generic_to_shared(&s.mbar[g]);
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb));
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < 32) {
        const uint32_t a = (uint32_t)__cvta_generic_to_shared(&s.taddr);
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(a), "n"(kTcCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the staged weights, for the tensor cores
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s.taddr;
    const uint32_t d = tmem + group * kMlpHid;               // the tile's accumulator columns
    const uint32_t dl = d + ((uint32_t)(warp * 32) << 16);   // this warp's lanes of them
    uint8_t *Ah = s.Ah[group], *Al = s.Al[group];
    unsigned long long *mbar = &s.mbar[group];
    const float b3 = s.b3;
    uint32_t parity = 0;
    bool failed = false;
    const int64_t tiles = (n + kTcRows - 1) / kTcRows, step = (int64_t)gridDim.x * kTcGroups;
    // row `tid` of a tile's inputs; the next tile's are loaded while the
    // current tile's products run
    auto load_row = [&](int64_t tile, float f[kMlpIn]) {
        const int64_t row = tile * kTcRows + tid;
        const bool in = tile < tiles && row < n;
        if constexpr (VEC) {
#pragma unroll
            for (int i = 0; i < kMlpIn; i += 4) {
                const float4 v = in ? __ldcs(reinterpret_cast<const float4 *>(X + row * kMlpIn + i))
                                    : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                f[i] = v.x;
                f[i + 1] = v.y;
                f[i + 2] = v.z;
                f[i + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < kMlpIn; ++i) f[i] = in ? __ldcs(X + row * kMlpIn + i) : 0.0f;
        }
    };
    float fin[kMlpIn];
    int64_t tile = (int64_t)blockIdx.x * kTcGroups + group;
    load_row(tile, fin);
    for (; tile < tiles; tile += step) {
        const int64_t row = tile * kTcRows + tid;
        // inputs of row `tid` and three 1s (the bias columns), split into BF16
        // hi and lo (1 is exact: its lo part is 0)
        {
            uint32_t h[8], l[8];
#pragma unroll
            for (int i = 0; i < 6; ++i) split_bf16x2(fin[2 * i], fin[2 * i + 1], h[i], l[i]);
            h[6] = 0x3F803F80u;
            h[7] = 0x00003F80u;
            l[6] = l[7] = 0u;
#pragma unroll
            for (int kg = 0; kg < 2; ++kg) {
                st_shared_v4(Ah + core_offset(tid, kg * 8, 16), h[4 * kg], h[4 * kg + 1], h[4 * kg + 2], h[4 * kg + 3]);
                st_shared_v4(Al + core_offset(tid, kg * 8, 16), l[4 * kg], l[4 * kg + 1], l[4 * kg + 2], l[4 * kg + 3]);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        // the group's rows are written, and its reads of the last tile's columns done
        if ((failed = group_or(group + 1, false))) break;
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            tc_mma(d, smem_desc(Ah, 128, 256), smem_desc(s.B1, 128, 256), 0u);
            tc_mma(d, smem_desc(Al, 128, 256), smem_desc(s.B1, 128, 256), 1u);
            tc_commit(mbar);
        }
        load_row(tile + step, fin);
        failed = __any_sync(0xffffffffu, !mbar_wait(mbar, parity, limit));
        parity ^= 1u;
        if (failed) {
            group_or(group + 1, true);
            break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // layer 1 epilogue (the bias is in the accumulator): ReLU, split ->
        // layer-2 A operand (row tid), over the inputs, which are consumed
#pragma unroll
        for (int c0 = 0; c0 < kMlpHid; c0 += 16) {
            uint32_t a[16];
            tmem_ld16(dl + c0, a);
            tmem_wait();
            uint32_t hh[8], ll[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                split_bf16x2(fmaxf(__uint_as_float(a[2 * i]), 0.0f), fmaxf(__uint_as_float(a[2 * i + 1]), 0.0f), hh[i],
                             ll[i]);
#pragma unroll
            for (int kg = 0; kg < 2; ++kg) {
                st_shared_v4(Ah + core_offset(tid, c0 + kg * 8, 64), hh[4 * kg], hh[4 * kg + 1], hh[4 * kg + 2],
                             hh[4 * kg + 3]);
                st_shared_v4(Al + core_offset(tid, c0 + kg * 8, 64), ll[4 * kg], ll[4 * kg + 1], ll[4 * kg + 2],
                             ll[4 * kg + 3]);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        if ((failed = group_or(group + 1, false))) break;
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {  // K-step ks: core matrices 2ks, 2ks + 1 along K
                const uint64_t b = smem_desc(s.B2 + ks * 256, 128, 1024);
                tc_mma(d, smem_desc(Ah + ks * 256, 128, 1024), b, ks > 0 ? 1u : 0u);
                tc_mma(d, smem_desc(Al + ks * 256, 128, 1024), b, 1u);
            }
            tc_mma(d, smem_desc(s.ones, 128, 256), smem_desc(s.B2b, 128, 256), 1u);  // + b2
            tc_commit(mbar);
        }
        failed = __any_sync(0xffffffffu, !mbar_wait(mbar, parity, limit));
        parity ^= 1u;
        if (failed) {
            if (tile + step < tiles) group_or(group + 1, true);
            break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // layer 2 epilogue (the bias is in the accumulator): ReLU, the 64 -> 1
        // dot product
        float z = b3;
#pragma unroll
        for (int c0 = 0; c0 < kMlpHid; c0 += 32) {
            uint32_t a[32];
            tmem_ld16(dl + c0, a);
            tmem_ld16(dl + c0 + 16, a + 16);
            tmem_wait();
#pragma unroll
            for (int c = 0; c < 32; c += 4) {
                const float4 w = *reinterpret_cast<const float4 *>(s.W3 + c0 + c);
                z = fmaf(w.x, fmaxf(__uint_as_float(a[c]), 0.0f), z);
                z = fmaf(w.y, fmaxf(__uint_as_float(a[c + 1]), 0.0f), z);
                z = fmaf(w.z, fmaxf(__uint_as_float(a[c + 2]), 0.0f), z);
                z = fmaf(w.w, fmaxf(__uint_as_float(a[c + 3]), 0.0f), z);
            }
        }
        if (row < n) logits[row] = z;
    }
    if (failed) {
        // a product did not complete in time: report it, and give it a bounded
        // while to land before TMEM is released
        if ((tid & 31) == 0) atomicOr(status, 1u);
        mbar_wait(mbar, parity ^ 1u, kTcWaitLimit);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTcCols));
}

int ensure_state(kf_context *ctx, MlpState **out)
{
    MlpState *&s = context_mlp_state(ctx);
    if (!s) {
        s = new MlpState;
        bool ok = cudaMalloc(&s->m, kMlpParams * sizeof(float)) == cudaSuccess &&
                  cudaMalloc(&s->v, kMlpParams * sizeof(float)) == cudaSuccess &&
                  cudaMalloc(&s->loss, sizeof(float)) == cudaSuccess &&
                  cudaMalloc(&s->w32, kMlpParams * sizeof(float)) == cudaSuccess &&
                  cudaMalloc(&s->W1, kW1Elems * sizeof(__nv_bfloat16)) == cudaSuccess &&
                  cudaMalloc(&s->W2, kW2Elems * sizeof(__nv_bfloat16)) == cudaSuccess &&
                  cudaMalloc(&s->status, sizeof(unsigned)) == cudaSuccess &&
                  zero_now(s->status, sizeof(unsigned)) == cudaSuccess;
        if (!ok) {
            destroy_mlp_state(s);
            s = nullptr;
            return set_error(ctx, KF_ERR_NOMEM, "could not allocate the proposal's scratch");
        }
    }
    *out = s;
    return KF_OK;
}

// Launch `kernel`, with programmatic dependent launch when `early`: the kernel
// may start while the launch before it on the stream still runs, and waits
// for it (griddepcontrol.wait) before it touches what that one writes.
template <class K, class... A>
cudaError_t launch_pdl(K kernel, unsigned grid, size_t smem, bool early, cudaStream_t stream, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kTrainThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Blocks of a gradient over `count` rows: one per tile, at most 2 per SM, each
// looping over its tiles.
unsigned grad_blocks(kf_context *ctx, int64_t count)
{
    return (unsigned)std::min<int64_t>((count + kTrainRows - 1) / kTrainRows, 2 * (int64_t)context_sm_count(ctx));
}

// Room for the partials of every block a gradient launches, and the kernel's
// shared memory (a per-device attribute).
int prepare_training(kf_context *ctx, MlpState *s)
{
    if (!s->partial && cudaMalloc(&s->partial, (size_t)2 * context_sm_count(ctx) * kPartLd * sizeof(float)) != cudaSuccess)
        return set_error(ctx, KF_ERR_NOMEM, "could not allocate the proposal's scratch");
    const cudaError_t e =
        cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
    return e == cudaSuccess ? KF_OK : cuda_error(ctx, e, "proposal training shared memory");
}

constexpr unsigned kReduceGrid = (kMlpParams + 1 + 31) / 32;

int64_t gcd64(int64_t a, int64_t b) { return b ? gcd64(b, a % b) : a; }

}  // namespace
}  // namespace kf

using namespace kf;

extern "C" {

int kf_proposal_gradient(kf_context *ctx, const float *weights, const float *features, const float *labels, int64_t n,
                         float *grad, float *loss, kf_stream stream_)
{
    if (!ctx) return KF_ERR_ARG;
    if (n < 1) return set_error(ctx, KF_ERR_ARG, "n must be >= 1");
    int rc;
    if ((rc = check_ptr(ctx, weights, 4, "weights")) || (rc = check_ptr(ctx, features, 4, "features")) ||
        (rc = check_ptr(ctx, labels, 4, "labels")) || (rc = check_ptr(ctx, grad, 4, "grad")))
        return rc;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    MlpState *s;
    if ((rc = ensure_state(ctx, &s))) return rc;
    if ((rc = prepare_training(ctx, s))) return rc;
    const unsigned blocks = grad_blocks(ctx, n);
    cudaError_t le = launch_pdl(mlp_grad_kernel, blocks, sizeof(TrainSmem), false, stream, weights, features, labels, n,
                                (int64_t)0, n, 1 % n, (int64_t)0, 1.0f / (float)n, s->partial);
    if (le == cudaSuccess)
        le = launch_pdl(mlp_reduce_kernel<false>, kReduceGrid, 0, true, stream, (const float *)s->partial, (int)blocks,
                        grad, s->loss, AdamArgs{});
    if (le != cudaSuccess) return cuda_error(ctx, le, "proposal gradient launch");
    if (loss) {
        float l = 0.0f;
        cudaMemcpyAsync(&l, s->loss, sizeof(float), cudaMemcpyDeviceToHost, stream);
        const cudaError_t e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) return cuda_error(ctx, e, "proposal gradient");
        *loss = l / (float)n;
    }
    return KF_OK;
}

int kf_proposal_train(kf_context *ctx, float *weights, const float *features, const float *labels, int64_t n, int epochs,
                      int batch, float learning_rate, float *epoch_loss, kf_stream stream_)
{
    if (!ctx) return KF_ERR_ARG;
    if (n < 1 || epochs < 0 || batch < 1 || !(learning_rate > 0.0f))
        return set_error(ctx, KF_ERR_ARG, "n >= 1, epochs >= 0, batch >= 1 and learning_rate > 0 required");
    int rc;
    if ((rc = check_ptr(ctx, weights, 4, "weights")) || (rc = check_ptr(ctx, features, 4, "features")) ||
        (rc = check_ptr(ctx, labels, 4, "labels")))
        return rc;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    MlpState *s;
    if ((rc = ensure_state(ctx, &s))) return rc;
    if ((rc = prepare_training(ctx, s))) return rc;
    cudaMemsetAsync(s->m, 0, kMlpParams * sizeof(float), stream);
    cudaMemsetAsync(s->v, 0, kMlpParams * sizeof(float), stream);
    // epoch order: sample = (j P + off) mod n with P coprime to n
    int64_t P = 1000003;
    while (gcd64(P, n) != 1) P += 2;
    int t = 0;
    for (int ep = 0; ep < epochs; ++ep) {
        cudaMemsetAsync(s->loss, 0, sizeof(float), stream);
        const int64_t off = (int64_t)ep * 7919 % n;
        for (int64_t b0 = 0; b0 < n; b0 += batch) {
            const int64_t cnt = std::min<int64_t>(batch, n - b0);
            const unsigned blocks = grad_blocks(ctx, cnt);
            // an epoch's first gradient follows a memset (or the caller's work), whose end it awaits whole
            cudaError_t le = launch_pdl(mlp_grad_kernel, blocks, sizeof(TrainSmem), b0 > 0, stream,
                                        (const float *)weights, features, labels, n, b0, cnt, P % n, off,
                                        1.0f / (float)cnt, s->partial);
            if (le == cudaSuccess)
                le = launch_pdl(mlp_reduce_kernel<true>, kReduceGrid, 0, true, stream, (const float *)s->partial,
                                (int)blocks, (float *)nullptr, s->loss,
                                AdamArgs{weights, s->m, s->v, ++t, learning_rate, 0.9f, 0.999f, 1e-8f});
            if (le != cudaSuccess) return cuda_error(ctx, le, "proposal training launch");
        }
        if (epoch_loss) {
            float l = 0.0f;
            cudaMemcpyAsync(&l, s->loss, sizeof(float), cudaMemcpyDeviceToHost, stream);
            const cudaError_t e = cudaStreamSynchronize(stream);
            if (e != cudaSuccess) return cuda_error(ctx, e, "proposal training");
            epoch_loss[ep] = l / (float)n;
        }
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? KF_OK : cuda_error(ctx, e, "proposal training");
}

int kf_proposal_load(kf_context *ctx, const float *weights, kf_stream stream_)
{
    if (!ctx) return KF_ERR_ARG;
    int rc;
    if ((rc = check_ptr(ctx, weights, 4, "weights"))) return rc;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    MlpState *s;
    if ((rc = ensure_state(ctx, &s))) return rc;
    cudaMemcpyAsync(s->w32, weights, kMlpParams * sizeof(float), cudaMemcpyDeviceToDevice, stream);
    to_bf16_kernel<<<8, 256, 0, stream>>>(s->w32, s->W1, s->W2);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(ctx, e, "proposal load");
    s->loaded = true;
    return KF_OK;
}

int kf_load_proposal(kf_context *ctx, const void *weights, size_t bytes)
{
    if (!ctx) return KF_ERR_ARG;
    if (bytes != kMlpParams * sizeof(float))
        return set_error(ctx, KF_ERR_ARG, "weights must be %zu bytes (%d FP32 parameters), got %zu",
                         (size_t)kMlpParams * sizeof(float), kMlpParams, bytes);
    return kf_proposal_load(ctx, static_cast<const float *>(weights), nullptr);
}

int kf_proposal_score_with(kf_context *ctx, const float *features, int64_t n, float *logits, int engine,
                           kf_stream stream_)
{
    if (!ctx) return KF_ERR_ARG;
    if (!proposal_loaded(ctx)) return set_error(ctx, KF_ERR_ARG, "no proposal weights loaded (kf_proposal_load)");
    if (n < 0) return set_error(ctx, KF_ERR_ARG, "n must be >= 0");
    if (engine != KF_SCORE_AUTO && engine != KF_SCORE_MMA_SYNC && engine != KF_SCORE_TCGEN05)
        return set_error(ctx, KF_ERR_ARG, "engine must be KF_SCORE_AUTO, KF_SCORE_MMA_SYNC or KF_SCORE_TCGEN05");
    if (n == 0) return KF_OK;
    int rc;
    if ((rc = check_ptr(ctx, features, 4, "features")) || (rc = check_ptr(ctx, logits, 4, "logits"))) return rc;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    MlpState *s = context_mlp_state(ctx);
    DeviceGuard dg(context_device(ctx));
    if (engine == KF_SCORE_AUTO) engine = n >= kScoreTcMinRows ? KF_SCORE_TCGEN05 : KF_SCORE_MMA_SYNC;
    cudaError_t e;
    if (engine == KF_SCORE_TCGEN05) {
        const auto kern = reinterpret_cast<uintptr_t>(features) % 16 ? mlp_score_tc_kernel<false> : mlp_score_tc_kernel<true>;
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TcSmem))) !=
            cudaSuccess)
            return cuda_error(ctx, e, "tcgen05 scoring shared memory");
        const int64_t tiles = (n + kTcRows - 1) / kTcRows;
        const unsigned grid = (unsigned)std::min<int64_t>((tiles + kTcGroups - 1) / kTcGroups,
                                                          (int64_t)context_sm_count(ctx) * kTcCtasPerSm);
        kern<<<grid, kTcThreads, sizeof(TcSmem), stream>>>(s->w32, features, n, logits, s->status, s->wait_limit);
    } else {
        if ((e = cudaFuncSetAttribute(mlp_score_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sizeof(ScoreSmem))) != cudaSuccess)
            return cuda_error(ctx, e, "scoring shared memory");
        const int64_t chunks = (n + 31) / 32;
        const unsigned grid = (unsigned)std::min<int64_t>((chunks + kScoreWarps - 1) / kScoreWarps,
                                                          (int64_t)context_sm_count(ctx) * 8);
        mlp_score_kernel<<<grid, 32 * kScoreWarps, sizeof(ScoreSmem), stream>>>(s->W1, s->W2, s->w32, features, n,
                                                                                logits);
    }
    e = cudaGetLastError();
    return e == cudaSuccess ? KF_OK : cuda_error(ctx, e, "proposal score launch");
}

int kf_proposal_score(kf_context *ctx, const float *features, int64_t n, float *logits, kf_stream stream)
{
    return kf_proposal_score_with(ctx, features, n, logits, KF_SCORE_AUTO, stream);
}

// For tests, not in kf.h: the polls after which a tcgen05 scoring wait of this
// context gives up (0: at once).  Weights must have been loaded.
int kf_test_score_wait_limit(kf_context *ctx, uint32_t polls)
{
    if (!ctx || !proposal_loaded(ctx)) return KF_ERR_ARG;
    context_mlp_state(ctx)->wait_limit = polls;
    return KF_OK;
}

int kf_proposal_status(kf_context *ctx, int *expired)
{
    if (!ctx || !expired) return KF_ERR_ARG;
    *expired = 0;
    MlpState *s = context_mlp_state(ctx);
    if (!s) return KF_OK;
    DeviceGuard dg(context_device(ctx));
    unsigned v = 0;
    const cudaError_t e = cudaMemcpy(&v, s->status, sizeof v, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_error(ctx, e, "proposal status");
    *expired = v != 0;
    return KF_OK;
}

}  // extern "C"
