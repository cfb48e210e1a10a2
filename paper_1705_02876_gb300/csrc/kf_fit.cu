// Kalman-filter track fit on sm_103a: one thread per track (Section 4.2),
// state and packed local covariance (kf_math.cuh) in registers, structure-of-arrays inputs read
// coalesced (Section 4.1: element (i, j) of consecutive tracks is contiguous).
#include <algorithm>
#include <mutex>
#include <set>
#include <utility>

#include "kf.h"
#include "kf_fit.cuh"

namespace kf {

namespace {

__device__ __forceinline__ void cp_async4(float *dst, const float *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
#ifdef __CUDACC__
__device__ __forceinline__ void prefetch_l2(const float *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
#endif
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Fit track base + off over every layer in order (the steps and stop rules are
// those of kf_fit_tracks in kf.h).  base is the block's: the addresses of every
// array are then a uniform pointer and the thread's offset.  A layer's hit is
// loaded ahead of its update: DEPTH = 1 into registers, at the start of the
// layer (the step and the transport, 250 instructions, cover the latency; a
// layer earlier cost nine registers and as many moves a layer); DEPTH >= 2
// layers ahead, by asynchronous copies (cp.async, one commit group per layer,
// empty for a layer without a hit) into this thread's column of a ring of
// DEPTH + 1 shared-memory stages of 9 floats each ([stage * 9 + i][stride]),
// so that the loads in flight hold no registers.  A non-finite value in a
// used hit makes the chi2 increment non-finite, or makes S fail its positive
// definiteness test, so the hit is tested only then.
// Without DEFER (the plain kernel's small batches and single events, and the
// tracks put off, which lie apart: few warps wait for DRAM with nothing to do)
// the next layer's hit goes to L2 a layer ahead.  Events of 5,000 tracks, one
// launch each, not in L2: 12.7 us, 14.8 without; of 20,000 14.8 and 15.9.
// DEFER: a track outside the pT bounds on the first layer, and any other at the
// first update that needs extended precision, is given up and true returned
// (nothing is written).
template <int DEPTH, bool DEFER, class OFF>
__device__ __forceinline__ bool fit_track(const FitGeom &g, const Routing &rt, const FitIO &io, int64_t base, OFF off,
                                          float *slot, int stride, float *ring = nullptr)
{
    const int64_t T = io.T;
    const float *seed_state = io.seed_state + base, *seed_cov = io.seed_cov + base;
    const float *hp = io.hit_pos + base;  // layer l, component i: hp[(3 l + i) T + off]
    const float *hc = io.hit_cov + base;
    const uint32_t mask = __ldcs(io.hit_mask + base + off);
    float m[3] = {0, 0, 0}, v[6] = {0, 0, 0, 0, 0, 0};
    auto load_hit = [&](bool has) {
        if (has) {
#pragma unroll
            for (int i = 0; i < 3; ++i) m[i] = __ldcs(hp + i * T + off);
#pragma unroll
            for (int i = 0; i < 6; ++i) v[i] = __ldcs(hc + i * T + off);
        }
        hp += 3 * T;
        hc += 6 * T;
    };
    // DEPTH >= 2: layer l's hit goes to stage l % (DEPTH + 1); stage_in is the
    // stage of the next layer to issue, stage_out that of the next to use
    int stage_in = 0, stage_out = 0, l_in = 0;
    auto issue = [&]() {
        if (l_in < g.L && ((mask >> l_in) & 1u)) {
            float *st = ring + stage_in * 9 * stride;
#pragma unroll
            for (int i = 0; i < 3; ++i) cp_async4(st + i * stride, hp + i * T + off);
#pragma unroll
            for (int i = 0; i < 6; ++i) cp_async4(st + (3 + i) * stride, hc + i * T + off);
        }
        cp_async_commit();
        ++l_in;
        hp += 3 * T;
        hc += 6 * T;
        stage_in = stage_in == DEPTH ? 0 : stage_in + 1;
    };
    float sx[6], sc[21];
#pragma unroll
    for (int i = 0; i < 6; ++i) sx[i] = __ldcs(seed_state + i * T + off);
#pragma unroll
    for (int i = 0; i < 21; ++i) sc[i] = __ldcs(seed_cov + i * T + off);
    const float qkb = (float)(io.charge + base)[off] * g.qk;
    if constexpr (DEPTH == 1) {
        load_hit(mask & 1u);  // the seed's loads are in flight
    } else {
#pragma unroll
        for (int k = 0; k < DEPTH; ++k) issue();
    }
    uint32_t flags = (all_finite<6>(sx) && all_finite<21>(sc)) ? 0u : (uint32_t)KF_FLAG_NAN_INPUT;
    float chi2 = 0.0f;
    int nhits = 0;
    Local p;
    float c[15], pn;
    bool deferred = false;
    if (!flags) flags = enter_local<DEFER>(sx, sc, qkb, g.r[0], g.inv_r[0], g.z_half, rt, slot, stride, p, c, pn);
    if (DEFER && flags == kPutOff) {
        deferred = true;
        flags = 0u;
    }
    const bool at_seed = flags != 0u;  // no layer reached
    if (!at_seed && !deferred) {
        for (int l = 0; l < g.L; ++l) {
            const bool has = (mask >> l) & 1u;
            if constexpr (DEPTH == 1) {
                if (l > 0) load_hit(has);
                if (!DEFER && l + 1 < g.L && ((mask >> (l + 1)) & 1u)) {
#pragma unroll
                    for (int i = 0; i < 3; ++i) prefetch_l2(hp + i * T + off);
#pragma unroll
                    for (int i = 0; i < 6; ++i) prefetch_l2(hc + i * T + off);
                }
            } else {
                issue();                 // layer l + DEPTH
                cp_async_wait<DEPTH>();  // layer l's group has landed
                if (has) {
                    const float *st = ring + stage_out * 9 * stride;
#pragma unroll
                    for (int i = 0; i < 3; ++i) m[i] = st[i * stride];
#pragma unroll
                    for (int i = 0; i < 6; ++i) v[i] = st[(3 + i) * stride];
                }
                stage_out = stage_out == DEPTH ? 0 : stage_out + 1;
            }
            if (l > 0) {
                LocalJac J;
                const uint32_t stop = step_local(p, qkb, g.r[l], g.inv_r[l], g.z_half, J, pn);
                if (stop) {
                    flags |= stop;
                    break;
                }
                transport_local(J, c);
            }
            scatter_local(p, noise_local(p, pn, g.xx0[l]), c);
            if (has) {
                float d = 0.0f;
                const int st = update_local<DEFER>(p, c, m, v, rt, &d, slot, stride);
                if (DEFER && st == 4) {
                    deferred = true;
                    break;
                }
                if (st == 1 || !isfinite(d)) {
                    if (!all_finite<3>(m) || !all_finite<6>(v)) {
                        flags |= KF_FLAG_NAN_INPUT;
                        break;
                    }
                }
                if (st == 1) {
                    flags |= KF_FLAG_INVERSION_FAILED;
                } else {
                    chi2 += d;
                    ++nhits;
                    if (st >= 2) flags |= KF_FLAG_FP64_PATH;
                    if (st == 3) flags |= KF_FLAG_PSD_REPAIRED;
                }
            }
        }
    }
    if constexpr (DEPTH > 1) cp_async_wait<0>();
    if (DEFER && deferred) return true;
    float x[6], c6[21];
    if (at_seed || (flags & KF_FLAG_NAN_INPUT)) {  // a track with bad input returns its seed
#pragma unroll
        for (int i = 0; i < 6; ++i) x[i] = seed_state[i * T + off];
#pragma unroll
        for (int i = 0; i < 21; ++i) c6[i] = seed_cov[i * T + off];
        chi2 = 0.0f;
        nhits = 0;
    } else {
        leave_local(p, c, x, c6);
    }
    float *out_state = io.out_state + base, *out_cov = io.out_cov + base;
#pragma unroll
    for (int i = 0; i < 6; ++i) __stcs(out_state + i * T + off, x[i]);
#pragma unroll
    for (int i = 0; i < 21; ++i) __stcs(out_cov + i * T + off, c6[i]);
    __stcs(io.out_chi2 + base + off, chi2);
    (io.out_ndof + base)[off] = (int16_t)(3 * nhits - 6);
    (io.out_flags + base)[off] = flags;
    return false;
}

}  // namespace

#ifdef __CUDACC__  // tests compile the above for the host
namespace {

// One thread per track over [t_begin, t_end), the updates in extended precision
// in line.  Two blocks of 256 threads per SM: at 128 registers (162 uncapped)
// 1,000,000 tracks take 205 us (212 without the prefetch, 255 uncapped).
__global__ void __launch_bounds__(256, 2) fit_plain_kernel(const FitGeom g, const Routing rt, const FitIO io,
                                                         int64_t t_begin, int64_t t_end)
{
    extern __shared__ float slots[];
    const int64_t t = t_begin + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < t_end) fit_track<1, false>(g, rt, io, t - threadIdx.x, threadIdx.x, slots + threadIdx.x, blockDim.x);
}

// One thread per track over the whole batch (Section 4.2: fill the GPU with the
// tracks of many events in one launch).  MINB > 1 caps the registers per
// thread at 65536 / (BLOCK * MINB) to raise occupancy.  DEPTH >= 2 keeps the
// hit ring in dynamic shared memory (ring_bytes(...)).
//
// An update in extended precision (float-float: some 1,100 instructions; FP64:
// a pipe 64 times narrower than the FP32 one) takes as long for one lane of a
// warp as for 32, so a track that needs one is put off: its flags are set to
// kPutOff and *work to the fit's tag, and fit_extended_kernel, launched behind,
// fits these tracks from their seeds in full warps (no tag: it returns at
// once; the tag of a fit replayed from a graph may stand from an earlier
// replay, and the kernel then finds no marked track).  With one track in eight
// outside the pT bounds (1,000,000 tracks, pT log-uniform 0.24 to 500 GeV)
// nearly every warp holds one and stops for it at every layer: 7.09 ms in line
// in FP64, 1.03 ms put off in FP64, 0.31 ms put off in float-float (0.70 in
// line).  Without that code this kernel also needs fewer registers (80 to 96,
// no spills).
template <int BLOCK, int MINB, int DEPTH>
__global__ void __launch_bounds__(BLOCK, MINB) fit_kernel(const FitGeom g, const Routing rt, const FitIO io,
                                                           unsigned *work, unsigned tag)
{
    extern __shared__ float ring[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int64_t base = (int64_t)blockIdx.x * BLOCK;
    const unsigned off = threadIdx.x;
    bool put_off = false;
    if (base + off < io.T) put_off = fit_track<DEPTH, true>(g, rt, io, base, off, nullptr, BLOCK, ring + off);
    if (put_off) (io.out_flags + base)[off] = kPutOff;
    if (__any_sync(0xffffffffu, put_off) && (off & 31u) == 0) *work = tag;
}

// The tracks put off by the launch before: a block gathers them from the flags
// of its chunks of the batch until it has one per thread, and fits those.  Two
// blocks of 256 threads per SM: the fewer blocks gather, the fewer end on a part
// of one (1,000,000 stress tracks: 307 us in all; 324 with four blocks of 128,
// 330 and 342 with 64 and 32 threads).
constexpr int kExtBlock = 256;
__global__ void __launch_bounds__(kExtBlock, 2) fit_extended_kernel(const FitGeom g, const Routing rt, const FitIO io,
                                                                     const unsigned *work, unsigned tag)
{
    __shared__ float slots[kSlotSize * kExtBlock];
    __shared__ int64_t queue[2 * kExtBlock];
    __shared__ int queued;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (__ldcg(work) != tag) return;
    if (threadIdx.x == 0) queued = 0;
    __syncthreads();
    const int64_t chunks = (io.T + kExtBlock - 1) / kExtBlock;
    for (int64_t ch = blockIdx.x; ch < chunks; ch += gridDim.x) {
        const int64_t t = ch * kExtBlock + threadIdx.x;
        if (t < io.T && __ldcg(io.out_flags + t) == kPutOff) queue[atomicAdd(&queued, 1)] = t;
        __syncthreads();
        const bool last = ch + gridDim.x >= chunks;
        int n = queued;
        while (n >= kExtBlock || (last && n > 0)) {  // uniform over the block
            const int take = min(n, kExtBlock);
            n -= take;
            if ((int)threadIdx.x < take)
                fit_track<1, false>(g, rt, io, 0, queue[n + threadIdx.x], slots + threadIdx.x, kExtBlock);
        }
        __syncthreads();
        if (threadIdx.x == 0) queued = n;
        __syncthreads();
    }
}

using FitFn = void (*)(FitGeom, Routing, FitIO, unsigned *, unsigned);

// Dynamic shared memory of a shape: DEPTH + 1 stages of 9 floats per thread.
constexpr size_t ring_bytes(int block, int depth) { return depth > 1 ? (size_t)(depth + 1) * 9 * block * 4 : 0; }

// (block, register cap, hit prefetch depth) shapes the autotuner chooses
// from; cap 0 = none.  A cap of R registers is
// __launch_bounds__(BLOCK, 65536 / (R * BLOCK)).
struct Shape {
    int block, cap, depth;
    FitFn fn;
};
const Shape kShapes[] = {
    {32, 0, 1, fit_kernel<32, 1, 1>},     {64, 0, 1, fit_kernel<64, 1, 1>},
    {128, 0, 1, fit_kernel<128, 1, 1>},   {256, 0, 1, fit_kernel<256, 1, 1>},
    {32, 168, 1, fit_kernel<32, 12, 1>},  {64, 168, 1, fit_kernel<64, 6, 1>},
    {128, 168, 1, fit_kernel<128, 3, 1>}, {32, 128, 1, fit_kernel<32, 16, 1>},
    {64, 128, 1, fit_kernel<64, 8, 1>},   {128, 128, 1, fit_kernel<128, 4, 1>},
    {256, 128, 1, fit_kernel<256, 2, 1>}, {32, 96, 1, fit_kernel<32, 20, 1>},
    {64, 96, 1, fit_kernel<64, 10, 1>},   {128, 96, 1, fit_kernel<128, 5, 1>},
    {32, 80, 1, fit_kernel<32, 24, 1>},   {64, 80, 1, fit_kernel<64, 12, 1>},
    {128, 80, 1, fit_kernel<128, 6, 1>},  {256, 80, 1, fit_kernel<256, 3, 1>},
    {32, 128, 2, fit_kernel<32, 16, 2>},  {64, 128, 2, fit_kernel<64, 8, 2>},
    {128, 128, 2, fit_kernel<128, 4, 2>}, {256, 128, 2, fit_kernel<256, 2, 2>},
    {32, 96, 2, fit_kernel<32, 20, 2>},   {64, 96, 2, fit_kernel<64, 10, 2>},
    {128, 96, 2, fit_kernel<128, 5, 2>},  {32, 128, 4, fit_kernel<32, 16, 4>},
    {64, 128, 4, fit_kernel<64, 8, 4>},   {128, 128, 4, fit_kernel<128, 4, 4>},
    {256, 128, 4, fit_kernel<256, 2, 4>}, {32, 96, 4, fit_kernel<32, 20, 4>},
    {64, 96, 4, fit_kernel<64, 10, 4>},   {128, 96, 4, fit_kernel<128, 5, 4>},
};

const Shape *find_shape(int block, int cap, int depth)
{
    for (const Shape &sh : kShapes)
        if (sh.block == block && sh.cap == cap && sh.depth == depth) return &sh;
    return nullptr;
}

// Allow a shape's dynamic shared memory on the current device.  The opt-in
// is a per-device function attribute, so it is remembered per (device,
// shape), under a lock: several host threads may launch at once.
cudaError_t prepare_shape(const Shape *sh)
{
    const size_t bytes = ring_bytes(sh->block, sh->depth);
    if (!bytes) return cudaSuccess;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    static std::mutex mu;
    static std::set<std::pair<int, const Shape *>> done;
    std::lock_guard<std::mutex> lock(mu);
    if (done.count({dev, sh})) return cudaSuccess;
    e = cudaFuncSetAttribute(sh->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) done.insert({dev, sh});
    return e;
}

}  // namespace

cudaError_t launch_fit_plain(const FitGeom &g, const Routing &rt, const FitIO &io, int64_t t_begin,
                             int64_t t_end, int block, cudaStream_t stream)
{
    if (t_end <= t_begin) return cudaSuccess;
    const int64_t n = t_end - t_begin;
    const unsigned grid = (unsigned)((n + block - 1) / block);
    fit_plain_kernel<<<grid, block, kSlotSize * block * sizeof(float), stream>>>(g, rt, io, t_begin, t_end);
    return cudaGetLastError();
}

int fit_shape_usable(int block, int cap, int depth)
{
    const Shape *sh = find_shape(block, cap, depth);
    if (!sh) return 0;
    return prepare_shape(sh) == cudaSuccess ? 1 : -1;
}

int fit_shapes(int *blocks, int *caps, int *depths, int max_n)
{
    int n = 0;
    for (const Shape &sh : kShapes)
        if (n < max_n) {
            blocks[n] = sh.block;
            caps[n] = sh.cap;
            depths[n] = sh.depth;
            ++n;
        }
    return n;
}

cudaError_t launch_fit_tuned(const FitGeom &g, const Routing &rt, const FitIO &io, int block, int cap, int depth,
                                  int sm_count, unsigned *work, unsigned tag, cudaStream_t stream)
{
    const Shape *sh = find_shape(block, cap, depth);
    if (!sh) return cudaErrorInvalidValue;
    cudaError_t e = prepare_shape(sh);
    if (e != cudaSuccess) return e;
    // A float-float gain takes three times an FP32 update and may be asked of
    // any share of the tracks, which a fit from the seed anew pays for only if
    // they are few.  1,000,000 tracks with gain_max 1, 100 and 10,000 (all, 76%
    // and none of them): 657, 250 and 205 us in line, 712, 401 and 178 put off.
    if (rt.mode == 1 && rt.gain_max > 0.0f) return launch_fit_plain(g, rt, io, 0, io.T, block, stream);
    const int64_t grid = (io.T + block - 1) / block;
    if (grid > INT32_MAX) return cudaErrorInvalidConfiguration;
    sh->fn<<<(unsigned)grid, block, ring_bytes(block, depth), stream>>>(g, rt, io, work, tag);
    if ((e = cudaGetLastError()) != cudaSuccess || rt.mode == 0) return e;  // without routing no track is put off
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min<int64_t>((io.T + kExtBlock - 1) / kExtBlock, (int64_t)sm_count * 2));
    cfg.blockDim = dim3(kExtBlock);
    cfg.stream = stream;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fit_extended_kernel, g, rt, io, (const unsigned *)work, tag);
}
#endif  // __CUDACC__

}  // namespace kf
