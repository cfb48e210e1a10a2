// Track-fit kernels: shared declarations between the kernels and the C-ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kf_math.cuh"

namespace kf {

constexpr int kMaxLayers = 32;

struct FitGeom {
    int L;
    float z_half;
    float qk;  // k * Bz; a track's curvature is charge * qk / pT
    float r[kMaxLayers];
    float inv_r[kMaxLayers];
    float xx0[kMaxLayers];
};

struct FitIO {
    int64_t T;  // row stride of every [..][T] array (tracks in the batch)
    const float *seed_state;
    const float *seed_cov;
    const int8_t *charge;
    const float *hit_pos;
    const float *hit_cov;
    const uint32_t *hit_mask;
    float *out_state;
    float *out_cov;
    float *out_chi2;
    int16_t *out_ndof;
    uint32_t *out_flags;
};

// A launch shape of the fit: threads per block, register cap (0 = none)
// and hit prefetch depth (layers ahead).
struct FitShape {
    int block, cap, depth;
};

// Launchers (kf_fit.cu).  All enqueue on `stream` and return the launch error.
cudaError_t launch_fit_plain(const FitGeom &g, const Routing &rt, const FitIO &io, int64_t t_begin,
                             int64_t t_end, int block, cudaStream_t stream);
// The fit of the whole batch: a kernel of blocks of `block` threads with
// registers capped at `cap` per thread (0 = no cap), hits loaded `depth` layers
// ahead (1: registers; 2, 4: a cp.async ring in shared memory), which writes
// `tag` to *work when a track needs extended precision, and with routing a
// second one for those tracks; or, with routing and gain_max > 0, the plain
// kernel in blocks of `block` threads.  *work is the launch's own until it has
// run; what it holds before does not matter, as long as each launch on it has
// another tag than the one before.
cudaError_t launch_fit_tuned(const FitGeom &g, const Routing &rt, const FitIO &io, int block, int cap, int depth,
                             int sm_count, unsigned *work, unsigned tag, cudaStream_t stream);
// 1 if this shape can be launched on the current device, 0 if it is not
// compiled in, -1 if its shared-memory opt-in failed.
int fit_shape_usable(int block, int cap, int depth);
// The (block, cap, depth) shapes compiled in; returns how many were written.
int fit_shapes(int *blocks, int *caps, int *depths, int max_n);

}  // namespace kf
