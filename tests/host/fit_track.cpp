// The fit of one track (fit_track of csrc/kf_fit.cu, hits loaded at their layer)
// compiled for the host, recording which hits it reads
// or fetches ahead.
#include "cuda_shim.h"

#define __CUDA_RUNTIME_H__  // the CUDA runtime's header is not needed
typedef int cudaError_t;
typedef void *cudaStream_t;
static unsigned long __cvta_generic_to_shared(const void *) { return 0; }

static const float *rec_base[2];
static int64_t rec_row[2], rec_tracks;  // floats per layer of hit_pos, hit_cov
static uint32_t *rec_read;
static void record(const float *p)
{
    for (int k = 0; k < 2; ++k) {
        const int64_t i = p - rec_base[k];
        if (i >= 0 && i < 32 * rec_row[k]) rec_read[i % rec_tracks] |= 1u << (i / rec_row[k]);
    }
}
static void record(const uint32_t *) {}
template <class T>
static T __ldcs(const T *p)
{
    record(p);
    return *p;
}
static void prefetch_l2(const float *p) { record(p); }
template <class T>
static void __stcs(T *p, T v)
{
    *p = v;
}

#include "kf_fit.cu"

using namespace kf;

// Fit n tracks; hits_read [n]: the layers whose hits were read.  hit_pos and
// hit_cov are 32 layers apart in one block, so that the two cannot be confused.
extern "C" void host_fit(int L, const float *r, const float *xx0, float z_half, float qk, int64_t n, const float *seed_state,
                         const float *seed_cov, const int8_t *charge, const float *hit_pos, const float *hit_cov,
                         const uint32_t *mask, float *state, float *cov, float *chi2, int16_t *ndof, uint32_t *flags,
                         uint32_t *hits_read)
{
    FitGeom g{};
    g.L = L;
    g.z_half = z_half;
    g.qk = qk;
    for (int l = 0; l < L; ++l) {
        g.r[l] = r[l];
        g.inv_r[l] = 1.0f / r[l];
        g.xx0[l] = xx0[l];
    }
    Routing rt{};
    rt.mode = 1;
    rt.det_min = 6.75f / 1e4f;
    rt.pt_lo2 = 0.25f * 0.25f;
    rt.pt_hi2 = 200.0f * 200.0f;
    const FitIO io{n, seed_state, seed_cov, charge, hit_pos, hit_cov, mask, state, cov, chi2, ndof, flags};
    rec_base[0] = hit_pos;
    rec_base[1] = hit_cov;
    rec_row[0] = 3 * n;
    rec_row[1] = 6 * n;
    rec_tracks = n;
    rec_read = hits_read;
    for (int64_t t = 0; t < n; ++t) {
        float slot[kSlotSize];
        hits_read[t] = 0;
        fit_track<1, false>(g, rt, io, t, 0, slot, 1);
    }
}
