// The per-track arithmetic of csrc/kf_math.cuh compiled for the host, for tests
// of single steps without a GPU.
#include "cuda_shim.h"

#include "kf_math.cuh"

using namespace kf;

static Routing routing(const float *opt)  // routed, cond_max, pt_lo, pt_hi, gain_max
{
    Routing rt{};
    rt.mode = (int)opt[0];
    rt.det_min = 6.75f / opt[1];
    rt.pt_lo2 = opt[2] * opt[2];
    rt.pt_hi2 = opt[3] * opt[3];
    rt.gain_max = opt[4];
    return rt;
}

// enter_local of n seeds [6][n], [21][n] to radius r: flags [n] and the local
// covariances [15][n].
extern "C" void host_enter(int64_t n, const float *state, const float *cov, const int8_t *charge, float qk, float r,
                           float z_half, const float *opt, float *out, uint32_t *flags)
{
    const Routing rt = routing(opt);
    for (int64_t t = 0; t < n; ++t) {
        float x[6], c6[21], c[15], slot[kSlotSize], pn;
        for (int i = 0; i < 6; ++i) x[i] = state[i * n + t];
        for (int i = 0; i < 21; ++i) c6[i] = cov[i * n + t];
        Local p{};
        flags[t] = enter_local(x, c6, charge[t] * qk, r, 1.0f / r, z_half, rt, slot, 1, p, c, pn);
        for (int i = 0; i < 15; ++i) out[i * n + t] = flags[t] ? NAN : c[i];
    }
}

// One update on the slot by the routine of `kind` (1 float-float gain, 2 FP64,
// 3 float-float): n of x [6][n] (position, q1, q2, pz), c [15][n], nx and ny,
// hits m [3][n] and v [6][n]; x and c in place, chi2 and the routine's result.
extern "C" void host_slot_update(int kind, int64_t n, float *x, float *c, const float *nrm, const float *m, const float *v,
                                 float *chi2, int32_t *st)
{
    for (int64_t t = 0; t < n; ++t) {
        float s[kSlotSize] = {};
        for (int i = 0; i < 6; ++i) s[kSlotX + i] = x[i * n + t];
        for (int i = 0; i < 15; ++i) s[kSlotC + i] = c[i * n + t];
        for (int i = 0; i < 3; ++i) s[kSlotM + i] = m[i * n + t];
        for (int i = 0; i < 6; ++i) s[kSlotV + i] = v[i * n + t];
        s[kSlotFrame + 2] = nrm[t];
        s[kSlotFrame + 3] = nrm[n + t];
        st[t] = update_ext(s, 1, kind);
        for (int i = 0; i < 6; ++i) x[i * n + t] = s[kSlotX + i];
        for (int i = 0; i < 15; ++i) c[i * n + t] = s[kSlotC + i];
        chi2[t] = s[kSlotChi2];
    }
}

// update_local of the same arrays, q1, q2 as given; st as it returns.
extern "C" void host_update(int64_t n, float *x, float *c, const float *nrm, const float *m, const float *v,
                            const float *opt, float *chi2, int32_t *st)
{
    const Routing rt = routing(opt);
    for (int64_t t = 0; t < n; ++t) {
        float cl[15], ml[3], vl[6], slot[kSlotSize];
        Local p{x[t], x[n + t], x[2 * n + t], x[3 * n + t], x[4 * n + t], x[5 * n + t], 1.0f, 0.0f, nrm[t], nrm[n + t]};
        for (int i = 0; i < 15; ++i) cl[i] = c[i * n + t];
        for (int i = 0; i < 3; ++i) ml[i] = m[i * n + t];
        for (int i = 0; i < 6; ++i) vl[i] = v[i * n + t];
        st[t] = update_local(p, cl, ml, vl, rt, &chi2[t], slot, 1);
        const float out[6] = {p.x, p.y, p.z, p.q1, p.q2, p.pz};
        for (int i = 0; i < 6; ++i) x[i * n + t] = out[i];
        for (int i = 0; i < 15; ++i) c[i * n + t] = cl[i];
    }
}
