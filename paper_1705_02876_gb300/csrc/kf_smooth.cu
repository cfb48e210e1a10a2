// The Kalman smoother on sm_103a: the forward fit (Sections 2, 2.1 and 4.2)
// followed, in the same thread, by the backward Rauch-Tung-Striebel pass that
// gives at every layer the estimate using all of the track's hits (Section 2
// names a final fit with a smoother as the step after building).
//
// Both passes work in the local coordinates (t, z, q1, q2, pz) of kf_math.cuh,
// where the covariances are 5x5 and positive definite.  With G the Jacobian
// from layer l to layer l+1 and Q the scattering noise added at layer l+1:
//   A_l  = Cf_l G^T Cp_{l+1}^-1 = G^-1 (I - K), K = Q Cp_{l+1}^-1  (Cp = G Cf G^T + Q),
//   xs_l = xf_l + A_l (xs_{l+1} - xp_{l+1}),
//   Cs_l = Cf_l + A_l (Cs_{l+1} - Cp_{l+1}) A_l^T.
// The second form is the one computed: Cp^-1 (an L D L^T factorisation) only
// multiplies the scattering noise, so the FP32 rounding that Cp's correlations
// amplify enters A scaled by |Q| / |Cp|.  K has the three momentum rows only,
// and G^-1 has the form of G itself (a step back along the helix), so that
// the covariance goes through the transport of the forward pass.  The forward
// pass writes the filtered coordinates, their covariance and frames (25 floats)
// of every layer to the output arrays; the backward pass reads them, repeats the
// step to layer l+1 (xp, G and Q come out the same, bit for bit) and overwrites
// them with the smoothed estimate.  Nothing else is stored: they are read back
// while still in L2, and each output line reaches DRAM once, smoothed.
#include "kf.h"
#include "kf_api_internal.h"
#include "kf_fit.cuh"

namespace kf {

struct SmoothState {};  // the smoother keeps no scratch

void destroy_smooth_state(SmoothState *s) { delete s; }

namespace {

struct SmoothIO {
    int64_t T;
    const float *seed_state, *seed_cov;
    const int8_t *charge;
    const float *hit_pos, *hit_cov;
    const uint32_t *hit_mask;
    float *out_state, *out_cov;  // [L][6][T], [L][21][T]
    int16_t *out_reached;
    uint32_t *out_flags;
};

// Registers capped at 128 (four blocks, 16 warps per SM).  Bound by FP32 issue:
// 1,474 warp instructions per 32 track-layers, 62% of the issue slots (500,000
// tracks of 10 layers: 0.355 ms on the 6x6 covariance, 0.297 ms now; 1.56 KB
// per track at the copy bandwidth would take 0.115 ms).
__global__ void __launch_bounds__(128, 4) smooth_kernel(const FitGeom g, const Routing rt, const SmoothIO io)
{
    extern __shared__ float slots[];
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= io.T) return;
    const int64_t T = io.T;
    const int L = g.L;
    float *slot = slots + threadIdx.x;
    const int stride = blockDim.x;
    float *os = io.out_state + t, *oc = io.out_cov + t;  // layer l, component i: os[(6 l + i) T], oc[(21 l + i) T]

    // ---- forward: the fit, keeping every layer
    const float qkb = (float)io.charge[t] * g.qk;
    const uint32_t mask = io.hit_mask[t];
    float m[3] = {0, 0, 0}, v[6] = {0, 0, 0, 0, 0, 0};
    const float *hp = io.hit_pos + t, *hc = io.hit_cov + t;
    auto load_hit = [&](float mm[3], float vv[6]) {
#pragma unroll
        for (int i = 0; i < 3; ++i) mm[i] = __ldcs(hp + i * T);
#pragma unroll
        for (int i = 0; i < 6; ++i) vv[i] = __ldcs(hc + i * T);
    };
    Local p{};
    float c[15], pn;
    uint32_t flags;
    bool go;
    {
        float x6[6], c6[21];
#pragma unroll
        for (int i = 0; i < 6; ++i) x6[i] = __ldcs(io.seed_state + i * T + t);
#pragma unroll
        for (int i = 0; i < 21; ++i) c6[i] = __ldcs(io.seed_cov + i * T + t);
        if (mask & 1u) load_hit(m, v);
        flags = (all_finite<6>(x6) && all_finite<21>(c6)) ? 0u : (uint32_t)KF_FLAG_NAN_INPUT;
        if (!flags) flags = enter_local(x6, c6, qkb, g.r[0], g.inv_r[0], g.z_half, rt, slot, stride, p, c, pn);
        go = flags == 0u;
    }
    int K = 0;
    for (int l = 0; l < L && go; ++l) {
        const bool has = (mask >> l) & 1u;
        if (l > 0 && has) load_hit(m, v);  // the step and the transport cover the latency
        hp += 3 * T;
        hc += 6 * T;
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
            const int st = update_local(p, c, m, v, rt, &d, slot, stride);
            // a non-finite hit value fails the update or makes d non-finite
            if ((st == 1 || !isfinite(d)) && (!all_finite<3>(m) || !all_finite<6>(v))) {
                flags |= KF_FLAG_NAN_INPUT;
                K = 0;
                break;
            }
            if (st == 1) flags |= KF_FLAG_INVERSION_FAILED;
            if (st >= 2) flags |= KF_FLAG_FP64_PATH;
            if (st == 3) flags |= KF_FLAG_PSD_REPAIRED;
        }
        K = l + 1;
        if (K < L) {  // filtered: the coordinates, their covariance and frames
            const float x[6] = {p.x, p.y, p.z, p.q1, p.q2, p.pz};
#pragma unroll
            for (int i = 0; i < 6; ++i) os[(int64_t)(6 * l + i) * T] = x[i];
#pragma unroll
            for (int i = 0; i < 15; ++i) oc[(int64_t)(21 * l + i) * T] = c[i];
            oc[(int64_t)(21 * l + 15) * T] = p.nx;
            oc[(int64_t)(21 * l + 16) * T] = p.ny;
            oc[(int64_t)(21 * l + 17) * T] = p.f0;
            oc[(int64_t)(21 * l + 18) * T] = p.f1;
        }
    }
    io.out_reached[t] = (int16_t)K;

    // ---- backward: p, c are the smoothed estimate of layer l + 1
    auto write = [&](int l) {
        float x6[6], c6[21];
        leave_local(p, c, x6, c6);
#pragma unroll
        for (int i = 0; i < 6; ++i) __stcs(os + (int64_t)(6 * l + i) * T, x6[i]);
#pragma unroll
        for (int i = 0; i < 21; ++i) __stcs(oc + (int64_t)(21 * l + i) * T, c6[i]);
    };
    if (K > 0) write(K - 1);
    for (int l = K - 2; l >= 0; --l) {
        Local f;
        float cf[15];
        {
            const float *a = os + (int64_t)(6 * l) * T, *b = oc + (int64_t)(21 * l) * T;
            // the filtered estimate's last read
            f = Local{__ldlu(a),         __ldlu(a + T),      __ldlu(a + 2 * T),  __ldlu(a + 3 * T),  __ldlu(a + 4 * T),
                      __ldlu(a + 5 * T), __ldlu(b + 17 * T), __ldlu(b + 18 * T), __ldlu(b + 15 * T), __ldlu(b + 16 * T)};
#pragma unroll
            for (int i = 0; i < 15; ++i) cf[i] = __ldlu(b + i * T);
        }
        // the prediction of layer l+1, as the forward pass made it (the track
        // reached layer l+1 there)
        Local q = f;
        LocalJac J, B;
        float cp[15], cn0;
        step_local(q, qkb, g.r[l + 1], g.inv_r[l + 1], INFINITY, J, pn, &B, &cn0);
#pragma unroll
        for (int i = 0; i < 15; ++i) cp[i] = cf[i];
        transport_local(J, cp);
        const float t2 = noise_local(q, pn, g.xx0[l + 1]);
        scatter_local(q, t2, cp);
        float D[15];
#pragma unroll
        for (int i = 0; i < 15; ++i) D[i] = c[i] - cp[i];
        // det G, the ratio of the momentum's normal components (a step keeps the
        // phase-space flux through the layers), must not vanish; pn = pT |cn|
        bool ok = cn0 * cn0 * fmaf(f.q1, f.q1, f.q2 * f.q2) > 1e-12f * pn * pn;
        // Cp = Lc diag(dg) Lc^T (unit lower Lc, kept in cp's strict triangle)
        float idg[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            float dj = cp[pk(j, j)];
#pragma unroll
            for (int k = 0; k < j; ++k) dj = fmaf(-cp[pk(j, k)] * cp[pk(j, k)], cp[pk(k, k)], dj);
            ok = ok && dj > 0.0f;
            cp[pk(j, j)] = dj;
            idg[j] = __fdividef(1.0f, dj);
#pragma unroll
            for (int i = j + 1; i < 5; ++i) {
                float u = cp[pk(i, j)];
#pragma unroll
                for (int k = 0; k < j; ++k) u = fmaf(-cp[pk(i, k)] * cp[pk(k, k)], cp[pk(j, k)], u);
                cp[pk(i, j)] = u * idg[j];
            }
        }
        if (!ok) {  // no smoothing across this layer: keep the filtered estimate
            flags |= KF_FLAG_INVERSION_FAILED;
            p = f;
#pragma unroll
            for (int i = 0; i < 15; ++i) c[i] = cf[i];
        } else {
            // K = Q Cp^-1, rows q1, q2, pz: one solve per row
            const float tu = -t2 * q.q1, tv = -t2 * q.q2;
            const float q6[6] = {t2 * fmaf(q.q2, q.q2, q.pz * q.pz), tu * q.q2, t2 * fmaf(q.q1, q.q1, q.pz * q.pz),
                                 tu * q.pz, tv * q.pz, t2 * fmaf(q.q1, q.q1, q.q2 * q.q2)};
            float Kr[3][5];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                float w[5] = {0.0f, 0.0f, q6[k == 0 ? 0 : k == 1 ? 1 : 3], q6[k == 0 ? 1 : k == 1 ? 2 : 4],
                              q6[k == 0 ? 3 : k == 1 ? 4 : 5]};
#pragma unroll
                for (int i = 3; i < 5; ++i)
#pragma unroll
                    for (int j = 2; j < i; ++j) w[i] = fmaf(-cp[pk(i, j)], w[j], w[i]);
#pragma unroll
                for (int i = 2; i < 5; ++i) w[i] *= idg[i];
#pragma unroll
                for (int i = 3; i >= 0; --i)
#pragma unroll
                    for (int j = i + 1; j < 5; ++j) w[i] = fmaf(-cp[pk(j, i)], w[j], w[i]);
#pragma unroll
                for (int i = 0; i < 5; ++i) Kr[k][i] = w[i];
            }
            // state: d = (I - K) (xs' - xp), then the step back
            const float e0 = p.x - q.x, e1 = p.y - q.y;
            const float dl[5] = {fmaf(q.nx, e1, -q.ny * e0), p.z - q.z, p.q1 - q.q1, p.q2 - q.q2, p.pz - q.pz};
            float d[5] = {dl[0], dl[1], dl[2], dl[3], dl[4]};
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int j = 0; j < 5; ++j) d[2 + k] = fmaf(-Kr[k][j], dl[j], d[2 + k]);
            const float dt = fmaf(B.A0, d[0], fmaf(B.A1, d[2], B.A2 * d[3]));
            const float la = fmaf(B.L0, d[0], fmaf(B.L1, d[2], B.L2 * d[3]));
            // covariance: (I - K) (Cs' - Cp) (I - K)^T, then the step back.
            // Where layer l + 1 is crossed almost along its surface, t at layer
            // l is a small difference of large terms: its row is taken from
            // A's row a as a whole, u = D a (from (I - K) D (I - K)^T, whose
            // roundings B's entries scale, the t variance of a looper came out
            // 4% off).
            float ct[5];
            {
                float a[5], b[5], u[5];  // t = a . delta, lambda = b . delta
#pragma unroll
                for (int j = 0; j < 5; ++j) {
                    a[j] = fmaf(-B.A1, Kr[0][j], fmaf(-B.A2, Kr[1][j], j == 0 ? B.A0 : j == 2 ? B.A1 : j == 3 ? B.A2 : 0.0f));
                    b[j] = fmaf(-B.L1, Kr[0][j], fmaf(-B.L2, Kr[1][j], j == 0 ? B.L0 : j == 2 ? B.L1 : j == 3 ? B.L2 : 0.0f));
                }
                float ul = 0.0f;
                ct[0] = 0.0f;
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    u[i] = 0.0f;
#pragma unroll
                    for (int j = 0; j < 5; ++j) u[i] = fmaf(a[j], D[pk(i, j)], u[i]);
                    ct[0] = fmaf(a[i], u[i], ct[0]);
                    ul = fmaf(b[i], u[i], ul);
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    ct[2 + k] = u[2 + k];
#pragma unroll
                    for (int i = 0; i < 5; ++i) ct[2 + k] = fmaf(-Kr[k][i], u[i], ct[2 + k]);
                }
                ct[1] = fmaf(B.jp, ct[4], fmaf(B.lz, ul, u[1]));
                ct[2] = fmaf(B.W1, ul, ct[2]);
                ct[3] = fmaf(B.W2, ul, ct[3]);
            }
            float E[3][5];
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int j = 0; j < 5; ++j) {
                    float acc = 0.0f;
#pragma unroll
                    for (int i = 0; i < 5; ++i) acc = fmaf(Kr[k][i], D[pk(i, j)], acc);
                    E[k][j] = acc;
                }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
#pragma unroll
                for (int j = 0; j < 2; ++j) D[pk(2 + k, j)] -= E[k][j];
#pragma unroll
                for (int h = 0; h <= k; ++h) {
                    float acc = D[pk(2 + k, 2 + h)] - E[k][2 + h] - E[h][2 + k];
#pragma unroll
                    for (int i = 0; i < 5; ++i) acc = fmaf(E[k][i], Kr[h][i], acc);
                    D[pk(2 + k, 2 + h)] = acc;
                }
            }
            transport_local(B, D);
#pragma unroll
            for (int i = 0; i < 5; ++i) D[pk(i, 0)] = ct[i];
            p = Local{fmaf(-f.ny, dt, f.x),
                      fmaf(f.nx, dt, f.y),
                      f.z + fmaf(B.jp, d[4], fmaf(B.lz, la, d[1])),
                      f.q1 + fmaf(B.W1, la, d[2]),
                      f.q2 + fmaf(B.W2, la, d[3]),
                      f.pz + d[4],
                      f.f0,
                      f.f1,
                      f.nx,
                      f.ny};
#pragma unroll
            for (int i = 0; i < 15; ++i) c[i] = cf[i] + D[i];
        }
        write(l);
    }
    // layers not reached (and every layer of a track with a non-finite input)
    for (int l = K; l < L; ++l) {
#pragma unroll
        for (int i = 0; i < 6; ++i) os[(int64_t)(6 * l + i) * T] = NAN;
#pragma unroll
        for (int i = 0; i < 21; ++i) oc[(int64_t)(21 * l + i) * T] = NAN;
    }
    io.out_flags[t] = flags;
}

}  // namespace
}  // namespace kf

using namespace kf;

extern "C" int kf_smooth_tracks(kf_context *ctx, const kf_geometry *geom, int64_t n_tracks, const float *seed_state,
                                const float *seed_cov, const int8_t *charge, const float *hit_pos, const float *hit_cov,
                                const uint32_t *hit_mask, float *out_state, float *out_cov, int16_t *out_reached,
                                uint32_t *out_flags, const kf_options *opt, kf_stream stream_)
{
    if (!ctx) return KF_ERR_ARG;
    kf_options o;
    if (opt) o = *opt;
    else kf_options_default(&o);
    int rc;
    FitGeom g;
    if ((rc = check_geometry(ctx, geom, &g))) return rc;
    if ((rc = check_options(ctx, o))) return rc;
    if (n_tracks < 0 || n_tracks > (int64_t(1) << 36))
        return set_error(ctx, KF_ERR_ARG, "n_tracks %lld out of range", (long long)n_tracks);
    if (n_tracks == 0) return KF_OK;
    if ((rc = check_ptr(ctx, seed_state, 4, "seed_state")) || (rc = check_ptr(ctx, seed_cov, 4, "seed_cov")) ||
        (rc = check_ptr(ctx, charge, 1, "charge")) || (rc = check_ptr(ctx, hit_pos, 4, "hit_pos")) ||
        (rc = check_ptr(ctx, hit_cov, 4, "hit_cov")) || (rc = check_ptr(ctx, hit_mask, 4, "hit_mask")) ||
        (rc = check_ptr(ctx, out_state, 4, "out_state")) || (rc = check_ptr(ctx, out_cov, 4, "out_cov")) ||
        (rc = check_ptr(ctx, out_reached, 2, "out_reached")) || (rc = check_ptr(ctx, out_flags, 4, "out_flags")))
        return rc;
    DeviceGuard dg(context_device(ctx));
    SmoothIO io{n_tracks, seed_state, seed_cov, charge, hit_pos, hit_cov, hit_mask,
                out_state, out_cov, out_reached, out_flags};
    const unsigned blocks = (unsigned)((n_tracks + 127) / 128);
    smooth_kernel<<<blocks, 128, kSlotSize * 128 * sizeof(float), reinterpret_cast<cudaStream_t>(stream_)>>>(
        g, make_routing(o), io);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? KF_OK : cuda_error(ctx, e, "smoother launch");
}
