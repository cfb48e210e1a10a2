// Per-track Kalman-filter arithmetic in registers (Sections 2, 2.1 and 4.2 of
// arXiv:1705.02876): one thread owns one track, its position, momentum and the
// packed covariance c[15] of its local coordinates (from a seed, the Cartesian
// state x[6] and c[21]); every function below works on those registers.
//
// Packed symmetric storage: lower triangle row by row, index(i,j) = i(i+1)/2+j.
#pragma once

#include <stdint.h>

#include "kf.h"

namespace kf {

constexpr float kField = 0.00299792458f;  // GeV / (cm T)

__host__ __device__ constexpr int pk(int i, int j) { return i >= j ? i * (i + 1) / 2 + j : j * (j + 1) / 2 + i; }

// 0 * v is 0 for finite v and NaN otherwise
template <int N>
__device__ __forceinline__ bool all_finite(const float *v)
{
    float acc = 0.0f;
#pragma unroll
    for (int i = 0; i < N; ++i) acc = fmaf(0.0f, v[i], acc);
    return acc == 0.0f;
}

// Divisions on the FP32 path use __fdividef (reciprocal approximation and a
// multiply, within 2 ulp for divisors of magnitude 2^-126..2^126, which every
// divisor here is) in place of the IEEE-rounded sequence.

// Helix propagation to the first forward crossing of radius r (uniform field
// along z; transverse path length s, omega = q k Bz / pT).  Writing
// tau = tan(omega s / 2), the crossing condition |P(s)|^2 = r^2 is the
// quadratic  B' tau^2 + omega u tau - omega^2 D / 4 = 0  with
// u = P.t, w = P x t, D = r^2 - |P|^2, B' = 1 + omega w - omega^2 D / 4.
// Its roots are omega (-u +- sqrt(Q)) / (2 B'), Q = u^2 + D B'.  The root
// rationalised to tau = omega sigma / 2, sigma = D / (u + sqrt(Q)), stays
// exact as omega -> 0 (sigma is then the straight-line path length) and is
// the first crossing whenever u + sqrt(Q) > 0: for B' > 0 the other root lies
// beyond half a turn, for B' < 0 (a start past the circle's closest approach
// to the axis, crossing towards its farthest point) both roots share a sign
// and this one is the smaller.  sin and cos of the turning angle are rational
// in tau, so only one atan (for z) is evaluated.  A start moving inwards with
// u + sqrt(Q) <= 0 takes the general two-root path.  Returns false if the
// cylinder is not reached.
//
// crossing() solves for the turn of a start (x, y) moving along (tx, ty):
// the transverse path length s, and with the turning angle phi = om s
// a = sin(phi) / om, b = (1 - cos(phi)) / om, sn = sin(phi), c = cos(phi).
struct Turn {
    float s, a, b, sn, c;
};
__device__ __forceinline__ bool crossing(float x, float y, float tx, float ty, float om, float pt2, float r, Turn &t)
{
    const float u = fmaf(x, tx, y * ty);
    const float w = fmaf(x, ty, -y * tx);
    const float D = fmaf(r, r, -fmaf(x, x, y * y));
    const float Bp = fmaf(-0.25f * om * om, D, fmaf(om, w, 1.0f));
    const float Qd = fmaf(u, u, D * Bp);
    const float sq = sqrtf(Qd), den = u + sq;
    // one test for the common case: a missed cylinder (Qd < 0) or no transverse
    // momentum makes den NaN
    float sigma = __fdividef(D, den);
    float tau = 0.5f * om * sigma;
    const float t2 = tau * tau;
    float s;
    if (den > 0.0f && t2 < 0.0625f) {
        // atan(tau)/tau: its Taylor series sum_k (-t2)^k / (2k+1) to t2^6 for
        // |tau| < 1/4 (truncation below 3e-10)
        float ratio = fmaf(t2, -1.0f / 13.0f, 1.0f / 11.0f);
        ratio = fmaf(t2, -ratio, 1.0f / 9.0f);
        ratio = fmaf(t2, -ratio, 1.0f / 7.0f);
        ratio = fmaf(t2, -ratio, 1.0f / 5.0f);
        ratio = fmaf(t2, -ratio, 1.0f / 3.0f);
        ratio = fmaf(t2, -ratio, 1.0f);
        s = sigma * ratio;
    } else if (!(Qd >= 0.0f) || !(pt2 > 0.0f)) {
        return false;
    } else if (den > 0.0f) {
        s = sigma * (atanf(tau) / tau);  // a wide turn
    } else {
        // A start moving inwards: both roots of the quadratic, each mapped to
        // its smallest positive path length.
        if (om == 0.0f) return false;
        const float period = 6.283185307179586f / fabsf(om);
        float best = INFINITY;
        for (int sgn = -1; sgn <= 1; sgn += 2) {
            float phi;
            if (Bp != 0.0f) {
                const float tr = om * (-u + sgn * copysignf(sq, om)) / (2.0f * Bp);
                phi = 2.0f * atanf(tr);
            } else {
                phi = sgn < 0 ? 2.0f * atanf(om * D / (4.0f * u)) : copysignf(3.14159265358979f, om);
            }
            float sk = phi / om;
            if (sk <= 0.0f) sk += period;
            best = fminf(best, sk);
        }
        s = best;
        tau = tanf(0.5f * om * s);
        sigma = om != 0.0f ? 2.0f * tau / om : s;
        if (!(s < INFINITY)) return false;
    }
    const float g = __fdividef(1.0f, fmaf(tau, tau, 1.0f));
    t.s = s;
    t.a = sigma * g;
    t.b = sigma * tau * g;
    t.sn = 2.0f * tau * g;
    t.c = fmaf(-tau, t.sn, 1.0f);
    return true;
}

struct Routing {
    int mode;        // 0 FP32, 1 routed
    float det_min;   // 27 / (4 cond_max): the least det of S's correlation matrix done in FP32
    float pt_lo2, pt_hi2;  // squares of the pT bounds
    float gain_max;  // information-gain threshold: C_ii / V_ii above it routes the gain
};

// A track whose updates run in extended precision whatever its hits are.
__device__ __forceinline__ bool outside_pt(float pt2, const Routing &rt)
{
    return rt.mode == 1 && (pt2 < rt.pt_lo2 || pt2 > rt.pt_hi2);
}

// What a fit that puts such tracks off (DEFER below) gets in place of flags.
constexpr uint32_t kPutOff = 0x80000000u;

// The extended-precision paths are out of line and rare.  A non-inlined
// function's registers count towards the kernel's allocation, so these work
// from a per-thread slot of shared memory ([kSlotSize][stride] floats,
// thread-major so that a warp's accesses hit distinct banks), reading and
// writing the covariance one row at a time: the kernel keeps the register
// budget of the FP32 main path.
constexpr int kSlotX = 0, kSlotC = 6, kSlotM = 27, kSlotV = 30, kSlotChi2 = 36, kSlotSize = 37;
constexpr int kSlotFrame = kSlotC + 15;  // f0, f1, nx, ny

struct SlotRef {
    float *p;
    int stride;
    __device__ __forceinline__ float &x(int i) const { return p[(kSlotX + i) * stride]; }
    __device__ __forceinline__ float &c(int i, int j) const { return p[(kSlotC + pk(i, j)) * stride]; }
    __device__ __forceinline__ float &m(int i) const { return p[(kSlotM + i) * stride]; }
    __device__ __forceinline__ float &v(int i) const { return p[(kSlotV + i) * stride]; }
    __device__ __forceinline__ float &chi2() const { return p[kSlotChi2 * stride]; }
    __device__ __forceinline__ float n(int i) const { return p[(kSlotFrame + 2 + i) * stride]; }
};

// The slow paths work in the same local coordinates as the FP32 update
// (below): n = (x, y)/|(x, y)| at the predicted position, t = z x n; the slot
// holds the position, the momentum (q1, q2, pz), the 15 floats of the local
// covariance, packed over u = 0 t, 1 z, 2 q1, 3 q2, 4 pz, and the frame's n.

// C_l -= K C_l[{t, z}, :] in place on the slot's local block, row u's gain
// (kt[u], kz[u]) against the original t and z columns: rows and, within a
// row, columns descending read only entries not yet rewritten, except the
// original (z, t) entry, kept for row t.
template <class R>
__device__ __forceinline__ void slot_local_downdate(const SlotRef &sl, const R kt[5], const R kz[5])
{
    float *c = sl.p + kSlotC * sl.stride;
    auto C = [&](int i, int j) -> float & { return c[pk(i, j) * sl.stride]; };
    const R zt = (R)C(1, 0);
#pragma unroll 1
    for (int u = 4; u >= 0; --u)
#pragma unroll 1
        for (int w = u; w >= 0; --w) {
            const R ctw = (R)C(w, 0);
            const R czw = w > 0 ? (R)C(w, 1) : u > 0 ? (R)C(1, 0) : zt;
            C(u, w) = (float)((R)C(u, w) - (kt[u] * ctw + kz[u] * czw));
        }
}

// The update in FP64 on the slot: the factorisation and the two scalar
// updates of update_local (below); then the PSD repair: a variance that
// cancellation drove to zero or below is clamped to 1e-12 of the trace
// (correlations are left alone).  Returns 2, 3 (repaired) or 1 (S not positive
// definite).  The FP64 pipe takes a warp instruction every 16 cycles of the SM,
// so the form with the fewest of them is used: some 130 and the conversions
// (an adjugate of S, and a gain with three columns, needed about 250).
static __device__ __noinline__ int update_fp64(float *slot_p, int stride)
{
    const SlotRef sl{slot_p, stride};
    double nx = sl.n(0), ny = sl.n(1);
    {  // the frame's n, normalised to FP64 (one Newton step)
        const double h = fma(-0.5, fma(nx, nx, ny * ny), 1.5);
        nx *= h;
        ny *= h;
    }
    double vt, vz, l, ia, it, iz;
    {
        const double v0 = sl.v(0), v1 = sl.v(1), v2 = sl.v(2), v3 = sl.v(3), v4 = sl.v(4);
        const double nn = nx * nx, tt = ny * ny, nt = nx * ny;
        const double vnn = fma(nn, v0, fma(2.0 * nt, v1, tt * v2));
        const double vnt = fma(nt, v2 - v0, (nn - tt) * v1);
        const double vtt = fma(tt, v0, fma(-2.0 * nt, v1, nn * v2));
        const double vnz = fma(nx, v3, ny * v4), vtz = fma(nx, v4, -ny * v3);
        ia = 1.0 / vnn;
        vt = vnt * ia;
        vz = vnz * ia;
        const double dt = fma(-vnt, vt, (double)sl.c(0, 0) + vtt);
        it = 1.0 / dt;
        const double e = fma(-vnt, vz, (double)sl.c(1, 0) + vtz);
        l = e * it;
        const double dz = fma(-l, e, fma(-vnz, vz, (double)sl.c(1, 1) + (double)sl.v(5)));
        if (!(vnn > 0.0 && dt > 0.0 && dz > 0.0 && dz < INFINITY)) return 1;
        iz = 1.0 / dz;
    }
    const double X0 = sl.x(0), X1 = sl.x(1);
    const double d0 = (double)sl.m(0) - X0, d1 = (double)sl.m(1) - X1;
    const double rn = fma(nx, d0, ny * d1);
    const double r1 = fma(-vt, rn, fma(nx, d1, -ny * d0));
    const double r2 = fma(-l, r1, fma(-vz, rn, (double)sl.m(2) - (double)sl.x(2)));
    const double w1 = r1 * it, w2 = r2 * iz;
    sl.chi2() = (float)fma(rn * rn, ia, fma(r1, w1, r2 * w2));
    const double b0 = fma(-l, (double)sl.c(0, 0), (double)sl.c(1, 0));
    // rows descending and, in a row, columns descending read only entries not
    // yet rewritten (b0 is kept); rolled, for the callers' registers
#pragma unroll 1
    for (int u = 4; u >= 0; --u) {
        const double a = sl.c(u, 0), b = u ? fma(-l, a, (double)sl.c(u, 1)) : b0;
        const double dx = fma(a, w1, b * w2);
        if (u == 0) {
            sl.x(0) = (float)fma(-ny, dx, X0);
            sl.x(1) = (float)fma(nx, dx, X1);
        } else {
            sl.x(u + 1) = (float)((double)sl.x(u + 1) + dx);
        }
        const double ka = -a * it, kb = -b * iz;
#pragma unroll 1
        for (int w = u; w >= 0; --w) {
            const double aw = sl.c(w, 0), bw = w ? fma(-l, aw, (double)sl.c(w, 1)) : b0;
            sl.c(u, w) = (float)fma(ka, aw, fma(kb, bw, (double)sl.c(u, w)));
        }
    }
    float tr = 0.0f;
    bool rep = false;
#pragma unroll
    for (int u = 0; u < 5; ++u) {
        tr += fabsf(sl.c(u, u));
        rep = rep || !(sl.c(u, u) > 0.0f);
    }
    if (!rep) return 2;
#pragma unroll 1
    for (int u = 0; u < 5; ++u)
        if (!(sl.c(u, u) > 0.0f)) sl.c(u, u) = 1e-12f * tr;
    return 3;
}

// Float-float arithmetic: a value is hi + lo with |lo| <= ulp(hi)/2, about 48
// significant bits carried on the FP32 pipe.  Error-free transformations
// (Knuth's two-sum, Dekker's fast two-sum, the FMA two-product) use the _rn
// intrinsics, which the compiler never contracts or reassociates.
struct ff {
    float hi, lo;
};
__device__ __forceinline__ ff two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ ff fast_two_sum(float a, float b)  // |a| >= |b|
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ ff two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ ff ff_add(ff x, ff y)
{
    const ff s = two_sum(x.hi, y.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo)));
}
__device__ __forceinline__ ff ff_mul(ff x, ff y)
{
    const ff p = two_prod(x.hi, y.hi);
    return fast_two_sum(p.hi, __fmaf_rn(x.hi, y.lo, __fmaf_rn(x.lo, y.hi, p.lo)));
}
__device__ __forceinline__ ff ff_neg(ff x) { return {-x.hi, -x.lo}; }
// a*b - c*d for float-float operands
__device__ __forceinline__ ff ff_det2(ff a, ff b, ff c, ff d) { return ff_add(ff_mul(a, b), ff_neg(ff_mul(c, d))); }
// sum_k s_k * c_k with float-float s and plain float c, accurate to float-float
__device__ __forceinline__ ff ff_dot3(ff s0, ff s1, ff s2, float c0, float c1, float c2)
{
    const ff p0 = two_prod(s0.hi, c0), p1 = two_prod(s1.hi, c1), p2 = two_prod(s2.hi, c2);
    const ff t0 = two_sum(p0.hi, p1.hi);
    const ff t1 = two_sum(t0.hi, p2.hi);
    float err = __fadd_rn(__fadd_rn(p0.lo, p1.lo), __fadd_rn(p2.lo, __fadd_rn(t0.lo, t1.lo)));
    err = __fmaf_rn(s0.lo, c0, __fmaf_rn(s1.lo, c1, __fmaf_rn(s2.lo, c2, err)));
    return fast_two_sum(t1.hi, err);
}

// Update on the slot with the gain formed in float-float, in the local frame
// of update_fp64: S (n, t, z) from the FP32 local entries (the entries that
// add C and V exact two-sums), S^-1 by adjugate / determinant, the gain's rows
// (C_ut, C_uz) S^-1 rounded to FP32, x += K r and C -= K C[{t, z}, :] in FP32;
// chi2 = r^T S^-1 r.  Returns 2, or 1 if S is not positive definite.
static __device__ __noinline__ int update_ff(float *slot_p, int stride)
{
    const SlotRef sl{slot_p, stride};
    const float X0 = sl.x(0), X1 = sl.x(1);
    const float nx = sl.n(0), ny = sl.n(1);
    auto L = [&](int i, int j) -> float & { return sl.c(i, j); };
    const float v0 = sl.v(0), v1 = sl.v(1), v2 = sl.v(2), v3 = sl.v(3), v4 = sl.v(4);
    const ff a{fmaf(nx * nx, v0, fmaf(2.0f * nx * ny, v1, ny * ny * v2)), 0.0f};
    const ff b{fmaf(nx * ny, v2 - v0, (nx * nx - ny * ny) * v1), 0.0f};
    const ff d{fmaf(nx, v3, ny * v4), 0.0f};
    const ff cc = two_sum(L(0, 0), fmaf(ny * ny, v0, fmaf(-2.0f * nx * ny, v1, nx * nx * v2)));
    const ff e = two_sum(L(1, 0), fmaf(nx, v4, -ny * v3)), f = two_sum(L(1, 1), sl.v(5));
    const ff i00 = ff_det2(cc, f, e, e), i10 = ff_det2(d, e, b, f), i11 = ff_det2(a, f, d, d);
    const ff i20 = ff_det2(b, e, cc, d), i21 = ff_det2(b, d, a, e), i22 = ff_det2(a, cc, b, b);
    const ff det = ff_add(ff_mul(a, i00), ff_add(ff_mul(b, i10), ff_mul(d, i20)));
    if (!(a.hi > 0.0f) || !(i22.hi > 0.0f) || !(det.hi > 0.0f)) return 1;
    // 1/det: one Newton step on the FP32 reciprocal, r + r (1 - det r)
    const float rc = 1.0f / det.hi;
    const ff one_minus = ff_add(ff{1.0f, 0.0f}, ff_neg(ff_mul(det, ff{rc, 0.0f})));
    const ff id = ff_add(ff{rc, 0.0f}, ff_mul(one_minus, ff{rc, 0.0f}));
    const ff s00 = ff_mul(i00, id), s10 = ff_mul(i10, id), s11 = ff_mul(i11, id);
    const ff s20 = ff_mul(i20, id), s21 = ff_mul(i21, id), s22 = ff_mul(i22, id);
    const float d0 = sl.m(0) - X0, d1 = sl.m(1) - X1;
    const ff rn = two_sum(nx * d0, ny * d1), rt = two_sum(nx * d1, -ny * d0), rz = two_sum(sl.m(2), -sl.x(2));
    const ff q0 = ff_add(ff_mul(s00, rn), ff_add(ff_mul(s10, rt), ff_mul(s20, rz)));
    const ff q1 = ff_add(ff_mul(s10, rn), ff_add(ff_mul(s11, rt), ff_mul(s21, rz)));
    const ff q2 = ff_add(ff_mul(s20, rn), ff_add(ff_mul(s21, rt), ff_mul(s22, rz)));
    const ff chi = ff_add(ff_mul(rn, q0), ff_add(ff_mul(rt, q1), ff_mul(rz, q2)));
    sl.chi2() = __fadd_rn(chi.hi, chi.lo);
    const float rrn = __fadd_rn(rn.hi, rn.lo), rrt = __fadd_rn(rt.hi, rt.lo), rrz = __fadd_rn(rz.hi, rz.lo);
    const ff zero{0.0f, 0.0f};
    float kt[5], kz[5];
    for (int u = 0; u < 5; ++u) {
        const float ct = L(u, 0), cz = L(u, 1);
        const ff knf = ff_dot3(s10, s20, zero, ct, cz, 0.0f);
        const ff ktf = ff_dot3(s11, s21, zero, ct, cz, 0.0f);
        const ff kzf = ff_dot3(s21, s22, zero, ct, cz, 0.0f);
        kt[u] = __fadd_rn(ktf.hi, ktf.lo);
        kz[u] = __fadd_rn(kzf.hi, kzf.lo);
        const float dx = fmaf(__fadd_rn(knf.hi, knf.lo), rrn, fmaf(kt[u], rrt, kz[u] * rrz));
        if (u == 0) {
            sl.x(0) = fmaf(-ny, dx, X0);
            sl.x(1) = fmaf(nx, dx, X1);
        } else {
            sl.x(u + 1) += dx;
        }
    }
    slot_local_downdate<float>(sl, kt, kz);
    return 2;
}

// The whole update in float-float: update_fp64 to some 2^-45 of its terms
// instead of 2^-52.  What a hit leaves of a variance C is about V: a result is
// off by 2^-45 C / V of itself, so that with C below kWideGain V (and S well
// conditioned, the caller's test) the FP32 results are those of the FP64 update
// but for rounding ties.  Some 1,100 FP32 instructions, about a tenth of the
// time of the FP64 pipe's 280.  Returns as update_fp64 does, or 0 with nothing
// written where C is larger.
constexpr float kWideGain = 1048576.0f;  // 2^20: 2^-25, half an FP32 half-ulp
__device__ __forceinline__ ff ff_sub(ff x, ff y) { return ff_add(x, ff_neg(y)); }
__device__ __forceinline__ ff ff_addf(ff x, float y)
{
    const ff s = two_sum(x.hi, y);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, x.lo));
}
__device__ __forceinline__ ff ff_mulf(ff x, float y)
{
    const ff p = two_prod(x.hi, y);
    return fast_two_sum(p.hi, __fmaf_rn(x.lo, y, p.lo));
}
__device__ __forceinline__ ff ff_rcp(ff x)  // Newton from the FP32 reciprocal r: r (1 + e + e^2), e = 1 - x r
{
    const float r = __fdividef(1.0f, x.hi);
    const float e = __fmaf_rn(-x.lo, r, __fmaf_rn(-x.hi, r, 1.0f));
    return fast_two_sum(r, __fmul_rn(r, __fmaf_rn(e, e, e)));
}
__device__ __forceinline__ float ff_round(ff x, float y) { return ff_addf(x, y).hi; }  // x + y to FP32

static __device__ __noinline__ int update_wide(float *slot_p, int stride)
{
    const SlotRef sl{slot_p, stride};
    ff nx{sl.n(0), 0.0f}, ny{sl.n(1), 0.0f};
    {  // the frame's n, normalised (one Newton step)
        const ff a = two_prod(nx.hi, nx.hi), b = two_prod(ny.hi, ny.hi);
        const ff s = ff_addf(ff_add(a, b), -1.0f);
        const float h = -0.5f * s.hi;
        nx = fast_two_sum(nx.hi, __fmul_rn(nx.hi, h));
        ny = fast_two_sum(ny.hi, __fmul_rn(ny.hi, h));
    }
    ff vt, vz, l, ia, it, iz;
    {
        const float v0 = sl.v(0), v1 = sl.v(1), v2 = sl.v(2), v3 = sl.v(3), v4 = sl.v(4);
        const ff nn = ff_mul(nx, nx), tt = ff_mul(ny, ny), nt = ff_mul(nx, ny);
        const ff x2 = ff_mulf(nt, 2.0f * v1);
        const ff vnn = ff_add(ff_add(ff_mulf(nn, v0), ff_mulf(tt, v2)), x2);
        const ff vnt = ff_add(ff_mul(nt, two_sum(v2, -v0)), ff_mulf(ff_sub(nn, tt), v1));
        const ff vtt = ff_sub(ff_add(ff_mulf(tt, v0), ff_mulf(nn, v2)), x2);
        const ff vnz = ff_add(ff_mulf(nx, v3), ff_mulf(ny, v4)), vtz = ff_sub(ff_mulf(nx, v4), ff_mulf(ny, v3));
        ia = ff_rcp(vnn);
        vt = ff_mul(vnt, ia);
        vz = ff_mul(vnz, ia);
        // V given n, and what C adds
        const ff ut = ff_sub(vtt, ff_mul(vnt, vt)), uz = ff_sub(vtz, ff_mul(vnt, vz));
        const ff dt = ff_addf(ut, sl.c(0, 0));
        it = ff_rcp(dt);
        const ff e = ff_addf(uz, sl.c(1, 0));
        l = ff_mul(e, it);
        const ff dz = ff_sub(ff_sub(two_sum(sl.c(1, 1), sl.v(5)), ff_mul(vnz, vz)), ff_mul(l, e));
        iz = ff_rcp(dz);
        if (!(vnn.hi > 0.0f && dt.hi > 0.0f && dz.hi > 0.0f && dz.hi < INFINITY)) return 1;
        // V's z pivot, given n and t
        const float uzz = fmaf(-__fdividef(uz.hi, ut.hi), uz.hi, fmaf(-vnz.hi, vz.hi, sl.v(5)));
        if (!(sl.c(0, 0) < kWideGain * ut.hi && sl.c(1, 1) < kWideGain * uzz)) return 0;
    }
    const float X0 = sl.x(0), X1 = sl.x(1), X2 = sl.x(2);
    ff w1, w2;
    {
        const ff d0 = two_sum(sl.m(0), -X0), d1 = two_sum(sl.m(1), -X1);
        const ff rn = ff_add(ff_mul(nx, d0), ff_mul(ny, d1));
        const ff r1 = ff_sub(ff_sub(ff_mul(nx, d1), ff_mul(ny, d0)), ff_mul(vt, rn));
        const ff r2 = ff_sub(ff_sub(two_sum(sl.m(2), -X2), ff_mul(vz, rn)), ff_mul(l, r1));
        w1 = ff_mul(r1, it);
        w2 = ff_mul(r2, iz);
        const ff chi = ff_add(ff_mul(ff_mul(rn, rn), ia), ff_add(ff_mul(r1, w1), ff_mul(r2, w2)));
        sl.chi2() = __fadd_rn(chi.hi, chi.lo);
    }
    float a[5];
    ff b[5];
#pragma unroll
    for (int u = 0; u < 5; ++u) {
        a[u] = sl.c(u, 0);
        b[u] = ff_addf(ff_neg(ff_mulf(l, a[u])), sl.c(u, 1));
        const ff dx = ff_add(ff_mulf(w1, a[u]), ff_mul(b[u], w2));
        if (u == 0) {
            sl.x(0) = ff_round(ff_neg(ff_mul(ny, dx)), X0);
            sl.x(1) = ff_round(ff_mul(nx, dx), X1);
        } else {
            sl.x(u + 1) = ff_round(dx, u == 1 ? X2 : sl.x(u + 1));
        }
    }
    float tr = 0.0f;
    bool rep = false;
#pragma unroll
    for (int u = 0; u < 5; ++u) {
        const ff ka = ff_mulf(it, -a[u]), kb = ff_mul(ff_neg(b[u]), iz);
#pragma unroll
        for (int w = 0; w <= u; ++w) {
            const ff p = two_prod(ka.hi, a[w]), q = two_prod(kb.hi, b[w].hi);
            const ff s = two_sum(sl.c(u, w), p.hi), t = two_sum(s.hi, q.hi);
            const float lo = __fadd_rn(__fadd_rn(s.lo, t.lo), __fadd_rn(__fmaf_rn(ka.lo, a[w], p.lo),
                                                                        __fmaf_rn(kb.hi, b[w].lo, __fmaf_rn(kb.lo, b[w].hi, q.lo))));
            const float v = __fadd_rn(t.hi, lo);
            sl.c(u, w) = v;
            if (u == w) {
                tr += fabsf(v);
                rep = rep || !(v > 0.0f);
            }
        }
    }
    if (!rep) return 2;
#pragma unroll 1
    for (int u = 0; u < 5; ++u)
        if (!(sl.c(u, u) > 0.0f)) sl.c(u, u) = 1e-12f * tr;
    return 3;
}

static __device__ __noinline__ int update_ext(float *slot, int stride, int kind)
{
    if (kind == 3) {
        const int st = update_wide(slot, stride);
        if (st) return st;
        kind = 2;
    }
    return kind == 2 ? update_fp64(slot, stride) : update_ff(slot, stride);
}

// ---------------------------------------------------------------------------
// The filter on the covariance of a track's local coordinates.  On a
// cylinder the crossing cannot move along the radial direction, so the
// covariance has five dimensions, not six: (t, z, q1, q2, pz), the position
// along t = z x n and along z, and the momentum.  The transverse momentum is
// kept in a frame that turns with the track: p = F (q1, q2), F the rotation
// (f0, -f1; f1, f0).  F is turned by the angle the helix turns the momentum
// by, so q1 and q2 do not change along a helix and the Jacobian from one layer
// to the next is the identity but for one row and a rank-one term:
//   lambda = L . (dt, dq1, dq2)   (the turning angle's change over omega)
//   t'     = A . (dt, dq1, dq2)
//   z'     = z + jp pz + lz lambda,  q' = q + W lambda,  pz' = pz,
// with that, e the unit direction and its left normal before the step, that',
// e' after it, n0, t0 and n1 the layers' frames, cn = n1 . that',
// se = n1 . e', W = omega (q2, -q1), jp = s / pT, lz = pz / pT,
//   A0 = (that' . n0) / cn,  (A1, A2) = (b that + a e) / (pT cn),
//   L0 = -(n1 . t0) / cn,    (L1, L2) = -((a + b k) that + (a k - b) e) / pT, k = se / cn
// (that and e in the turning frame: (q1, q2) / pT and (-q2, q1) / pT); the
// terms in s of the Cartesian Jacobian cancel.  The transport is 67 FP32
// instructions (178 on the Cartesian block structure), its Jacobian some 30
// (90), and the update needs no rotation in and out.  F starts along the
// momentum: the covariance of a stiff track is wide along it (curvature) and
// narrow across, and entries that mix the two would carry the rounding of the
// wide one.  Every sum of products below is written with fmaf, so that the
// rounding does not depend on what the code is inlined into.
struct Local {
    float x, y, z, q1, q2, pz;  // position and momentum, p = F (q1, q2)
    float f0, f1;               // F: cosine and sine
    float nx, ny;               // n of the last layer reached
};
// Packed local covariance: index pk(i, j) over 0 t, 1 z, 2 q1, 3 q2, 4 pz.

struct LocalJac {
    float A0, A1, A2, L0, L1, L2, W1, W2, jp, lz;
};

// Step to radius r = 1 / inv_r.  0 and the new position, frames, Jacobian and
// pn = |p . n| there; or, with p as it was, KF_FLAG_UNREACHABLE, or
// KF_FLAG_LEFT_BARREL when the crossing lies beyond z_half.
// With B, the Jacobian of the step back too: the same formulas from n1 to n0
// by the angle -phi (an inverse of J itself loses its digits near a tangential
// crossing), and cn_start = n0 . that.
__device__ __forceinline__ uint32_t step_local(Local &p, float qkb, float r, float inv_r, float z_half, LocalJac &J,
                                               float &pn, LocalJac *B = nullptr, float *cn_start = nullptr)
{
    const float pt2 = fmaf(p.q1, p.q1, p.q2 * p.q2);
    const float ipt = rsqrtf(pt2);
    const float om = qkb * ipt;
    const float tx = fmaf(p.f0, p.q1, -p.f1 * p.q2) * ipt, ty = fmaf(p.f1, p.q1, p.f0 * p.q2) * ipt;
    Turn t;
    if (!crossing(p.x, p.y, tx, ty, om, pt2, r, t)) return KF_FLAG_UNREACHABLE;
    J.jp = t.s * ipt;
    const float z = fmaf(p.pz, J.jp, p.z);
    if (fabsf(z) > z_half) return KF_FLAG_LEFT_BARREL;
    p.z = z;
    p.x += fmaf(tx, t.a, ty * t.b);
    p.y += fmaf(ty, t.a, -tx * t.b);
    const float ux = fmaf(tx, t.c, ty * t.sn), uy = fmaf(ty, t.c, -tx * t.sn);  // that'
    const float g0 = fmaf(p.f0, t.c, p.f1 * t.sn);
    p.f1 = fmaf(p.f1, t.c, -p.f0 * t.sn);
    p.f0 = g0;
    const float nx = p.x * inv_r, ny = p.y * inv_r;
    if (B) {
        const float cn0 = fmaf(p.nx, tx, p.ny * ty), se0 = fmaf(p.ny, tx, -p.nx * ty);
        const float icn0 = __fdividef(1.0f, cn0), i2 = ipt * ipt, k = se0 * icn0;
        const float al = -i2 * fmaf(t.b, k, -t.a), be = i2 * fmaf(t.a, k, t.b);
        const float ga = i2 * icn0 * t.b, de = -i2 * icn0 * t.a;
        *B = LocalJac{fmaf(tx, nx, ty * ny) * icn0, fmaf(ga, p.q1, -de * p.q2), fmaf(ga, p.q2, de * p.q1),
                      fmaf(p.nx, ny, -p.ny * nx) * icn0, fmaf(al, p.q1, -be * p.q2), fmaf(al, p.q2, be * p.q1),
                      om * p.q2, -om * p.q1, -J.jp, p.pz * ipt};
        *cn_start = cn0;
    }
    const float cn = fmaf(nx, ux, ny * uy), se = fmaf(ny, ux, -nx * uy);
    const float icn = __fdividef(1.0f, cn);
    J.A0 = fmaf(ux, p.nx, uy * p.ny) * icn;
    J.L0 = fmaf(nx, p.ny, -ny * p.nx) * icn;
    p.nx = nx;
    p.ny = ny;
    const float i2 = ipt * ipt, k = se * icn;
    const float al = -i2 * fmaf(t.b, k, t.a), be = i2 * fmaf(-t.a, k, t.b);
    J.L1 = fmaf(al, p.q1, -be * p.q2);
    J.L2 = fmaf(al, p.q2, be * p.q1);
    const float ga = i2 * icn * t.b, de = i2 * icn * t.a;
    J.A1 = fmaf(ga, p.q1, -de * p.q2);
    J.A2 = fmaf(ga, p.q2, de * p.q1);
    J.W1 = om * p.q2;
    J.W2 = -om * p.q1;
    J.lz = p.pz * ipt;
    pn = fabsf(cn) * pt2 * ipt;
    return 0u;
}

// c <- J c J^T
__device__ __forceinline__ void transport_local(const LocalJac &J, float c[15])
{
    constexpr int T = 0, Z = 1, U = 2, V = 3, P = 4;
    auto row = [&](float a0, float a1, float a2, int i) {
        return fmaf(a0, c[pk(T, i)], fmaf(a1, c[pk(U, i)], a2 * c[pk(V, i)]));
    };
    // covariances of lambda and of t' with the old coordinates
    const float lt = row(J.L0, J.L1, J.L2, T), lz = row(J.L0, J.L1, J.L2, Z), lu = row(J.L0, J.L1, J.L2, U);
    const float lv = row(J.L0, J.L1, J.L2, V), lp = row(J.L0, J.L1, J.L2, P);
    const float at = row(J.A0, J.A1, J.A2, T), az = row(J.A0, J.A1, J.A2, Z), au = row(J.A0, J.A1, J.A2, U);
    const float av = row(J.A0, J.A1, J.A2, V), ap = row(J.A0, J.A1, J.A2, P);
    const float ll = fmaf(J.L0, lt, fmaf(J.L1, lu, J.L2 * lv));
    const float tl = fmaf(J.A0, lt, fmaf(J.A1, lu, J.A2 * lv));
    c[pk(T, T)] = fmaf(J.A0, at, fmaf(J.A1, au, J.A2 * av));
    c[pk(U, T)] = fmaf(J.W1, tl, au);
    c[pk(V, T)] = fmaf(J.W2, tl, av);
    c[pk(P, T)] = ap;
    c[pk(Z, T)] = fmaf(J.jp, ap, fmaf(J.lz, tl, az));
    // y = z + jp pz, then z' = y + lz lambda
    const float yp = fmaf(J.jp, c[pk(P, P)], c[pk(P, Z)]);
    const float yl = fmaf(J.jp, lp, lz), zl = fmaf(J.lz, ll, yl);
    const float yy = fmaf(J.jp, c[pk(P, Z)] + yp, c[pk(Z, Z)]);
    c[pk(Z, Z)] = fmaf(J.lz, yl + zl, yy);
    c[pk(U, Z)] = fmaf(J.jp, c[pk(P, U)], fmaf(J.lz, lu, fmaf(J.W1, zl, c[pk(U, Z)])));
    c[pk(V, Z)] = fmaf(J.jp, c[pk(P, V)], fmaf(J.lz, lv, fmaf(J.W2, zl, c[pk(V, Z)])));
    c[pk(P, Z)] = fmaf(J.lz, lp, yp);
    const float u1 = fmaf(J.W1, ll, lu), v1 = fmaf(J.W2, ll, lv);  // of lambda with q'
    c[pk(U, U)] = fmaf(J.W1, lu + u1, c[pk(U, U)]);
    c[pk(V, U)] = fmaf(J.W2, lu, fmaf(J.W1, v1, c[pk(V, U)]));
    c[pk(V, V)] = fmaf(J.W2, lv + v1, c[pk(V, V)]);
    c[pk(P, U)] = fmaf(J.W1, lp, c[pk(P, U)]);
    c[pk(P, V)] = fmaf(J.W2, lp, c[pk(P, V)]);
}

// The bending plane's block of enter_local (tt, q2 t, q2 q2) in float-float, on
// the slot: the covariance of (x, y, px, py), packed, then the rows t and q2
// over them; the block is left at the slot's start.
static __device__ __noinline__ void enter_wide(float *s, int stride)
{
    auto dot = [&](const ff m[4], int row) {  // the row . m
        ff p[4];
        float lo = 0.0f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float v = s[(row + j) * stride];
            p[j] = two_prod(m[j].hi, v);
            lo = __fadd_rn(lo, __fmaf_rn(m[j].lo, v, p[j].lo));
        }
        const ff a = two_sum(p[0].hi, p[1].hi), b = two_sum(a.hi, p[2].hi), c = two_sum(b.hi, p[3].hi);
        return two_sum(c.hi, __fadd_rn(lo, __fadd_rn(a.lo, __fadd_rn(b.lo, c.lo))));
    };
    constexpr int T = 10, Q = 14;
    float out[3];
#pragma unroll 1
    for (int row = T; row <= Q; row += Q - T) {
        ff m[4];  // the row times the covariance
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const ff col[4] = {{s[pk(0, i) * stride], 0.0f}, {s[pk(1, i) * stride], 0.0f},
                               {s[pk(2, i) * stride], 0.0f}, {s[pk(3, i) * stride], 0.0f}};
            m[i] = dot(col, row);
        }
        if (row == T) out[0] = dot(m, T).hi;
        out[row == T ? 1 : 2] = dot(m, Q).hi;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) s[i * stride] = out[i];
}

// The step from a start anywhere (a seed) with a full 6x6 covariance onto the
// first layer; the turning frame starts along the seed's momentum.  Returns as
// step_local does.  The rows of the Jacobian are those of LocalJac with a
// displacement (dx, dy) in place of the start's dt (lambda = -n1 . (dx, dy) / cn
// + ..., t' = that' x (dx, dy) / cn + ...), on the Cartesian coordinates, so that
// an entry of the local covariance comes from the seed's in one pass.
// A hit after a seed shrinks q2's variance to what t leaves of it, a small
// difference of the bending plane's three entries: their sums run from the
// positions' terms to the momenta's, which exceed them, and are in float-float
// for a track outside the pT bounds, whose updates are too.  (Through the 6x6
// covariance on the layer, rotated, an entry had some ten roundings.  Error of
// the fitted covariance against 64 bits, five hits, pT 0.5 to 10 GeV: 11.6e-6,
// now 9.3e-6; pT 0.24 to 500 GeV: 6.0e-4, with the sums alone 4.7e-4, now
// 3.9e-4; three hits 3.9e-4, 3.0e-4, 2.5e-4.)
// DEFER: kPutOff for such a track, which is left where it was.
template <bool DEFER = false>
__device__ __forceinline__ uint32_t enter_local(const float x[6], const float c6[21], float qkb, float r, float inv_r,
                                                float z_half, const Routing &rt, float *slot, int stride, Local &p,
                                                float c[15], float &pn)
{
    const float pt2 = fmaf(x[3], x[3], x[4] * x[4]);
    const float ipt = rsqrtf(pt2);
    const float om = qkb * ipt;
    const float tx = x[3] * ipt, ty = x[4] * ipt;
    Turn t;
    if (!crossing(x[0], x[1], tx, ty, om, pt2, r, t)) return KF_FLAG_UNREACHABLE;
    const float jp = t.s * ipt;
    const float z1 = fmaf(x[5], jp, x[2]);
    if (fabsf(z1) > z_half) return KF_FLAG_LEFT_BARREL;
    const bool wide = outside_pt(pt2, rt);
    if (DEFER && wide) return kPutOff;
    const float x1 = x[0] + fmaf(tx, t.a, ty * t.b), y1 = x[1] + fmaf(ty, t.a, -tx * t.b);
    const float ux = fmaf(tx, t.c, ty * t.sn), uy = fmaf(ty, t.c, -tx * t.sn);  // that'
    const float nx = x1 * inv_r, ny = y1 * inv_r;
    const float cn = fmaf(nx, ux, ny * uy), se = fmaf(ny, ux, -nx * uy);
    const float icn = __fdividef(1.0f, cn), k = se * icn;
    const float lx = -nx * icn, ly = -ny * icn;
    const float l1 = -ipt * fmaf(t.b, k, t.a), l2 = -ipt * fmaf(t.a, k, -t.b);
    const float a1 = ipt * icn * t.b, a2 = ipt * icn * t.a;
    const float l3 = fmaf(l1, tx, -l2 * ty), l4 = fmaf(l1, ty, l2 * tx);
    const float lz = x[5] * ipt;
    // rows over (x, y, px, py): t, q2 and z (which has 1 for z and jp for pz
    // too); q1's is (tx, ty) over (px, py)
    const float T[4] = {-uy * icn, ux * icn, fmaf(a1, tx, -a2 * ty), fmaf(a1, ty, a2 * tx)};
    const float Q[4] = {-qkb * lx, -qkb * ly, fmaf(-qkb, l3, -ty), fmaf(-qkb, l4, tx)};
    const float Z[4] = {lz * lx, lz * ly, lz * l3, lz * l4};
    auto row4 = [&](const float *v, int j) {
        return fmaf(v[3], c6[pk(4, j)], fmaf(v[2], c6[pk(3, j)], fmaf(v[1], c6[pk(1, j)], v[0] * c6[pk(0, j)])));
    };
    float tc[6], zc[6], uc[6], vc[6];  // the rows times the covariance
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        tc[j] = row4(T, j);
        zc[j] = fmaf(jp, c6[pk(5, j)], c6[pk(2, j)] + row4(Z, j));
        uc[j] = fmaf(ty, c6[pk(4, j)], tx * c6[pk(3, j)]);
        vc[j] = row4(Q, j);
    }
    auto on4 = [&](const float *m, const float *v) {
        return fmaf(m[4], v[3], fmaf(m[3], v[2], fmaf(m[1], v[1], m[0] * v[0])));
    };
    auto onz = [&](const float *m) { return fmaf(m[5], jp, m[2] + on4(m, Z)); };
    auto onu = [&](const float *m) { return fmaf(m[4], ty, m[3] * tx); };
    c[pk(0, 0)] = on4(tc, T);
    c[pk(1, 0)] = onz(tc);
    c[pk(1, 1)] = onz(zc);
    c[pk(2, 0)] = onu(tc);
    c[pk(2, 1)] = onu(zc);
    c[pk(2, 2)] = onu(uc);
    c[pk(3, 0)] = on4(tc, Q);
    c[pk(3, 1)] = on4(zc, Q);
    c[pk(3, 2)] = on4(uc, Q);
    c[pk(3, 3)] = on4(vc, Q);
    c[pk(4, 0)] = tc[5];
    c[pk(4, 1)] = zc[5];
    c[pk(4, 2)] = uc[5];
    c[pk(4, 3)] = vc[5];
    c[pk(4, 4)] = c6[pk(5, 5)];
    if constexpr (!DEFER) {
        if (wide) {
            constexpr int P[4] = {0, 1, 3, 4};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j <= i; ++j) slot[pk(i, j) * stride] = c6[pk(P[i], P[j])];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                slot[(10 + i) * stride] = T[i];
                slot[(14 + i) * stride] = Q[i];
            }
            enter_wide(slot, stride);
            c[pk(0, 0)] = slot[0];
            c[pk(3, 0)] = slot[stride];
            c[pk(3, 3)] = slot[2 * stride];
        }
    }
    p = Local{x1, y1, z1, pt2 * ipt, 0.0f, x[5], ux, uy, nx, ny};
    pn = fabsf(cn) * pt2 * ipt;
    return 0u;
}

// The momentum noise of a thin layer, theta0^2 (|p|^2 I3 - p p^T) (Highland,
// beta = 1, path x_over_x0 / |cos(incidence)|): theta0^2.
__device__ __forceinline__ float noise_local(const Local &p, float pn, float x_over_x0)
{
    if (!(x_over_x0 > 0.0f)) return 0.0f;
    const float ip = rsqrtf(fmaf(p.pz, p.pz, fmaf(p.q1, p.q1, p.q2 * p.q2)));
    const float xx0 = __fdividef(x_over_x0, pn * ip);
    const float lg = fmaf(0.038f, __logf(xx0), 1.0f);
    return (0.0136f * 0.0136f) * (ip * ip) * xx0 * (lg * lg);
}

// That noise, theta2 = theta0^2, added to the momentum block.
__device__ __forceinline__ void scatter_local(const Local &p, float theta2, float c[15])
{
    const float tu = -theta2 * p.q1, tv = -theta2 * p.q2;
    c[pk(2, 2)] = fmaf(theta2, fmaf(p.q2, p.q2, p.pz * p.pz), c[pk(2, 2)]);
    c[pk(3, 2)] = fmaf(tu, p.q2, c[pk(3, 2)]);
    c[pk(3, 3)] = fmaf(theta2, fmaf(p.q1, p.q1, p.pz * p.pz), c[pk(3, 3)]);
    c[pk(4, 2)] = fmaf(tu, p.pz, c[pk(4, 2)]);
    c[pk(4, 3)] = fmaf(tv, p.pz, c[pk(4, 3)]);
    c[pk(4, 4)] = fmaf(theta2, fmaf(p.q1, p.q1, p.q2 * p.q2), c[pk(4, 4)]);
}

// Update with a 3-D hit (Section 2.1: 3x3 measurement covariance V).
//   S = C_xx + V, K = C[:, 0:3] S^-1, x += K r, C -= K C[0:3, :],
//   dchi2 = r^T S^-1 r.
//
// In (n, t, z) C has no radial row, and the exactly known radial direction
// does not mix with the uncertain tangential one, which in x/y share every
// entry (FP32 could not resolve the gain of an update that shrinks the
// covariance by orders of magnitude, a hit after a diffuse seed).  S is
// factorised in the order n, t, z: with vt = V_nt / V_nn, vz = V_nz / V_nn the
// hit's t and z given its n, S's t pivot dt, its z pivot dz and l = S_zt' / dt,
// three residuals rn, r1, r2 with variances V_nn, dt, dz,
//   chi2 = rn^2 / V_nn + r1^2 / dt + r2^2 / dz,
// and the gain is two scalar updates with the columns C_t and C_z - l C_t.
// det S = V_nn dt dz, positive definite when all three pivots are positive.
// Routing (mode 1):
//   * the whole update is redone in FP64 with a PSD repair (update_fp64) when
//     S is not positive definite in FP32, when the determinant of its
//     correlation matrix R = D^-1/2 S D^-1/2 (D = diag S) is below
//     27 / (4 cond_max) (R's eigenvalues sum to 3, so that this bounds
//     cond_2(R) by cond_max on the FP32 path; the spread of S's diagonal, V_nn
//     << C_zz, is harmless);
//   * else, when pT lies outside [pt_lo, pt_hi], it is redone in float-float
//     (update_wide), or in FP64 after all where the hit is more than a million
//     times as precise as the prediction (kWideGain, against V's t and z pivots);
//   * with gain_max > 0, the gain is formed in float-float (update_ff) when
//     C_ii > gain_max V_ii for some i.
// Returns 0 updated in FP32, 2 updated with extended-precision arithmetic,
// 3 updated in FP64 with a PSD repair, 1 failed (S not positive definite).
// DEFER: an update that needs extended precision is left undone, 4 returned.
template <bool DEFER = false>
__device__ __forceinline__ int update_local(Local &p, float c[15], const float m[3], const float v[6],
                                            const Routing &rt, float *dchi2, float *slot, int stride)
{
    const float nx = p.nx, ny = p.ny;
    const float nn = nx * nx, tt = ny * ny, nt = nx * ny;
    const float vnn = fmaf(nn, v[0], fmaf(2.0f * nt, v[1], tt * v[2]));
    const float vnt = fmaf(nt, v[2] - v[0], fmaf(nx, nx, -tt) * v[1]);
    const float vtt = fmaf(tt, v[0], fmaf(-2.0f * nt, v[1], nn * v[2]));
    const float vnz = fmaf(nx, v[3], ny * v[4]), vtz = fmaf(nx, v[4], -ny * v[3]);
    const float stt = c[pk(0, 0)] + vtt, szz = c[pk(1, 1)] + v[5];
    const float ia = __fdividef(1.0f, vnn);
    const float vt = vnt * ia, vz = vnz * ia;
    const float dt = fmaf(-vnt, vt, stt);
    const float it = __fdividef(1.0f, dt);
    const float e = fmaf(-vnt, vz, c[pk(1, 0)] + vtz);
    const float l = e * it;
    const float dz = fmaf(-l, e, fmaf(-vnz, vz, szz));
    // an infinite V_zz must not pass: the caller tells a bad hit by the failure
    const bool pd = vnn > 0.0f && dt > 0.0f && dz > 0.0f && dz < INFINITY;
    int kind = 0;
    if (rt.mode == 1) {
        const bool ill = !pd || dt * dz <= rt.det_min * (stt * szz);
        const float pt2 = fmaf(p.q1, p.q1, p.q2 * p.q2);
        if (ill)
            kind = 2;
        else if (outside_pt(pt2, rt))
            kind = 3;
        else if (rt.gain_max > 0.0f)  // one test (|): the lanes it holds for reach the call together
            kind = (tt * c[pk(0, 0)] > rt.gain_max * v[0]) | (nn * c[pk(0, 0)] > rt.gain_max * v[2]) |
                   (c[pk(1, 1)] > rt.gain_max * v[5]);
    } else if (!pd) {
        return 1;
    }
    if constexpr (DEFER) {
        if (kind) return 4;
    }
    if (kind) {
        float *s = slot;
        const float x[6] = {p.x, p.y, p.z, p.q1, p.q2, p.pz};
#pragma unroll
        for (int i = 0; i < 6; ++i) s[(kSlotX + i) * stride] = x[i];
#pragma unroll
        for (int i = 0; i < 15; ++i) s[(kSlotC + i) * stride] = c[i];
#pragma unroll
        for (int i = 0; i < 3; ++i) s[(kSlotM + i) * stride] = m[i];
#pragma unroll
        for (int i = 0; i < 6; ++i) s[(kSlotV + i) * stride] = v[i];
        s[(kSlotFrame + 2) * stride] = nx;
        s[(kSlotFrame + 3) * stride] = ny;
        const int st = update_ext(slot, stride, kind);
        if (st == 1) return 1;
        p.x = s[kSlotX * stride];
        p.y = s[(kSlotX + 1) * stride];
        p.z = s[(kSlotX + 2) * stride];
        p.q1 = s[(kSlotX + 3) * stride];
        p.q2 = s[(kSlotX + 4) * stride];
        p.pz = s[(kSlotX + 5) * stride];
#pragma unroll
        for (int i = 0; i < 15; ++i) c[i] = s[(kSlotC + i) * stride];
        *dchi2 = s[kSlotChi2 * stride];
        return st;
    }
    const float iz = __fdividef(1.0f, dz);
    const float d0 = m[0] - p.x, d1 = m[1] - p.y;
    const float rn = fmaf(nx, d0, ny * d1);
    const float r1 = fmaf(-vt, rn, fmaf(nx, d1, -ny * d0));
    const float r2 = fmaf(-l, r1, fmaf(-vz, rn, m[2] - p.z));
    const float w1 = r1 * it, w2 = r2 * iz;
    *dchi2 = fmaf(rn * rn, ia, fmaf(r1, w1, r2 * w2));
    float a[5], b[5];  // the columns of the two scalar updates, and their gains
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        a[i] = c[pk(i, 0)];
        b[i] = fmaf(-l, a[i], c[pk(i, 1)]);
    }
    const float dx = fmaf(a[0], w1, b[0] * w2);
    p.x = fmaf(-ny, dx, p.x);
    p.y = fmaf(nx, dx, p.y);
    p.z += fmaf(a[1], w1, b[1] * w2);
    p.q1 += fmaf(a[2], w1, b[2] * w2);
    p.q2 += fmaf(a[3], w1, b[3] * w2);
    p.pz += fmaf(a[4], w1, b[4] * w2);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const float ka = -a[i] * it, kb = -b[i] * iz;
#pragma unroll
        for (int j = 0; j <= i; ++j) c[pk(i, j)] = fmaf(ka, a[j], fmaf(kb, b[j], c[pk(i, j)]));
    }
    return 0;
}

// The Cartesian state and covariance (packed 6x6) of local coordinates.
__device__ __forceinline__ void leave_local(const Local &p, const float c[15], float x[6], float c6[21])
{
    const float f0 = p.f0, f1 = p.f1;
    x[0] = p.x;
    x[1] = p.y;
    x[2] = p.z;
    x[3] = fmaf(f0, p.q1, -f1 * p.q2);
    x[4] = fmaf(f1, p.q1, f0 * p.q2);
    x[5] = p.pz;
    auto px = [&](int j) { return fmaf(f0, c[pk(2, j)], -f1 * c[pk(3, j)]); };
    auto py = [&](int j) { return fmaf(f1, c[pk(2, j)], f0 * c[pk(3, j)]); };
    const float lt[4] = {c[pk(1, 0)], px(0), py(0), c[pk(4, 0)]};
    c6[pk(0, 0)] = p.ny * p.ny * c[pk(0, 0)];
    c6[pk(1, 0)] = -p.nx * p.ny * c[pk(0, 0)];
    c6[pk(1, 1)] = p.nx * p.nx * c[pk(0, 0)];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        c6[pk(i + 2, 0)] = -p.ny * lt[i];
        c6[pk(i + 2, 1)] = p.nx * lt[i];
    }
    c6[pk(2, 2)] = c[pk(1, 1)];
    c6[pk(3, 2)] = px(1);
    c6[pk(4, 2)] = py(1);
    c6[pk(5, 2)] = c[pk(4, 1)];
    const float uu = px(2), uv = px(3), vu = py(2), vv = py(3);
    c6[pk(3, 3)] = fmaf(f0, uu, -f1 * uv);
    c6[pk(4, 3)] = fmaf(f0, vu, -f1 * vv);
    c6[pk(4, 4)] = fmaf(f1, vu, f0 * vv);
    c6[pk(5, 3)] = px(4);
    c6[pk(5, 4)] = py(4);
    c6[pk(5, 5)] = c[pk(4, 4)];
}

}  // namespace kf
