// Floating-point operations of one layer of the fit (step_local,
// transport_local, noise_local, scatter_local and update_local of
// csrc/kf_math.cuh), counted by compiling that source with a scalar that
// counts: an addition, multiplication, reciprocal, square root or logarithm is
// one, a fused multiply-add two.  Sign flips, comparisons, fabs and copies are
// not counted.
#include <math.h>
#include <stdint.h>

typedef float plain_float;
static unsigned long long n_ops;

struct Counted {
    plain_float v;
    Counted() = default;
    constexpr Counted(plain_float x) : v(x) {}
    constexpr Counted(double x) : v((plain_float)x) {}
    constexpr Counted(int x) : v((plain_float)x) {}
    operator double() const { return v; }
};
static Counted counted(int n, plain_float v)
{
    n_ops += n;
    return Counted(v);
}
#define BINARY(op, n, R, mk)                                                                            \
    inline R operator op(Counted a, Counted b) { return mk(n, a.v op b.v); }                            \
    inline R operator op(Counted a, plain_float b) { return mk(n, a.v op b); }                          \
    inline R operator op(plain_float a, Counted b) { return mk(n, a op b.v); }
#define PLAIN(n, x) (x)
BINARY(+, 1, Counted, counted)
BINARY(-, 1, Counted, counted)
BINARY(*, 1, Counted, counted)
BINARY(/, 2, Counted, counted)
BINARY(<, 0, bool, PLAIN)
BINARY(>, 0, bool, PLAIN)
BINARY(<=, 0, bool, PLAIN)
BINARY(>=, 0, bool, PLAIN)
BINARY(==, 0, bool, PLAIN)
BINARY(!=, 0, bool, PLAIN)
inline Counted operator-(Counted a) { return Counted(-a.v); }
inline Counted &operator+=(Counted &a, Counted b) { return a = a + b; }
inline Counted &operator*=(Counted &a, Counted b) { return a = a * b; }

#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
static Counted c_fma(Counted a, Counted b, Counted c) { return counted(2, ::fmaf(a.v, b.v, c.v)); }
static Counted c_div(Counted a, Counted b) { return counted(a.v == 1.0f || a.v == -1.0f ? 1 : 2, a.v / b.v); }
static Counted c_rsqrt(Counted a) { return counted(1, 1.0f / ::sqrtf(a.v)); }
static Counted c_sqrt(Counted a) { return counted(1, ::sqrtf(a.v)); }
static Counted c_log(Counted a) { return counted(1, ::logf(a.v)); }
static Counted c_atan(Counted a) { return counted(1, ::atanf(a.v)); }
static Counted c_tan(Counted a) { return counted(1, ::tanf(a.v)); }
static Counted c_abs(Counted a) { return Counted(::fabsf(a.v)); }
static Counted c_min(Counted a, Counted b) { return Counted(::fminf(a.v, b.v)); }
static Counted c_copysign(Counted a, Counted b) { return Counted(::copysignf(a.v, b.v)); }
static Counted c_add(Counted a, Counted b) { return a + b; }
static Counted c_sub(Counted a, Counted b) { return a - b; }
static Counted c_mul(Counted a, Counted b) { return a * b; }
#define fmaf c_fma
#define __fdividef c_div
#define rsqrtf c_rsqrt
#define sqrtf c_sqrt
#define __logf c_log
#define atanf c_atan
#define tanf c_tan
#define fabsf c_abs
#define fminf c_min
#define copysignf c_copysign
#define __fadd_rn c_add
#define __fsub_rn c_sub
#define __fmul_rn c_mul
#define __fmaf_rn c_fma
#define float Counted
#include "kf.h"
#include "kf_math.cuh"
#undef float

using namespace kf;

// Of n tracks over L layers: counts[0] the operations of layers 1 .. L - 1,
// counts[1] how many of those layers were reached, counts[2] the operations of
// the first layer and of writing the result.
extern "C" void host_count(int L, const plain_float *r, const plain_float *xx0, plain_float z_half, plain_float qk, int64_t n,
                           const plain_float *seed_state, const plain_float *seed_cov, const int8_t *charge,
                           const plain_float *hit_pos, const plain_float *hit_cov, unsigned long long *counts)
{
    Routing rt{};
    rt.mode = 1;
    rt.det_min = 6.75f / 1e4f;
    rt.pt_lo2 = 0.25f * 0.25f;
    rt.pt_hi2 = 200.0f * 200.0f;
    counts[0] = counts[1] = counts[2] = 0;
    for (int64_t t = 0; t < n; ++t) {
        Counted x[6], c6[21], c[15], slot[kSlotSize], pn, d;
        for (int i = 0; i < 6; ++i) x[i] = seed_state[i * n + t];
        for (int i = 0; i < 21; ++i) c6[i] = seed_cov[i * n + t];
        const Counted qkb(charge[t] * qk);
        Local p{};
        for (int l = 0; l < L; ++l) {
            Counted m[3], v[6];
            for (int i = 0; i < 3; ++i) m[i] = hit_pos[(3 * l + i) * n + t];
            for (int i = 0; i < 6; ++i) v[i] = hit_cov[(6 * l + i) * n + t];
            n_ops = 0;
            if (l == 0) {
                if (enter_local(x, c6, qkb, r[0], 1.0f / r[0], z_half, rt, slot, 1, p, c, pn)) break;
            } else {
                LocalJac J;
                if (step_local(p, qkb, r[l], 1.0f / r[l], z_half, J, pn)) break;
                transport_local(J, c);
            }
            scatter_local(p, noise_local(p, pn, xx0[l]), c);
            if (update_local(p, c, m, v, rt, &d, slot, 1)) break;
            counts[l == 0 ? 2 : 0] += n_ops;
            counts[1] += l > 0;
        }
        n_ops = 0;
        leave_local(p, c, x, c6);
        counts[2] += n_ops;
    }
}
