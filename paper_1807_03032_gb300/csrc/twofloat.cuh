// twofloat.cuh -- two-float arithmetic (a value as an unevaluated sum hi + lo
// of floats) of the setup kernels, and the TTI coefficients formed with it.
// Every operation is rounded by itself, so the host compiler's build of this
// header (-ffp-contract=off) gives the bits of the device's.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define FD_TF __device__ __forceinline__
#else
#define FD_TF static inline
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __frcp_rn(float a) { return 1.0f / a; }
static inline float __fsqrt_rn(float a) { return sqrtf(a); }
#endif

namespace fdsweep {

// The error-free transformations TwoSum (Knuth) and TwoProduct (by FMA).
struct TwoFloat {
    float hi, lo;
};

FD_TF TwoFloat two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return TwoFloat{s, e};
}

FD_TF TwoFloat quick_two_sum(float a, float b) {  // |a| >= |b| or a = 0
    const float s = __fadd_rn(a, b);
    return TwoFloat{s, __fsub_rn(b, __fsub_rn(s, a))};
}

FD_TF TwoFloat tf_mul(TwoFloat a, TwoFloat b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
    return quick_two_sum(p, e);
}

FD_TF TwoFloat tf_add(TwoFloat a, TwoFloat b) {
    const TwoFloat s = two_sum(a.hi, b.hi);
    return quick_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}

// Whether every value within 2^-42 of v's size around v rounds to one float
// (Ziv's rounding test); *f receives it.
FD_TF bool rounds_surely(TwoFloat v, float *f) {
    constexpr float E = 0x1p-42f;
    *f = __fadd_rn(v.hi, fmaf(v.hi, E, v.lo));
    return *f == __fadd_rn(v.hi, fmaf(v.hi, -E, v.lo));
}

// sin x and cos x as two-floats for |x| <= kSincosRange, to about 2^-44 of
// their size: x - k pi/2 with pi/2 as three floats and exact products (Cody
// and Waite's reduction), then the Taylor series on [-pi/4, pi/4], the last
// terms in plain FP32 and the leading ones in two-float arithmetic.  False
// where the reduction cancels too many digits for that: its error is at most
// 2^-63, and 2^-70 within one turn of 0, where a remainder below 2^-20 leaves
// nothing to round in the first sums (the nearest floats to 90, 180, 270 and 360
// degrees, axes that models do use, are 2^-24, 2^-23, 2^-26 and 2^-22 from them).
constexpr float kSincosRange = 1000.f;
FD_TF bool sincos_two_float(float x, TwoFloat *sine, TwoFloat *cosine) {
    const float k = rintf(__fmul_rn(x, 0x1.45f306p-1f));  // x / (pi/2)
    constexpr float P1 = 0x1.921fb6p+0f, P2 = -0x1.777a5cp-25f, P3 = -0x1.ee59dap-50f;
    const float p1 = __fmul_rn(k, P1), p1l = fmaf(k, P1, -p1);
    const TwoFloat t1 = two_sum(__fsub_rn(x, p1), -p1l);  // x - p1 is exact
    const float p2 = __fmul_rn(k, P2), p2l = fmaf(k, P2, -p2);
    const TwoFloat t2 = two_sum(t1.hi, -p2);
    const TwoFloat r =
        quick_two_sum(t2.hi, __fsub_rn(__fadd_rn(t1.lo, t2.lo), fmaf(k, P3, p2l)));
    const TwoFloat z = tf_mul(r, r);
    const float y = z.hi;
    // sin r = r + r z (-1/3! + z (1/5! + z (-1/7! + z (1/9! - ... - z^3 / 15!))))
    const float u = fmaf(y, fmaf(y, fmaf(y, -1.f / 1307674368000.f, 1.f / 6227020800.f),
                                 -1.f / 39916800.f), 1.f / 362880.f);
    TwoFloat q = tf_add(TwoFloat{-0x1.a01a02p-13f, 0x1.7f97fap-39f},
                        TwoFloat{__fmul_rn(y, u), 0.f});
    q = tf_add(TwoFloat{0x1.111112p-7f, -0x1.dddddep-32f}, tf_mul(z, q));
    q = tf_add(TwoFloat{-0x1.555556p-3f, 0x1.555556p-28f}, tf_mul(z, q));
    const TwoFloat s = tf_add(r, tf_mul(r, tf_mul(z, q)));
    // cos r = 1 + z (-1/2! + z (1/4! + z (-1/6! + z (1/8! - ... + z^3 / 14!))))
    const float v = fmaf(y, fmaf(y, fmaf(y, -1.f / 87178291200.f, 1.f / 479001600.f),
                                 -1.f / 3628800.f), 1.f / 40320.f);
    TwoFloat g = tf_add(TwoFloat{-0x1.6c16c2p-10f, 0x1.27d27ep-35f},
                        TwoFloat{__fmul_rn(y, v), 0.f});
    g = tf_add(TwoFloat{0x1.555556p-5f, -0x1.555556p-30f}, tf_mul(z, g));
    g = tf_add(TwoFloat{-0.5f, 0.f}, tf_mul(z, g));
    const TwoFloat c = tf_add(TwoFloat{1.f, 0.f}, tf_mul(z, g));
    const int quadrant = (int)k & 3;
    TwoFloat a = (quadrant & 1) ? c : s, b = (quadrant & 1) ? s : c;
    if (quadrant & 2) a = TwoFloat{-a.hi, -a.lo};
    if ((quadrant + 1) & 2) b = TwoFloat{-b.hi, -b.lo};
    *sine = a;
    *cosine = b;
    return fabsf(r.hi) >= 0x1p-20f || k == 0.f || (fabsf(k) <= 4.f && fabsf(r.hi) >= 0x1p-27f);
}

// n = (sin theta cos phi, sin theta sin phi, cos theta) of one point: the FP64
// functions and products rounded once.  The two-float values decide it wherever
// their error cannot change the rounding (all but about one point in 2^16); the
// others, angles beyond kSincosRange and components below 2^-80 take FP64.
FD_TF void axis_of(float th, float ph, float *nx, float *ny, float *nz) {
    if (fabsf(th) <= kSincosRange && fabsf(ph) <= kSincosRange) {
        TwoFloat st, ct, sp, cp;
        bool sure = sincos_two_float(th, &st, &ct);
        sure &= sincos_two_float(ph, &sp, &cp);
        const TwoFloat x = tf_mul(st, cp), y = tf_mul(st, sp);
        sure &= fabsf(x.hi) >= 0x1p-80f || st.hi == 0.f;
        sure &= fabsf(y.hi) >= 0x1p-80f || st.hi == 0.f || sp.hi == 0.f;
        sure &= rounds_surely(x, nx);
        sure &= rounds_surely(y, ny);
        sure &= rounds_surely(ct, nz);
        if (sure) return;
    }
    double st, ct, sp, cp;
    sincos((double)th, &st, &ct);
    sincos((double)ph, &sp, &cp);
    *nx = (float)(st * cp);
    *ny = (float)(st * sp);
    *nz = (float)ct;
}

// sqrt(1 + 2 delta), the FP64 root rounded once: 1 + 2 delta as an exact
// two-float, the FP32 root corrected by its exact residual to about 2^-45 of
// its size; FP64 where that does not decide the rounding.
FD_TF float anellipticity_root(float delta) {
    const TwoFloat x = two_sum(1.f, 2.f * delta);
    if (x.hi > 0.f) {
        const float r = __fsqrt_rn(x.hi);
        const float c = __fmul_rn(__fadd_rn(fmaf(-r, r, x.hi), x.lo), __frcp_rn(2.f * r));
        float s;
        if (rounds_surely(TwoFloat{r, c}, &s)) return s;
    }
    return (float)sqrt(fmax(0.0, 1.0 + 2.0 * (double)delta));
}

// The nearest float to (A + a) / (X + x) for two-float numerator and
// denominator (X > 0): q = A (1/X) is within two units of the answer; the
// residual (A + a) - q (X + x), whose leading part A - q X FMA forms to 2^-47
// of A, times 1/X is the remaining correction, and q plus it is rounded once
// (Markstein's final step).  The result can differ from exact rounding only
// when the quotient lies within about 2^-44 of its size of a rounding midpoint:
// 11 of 4e8 random quotients of the setup's range, by at most 4.2e-8 units,
// against 13 and as much with q a full-precision division.
FD_TF float div_two_float_rn(float A, float a, float X, float x) {
    const float y = __frcp_rn(X);
    const float q = __fmul_rn(A, y);
    float r = fmaf(-q, X, A);
    r = __fadd_rn(r, a);
    r = fmaf(-q, x, r);
    return fmaf(r, y, q);
}

}  // namespace fdsweep
