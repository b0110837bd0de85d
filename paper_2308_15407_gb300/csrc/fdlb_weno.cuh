// WENO-5 face values (Sec. III B 2) of the update kernel, in the differences of the stencil.
//
// With the first differences d1..d4 and second differences e1..e3 of the five upwind nodes
// (a, b, c, d, e) the indicators are 13/12 e_q^2 + 1/4 q_q^2 with q1 = e1 + 2 d2, q2 = d2 + d3,
// q3 = e3 - 2 d3, and the candidates are offsets from c,
//   F1 = c + (5 d2 - 2 d1)/6,   F2 = c + (d2 + 2 d3)/6,   F3 = c + (4 d3 - d4)/6,
// which differ by third differences: F2 - F1 = (e2 - e1)/3, F3 - F2 = -(e3 - e2)/6.  With
// m_1 = (s2 s3)^2 and so on (omega~_q = delta_q/s_q^2 times a common factor, delta_q = 1 : 6 : 3)
//   face = c + (m1 (5 d2 - 2 d1) + 6 m2 (d2 + 2 d3) + 3 m3 (4 d3 - d4))/(6 (m1 + 6 m2 + 3 m3))
//        = c + (d2 + 2 d3 - (2 m1 (e2 - e1) + 3 m3 (e3 - e2))/(m1 + 6 m2 + 3 m3))/6.
// No epsilon; a vanishing indicator takes the weight in the limit.
//
// FP32: the first form, 46 instructions against 61 of the candidates and normalised weights.  Each
// offset carries its own weight, so next to a front, where d2 + 2 d3 holds a jump, no two terms of the
// jump's size cancel: 6e-8 of the face for jumps of 1e2 between neighbouring nodes (the second form, 42
// instructions: 1e-5, and no digit from jumps of 1e7 on; the sum of weighted candidates: 5e-7).
//
// FP64: the pipe issues one warp instruction per 64 to 76 cycles and scheduler on this GPU, so
// where the stencil is smooth only what carries the value is FP64: the differences (exact
// cancellation), F2 and the final sum of the second form, 11 instructions instead of 75.  The weights
// multiply third differences and run in double-float (quotient to 3e-14): the face's error from them is
// at most 1.3e-14 of the largest third difference, so with third differences up to 2^-WENO_SMOOTH |c|
// it is two roundings of c at most.  A rougher stencil takes the first form, all in FP64.
// Largest error over 1e5 stencils each, relative to the face, against 64 mantissa bits (weighted candidates in
// FP64 -> this form): smooth (steps of 0.01 to 0.4 in exp(sin x / 2)) 5.6e-16 -> 3.3e-16; ratios of 1.01 to 3
// between neighbours with 1 % noise 7.4e-16 -> 5.6e-16 (5 and 10: 6.3e-16 -> 8.1e-16); fronts of 3 to 1e12
// 8.8e-16 -> 1.1e-16.  Double-float weights everywhere: 5e-14 at a ratio of 3, 3e-12 at a front of 1e2.
#pragma once
#include "fdlb_df.cuh"

namespace fdlb {

__device__ __forceinline__ float weno_face(float a, float b, float c, float d, float e) {
    const float d1 = b - a, d2 = c - b, d3 = d - c, d4 = e - d;
    const float e1 = d2 - d1, e2 = d3 - d2, e3 = d4 - d3;
    const float q1 = fmaf(2.0f, d2, e1), q2 = d2 + d3, q3 = fmaf(-2.0f, d3, e3);
    const float k = 13.0f / 3.0f;
    const float s1 = fmaf(k * e1, e1, q1 * q1), s2 = fmaf(k * e2, e2, q2 * q2), s3 = fmaf(k * e3, e3, q3 * q3);
    // scaled by the largest, so that the fourth powers stay in range: up to 2^60, since next to a front the
    // largest is 1e-30 of that, and times the offsets of a velocity tail it has to stay a normal number
    const float smax = fmaxf(s1, fmaxf(s2, s3));
    const float r = rcp_approx(fmaxf(smax, 4e-30f)) * 0x1p15f;
    const float a1 = s1 * r, a2 = s2 * r, a3 = s3 * r;
    const float p1 = a1 * a1, p2 = a2 * a2, p3 = a3 * a3;
    float m1 = p2 * p3, m2 = p1 * p3, m3 = p1 * p2;
    float w2 = 6.0f * m2, w3 = 3.0f * m3, sum = (m1 + w2) + w3;
    if (sum < 0x1p60f * 1e-30f) {
        if (smax < 4e-30f) {
            // uniform to FP32 resolution: the candidates agree, the ideal weights are the limit
            m1 = m2 = m3 = 1.0f;
        } else {
            // two indicators vanish relative to the third: weight on the smallest
            const float smin = fminf(s1, fminf(s2, s3));
            m1 = s1 == smin ? 1.0f : 0.0f;
            m2 = s2 == smin ? 1.0f : 0.0f;
            m3 = s3 == smin ? 1.0f : 0.0f;
        }
        w2 = 6.0f * m2;
        w3 = 3.0f * m3;
        sum = (m1 + w2) + w3;
    }
    // six times the candidates' offsets from c, each times its own weight
    const float o1 = fmaf(-2.0f, d1, 5.0f * d2), o2 = fmaf(2.0f, d3, d2), o3 = fmaf(4.0f, d3, -d4);
    return fmaf(fmaf(m1, o1, fmaf(w2, o2, w3 * o3)), rcp_approx(sum) * (1.0f / 6.0f), c);
}

constexpr int WENO_SMOOTH = 6;

// The face of a stencil that is not smooth, the first form, all of it in FP64, from the differences.  (The
// offsets' weights are eighth powers of differences, those beyond 2^-60 .. 2^100 are scaled first: with the
// largest at 2^-t and the smooth side at 2^-(t + r), the numerator is 2^-(9 t + 5 r), and a full number for all
// jumps up to 2^96.)
__device__ __forceinline__ double weno_face_rough(double a, double b, double c, double d, double e) {
    double d1 = b - a, d2 = c - b, d3 = d - c, d4 = e - d;
    const int top = max(max(__double2hiint(d1) & 0x7fffffff, __double2hiint(d2) & 0x7fffffff),
                        max(__double2hiint(d3) & 0x7fffffff, __double2hiint(d4) & 0x7fffffff));
    const double o1 = fma(-2.0, d1, 5.0 * d2), o2 = fma(2.0, d3, d2), o3 = fma(4.0, d3, -d4);
    if ((unsigned)(top - (963 << 20)) > (160u << 20)) {
        const double sc = __hiloint2double(max((2045 << 20) - (top & 0x7ff00000), 1 << 20), 0);
        d1 *= sc;
        d2 *= sc;
        d3 *= sc;
        d4 *= sc;
    }
    const double e1 = d2 - d1, e2 = d3 - d2, e3 = d4 - d3;
    const double q1 = fma(2.0, d2, e1), q2 = d2 + d3, q3 = fma(-2.0, d3, e3), k = 13.0 / 3.0;
    const double s1 = fma(k * e1, e1, q1 * q1), s2 = fma(k * e2, e2, q2 * q2), s3 = fma(k * e3, e3, q3 * q3);
    const double s12 = s1 * s2, s13 = s1 * s3, s23 = s2 * s3;
    double m1 = s23 * s23, m2 = s13 * s13, m3 = s12 * s12;
    if (!(__double2hiint(m1) | __double2hiint(m2) | __double2hiint(m3))) {
        // two indicators vanish (or underflow): weight on the smallest ones
        const double smin = fmin(s1, fmin(s2, s3));
        m1 = s1 == smin ? 1.0 : 0.0;
        m2 = s2 == smin ? 1.0 : 0.0;
        m3 = s3 == smin ? 1.0 : 0.0;
    }
    const double w2 = 6.0 * m2, w3 = 3.0 * m3;
    return fma(fma(m1, o1, fma(w2, o2, w3 * o3)) / ((m1 + w2) + w3), 1.0 / 6.0, c);
}

// The face where the stencil is smooth; rough: it is not, and the value has to come from weno_face_rough.
__device__ __forceinline__ double weno_face_smooth(double a, double b, double c, double d, double e, bool& rough) {
    const double d1 = b - a, d2 = c - b, d3 = d - c, d4 = e - d;
    const double e1 = d2 - d1, e2 = d3 - d2, e3 = d4 - d3;
    const double X = fma(2.0, d3, d2);
    const int top = max(max(__double2hiint(d1) & 0x7fffffff, __double2hiint(d2) & 0x7fffffff),
                        max(__double2hiint(d3) & 0x7fffffff, __double2hiint(d4) & 0x7fffffff));
    rough = false;
    if (top >= 0x7ff00000) return (a + b) + (c + d) + e;      // not finite: stays not finite
    const int eb = ((top >> 20) - 127) << 20;
    if (top < (128 << 20)) {
        // no difference above 2^-895: ideal weights, (2 (e2 - e1) + 3 (e3 - e2))/10
        return fma(X - 0.1 * (fma(2.0, e2 - e1, 3.0 * (e3 - e2))), 1.0 / 6.0, c);
    }
    const df D2 = split_scaled(d2, eb), D3 = split_scaled(d3, eb);
    const df E1 = split_scaled(e1, eb), E2 = split_scaled(e2, eb), E3 = split_scaled(e3, eb);
    const df T1 = plus(E2, -E1), T2 = plus(E3, -E2);
    // the larger third difference as the high word of a double, against that of c
    const uint32_t third = (__float_as_uint(fmaxf(fabsf(T1.hi), fabsf(T2.hi))) >> 3) + (uint32_t)eb;
    rough = third + (WENO_SMOOTH << 20) > ((uint32_t)__double2hiint(c) & 0x7fffffffu);
    const df q1 = plus(E1, df{2.0f * D2.hi, 2.0f * D2.lo}), q2 = plus(D2, D3), q3 = plus(E3, df{-2.0f * D3.hi, -2.0f * D3.lo});
    // indicators times 12/13: e^2 + 3/13 q^2
    const df k = r_c(3.0 / 13.0, df{});
    const df s1 = plus(sqr_u(E1), mul_u(k, sqr_u(q1))), s2 = plus(sqr_u(E2), mul_u(k, sqr_u(q2)));
    const df s3 = plus(sqr_u(E3), mul_u(k, sqr_u(q3)));
    const df p1 = sqr_u(s1), p2 = sqr_u(s2), p3 = sqr_u(s3);
    df m1 = mul_u(p2, p3), m2 = mul_u(p1, p3), m3 = mul_u(p1, p2);
    if (!(fmaxf(m1.hi, fmaxf(m2.hi, m3.hi)) >= 1e-30f)) {
        // two indicators far below the third: (s_min/s_q)^2, or the vanishing ones alone
        const float smin = fminf(s1.hi, fminf(s2.hi, s3.hi));
        if (smin == 0.0f) {
            m1 = {s1.hi == 0.0f ? 1.0f : 0.0f, 0.0f};
            m2 = {s2.hi == 0.0f ? 1.0f : 0.0f, 0.0f};
            m3 = {s3.hi == 0.0f ? 1.0f : 0.0f, 0.0f};
        } else {
            const df sm = s1.hi == smin ? s1 : (s2.hi == smin ? s2 : s3);
            m1 = sqr_u(div_u(sm, s1));
            m2 = sqr_u(div_u(sm, s2));
            m3 = sqr_u(div_u(sm, s3));
        }
    }
    const df m33 = scale_u(m3, 3.0f);
    const df sum = plus(plus(m1, m33), scale_u(m2, 6.0f));
    const df num = plus(mul_u(df{2.0f * m1.hi, 2.0f * m1.lo}, T1), mul_u(m33, T2));
    const df corr = div_u(num, sum);
    return fma((X - join_scaled(corr.hi, eb)) - join_scaled(corr.lo, eb), 1.0 / 6.0, c);
}

__device__ __forceinline__ double weno_face(double a, double b, double c, double d, double e) {
    bool rough;
    const double f = weno_face_smooth(a, b, c, d, e, rough);
    return rough ? weno_face_rough(a, b, c, d, e) : f;
}

}  // namespace fdlb
