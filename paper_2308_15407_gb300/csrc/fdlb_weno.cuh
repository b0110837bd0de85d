// WENO-5 face values (Sec. III B 2) of the update kernel, in the differences of the stencil.
//
// With the first differences d1..d4 and second differences e1..e3 of the five upwind nodes
// (a, b, c, d, e) the candidates differ from the middle one by third differences,
//   F1 = F2 - (e2 - e1)/3,   F2 = c + (d2 + 2 d3)/6,   F3 = F2 - (e3 - e2)/6,
// and the indicators are 13/12 e_q^2 + 1/4 q_q^2 with q1 = e1 + 2 d2, q2 = d2 + d3,
// q3 = e3 - 2 d3.  With m_1 = (s2 s3)^2 and so on (omega~_q = delta_q/s_q^2 times a common factor)
//   face = c + (d2 + 2 d3 - (2 m1 (e2 - e1) + 3 m3 (e3 - e2))/(m1 + 6 m2 + 3 m3))/6.
// No epsilon; a vanishing indicator takes the weight in the limit.
//
// FP32: 42 instructions against 61 of the three candidates and normalised weights, and the large
// part of the value, c, is never multiplied.
//
// FP64: the pipe issues one warp instruction per 64 to 76 cycles and scheduler on this GPU, so only
// what carries the value is FP64: the differences (exact cancellation), F2 and the final sum, 11
// instructions instead of 75.  The weights multiply third differences and run in double-float
// (float pairs, 2^-46): their relative error d gives the face an error d |e2 - e1|, below the
// rounding of c wherever the stencil is smoother than |e2 - e1| ~ 1e-2 c.
#pragma once
#include <stdint.h>

namespace fdlb {

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float weno_face(float a, float b, float c, float d, float e) {
    const float d1 = b - a, d2 = c - b, d3 = d - c, d4 = e - d;
    const float e1 = d2 - d1, e2 = d3 - d2, e3 = d4 - d3;
    const float q1 = fmaf(2.0f, d2, e1), q2 = d2 + d3, q3 = fmaf(-2.0f, d3, e3);
    const float k = 13.0f / 3.0f;
    const float s1 = fmaf(k * e1, e1, q1 * q1), s2 = fmaf(k * e2, e2, q2 * q2), s3 = fmaf(k * e3, e3, q3 * q3);
    // scaled by the largest, so that the fourth powers stay in range
    const float smax = fmaxf(s1, fmaxf(s2, s3));
    const float r = rcp_approx(fmaxf(smax, 4e-30f));
    const float a1 = s1 * r, a2 = s2 * r, a3 = s3 * r;
    const float p1 = a1 * a1, p2 = a2 * a2, p3 = a3 * a3;
    float m1 = p2 * p3, m2 = p1 * p3, m3 = p1 * p2;
    float sum = fmaf(6.0f, m2, fmaf(3.0f, m3, m1));
    if (sum < 1e-30f) {
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
        sum = fmaf(6.0f, m2, fmaf(3.0f, m3, m1));
    }
    const float num = fmaf(3.0f * m3, e3 - e2, (m1 + m1) * (e2 - e1));
    return fmaf(fmaf(-num, rcp_approx(sum), fmaf(2.0f, d3, d2)), 1.0f / 6.0f, c);
}

// ---- float pairs without the final normalisation (head and a tail of a few units in its last
// place), for the FP64 weights
struct fp2 {
    float h, l;
};
__device__ __forceinline__ fp2 p_add(fp2 a, fp2 b) {
    const float s = __fadd_rn(a.h, b.h);
    const float t = __fsub_rn(s, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
    return {s, __fadd_rn(e, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ fp2 p_neg(fp2 a) { return {-a.h, -a.l}; }
__device__ __forceinline__ fp2 p_mul(fp2 a, fp2 b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    return {p, __fmaf_rn(a.l, b.h, e)};
}
__device__ __forceinline__ fp2 p_sqr(fp2 a) {
    const float p = __fmul_rn(a.h, a.h);
    return {p, __fmaf_rn(__fadd_rn(a.h, a.h), a.l, __fmaf_rn(a.h, a.h, -p))};
}
__device__ __forceinline__ fp2 p_scale(fp2 a, float c) {
    const float p = __fmul_rn(a.h, c);
    return {p, __fmaf_rn(a.l, c, __fmaf_rn(a.h, c, -p))};
}
// a / b to ~1e-14 (one correction of the approximate quotient)
__device__ __forceinline__ fp2 p_div(fp2 a, fp2 b) {
    const float r = rcp_approx(b.h), q = __fmul_rn(a.h, r);
    const float t = __fadd_rn(__fmaf_rn(-q, b.h, a.h), __fmaf_rn(-q, b.l, a.l));
    return {q, __fmul_rn(t, r)};
}

// x / 2^(E - 1023) as a float pair (the tail rounded: 2^-49), eb = (E - 127) << 20, by integer
// operations (a conversion to or from double runs on the FP64 pipe).  Values below 2^-96 give 0.
__device__ __forceinline__ fp2 split_scaled(double x, int eb) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int t = (int)(hi & 0x7fffffffu) - eb;
    const uint32_t hb = __funnelshift_l(lo, (uint32_t)t, 3), sg = hi & 0x80000000u;
    // the 29 bits below the head, times the power of two of the double's last place
    const float tail = __fmul_rn(__uint2float_rn(lo & 0x1fffffffu), __uint_as_float(((hb & 0x7f800000u) - (52u << 23)) | sg));
    if (t < (54 << 20)) return {t < (31 << 20) ? 0.0f : __uint_as_float(hb | sg), 0.0f};
    return {__uint_as_float(hb | sg), tail};
}
// y 2^(E - 1023) as a double, eb as above.
__device__ __forceinline__ double join_scaled(float y, int eb) {
    const uint32_t b = __float_as_uint(y), m = b & 0x7fffffffu;
    const int t = (int)(m >> 3) + eb;
    if (m < 0x00800000u || t < (1 << 20)) return 0.0;
    return __hiloint2double((int)((uint32_t)t | (b & 0x80000000u)), (int)(m << 29));
}

__device__ __forceinline__ double weno_face(double a, double b, double c, double d, double e) {
    const double d1 = b - a, d2 = c - b, d3 = d - c, d4 = e - d;
    const double e1 = d2 - d1, e2 = d3 - d2, e3 = d4 - d3;
    const double X = fma(2.0, d3, d2);
    const int top = max(max(__double2hiint(d1) & 0x7fffffff, __double2hiint(d2) & 0x7fffffff),
                        max(__double2hiint(d3) & 0x7fffffff, __double2hiint(d4) & 0x7fffffff));
    if (top >= 0x7ff00000) return (a + b) + (c + d) + e;      // not finite: stays not finite
    fp2 corr;
    const int eb = ((top >> 20) - 127) << 20;
    if (top < (128 << 20)) {
        // no difference above 2^-895: ideal weights, (2 (e2 - e1) + 3 (e3 - e2))/10
        return fma(X - 0.1 * (fma(2.0, e2 - e1, 3.0 * (e3 - e2))), 1.0 / 6.0, c);
    }
    {
        const fp2 D2 = split_scaled(d2, eb), D3 = split_scaled(d3, eb);
        const fp2 E1 = split_scaled(e1, eb), E2 = split_scaled(e2, eb), E3 = split_scaled(e3, eb);
        const fp2 q1 = p_add(E1, {2.0f * D2.h, 2.0f * D2.l}), q2 = p_add(D2, D3), q3 = p_add(E3, {-2.0f * D3.h, -2.0f * D3.l});
        // indicators times 12/13: e^2 + 3/13 q^2
        const fp2 k = {3.0f / 13.0f, (float)(3.0 / 13.0 - (double)(3.0f / 13.0f))};
        const fp2 s1 = p_add(p_sqr(E1), p_mul(k, p_sqr(q1))), s2 = p_add(p_sqr(E2), p_mul(k, p_sqr(q2)));
        const fp2 s3 = p_add(p_sqr(E3), p_mul(k, p_sqr(q3)));
        const fp2 p1 = p_sqr(s1), p2 = p_sqr(s2), p3 = p_sqr(s3);
        fp2 m1 = p_mul(p2, p3), m2 = p_mul(p1, p3), m3 = p_mul(p1, p2);
        if (!(fmaxf(m1.h, fmaxf(m2.h, m3.h)) >= 1e-30f)) {
            // two indicators far below the third: (s_min/s_q)^2, or the vanishing ones alone
            const float smin = fminf(s1.h, fminf(s2.h, s3.h));
            if (smin == 0.0f) {
                m1 = {s1.h == 0.0f ? 1.0f : 0.0f, 0.0f};
                m2 = {s2.h == 0.0f ? 1.0f : 0.0f, 0.0f};
                m3 = {s3.h == 0.0f ? 1.0f : 0.0f, 0.0f};
            } else {
                const fp2 sm = s1.h == smin ? s1 : (s2.h == smin ? s2 : s3);
                m1 = p_sqr(p_div(sm, s1));
                m2 = p_sqr(p_div(sm, s2));
                m3 = p_sqr(p_div(sm, s3));
            }
        }
        const fp2 m33 = p_scale(m3, 3.0f);
        const fp2 sum = p_add(p_add(m1, m33), p_scale(m2, 6.0f));
        const fp2 T1 = p_add(E2, p_neg(E1)), T2 = p_add(E3, p_neg(E2));
        const fp2 num = p_add(p_mul({2.0f * m1.h, 2.0f * m1.l}, T1), p_mul(m33, T2));
        corr = p_div(num, sum);
    }
    return fma((X - join_scaled(corr.h, eb)) - join_scaled(corr.l, eb), 1.0 / 6.0, c);
}

}  // namespace fdlb
