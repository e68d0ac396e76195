// sturm.cuh -- Sturm counts of the Golub-Kahan tridiagonal in product form.
//
// For the 2n x 2n tridiagonal with zero diagonal and off-diagonals t_0, t_1, ... the leading
// principal minors of TGK - x I are p_0 = 1, p_1 = -x, p_{i+2} = -x p_{i+1} - t_i^2 p_i, and
// the number of negative pivots of its LDL^T factorisation is the number of sign changes in
// that sequence (Givens 1954; Wilkinson, The Algebraic Eigenvalue Problem, ch. 5).  Against the
// pivot recurrence q = -x - t^2 / q the chain of one term is a single FMA instead of a division
// (4 against about 45 cycles), and the whole term is a multiply, an FMA and a sign bit.
//
// Rounding: with p_{i+2} = (1 + d)(-x p_{i+1} - t_i^2 (1 + d') p_i) the factors (1 + d) can be
// moved into t^2, so the computed signs are those of the exact sequence for the same x and
// off-diagonals that differ relatively by at most two roundings of t^2 -- no looser than the
// pivot form.
//
// Range: |x| <= 1 and t^2 <= 1 by scaling, so minors shrink; both running minors are multiplied
// by the same power of two (exact) every few terms.  Over two terms they shrink at most by
// min(x^2, t^2); the callers keep t^2 >= kT2Floor, which is far below what moves a value, so
// that an exactly zero minor (x on a value of a leading block, which degenerate inputs do meet)
// is followed by a nonzero one.  A zero minor counts as positive: whichever sign it is given,
// the changes before and after it add up to one.
#pragma once

#include "common.cuh"

namespace nla {

constexpr float kT2FloorF = 0x1p-60f;   // 2^-30 of the bound in t: below FP32's resolution of the values
constexpr double kT2FloorD = 0x1p-120;  // 2^-60 of the bound

// Shift the sign of v into the history (newest in bit 0).
NLA_DEV unsigned push_sign(unsigned hist, float v) { return __funnelshift_l(__float_as_uint(v), hist, 1); }
NLA_DEV unsigned push_sign(unsigned hist, double v) {
    return __funnelshift_l((unsigned)__double2hiint(v), hist, 1);
}

// Multiply both minors by the power of two that brings the larger one to [1, 2).
NLA_DEV void rescale_pair(float &a, float &b) {
    const unsigned e = __float_as_uint(fmaxf(fabsf(a), fabsf(b))) & 0x7f800000u;
    const float s = __uint_as_float(0x7f000000u - e);
    a *= s;
    b *= s;
}
NLA_DEV void rescale_pair(double &a, double &b) {
    const unsigned ha = (unsigned)__double2hiint(a) & 0x7ff00000u, hb = (unsigned)__double2hiint(b) & 0x7ff00000u;
    const double s = __hiloint2double((int)(0x7fe00000u - max(ha, hb)), 0);
    a *= s;
    b *= s;
}

// Negative pivots of TGK - x I, t2[0 .. n2) = squares of the n2 = 2n - 1 off-diagonals
// (>= the floor above, <= 1), 0 < x <= 1.  t2 16-byte aligned.
NLA_DEV int sturm_neg(int n2, const float *__restrict__ t2, float x) {
    float a = 1.f, b = -x;  // p_i, p_{i+1}
    unsigned hist = 1u;     // signs of p_0 (0), p_1 (1)
    int neg = 1;
    int i = 0;
    // (FP32 keeps 2^-126 .. 2^127: four terms shrink by 2^-120 at most, so rescale every four)
    for (; i + 16 <= n2; i += 16) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float4 t = *reinterpret_cast<const float4 *>(t2 + i + 4 * u);
            a = fmaf(-x, b, -(t.x * a)), hist = push_sign(hist, a);
            b = fmaf(-x, a, -(t.y * b)), hist = push_sign(hist, b);
            a = fmaf(-x, b, -(t.z * a)), hist = push_sign(hist, a);
            b = fmaf(-x, a, -(t.w * b)), hist = push_sign(hist, b);
            rescale_pair(a, b);
        }
        neg += __popc((hist ^ (hist >> 1)) & 0xffffu);
    }
    for (; i < n2; ++i) {
        const float c = fmaf(-x, b, -(t2[i] * a));
        hist = push_sign(hist, c);
        neg += (hist ^ (hist >> 1)) & 1u;
        a = b;
        b = c;
        rescale_pair(a, b);
    }
    return neg;
}
NLA_DEV int sturm_neg(int n2, const double *__restrict__ t2, double x) {
    double a = 1.0, b = -x;
    unsigned hist = 1u;
    int neg = 1;
    int i = 0;
    // (eight terms shrink by 2^-480 at most: one rescaling per eight)
    for (; i + 16 <= n2; i += 16) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const double2 t = *reinterpret_cast<const double2 *>(t2 + i + 8 * u + 2 * w);
                a = fma(-x, b, -(t.x * a)), hist = push_sign(hist, a);
                b = fma(-x, a, -(t.y * b)), hist = push_sign(hist, b);
            }
            rescale_pair(a, b);
        }
        neg += __popc((hist ^ (hist >> 1)) & 0xffffu);
    }
    for (; i < n2; ++i) {
        const double c = fma(-x, b, -(t2[i] * a));
        hist = push_sign(hist, c);
        neg += (hist ^ (hist >> 1)) & 1u;
        a = b;
        b = c;
        rescale_pair(a, b);
    }
    return neg;
}

}  // namespace nla
