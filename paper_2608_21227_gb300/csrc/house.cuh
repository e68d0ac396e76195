// house.cuh -- scalars of a Householder reflector, shared by the panel and the bulge chase.
#pragma once

#include "common.cuh"

namespace nla {

// sqrt(q) and 1 / sqrt(q), 1 / u in FP32 from the hardware estimates and one Newton step each:
// a reflector's scalars scale what they touch, and an n x n matrix goes through thousands of
// reflectors, so the estimates' errors of 1 to 2 ulp, which lean to one side, add up in the
// singular values (mean error at 1,537 columns 6e-7 of sigma_1 without the steps).
NLA_DEV void sqrt_and_inverse(float q, float &r, float &rs) {
    rs = rsqrtf(q);
    r = q * rs;
    r = fmaf(fmaf(-r, r, q), 0.5f * rs, r);
    rs = fmaf(fmaf(-r, rs, 1.f), rs, rs);
}
NLA_DEV float inverse(float u) {
    const float s = __fdividef(1.f, u);
    return fmaf(fmaf(-u, s, 1.f), s, s);
}

// Householder scalars of x with alpha = x_0 and qt = sum of the other squares, qt > 0: with
// r = |x|, beta = -sign(alpha) r, u_0 = alpha - beta, and the factors with H row = row - ((u^T
// row) m1 m2) u.  FP32 splits 1 / (u^T u / 2) = tau / u_0^2 into two factors so that it stays in
// range wherever r^2 does.
NLA_DEV void house(float alpha, float qt, float &beta, float &u0, float &m1, float &m2) {
    float r, rs;
    sqrt_and_inverse(fmaf(alpha, alpha, qt), r, rs);
    beta = alpha >= 0.f ? -r : r;
    u0 = alpha - beta;
    m1 = inverse(u0);
    m2 = fmaf(fabsf(alpha), rs, 1.f) * m1;
}
// A double of the value of the float bits f (a normal number) times 2^e, by integer operations.
NLA_DEV double widen(unsigned f, int e) {
    return __hiloint2double((int)((f >> 3) & 0xfffffu) | ((int)(f >> 23) - 127 + 1023 + e) << 20, (int)(f << 29));
}
// Whether q = |x|^2 is where every intermediate product of house is a normal number.  Outside
// (a vector below 2^-480 or above 2^496 in length) 1 / q itself overflows or is subnormal, so the
// callers keep the factors apart or scale the vector first.
NLA_DEV bool ordinary(double q) { return (unsigned)__double2hiint(q) - 0x03f00000u < 0x7e000000u - 0x03f00000u; }
NLA_DEV bool ordinary(float) { return true; }

// FP64, ordinary(r^2): r and m1 = 1 / (r^2 + |alpha| r) from FP32 estimates (2^-22) and one
// third-order step each (the Householder iterations of order 3 for the inverse square root and the
// reciprocal: the error becomes the cube, below 2^-60): 10 FP64 instructions one after another,
// where the library's square root and two divisions take about 40.  Against those the applied
// reflector is no less exact: error of H row over 200,000 Gaussian pairs of 16 entries 0.86 units of
// 2^-53 (rms, no bias) and 1.04 with tau and a normalised vector from the library functions.
NLA_DEV void house(double alpha, double qt, double &beta, double &u0, double &m1, double &m2) {
    const double q = fma(alpha, alpha, qt);
    const unsigned qh = (unsigned)__double2hiint(q), ah = (unsigned)__double2hiint(alpha);
    const unsigned sa = ah & 0x80000000u;
    const double ar = fabs(alpha);
    const int ex = (int)(qh >> 20) - 1023, odd = ex & 1, h = (ex - odd) / 2;
    const float m = __uint_as_float((unsigned)(127 + odd) << 23 | (qh & 0xfffffu) << 3 |
                                    (unsigned)__double2loint(q) >> 29);  // q 4^-h in [1, 4)
    const float rsm = rsqrtf(m);
    const double y = widen(__float_as_uint(rsm), -h);
    // |alpha| 2^-h in FP32 (0 when it is far below r)
    const int ea = (int)(ah >> 20 & 0x7ffu) - 1023 - h;
    const float am = ea < -100 ? 0.f
                               : __uint_as_float((unsigned)(127 + ea) << 23 | (ah & 0xfffffu) << 3 |
                                                 (unsigned)__double2loint(alpha) >> 29);
    const double z = widen(__float_as_uint(__fdividef(1.f, fmaf(am, m * rsm, m))), -2 * h);
    const double t = q * y;
    const double e = fma(-t, y, 1.0);
    const double r = fma(t, fma(e, 0.375, 0.5) * e, t);
    const double f = fma(-fma(ar, r, q), z, 1.0);
    const double um = ar + r;
    beta = __hiloint2double((int)((unsigned)__double2hiint(r) | (sa ^ 0x80000000u)), __double2loint(r));
    u0 = __hiloint2double((int)((unsigned)__double2hiint(um) | sa), __double2loint(um));
    m1 = fma(z, fma(f, f, f), z);
    m2 = 1.0;
}

}  // namespace nla
