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
// FP32 keeps the factors apart everywhere.  What is left: (u^T row) m1 m2 overflows where a vector
// below 2^-63 meets coefficients above 2^62; below 2^-66 its norm has lost its digits anyway, and a
// test on the chain cost 3 % of the chase.
NLA_DEV bool ordinary(float) { return true; }

// The FP64 scalars, for an ordinary q only, start from FP32 estimates (2^-22) of
// q = alpha^2 + qt, r = |x| = sqrt(q), and take one third-order step each (the Householder
// iterations of order 3 for the inverse square root and the reciprocal: the error becomes the cube,
// below 2^-60).  FP64 instructions are what counts: about a dozen one after another, where the
// library's square root and two divisions take about 40.  The reflector is no less exact for it
// (Gaussian vectors of 9 to 23 entries, units of 2^-53, no bias): rms error of H row 0.86 in either
// form below, 1.04 with tau, the scale and a normalised vector from the library functions;
// tau (1 + |v|^2) / 2 - 1 of a stored vector 0.80 (house_tau) and 0.79.  tau and the scale as
// products of house's m1, u_0 and beta came to 1.96.
struct RootEstimate {
    double q, y;       // y ~ 1 / r
    float m, rsm, am;  // q 4^-h in [1, 4), its inverse root, |alpha| 2^-h (0 when it is far below r)
    int h;
    unsigned sign;     // of alpha
};
NLA_DEV RootEstimate root_estimate(double alpha, double qt) {
    RootEstimate e;
    e.q = fma(alpha, alpha, qt);
    const unsigned qh = (unsigned)__double2hiint(e.q), ah = (unsigned)__double2hiint(alpha);
    const int ex = (int)(qh >> 20) - 1023, odd = ex & 1;
    e.h = (ex - odd) / 2;
    e.sign = ah & 0x80000000u;
    e.m = __uint_as_float((unsigned)(127 + odd) << 23 | (qh & 0xfffffu) << 3 | (unsigned)__double2loint(e.q) >> 29);
    e.rsm = rsqrtf(e.m);
    e.y = widen(__float_as_uint(e.rsm), -e.h);
    const int ea = (int)(ah >> 20 & 0x7ffu) - 1023 - e.h;
    e.am = ea < -100 ? 0.f
                     : __uint_as_float((unsigned)(127 + ea) << 23 | (ah & 0xfffffu) << 3 |
                                       (unsigned)__double2loint(alpha) >> 29);
    return e;
}
NLA_DEV double with_sign(double magnitude, unsigned sign) {
    return __hiloint2double((int)((unsigned)__double2hiint(magnitude) | sign), __double2loint(magnitude));
}
// beta, u_0 and m1 = 1 / (r^2 + |alpha| r).
NLA_DEV void house(double alpha, double qt, double &beta, double &u0, double &m1, double &m2) {
    const RootEstimate s = root_estimate(alpha, qt);
    const double ar = fabs(alpha);
    const double z = widen(__float_as_uint(__fdividef(1.f, fmaf(s.am, s.m * s.rsm, s.m))), -2 * s.h);
    const double t = s.q * s.y;
    const double e = fma(-t, s.y, 1.0);
    const double r = fma(t, fma(e, 0.375, 0.5) * e, t);
    const double f = fma(-fma(ar, r, s.q), z, 1.0);
    beta = with_sign(r, s.sign ^ 0x80000000u);
    u0 = with_sign(ar + r, s.sign);
    m1 = fma(z, fma(f, f, f), z);
    m2 = 1.0;
}
// The same reflector as tau = (beta - alpha) / beta = 1 + |alpha| / r and scale = 1 / u_0, for a
// vector that is normalised to v_0 = 1; r gets a Newton step and |alpha| + r is never rounded.
NLA_DEV void house_tau(double alpha, double qt, double &beta, double &tau, double &scale) {
    const RootEstimate s = root_estimate(alpha, qt);
    const double ar = fabs(alpha);
    const double z = widen(__float_as_uint(__fdividef(1.f, fmaf(s.m, s.rsm, s.am))), -s.h);
    const double t = s.q * s.y;
    const double e = fma(-t, s.y, 1.0);
    const double p = fma(e, 0.375, 0.5) * e;
    const double r1 = fma(t, p, t);
    const double r = fma(fma(-r1, r1, s.q), widen(__float_as_uint(s.rsm), -s.h - 1), r1);
    const double f = fma(-r, z, fma(-ar, z, 1.0));
    beta = with_sign(r, s.sign ^ 0x80000000u);
    tau = fma(ar, fma(s.y, p, s.y), 1.0);
    scale = with_sign(fma(z, fma(f, f, f), z), s.sign);
}

}  // namespace nla
