// FP64 collision with most of its arithmetic in pairs of FP32 numbers.
//
// GB300 issues one FP64 instruction per warp and scheduler every 64 cycles (77
// with all four busy), an FP32 one every cycle; the plain FP64 collision (about
// 120 operations) is bound by that pipe by a factor of twenty over memory.
// Here a node takes 18 FP64 operations:
//   d_i  = f_i - w_i R      exact to FP64, R the density rounded to FP32;
//   f_i' = f_i + delta_i    the collision's increment (Eq. 6), rounded to FP64;
// and delta is computed from d in pairs h + l of FP32 numbers (48 bits; the
// sums and products of Dekker and Knuth), at about 900 FP32 operations.  d and
// delta are small where the flow is near equilibrium, so their 48 bits reach
// below the last bit of f; a node where they are not small (|d_i| > R/32, a flow
// above 0.094 lattice speeds, or R not from 2^-12 to 2^30) takes the plain FP64
// collision instead.  Up to that bound the populations' rms error stays below the
// plain collision's; at twice the bound it would not (see below).
//
// Measured, 25601 x 256 pressure channel: 313 us per sweep against 1455 us;
// the 18 FP64 operations alone take 225 us.  rms error of a population after
// one collision, relative to the density, against long double: 8e-18 to 1.6e-17
// for velocities of 1e-3 to 0.04 and 2.8e-17 at 0.08, against 3.4e-17 of the plain
// form (whose moments sum populations, not deviations); 4.4e-17 at 0.12, beyond the
// bound.  Density and momentum as before, 4 to 10 % more at non-equilibrium parts of
// 1 %.  Whole runs end closer to long double than with the plain form: 4 x 32
// periodic, 1000 steps, rms of the state 7.6e-17 against 3.1e-16.
//
// A flow beyond the bound pays for both forms.  us per step, against the plain
// collision alone: 200 x 20 pressure at a velocity of 0.114 20.4 / 12.9, 457 x 33 at
// 0.19 18.9 / 13.5, 300 x 128 at 0.33 23.1 / 21.0, 801 x 17 periodic at 0.21 10.3 /
// 8.8; within it 200 x 20 at 0.053 5.9 / 13.0.
//
// Host compilers see the same arithmetic (no fused contraction), so that its
// error can be measured there.
#pragma once

#include <cstdint>
#include <cstring>

#ifndef __CUDACC__
#include <cmath>
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace clb {
namespace pr {

#define CLB_HD __host__ __device__ __forceinline__

#ifdef __CUDA_ARCH__
CLB_HD float fadd(float a, float b) { return __fadd_rn(a, b); }
CLB_HD float fsub(float a, float b) { return __fsub_rn(a, b); }
CLB_HD float fmul(float a, float b) { return __fmul_rn(a, b); }
CLB_HD float ffma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
CLB_HD uint32_t bits(float a) { return __float_as_uint(a); }
CLB_HD float real(uint32_t a) { return __uint_as_float(a); }
CLB_HD uint32_t hi(double a) { return (uint32_t)__double2hiint(a); }
CLB_HD uint32_t lo(double a) { return (uint32_t)__double2loint(a); }
CLB_HD double real(uint32_t h, uint32_t l) { return __hiloint2double((int)h, (int)l); }
CLB_HD float to_float(int32_t a) { return __int2float_rn(a); }
CLB_HD int32_t to_int(float a) { return __float2int_rn(a); }
CLB_HD float recip(float a) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
CLB_HD double dadd(double a, double b) { return __dadd_rn(a, b); }
CLB_HD double dfma(double a, double b, double c) { return __fma_rn(a, b, c); }
#else
CLB_HD float fadd(float a, float b) { return a + b; }
CLB_HD float fsub(float a, float b) { return a - b; }
CLB_HD float fmul(float a, float b) { return a * b; }
CLB_HD float ffma(float a, float b, float c) { return fmaf(a, b, c); }
CLB_HD uint32_t bits(float a) {
    uint32_t u;
    memcpy(&u, &a, 4);
    return u;
}
CLB_HD float real(uint32_t a) {
    float f;
    memcpy(&f, &a, 4);
    return f;
}
CLB_HD uint64_t bits(double a) {
    uint64_t u;
    memcpy(&u, &a, 8);
    return u;
}
CLB_HD uint32_t hi(double a) { return (uint32_t)(bits(a) >> 32); }
CLB_HD uint32_t lo(double a) { return (uint32_t)bits(a); }
CLB_HD double real(uint32_t h, uint32_t l) {
    const uint64_t u = ((uint64_t)h << 32) | l;
    double d;
    memcpy(&d, &u, 8);
    return d;
}
CLB_HD float to_float(int32_t a) { return (float)a; }
CLB_HD int32_t to_int(float a) { return (int32_t)lrintf(a); }
CLB_HD float recip(float a) { return 1.0f / a; }
CLB_HD double dadd(double a, double b) { return a + b; }
CLB_HD double dfma(double a, double b, double c) { return fma(a, b, c); }
#endif

// h + l; normalised: |l| <= ulp(h)/2.  Sums leave their result unnormalised
// (|l| a few ulps of the larger operand), products want normalised operands.
struct P {
    float h, l;
};

// exact a + b = h + l (Knuth)
CLB_HD P two_sum(float a, float b) {
    const float s = fadd(a, b), z = fsub(s, a);
    return {s, fadd(fsub(a, fsub(s, z)), fsub(b, z))};
}
CLB_HD P add(P a, P b) {
    const P s = two_sum(a.h, b.h);
    return {s.h, fadd(s.l, fadd(a.l, b.l))};
}
CLB_HD P neg(P a) { return {-a.h, -a.l}; }
CLB_HD P sub(P a, P b) { return add(a, neg(b)); }
CLB_HD P norm(P a) {  // Dekker's fast two-sum: |h| >= |l|, or h = 0
    const float s = fadd(a.h, a.l);
    return {s, fsub(a.l, fsub(s, a.h))};
}
// operands normalised; the result is unnormalised by an ulp or two
CLB_HD P mul(P a, P b) {
    const float p = fmul(a.h, b.h);
    float e = ffma(a.h, b.h, -p);
    e = ffma(a.h, b.l, e);
    e = ffma(a.l, b.h, e);
    return {p, e};
}
CLB_HD P mad(P a, P b, P c) { return add(mul(a, b), c); }   // a b + c
CLB_HD P msub(P a, P b, P c) { return add(mul(neg(a), b), c); }  // c - a b
CLB_HD P twice(P a) { return {fmul(2.0f, a.h), fmul(2.0f, a.l)}; }
CLB_HD P scale(P a, float p2) { return {fmul(p2, a.h), fmul(p2, a.l)}; }  // by a power of two
// constants (folded at compile time, or on the host)
CLB_HD constexpr P pair_of(double v) { return {(float)v, (float)(v - (double)(float)v)}; }
// Whether a density can be split and collided with (2^-12 to 2^30), by its high
// word: a NaN, an infinity, a negative or another number out of FP32's range
// would come out of split as some finite one.
CLB_HD bool in_range(double v) {
    const uint32_t m = hi(v);
    return m >= (1011u << 20) && m < (1053u << 20);
}
// 1 / a for normalised a > 0: the FP32 reciprocal y and its correction
// y (e + e^2), e = 1 - a y formed with fused multiply-adds.
CLB_HD P inv(P a) {
    const float y = recip(a.h);
    const float e = ffma(-a.l, y, ffma(-a.h, y, 1.0f));
    return norm({y, fmul(y, ffma(e, e, e))});
}

// The double d as an FP32 pair, by its bits (a conversion instruction costs as
// much as an FP64 operation): h its leading 24 bits, l the other 29 rounded to
// 24.  m: the high word of |d|.  Magnitudes under 2^-73 become 2^-73, far below
// the last bit of the densities this is used at (R >= 2^-12), which spares the
// cases of zero and underflow.
CLB_HD P split(double d, uint32_t m) {
    const uint32_t u = hi(d), w = lo(d);
    m = m < (950u << 20) ? 950u << 20 : m;
    // an exponent field of 11 bits less 896, in 8 bits: its low 8 with the top one flipped
    const uint32_t t = (m << 3) | (w >> 29);
    const uint32_t h = (((t & 0x7fffffffu) | (u & 0x80000000u)) ^ 0x40000000u);
    const float s = real((h & 0xff800000u) - (52u << 23));  // the unit of the lower 29 bits, signed
    return {real(h), fmul(to_float((int32_t)(w & 0x1fffffffu)), s)};
}
CLB_HD P split(double d) { return split(d, hi(d) & 0x7fffffffu); }
// The normalised pair as a double: the double h, its bits moved on by l in
// units of h's last place among 53 bits (twice as many below a power of two,
// where the places are half as wide).  The sum h + l rounded to FP64, down to
// |h| = 2^-75; smaller ones, and 0, come out as something below 2^-74.
CLB_HD double join(P a) {
    const uint32_t u = bits(a.h), sign = u & 0x80000000u;
    const float s = real((0x99000000u - (u & 0x7f800000u)) | sign);  // 2^(52 - exponent), signed
    float p = fmul(a.l, s);
    if (p < 0.0f && (u << 9) == 0) p = fadd(p, p);
    const int32_t l = to_int(p);
    const uint32_t x = u << 29, y = x + (uint32_t)l;
    const uint32_t h = ((u & 0x7fffffffu) >> 3) + (896u << 20) + (uint32_t)(l >> 31) + (y < x ? 1u : 0u);
    return real(h | sign, y);
}

// Launch constants of the pair collision.
struct Const {
    P s3_12, s8_4, sv_4, sq_4;  // as KC
    P A, B, A316, CA;
    P fx, hfx;
    bool fits;                  // every constant is one that pairs can hold (fits)
};
// Whether a launch constant can be held and multiplied as a pair: below 2^40 in
// magnitude, so that the largest product of the rates, B (A316 B), stays in
// FP32's range and the reciprocal's.  (ny Kn from 1.3e-13 to 8e11; beyond, every
// node takes the plain FP64 collision.)
CLB_HD bool fits(double v) { return v < 0x1p40 && v > -0x1p40; }

// Densities of the populations f: R, about their sum (to 2^-19, each taken by
// the high word of its double), the deviations d from w_i R as pairs
// (normalised), and whether they are small enough for the pairs.
CLB_HD bool deviations(const double (&f)[9], float& R, P (&d)[9]) {
    // a positive double's high word as a float: eight times, less the exponents' offset
    float s = 0.0f;
    for (int i = 0; i < 9; ++i) {
        const float v = real(hi(f[i]) * 8u - (896u << 23));
        s = i ? fadd(s, v) : v;
    }
    R = s;
    const uint32_t u = bits(s), rh = (u >> 3) + (896u << 20);  // R as a double, by its bits
    const double Rd = real(rh, u << 29);
    uint32_t big = 0;
    for (int i = 0; i < 9; ++i) {
        const double w = i == 0 ? 4.0 / 9.0 : i < 5 ? 1.0 / 9.0 : 1.0 / 36.0;
        const double v = dfma(-w, Rd, f[i]);
        const uint32_t m = hi(v) & 0x7fffffffu;
        big = m > big ? m : big;
        d[i] = split(v, m);
    }
    // |d| <= R/32, compared as high words: a NaN, an infinity or a value out
    // of FP32's range (whose R means nothing) is above
    return R >= 2.4414062e-4f && R <= 1.07e9f && big < rh - (5u << 20);
}

struct Moments {
    P rho, drho, jx, jy;                       // rho = R + drho
    P kxx, kyy, nkxy, kxxy, kxyy, kxxyy;       // deviation parts (Eq. 8)
};
CLB_HD void moments(float R, const P (&d)[9], Moments& m) {
    const P a57 = add(d[5], d[7]), a68 = add(d[6], d[8]), p57 = sub(d[5], d[7]), p86 = sub(d[8], d[6]);
    m.nkxy = sub(a68, a57);
    m.kxxyy = add(a57, a68);
    m.kxxy = sub(p57, p86);
    m.kxyy = add(p57, p86);
    const P s13 = add(d[1], d[3]), s24 = add(d[2], d[4]);
    m.kxx = add(s13, m.kxxyy);
    m.kyy = add(s24, m.kxxyy);
    m.drho = norm(add(add(add(d[0], s13), s24), m.kxxyy));  // below 2^-18 R
    m.jx = norm(add(sub(d[1], d[3]), m.kxyy));
    m.jy = norm(add(sub(d[2], d[4]), m.kxxy));
    const P r = two_sum(R, m.drho.h);
    m.rho = norm({r.h, fadd(r.l, m.drho.l)});
}

// The collision's increments for the deviations d from w_i R (collide in
// clb_device.cuh, term by term; FORCE: body force along x and constant rates,
// else rates from rho_kn or, where that is null, from the node's density).
template <bool FORCE> CLB_HD void collide(float R, const P (&d)[9], const Const& c, const P* rho_kn, P (&o)[9]) {
    Moments m;
    moments(R, d, m);
    const P rho = m.rho, irho = inv(rho);
    P sv4 = c.sv_4, sq4 = c.sq_4;
    if (!FORCE) {
        const P q = norm(add(rho_kn ? *rho_kn : rho, c.B)), q4 = scale(q, 0.25f);
        const P hv = norm(add(scale(q, 0.5f), c.A));
        const P in = norm(add(mul(c.A316, q), {0.5f, 0.0f}));
        const P hq = norm(mad(q, in, c.CA));
        sv4 = norm(mul(q4, inv(hv)));
        sq4 = norm(mul(q4, inv(hq)));
    }
    P ux = mul(m.jx, irho);
    if (FORCE) ux = add(ux, c.hfx);
    ux = norm(ux);
    const P uy = norm(mul(m.jy, irho));
    const P ux2 = norm(mul(ux, ux)), uy2 = norm(mul(uy, uy)), uxy = norm(mul(ux, uy));
    const P ux_2 = twice(ux), uy_2 = twice(uy);
    const P third = mul({R, 0.0f}, pair_of(1.0 / 3.0));
    const P kxxf = norm(add(third, m.kxx)), kyyf = norm(add(third, m.kyy));
    const P t5u = norm(mad(rho, uxy, m.nkxy));
    P t3 = add(mul(rho, norm(add(ux2, uy2))), sub(mul(m.drho, pair_of(2.0 / 3.0)), add(m.kxx, m.kyy)));
    P t4 = add(mul(rho, norm(sub(ux2, uy2))), sub(m.kyy, m.kxx));
    P t5 = t5u;
    P t6 = mad(ux_2, t5u, msub(uy, kxxf, m.kxxy));
    P t7 = mad(uy_2, t5u, msub(ux, kyyf, m.kxyy));
    const P kxxy = norm(m.kxxy), kxyy = norm(m.kxyy);
    P t8 = add(mul(m.drho, pair_of(1.0 / 9.0)),
               mul(uxy, norm(add({fmul(3.0f, t5u.h), ffma(3.0f, t5u.l, ffma(3.0f, t5u.h, -fmul(3.0f, t5u.h)))}, m.nkxy))));
    t8 = mad(ux_2, kxyy, t8);
    t8 = mad(uy_2, kxxy, t8);
    t8 = sub(t8, mad(ux2, kyyf, mad(uy2, kxxf, m.kxxyy)));
    P rf{0.0f, 0.0f};
    if (FORCE) {
        rf = norm(mul(rho, c.fx));
        const P fu = mul(rf, ux), half = scale(rf, 0.5f);
        t3 = sub(t3, fu);
        t4 = sub(t4, fu);
        t5 = norm(msub(half, uy, t5));
        t6 = msub(rf, uxy, t6);
        t7 = msub(half, uy2, t7);
        t8 = msub(rf, norm(mul(ux, uy2)), t8);
    }
    const P g3 = norm(mul(c.s3_12, norm(t3)));
    const P g4 = norm(mul(sv4, norm(t4)));
    const P g5 = norm(mul(sv4, t5));
    const P g15 = {fmul(1.5f, g3.h), ffma(1.5f, g3.l, ffma(1.5f, g3.h, -fmul(1.5f, g3.h)))}, g42 = scale(g4, 0.5f);
    const P hp = norm(add(g15, g42)), hm = norm(sub(g15, g42));
    const P g6 = norm(add(mul(sq4, norm(t6)), neg(mad(uy, hp, mul(ux_2, g5)))));
    const P g7 = norm(add(mul(sq4, norm(t7)), neg(mad(ux, hm, mul(uy_2, g5)))));
    P b8 = mad(uy2, hp, twice(g3));
    b8 = mad(ux2, hm, b8);
    b8 = mad(scale(uxy, 4.0f), g5, b8);
    b8 = mad(uy_2, g6, b8);
    b8 = mad(ux_2, g7, b8);
    const P g8 = sub(mul(c.s8_4, norm(t8)), b8);
    // Eq. 6
    o[0] = scale(sub(g8, g3), 4.0f);
    const P ca = sub(g4, g3), s34 = neg(add(g3, g4)), ce = add(twice(g3), g8);
    const P n8 = neg(twice(g8)), c8 = add(ca, n8), e8 = add(s34, n8), g6_2 = twice(g6), g7_2 = twice(g7);
    o[1] = add(c8, g7_2);
    o[3] = sub(c8, g7_2);
    o[2] = add(e8, g6_2);
    o[4] = sub(e8, g6_2);
    const P e5 = add(ce, g5), e6 = sub(ce, g5), gp = add(g6, g7), gm = sub(g6, g7);
    o[5] = sub(e5, gp);
    o[7] = add(e5, gp);
    o[6] = sub(e6, gm);
    o[8] = add(e6, gm);
    if (FORCE) {  // S = T^-1 S^ (Eq. 9-10)
        const P q1 = scale(rf, 0.5f);                            // m1 / 2
        const P m3 = mul(scale(rf, 2.0f), ux);                   // = m4
        const P m5 = mul(rf, uy), m6 = mul(scale(rf, 2.0f), uxy), m7 = norm(mul(rf, uy2));
        const P m8 = twice(mul(m7, ux));
        const P x = scale(sub(m3, m8), 0.5f), y = sub(q1, scale(m7, 0.5f)), z = scale(m8, -0.5f), w = scale(m6, -0.5f);
        o[0] = add(o[0], sub(m8, m3));
        o[1] = add(o[1], add(x, y));
        o[3] = add(o[3], sub(x, y));
        o[2] = add(o[2], add(z, w));
        o[4] = add(o[4], sub(z, w));
        const P p56 = add(m5, m6), n56 = sub(m6, m5), p78 = add(m7, m8), n78 = sub(m8, m7);
        o[5] = add(o[5], scale(add(p56, p78), 0.25f));
        o[6] = add(o[6], scale(add(n56, n78), 0.25f));
        o[7] = add(o[7], scale(sub(n78, n56), 0.25f));
        o[8] = add(o[8], scale(sub(p78, p56), 0.25f));
    }
}

// Velocity of a node from its moments.
CLB_HD void velocity(const Moments& m, P& ux, P& uy) {
    const P irho = inv(m.rho);
    ux = norm(mul(m.jx, irho));
    uy = norm(mul(m.jy, irho));
}

// Moments 3..8 of the equilibrium (Eq. 11) without their parts linear in the
// density alone.
CLB_HD void eq_moments(P rho, P ux, P uy, P (&m)[9]) {
    const P ux2 = norm(mul(ux, ux)), uy2 = norm(mul(uy, uy)), u2 = norm(add(ux2, uy2)), third = pair_of(1.0 / 3.0);
    m[1] = norm(mul(rho, ux));
    m[2] = norm(mul(rho, uy));
    m[3] = norm(mul(rho, u2));
    m[4] = mul(rho, norm(sub(ux2, uy2)));
    m[5] = mul(m[1], uy);
    m[6] = mul(m[2], norm(add(third, ux2)));
    m[7] = mul(m[1], norm(add(third, uy2)));
    m[8] = add(mul(m[3], third), mul(norm(mul(m[1], ux)), uy2));
}

// f^eq_i(rho + dr, vx, vy) - f^eq_i(rho, ux, uy) of the nine populations: what
// the rebuilt end column (Sec. 3.2) adds to its neighbour's.
CLB_HD void eq_difference(P rho, P dr, P ux, P uy, P vx, P vy, P (&o)[9]) {
    P a[9], b[9], m[9];
    eq_moments(rho, ux, uy, a);
    eq_moments(norm(add(rho, dr)), vx, vy, b);
    for (int k = 1; k < 9; ++k) m[k] = sub(b[k], a[k]);
    m[3] = add(m[3], mul(dr, pair_of(2.0 / 3.0)));
    m[8] = add(m[8], mul(dr, pair_of(1.0 / 9.0)));
    o[0] = add(sub(dr, m[3]), m[8]);
    const P c = sub(m[3], twice(m[8])), x = twice(sub(m[1], m[7])), y = twice(sub(m[2], m[6]));
    const P p = add(c, m[4]), q = sub(c, m[4]);
    o[1] = scale(add(p, x), 0.25f);
    o[3] = scale(sub(p, x), 0.25f);
    o[2] = scale(add(q, y), 0.25f);
    o[4] = scale(sub(q, y), 0.25f);
    const P s56 = add(m[5], m[6]), n56 = sub(m[6], m[5]), s78 = add(m[7], m[8]), n78 = sub(m[8], m[7]);
    o[5] = scale(add(s56, s78), 0.25f);
    o[6] = scale(add(n56, n78), 0.25f);
    o[7] = scale(sub(n78, n56), 0.25f);
    o[8] = scale(sub(s78, s56), 0.25f);
}

#undef CLB_HD
}  // namespace pr
}  // namespace clb
