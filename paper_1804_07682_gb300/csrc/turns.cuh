// turns.cuh -- phases and their cosines in 64-bit integers, for the
// element-wise probability.
//
// The FP64 unit runs at 1/64 of the FP32 rate on this GPU and a conversion to
// or from double takes a slot of it; 32-bit integer multiplies run at half the
// FP32 rate.  So a phase x = c / E is formed as the fraction of x / pi (sin^2 x
// and sin 2x have period pi) in units of 2^-64, and cos 2x and sin 2x come from
// a table of 512 angles and two short series in the remainder, all in integers.
// c / pi is held to 2^-62 of itself and 1 / E to 2^-61, so the phase is good to
// its number of half-turns times 2^-60 (a double phase: 2^-52), and cos 2x to
// 2^-61.  Everything here also compiles for the host.
#pragma once

#include <stdint.h>

#include "turn_table.h"

namespace gna {

#if defined(__CUDACC__)
#define GNA_HD __host__ __device__ __forceinline__
#else
#define GNA_HD inline
#endif

// |c| / pi = m 2^(e - 64) with m in [2^63, 2^64) (or m = 0), and its sign.
struct TurnCoef {
    uint64_t m;
    int e;
    int neg;
};

// 1 / E = y 2^(-63 - e), y in (2^62, 2^63].
struct TurnRecip {
    uint64_t y;
    int e;
};

// x = c / E is taken in turns.cuh's arithmetic while |x| / pi < 2^30 and
// >= 2^-35; `shift` below is then within -32 .. 31.
GNA_HD bool turn_shift_ok(int shift) { return (unsigned)(shift + 32) < 64u; }

// Left shift that brings the 128-bit product m y to turns in units of 2^-64
// (its upper 64 bits): the number of half-turns is in (2^(shift-3), 2^(shift-1)].
GNA_HD int turn_shift(int ec, int ee) { return ec - ee + 1; }

GNA_HD uint32_t funnel_left(uint32_t lo, uint32_t hi, int n) {
#if defined(__CUDA_ARCH__)
    return __funnelshift_l(lo, hi, n);
#else
    return n ? (hi << n) | (lo >> (32 - n)) : hi;
#endif
}

// Reciprocal of the double with words (hi, lo), a positive normal number: the
// hardware's FP32 reciprocal of its leading 24 bits (24 bits of y0), then
// 1/E = y0 (1 + r + r^2), r = 1 - E y0 exact in the low 64 bits of the product.
// |r| < 2^-21, so the neglected r^3 is below 2^-62.
GNA_HD TurnRecip turn_recip(uint32_t hi, uint32_t lo) {
    const uint32_t mf = (funnel_left(lo, hi, 3) & 0x7fffffu) | 0x3f800000u;
    uint32_t yb;
#if defined(__CUDA_ARCH__)
    float yf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(__uint_as_float(mf)));
    yb = __float_as_uint(yf);
#else
    union {
        uint32_t u;
        float f;
    } a, b;
    a.u = mf;
    b.f = 1.0f / a.f;
    yb = b.u;
#endif
    const uint32_t y0 = yb - 0x3e800000u;  // y0 2^-24: linear in the bits on (1/2, 1], 2^24 at 1
    const uint32_t mh = (hi & 0xfffffu) | 0x100000u;
    const uint64_t p = (uint64_t)lo * y0 + ((uint64_t)(mh * y0) << 32);  // E y0 2^76 mod 2^64
    const int64_t r = (int64_t)(0 - p);
    const int32_t rh = (int32_t)(r >> 32);
    const int64_t t = r + (((int64_t)rh * rh) >> 12);
    const int64_t s = (int64_t)(int32_t)(t >> 32) * (int32_t)y0 + (int64_t)(((uint64_t)(uint32_t)t * y0) >> 32);
    TurnRecip o;
    o.y = ((uint64_t)y0 << 39) + (uint64_t)(s >> 5);
    o.e = (int)((hi >> 20) & 0x7ff) - 1023;
    return o;
}

// Fraction of the phase x / pi in units of 2^-64, for the shift of
// turn_shift().  The product of the two low words is left out: 2^-95 of the
// full scale of m y.
GNA_HD uint64_t turn_phase(uint64_t m, int neg, uint64_t y, int shift) {
    const uint32_t ml = (uint32_t)m, mh = (uint32_t)(m >> 32), yl = (uint32_t)y, yh = (uint32_t)(y >> 32);
    const uint64_t t = (uint64_t)ml * yh;
    const uint64_t t2 = (uint64_t)mh * yl + (uint32_t)t;
    const uint64_t h = (uint64_t)mh * yh + (t >> 32) + (t2 >> 32);
    const uint32_t w1 = (uint32_t)t2, w2 = (uint32_t)h, w3 = (uint32_t)(h >> 32);
    const bool right = shift < 0;  // then a whole word further down
    const uint32_t a2 = right ? 0u : w3, a1 = right ? w3 : w2, a0 = right ? w2 : w1;
    const int n = shift & 31;
    const uint64_t f = ((uint64_t)funnel_left(a1, a2, n) << 32) | funnel_left(a0, a1, n);
    return neg ? 0 - f : f;
}

// (a b) >> 64 without the product of the two low halves (an error of at most
// three units); |a|, |b| <= 2^63 and not both near it.
GNA_HD int64_t mul_hi(int64_t a, int64_t b) {
    const int32_t ah = (int32_t)(a >> 32), bh = (int32_t)(b >> 32);
    const int32_t al = (int32_t)((uint32_t)a >> 1), bl = (int32_t)((uint32_t)b >> 1);
    const int64_t mid = (int64_t)ah * bl + (int64_t)al * bh;
    return (int64_t)ah * bh + (mid >> 31);
}

// w = 2 pi d for the remainder d (|d| <= 2^-10 turns, `dd` = d 2^73):
// g = (1 - cos w) 2^69, s = sin w 2^69.
GNA_HD void turn_small(int64_t dd, int64_t& g, int64_t& s) {
    const int32_t dh = (int32_t)(dd >> 32), dl = (int32_t)((uint32_t)dd >> 1);
    const int64_t u = (int64_t)dh * dh + (((int64_t)dh * dl) >> 30);  // d^2 2^82
    const int32_t v = (int32_t)(u >> 32);                             // d^2 2^50, <= 2^30
    const int32_t c2 = (int32_t)GNA_TURN_C2_Q24 - (int32_t)(((int64_t)v * (int32_t)GNA_TURN_C3_Q24) >> 50);
    const int64_t c1 = GNA_TURN_C1_Q58 - (((int64_t)v * c2) >> 16);
    g = mul_hi(u, c1) >> 7;
    const int64_t s1 = GNA_TURN_S1_Q57 - (((int64_t)v * (int32_t)GNA_TURN_S2_Q24) >> 17);
    const int64_t s0 = GNA_TURN_S0_Q60 - (mul_hi(u, s1) >> 15);
    s = mul_hi(dd, s0);
}

// Nearest of the 512 angles to the fraction f, and the remainder times 2^73.
GNA_HD int turn_split(uint64_t f, int64_t& dd) {
    const uint32_t fh = (uint32_t)(f >> 32);
    const uint32_t k = (fh + (1u << 22)) >> 23;
    dd = (int64_t)((f - ((uint64_t)k << 55)) << 9);
    return (int)(k & 511u);
}

// (c g + z s) >> 64 and the like: two products summed before they are cut.
GNA_HD int64_t mul_hi2(int64_t a, int64_t b, int64_t c, int64_t d) {
    const int32_t ah = (int32_t)(a >> 32), bh = (int32_t)(b >> 32), ch = (int32_t)(c >> 32), dh = (int32_t)(d >> 32);
    const int32_t al = (int32_t)((uint32_t)a >> 1), bl = (int32_t)((uint32_t)b >> 1);
    const int32_t cl = (int32_t)((uint32_t)c >> 1), dl = (int32_t)((uint32_t)d >> 1);
    const int64_t mid = (int64_t)ah * bl + (int64_t)al * bh + (int64_t)ch * dl + (int64_t)cl * dh;
    return (int64_t)ah * bh + (int64_t)ch * dh + (mid >> 31);
}

// cos 2x and sin 2x times 2^62 from the table entry (c, z) of x's nearest angle.
GNA_HD int64_t turn_cos(int64_t c, int64_t z, int64_t g, int64_t s) { return c - (mul_hi2(c, g, z, s) >> 5); }
GNA_HD int64_t turn_sin(int64_t c, int64_t z, int64_t g, int64_t s) { return z + (mul_hi2(c, s, z, -g) >> 5); }

// Host: c / pi as mantissa, exponent and sign; false for a value that is not finite.
inline bool turn_coef(double c, TurnCoef& o) {
    union {
        double d;
        uint64_t u;
    } b;
    b.d = c;
    o.neg = (int)(b.u >> 63);
    const int ex = (int)((b.u >> 52) & 0x7ff);
    const uint64_t frac = b.u & 0xfffffffffffffull;
    if (ex == 0x7ff) return false;
    o.m = 0;
    o.e = 0;
    if (ex == 0 && frac == 0) return true;
    if (ex == 0) return false;  // subnormal: left to the double path
    const uint64_t m = (frac | (1ull << 52)) << 11;  // c = m 2^(ex - 1023 - 63)
    // m and the constant are in [2^63, 2^64): their product has 127 or 128 bits
    const uint64_t a = m, k = GNA_INV_PI_Q65;
    const uint64_t al = a & 0xffffffffu, ah = a >> 32, kl = k & 0xffffffffu, kh = k >> 32;
    const uint64_t ll = al * kl, lh = al * kh, hl = ah * kl, hh = ah * kh;
    const uint64_t mid = (ll >> 32) + (lh & 0xffffffffu) + (hl & 0xffffffffu);
    uint64_t hi = hh + (lh >> 32) + (hl >> 32) + (mid >> 32);
    const uint64_t lo = (mid << 32) | (ll & 0xffffffffu);
    // c / pi = (hi : lo) 2^(ex - 1023 - 63 - 65) = hi 2^(ex - 1023 - 64)
    int e = ex - 1023;
    if (!(hi >> 63)) {
        hi = (hi << 1) | (lo >> 63);
        e -= 1;
    }
    o.m = hi;
    o.e = e;
    return true;
}

}  // namespace gna
