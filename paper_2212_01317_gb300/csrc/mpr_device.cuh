// Device building blocks of the SV-MPR sweep: Philox4x32-10, the (0,1)
// uniform, and one Metropolis + over-relaxation update of a gap site.
#pragma once
#include <cstdint>

#include "mpr_internal.h"

namespace mpr {

constexpr float kTwoPi = 6.28318530717958647692f;

// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): ten rounds of two
// 32x32->64 multiplies; the key advances by the Weyl constants between rounds.
__device__ __forceinline__ void philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                              uint32_t k0, uint32_t k1, uint32_t out[4]) {
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const uint64_t pa = (uint64_t)0xD2511F53u * c0;
        const uint64_t pb = (uint64_t)0xCD9E8D57u * c2;
        c0 = (uint32_t)(pb >> 32) ^ c1 ^ k0;
        c1 = (uint32_t)pb;
        c2 = (uint32_t)(pa >> 32) ^ c3 ^ k1;
        c3 = (uint32_t)pa;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    out[0] = c0;
    out[1] = c1;
    out[2] = c2;
    out[3] = c3;
}

// The same generator with the round keys of key word 0 given (k0 + r W0 for
// r = 0 .. 9, taken from kernel parameters, where the XOR reads them
// directly); key word 1 advances in the loop.
__device__ __forceinline__ void philox4x32_10_rk(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                 const uint32_t (&rk0)[10], uint32_t k1,
                                                 uint32_t out[4]) {
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const uint64_t pa = (uint64_t)0xD2511F53u * c0;
        const uint64_t pb = (uint64_t)0xCD9E8D57u * c2;
        c0 = (uint32_t)(pb >> 32) ^ c1 ^ rk0[round];
        c1 = (uint32_t)pb;
        c2 = (uint32_t)(pa >> 32) ^ c3 ^ (k1 + (uint32_t)round * 0xBB67AE85u);
        c3 = (uint32_t)pa;
    }
    out[0] = c0;
    out[1] = c1;
    out[2] = c2;
    out[3] = c3;
}

// (((x >> 8) | 1) * 2^-24): an odd multiple of 2^-24 in (0,1), exact in FP32
// and equal to the oracle's value. Built from the bits: f = 1 + (x >> 9) 2^-23
// is a float with mantissa x >> 9, and f - (1 - 2^-24) = (2 (x >> 9) + 1)
// 2^-24 has at most 24 significant bits, so the one subtraction is exact
// (1 - 2^-24 is itself a float, 0x3F7FFFFF).
__device__ __forceinline__ float u01(uint32_t x) {
    return __uint_as_float(0x3F800000u | (x >> 9)) - 0.999999940395355224609375f;
}

// The same from two words at once: the shift and the exponent bits are one
// funnel shift (0x3F800000 = 0x7F << 23), the subtraction is packed.
__device__ __forceinline__ float2 u01_2(uint32_t x, uint32_t y) {
    return __fadd2_rn(make_float2(__uint_as_float(__funnelshift_r(x, 0x7Fu, 9)),
                                  __uint_as_float(__funnelshift_r(y, 0x7Fu, 9))),
                      make_float2(-0.999999940395355224609375f, -0.999999940395355224609375f));
}

__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }

// psi = atan2(S, C) for S >= 0, psi in [0, pi]: atan(t) = t P(t^2) on
// t = min/max of (|C|, S) in [0, 1], then the octant is restored. P is a
// degree-7 near-minimax fit (gen_atan_poly.py; |error| < 7e-8 on [0, 1]).
__device__ __forceinline__ float atan2_upper(float S, float C) {
    const float ax = fabsf(C);
    const float mn = fminf(ax, S), mx = fmaxf(ax, S);
    const float t = __fdividef(mn, mx);
    const float z = t * t;
    float p = -4.054566845e-03f;
    p = fmaf(p, z, 2.186295763e-02f);
    p = fmaf(p, z, -5.591232702e-02f);
    p = fmaf(p, z, 9.642197192e-02f);
    p = fmaf(p, z, -1.390862912e-01f);
    p = fmaf(p, z, 1.994656622e-01f);
    p = fmaf(p, z, -3.332985938e-01f);
    p = fmaf(p, z, 9.999993443e-01f);
    float a = t * p;
    a = (S > ax) ? (1.57079632679489662f - a) : a;
    return (C < 0.0f) ? (3.14159265358979324f - a) : a;
}

// 1 / x and 2^x of the hardware (PTX rcp / ex2, denormals flushed: x is a sum
// of cosines or sines here, never denormal, and 2^x is compared with numbers
// of at least 2^-24).
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// atan2_upper of two arguments, the polynomial in packed arithmetic.
__device__ __forceinline__ float2 atan2_upper_2(float2 S, float2 C) {
    const float ax = fabsf(C.x), ay = fabsf(C.y);
    const float2 mn = make_float2(fminf(ax, S.x), fminf(ay, S.y));
    const float2 t = __fmul2_rn(mn, make_float2(rcp_approx(fmaxf(ax, S.x)),
                                                rcp_approx(fmaxf(ay, S.y))));
    const float2 z = __fmul2_rn(t, t);
    float2 p = both(-4.054566845e-03f);
    p = __ffma2_rn(p, z, both(2.186295763e-02f));
    p = __ffma2_rn(p, z, both(-5.591232702e-02f));
    p = __ffma2_rn(p, z, both(9.642197192e-02f));
    p = __ffma2_rn(p, z, both(-1.390862912e-01f));
    p = __ffma2_rn(p, z, both(1.994656622e-01f));
    p = __ffma2_rn(p, z, both(-3.332985938e-01f));
    p = __ffma2_rn(p, z, both(9.999993443e-01f));
    float2 a = __fmul2_rn(t, p);
    const float2 h = __ffma2_rn(a, both(-1.0f), both(1.57079632679489662f));
    a = make_float2(S.x > ax ? h.x : a.x, S.y > ay ? h.y : a.y);
    const float2 g = __ffma2_rn(a, both(-1.0f), both(3.14159265358979324f));
    return make_float2(C.x < 0.0f ? g.x : a.x, C.y < 0.0f ? g.y : a.y);
}

// Sum of a pair's weighted changes as an unevaluated sum hi + lo.
struct Sum2 {
    float2 hi, lo;
    __device__ void add(float2 x, float w) {
        const float2 w2 = both(w);
        const float2 p = __fmul2_rn(x, w2);
        const float2 e = __ffma2_rn(x, w2, make_float2(-p.x, -p.y));        // x w = p + e
        const float2 s = __fadd2_rn(hi, p);
        const float2 t = __ffma2_rn(hi, both(-1.0f), s);
        const float2 a = __ffma2_rn(__ffma2_rn(t, both(-1.0f), s), both(-1.0f), hi);
        const float2 b = __ffma2_rn(t, both(-1.0f), p);                     // hi + p = s + a + b
        lo = __fadd2_rn(lo, __fadd2_rn(__fadd2_rn(a, b), e));
        hi = s;
    }
};

// Outcome of one site update: the new angle, the angle after the Metropolis
// move, the energy change, and whether the over-relaxation was applied.
struct SiteNew {
    float phi, mid, dE;
    bool refl;
};

// Outcome of a site's update in both realizations of a pair (.x, .y): the new
// angles, the angles after the Metropolis move, the energy change, and whether
// the over-relaxation was applied.
struct PairNew {
    float2 phi, mid, dE;
    bool refl0, refl1;
};

__device__ __forceinline__ void sincos_2(float2 x, float2& s, float2& c) {
    __sincosf(x.x, &s.x, &c.x);
    __sincosf(x.y, &s.y, &c.y);
}

// cos / sin of q times the final angle from those of q phi_a after the
// Metropolis move: after a reflection q phi'' = 2 psi - q phi_a with
// cos 2psi = (C^2 - S^2)/R^2, sin 2psi = 2CS/R^2.
__device__ __forceinline__ void final_cs(bool refl, float ca, float sa, float C, float S, float& c,
                                         float& s) {
    if (refl) {
        const float ir2 = __fdividef(1.0f, C * C + S * S);
        const float c2 = (C * C - S * S) * ir2;
        const float s2 = 2.0f * C * S * ir2;
        c = c2 * ca + s2 * sa;
        s = s2 * ca - c2 * sa;
    } else {
        c = ca;
        s = sa;
    }
}

}  // namespace mpr
