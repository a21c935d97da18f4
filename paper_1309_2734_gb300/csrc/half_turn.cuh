// The sine and cosine of fixed-point turns by the polynomials of sincospoly.h and sinpoly.h, two at a time in packed
// operations.
#pragma once

#include "sincospoly.h"
#include "sinpoly.h"

namespace cgh {
namespace dev {

__device__ __forceinline__ float2 f2(float a)
{
    return make_float2(a, a);
}

// sqrt(2) sin(pi r) and sqrt(2) cos(pi r) of two signed turns r (2^-32 turn): half the angle, so that s^2 - 1 and s c
// are minus the cosine and the sine of the whole turn without a quadrant (sincospoly.h).
template <int U>
__device__ __forceinline__ void half_turn2(const float2 (&turn)[U], float2 (&s)[U], float2 (&c)[U])
{
    float2 r[U], u[U], hs[U], hc[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
        r[j] = __fmul2_rn(turn[j], f2(2.3283064365386963e-10f));
        u[j] = __fmul2_rn(r[j], r[j]);
        hs[j] = f2(CGH_HSIN_4);
        hc[j] = f2(CGH_HCOS_4);
    }
#define CGH_HORNER(OUT, IN, COEF)                                                                                     \
    _Pragma("unroll") for (int j = 0; j < U; ++j) OUT[j] = __ffma2_rn(IN[j], u[j], f2(COEF));
    CGH_HORNER(hs, hs, CGH_HSIN_3)
    CGH_HORNER(hc, hc, CGH_HCOS_3)
    CGH_HORNER(hs, hs, CGH_HSIN_2)
    CGH_HORNER(hc, hc, CGH_HCOS_2)
    CGH_HORNER(hs, hs, CGH_HSIN_1)
    CGH_HORNER(hc, hc, CGH_HCOS_1)
    CGH_HORNER(hs, hs, CGH_HSIN_0)
    CGH_HORNER(c, hc, CGH_HCOS_0)
#undef CGH_HORNER
#pragma unroll
    for (int j = 0; j < U; ++j) s[j] = __fmul2_rn(r[j], hs[j]);
}

// x = -cos(2 pi r) and y = sin(2 pi r) of two signed turns r (2^-32 turn), folded to a quarter of a turn (sinpoly.h): one
// odd polynomial, whose last operation is a product, gives both to 2.8e-8 RMS; half_turn2's doubled angle to 8.5e-8 in
// two packed operations and six integer ones fewer.
template <int U>
__device__ __forceinline__ void quarter_turn2(const float2 (&turn)[U], float2 (&x)[U], float2 (&y)[U])
{
    float2 d[U], m[U], ud[U], um[U], hd[U], hm[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
        const float2 r = __fmul2_rn(turn[j], f2(2.3283064365386963e-10f));
        const float2 a = make_float2(fabsf(r.x), fabsf(r.y));
        const float2 b = __ffma2_rn(a, f2(-1.0f), f2(0.5f));
        d[j] = __fadd2_rn(a, f2(-0.25f));
        m[j] = make_float2(copysignf(fminf(a.x, b.x), r.x), copysignf(fminf(a.y, b.y), r.y));
        ud[j] = __fmul2_rn(d[j], d[j]);
        um[j] = __fmul2_rn(m[j], m[j]);
        hd[j] = hm[j] = f2(CGH_SIN_4);
    }
#define CGH_HORNER(COEF)                                                                                              \
    _Pragma("unroll") for (int j = 0; j < U; ++j) {                                                                   \
        hd[j] = __ffma2_rn(hd[j], ud[j], f2(COEF));                                                                   \
        hm[j] = __ffma2_rn(hm[j], um[j], f2(COEF));                                                                   \
    }
    CGH_HORNER(CGH_SIN_3)
    CGH_HORNER(CGH_SIN_2)
    CGH_HORNER(CGH_SIN_1)
    CGH_HORNER(CGH_SIN_0)
#undef CGH_HORNER
#pragma unroll
    for (int j = 0; j < U; ++j) {
        x[j] = __fmul2_rn(d[j], hd[j]);
        y[j] = __fmul2_rn(m[j], hm[j]);
    }
}

}  // namespace dev
}  // namespace cgh
