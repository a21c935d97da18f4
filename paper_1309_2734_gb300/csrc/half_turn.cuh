// The sine and cosine of fixed-point turns by the polynomials of sincospoly.h, two at a time in packed operations.
#pragma once

#include "sincospoly.h"

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

}  // namespace dev
}  // namespace cgh
