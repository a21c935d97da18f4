// f2: the spherical remainder at the centre of a tile of pixels, shared by the SIMT kernel (spherical.cu) and the
// tensor-core form (direct_mma.cu).
#pragma once

#include "device_util.cuh"

namespace cgh {
namespace dev {

// Error-free transformations on float pairs (hi + lo): Knuth's two-sum, Dekker's fast two-sum (|a| >= |b|).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

__device__ __forceinline__ void fast_two_sum(float a, float b, float &s, float &e)
{
    s = a + b;
    e = b - (s - a);
}

// The remainder at the thread tile's centre, d0 = Z h(U0) = -(Z / 2) v0^2 with v0 = sqrt(1 + U0) - 1 and
// U0 = (cx^2 + cy^2) (p / z)^2, in double-float arithmetic (float pairs, about 44 significant bits) from the
// point's (p / z)^2 and Z / 2 as pairs: a float alone would carry d0 only to ~1e-7 of itself, and d0 reaches
// hundreds of turns for close points on wide holograms.  Returns d0 - round(d0) (turns); v0, s0 = sqrt(1 + U0)
// and rs0 = 1 / s0 as floats.
__device__ __forceinline__ float sph_d0_frac(float cx, float cy, const float4 x, float &v0, float &s0, float &rs0)
{
    const float qh = fabsf(x.x), zh = fabsf(x.y), ql = x.z, zl = x.w;
    // R0 = cx^2 + cy^2, exact as a pair (half-integers below 2^17)
    const float px = cx * cx, ex = fmaf(cx, cx, -px);
    const float py = cy * cy, ey = fmaf(cy, cy, -py);
    float rh, rl;
    two_sum(px, py, rh, rl);
    fast_two_sum(rh, rl + (ex + ey), rh, rl);
    // U0 = R0 (p / z)^2 and 1 + U0
    float uh = rh * qh;
    float ul = fmaf(rh, qh, -uh) + fmaf(rh, ql, rl * qh);
    fast_two_sum(uh, ul, uh, ul);
    float oh, ol;
    two_sum(1.0f, uh, oh, ol);
    fast_two_sum(oh, ol + ul, oh, ol);
    // s0: one Newton step from the float estimate doubles its ~22 correct bits
    const float rs = rsqrtf(oh);
    const float y = oh * rs;
    float sh, sl;
    fast_two_sum(y, (fmaf(-y, y, oh) + ol) * (0.5f * rs), sh, sl);
    // v0 = s0 - 1 (exact subtraction), then d0 = -(Z / 2) v0^2
    float vh, vl;
    two_sum(sh, -1.0f, vh, vl);
    fast_two_sum(vh, vl + sl, vh, vl);
    const float wh = vh * vh, wl = fmaf(vh, vh, -wh) + 2.0f * vh * vl;
    float dh = zh * wh;
    float dl = fmaf(zh, wh, -dh) + fmaf(zh, wl, zl * wh);
    fast_two_sum(dh, dl, dh, dl);
    v0 = vh;
    s0 = sh;
    rs0 = rs;
    return -((dh - rintf(dh)) + dl);
}

}  // namespace dev
}  // namespace cgh
