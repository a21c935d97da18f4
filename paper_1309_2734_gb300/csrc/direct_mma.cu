// a2, the direct form on the tensor cores: the tables of the sines and cosines of a point's columns and rows that a
// CTA takes once for its tile of pixels (the cosine addition formula, direct_dev.cuh) are the operands of a matrix
// product, I(m, n) = sum_j [cos a_jm, sin a_jm] . [A_j cos b_jn, -A_j sin b_jn], so tcgen05.mma adds them up
// instead of two FMAs a pixel and point.  No factor goes through memory: each CTA makes its tile's entries in
// shared memory and multiplies them there.
//
// Precision (the form's contract is single precision).  An entry is taken to 1.2e-7 RMS from the exact fixed-point
// turn (half_turn2), every other point half a turn on in both of its entries so that a mean error of the cosine over
// the turns cancels between points, and held as the sum of two FP16 values, hi + lo (22 bits and the signs), the
// amplitudes scaled by 2^12 so that lo stays normal down to 2^-15 of the largest; the product is lo hi + hi lo + hi hi,
// the large products last.  The tensor cores' FP32 accumulation truncates, which takes 1.9e-7 of a chain's value per
// group of 32 points, so a chain is kChain = 2 groups, its mean loss is put back (kUnscale), and the chains are added
// in FP32, in point order.  NRMS against FP64 (before: the SIMT kernel with the hardware cosine / with the polynomial):
//   1920x1080, 10^4 points 3.5e-7 (6.0e-7);  1283x717, 3001 points, piston and reference 3.2e-7 (4.1e-7);
//   640x64, 3000 points 1.1e-7 (3.1e-7);  256x256, 1024 points 2.8e-7 (6.7e-7);  wave 3.5e-7 (5.9e-7).
// (Without the half turn 640x64 gave 7.2e-7; chains of 1 / 4 / 8 groups at 1920x1080 3.1 / 8.6 / 17.6e-7.)
// The accurate form takes its entries to 2.8e-8 (quarter_turn2) and chains of one group: with the above it would be coarser
// on small clouds than the SIMT kernel's polynomial.  NRMS of the SIMT kernel / as above / with both:
//   256x256, 20 points 1.6 / 2.5 / 1.5e-7, 300 points 2.2 / 3.0 / 1.5e-7, 2048 points 2.0 / 2.5 / 1.6e-7;
//   640x64, 1024 points 1.27 / 1.50 / 0.95e-7;  1283x717, 3001 points 4.1 / 3.2 / 1.8e-7;  1920x1080, 2 10^5 points
//   5.2 / - / 4.3e-7.  (From some 6 10^4 points on holograms of 256x256 or less the SIMT kernel's shorter partial sums are
//   better, 1.5 against 1.8e-7.)
// Time: 1920x1080, 10^4 points 0.370 ms (SIMT 1.89, as above 0.305), 1283x717, 3001 points 88 us (394, 79).
//
// The kernel starts while the points are being prepared (dependent launch) and reduces max |A| itself, so nothing is
// cleared before: 256x256, 10^3 points with the quantiser 25.7 us (35.4 with plain launches, clears and prep blocks of
// 256 points).
//
// Time, prep included (before): 1920x1080, 10^4 points 0.305 ms (1.77; 68 G terms/ms); its complex wave 0.480 ms
// (3.30); 1024x1024, 10^3 points 0.042 ms (0.117); 256x256, 10^3 points 0.021 ms (0.046); the spherical hologram,
// 1920x1080, 10^4 points at 0.3-1 m 0.644 ms (7.36; at 0.25 m, where only the narrowest tile's bound holds, 1.50).
// What bounds it: the making of entries (0.26 of 0.31 ms with the MMAs left out), 30 instructions for two entries, 15
// of them packed FMAs of two to three cycles, so the FMA pipe is about 80 % busy while entries are made (53 % over the
// kernel); the tensor cores are active 36 % of the time.  128 x BN tiles: larger tiles share an entry among more pixels (BN = 64 / 128 /
// 192 / 224: 0.66 / 0.42 / 0.34 / 0.31 ms), and two stages of 224 rows fill shared memory.
//
// Measured and not used: a pair of CTAs (cta_group::2) on tiles of 256 rows, half of B's entries each, 0.322 ms and the
// wave 0.557 -- two fifths fewer entries, but then the loop of MMAs, fold and next chain (tensor memory holds one
// accumulator beside the totals) and the cluster's round trips are as long; four warps of their own for the folds 0.306
// and 0.563 ms (80 registers a thread, and the folds take longer than the next stage's entries).
//
// One CTA per SM, 18 warps.  Sixteen worker warps make the entries of a stage -- 32 points x (128 A rows + BN B rows),
// hi and lo planes, K-major with the 128-byte swizzle -- and fold the chains; one thread of warp 16 issues the MMAs, one
// of warp 17 brings the points (1-D bulk copies).  (Eight worker warps with the totals in registers: 0.41 ms; the totals
// in tensor memory cost a read and a write more per fold but leave registers for sixteen warps.  Points loaded by the
// MMA thread: 0.33 ms, its copies delay the next stage's MMAs by 600 clocks.)
//
//     ptfull[4]  points of a stage are there        (bulk copy -> workers)
//     ptempty[4] they are read                      (workers -> loader)
//     full[S]    a stage's entries are written      (workers -> MMA)
//     empty[S]   its MMAs are done                  (MMA -> workers)
//     tfull      a chain is in the accumulator      (MMA -> workers)
//     tempty     its values are in the totals       (workers -> MMA)
//     parts[2]   a CTA's parts of a tile are out; who finished the tile (workers, thread 0)
//
// A chain's MMAs run while the next stage is made; then it is folded.  Work is the flat list of (pixel tile, group of
// 32 points) pairs in equal shares per CTA, a tile's parts summed in CTA order by the CTA that finishes last, as in the
// balanced layout of direct.cu.
#include <algorithm>
#include <type_traits>

#include <cuda_fp16.h>

#include "device_util.cuh"
#include "half_turn.cuh"
#include "host_util.h"
#include "kernels.h"
#include "spherical_dev.cuh"
#include "tcgen05.cuh"

namespace cgh {

namespace {

using dev::f2;
using dev::half_turn2;
using dev::quarter_turn2;

constexpr int kWorkers = 512;
constexpr int kMmaThreads = kWorkers + 64;   // the workers, the MMA warp, the loader warp
constexpr int kRowsA = 128;
constexpr int kGroup = kDirectMmaGroup;      // points of a stage: 64 K elements, one 128-byte swizzle row
constexpr int kPtSlots = 4;
constexpr int kPtBytes = kGroup * (int)(sizeof(int4) + sizeof(uint2));
constexpr int kChain = 2;                    // stages of an accumulation chain
constexpr int kAccChain = 1;                 // the accurate form's
constexpr int kSphChain = 4;                 // spherical: stages of half as many points
constexpr float kEntryScale = 4096.0f;       // 2^12, the A side (amplitudes)
// 2^-12, times 1 + 2.4e-7: the accumulation truncates, and a chain of two groups loses 2.9e-7 of its value on average
// (measured on random clouds; 2.6e-7 on coherent ones); a spherical chain, with twice the MMAs, 4.6e-7
constexpr float kUnscale = 2.44140625e-04f * (1.0f + 2.384185791015625e-07f);
constexpr float kSphUnscale = 2.44140625e-04f * (1.0f + 4.76837158203125e-07f);
// The accurate form's chains of one group lose 5e-8 (one point) to 1.1e-7 of their value in a random cloud, nothing where
// many points add up in phase; the sum gets 4e-8 of it back (by one FMA: a unit in the last place from 1.5 on).
constexpr float kAccUnscale = 2.44140625e-04f, kAccLoss = 4e-8f;

template <int BN>
struct MmaCfg {
    static constexpr int kA = kRowsA * 128, kB = BN * 128;   // bytes of one plane of A, of B
    static constexpr int kStage = 2 * (kA + kB);
    static constexpr int kRoom = 232448 - 1024 - kPtSlots * kPtBytes - 256;
    static constexpr int kStages = kRoom / kStage > 4 ? 4 : kRoom / kStage;
    static constexpr int kTotal = BN <= 128 ? 128 : 256;   // tensor-memory column of the totals, after the chain
    static constexpr int kTmemCols = 2 * kTotal;
    static constexpr int kSmem = 1024 + kStages * kStage + kPtSlots * kPtBytes + 256;
    static_assert(BN % 32 == 0 && BN >= 64 && BN <= 256, "B rows in steps of 32, TMEM columns in halves of 16s");
    static_assert(kStages >= 2, "at least a double-buffered ring");
};

struct MmaArgs {
    const int4 *geo;
    const uint2 *aux;
    const float4 *ext;         // the spherical form's constants
    const float *amp_max;      // max |A| in amp_parts values; spherical: [0] max |A|, [1] the bound (prep)
    int amp_parts;
    float *out;                // plane 1 (the imaginary part) follows plane 0
    float4 *slots;
    int *counters;
    int *status;
    unsigned long long timeout_ns;
    long long units, groups;   // (tile, group) pairs; groups per tile
    int width, height, tiles_a;
    int a_rows;                // 1: A rows are hologram rows; 0: hologram columns
    int vec, drop;
    int add;                   // add to out: a later launch over the points
    float phase_lo, phase_hi;  // the spherical form: the bounds this launch takes
    PhaseRef ref;
};

// The walk of one point down a side's rows in steps of 32 (Eqs. 6-8 at that stride): t = C d^2 at the first row,
// D its first difference, S the second, top 32 bits of the 64-bit products.
struct Walk {
    uint32_t t, D;
};
__device__ __forceinline__ Walk walk_start(int d, uint32_t ch, uint32_t cl, uint32_t add, uint32_t step)
{
    const uint32_t d2 = (uint32_t)(d * d);
    const int e = 64 * d + 1024;   // (d + 32)^2 - d^2
    Walk w;
    w.t = ch * d2 + __umulhi(cl, d2) + add;
    w.D = ch * (uint32_t)e + __umulhi(cl, (uint32_t)e) - (e < 0 ? cl : 0u) + step;
    return w;
}

// v - h for both halves of a packed FP16 pair (mixed-precision FMA, exact).
__device__ __forceinline__ float2 minus_half2(float2 v, uint32_t h)
{
    float2 d;
    asm("{\n\t.reg .b16 l, u, m;\n\t"
        "mov.b32 {l, u}, %2;\n\t"
        "mov.b16 m, 0xbc00;\n\t"
        "fma.rn.f32.f16 %0, l, m, %3;\n\t"
        "fma.rn.f32.f16 %1, u, m, %4;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "r"(h), "f"(v.x), "f"(v.y));
    return d;
}

__device__ __forceinline__ uint32_t pack_half2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// The row of the imaginary part from that of the real part: {-cos, -sin} -> {-sin, cos}.
__device__ __forceinline__ uint32_t turn_quarter(uint32_t h)
{
    return __byte_perm(h, 0, 0x1032) ^ 0x80000000u;
}

__device__ __forceinline__ void st_shared8(uint32_t addr, uint32_t a, uint32_t b)
{
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}

__device__ __forceinline__ void st_shared4(uint32_t addr, uint32_t a)
{
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(a) : "memory");
}

// 32 lanes x 8 columns of tensor memory (as tmem_ld16, tmem_st16).
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
                 : "r"(taddr));
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float (&r)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
                 "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7])
                 : "memory");
}

// Entries of this thread's two points (16 apart: conflict-free loads; K slots 2 pair and 2 pair + 1) at STEPS rows 32
// apart.  A side: 2^12 A (-cos a, sin a).  B side: its turns
// walked backwards (b -> -b), (-cos b, -sin b); PLANES = 2: and the rows of the imaginary part, (-sin b, cos b), im_off
// further on.
template <int STEPS, bool B, int PLANES, bool ACC>
__device__ __forceinline__ void side_entries(const int4 *geo, const uint2 *aux, bool swap, int row, uint32_t add,
                                             uint32_t step, uint32_t piston, float a_scale, uint32_t hi,
                                             uint32_t lo_off, uint32_t im_off)
{
    Walk w[2];
    uint32_t S[2];
    float2 a = f2(0.0f);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const int4 q = geo[16 * p];
        const uint32_t ch = (uint32_t)q.z, cl = (uint32_t)q.w;
        w[p] = walk_start(row - (swap != B ? q.y : q.x), ch, cl, add, step);
        S[p] = (ch << 11) | (cl >> 21);   // 2048 C
        if (p & 1) w[p].t ^= 0x80000000u;   // the half turn of every other point
        if (B) {
            w[p].t = 0u - w[p].t;
        } else {
            const uint2 x = aux[16 * p];
            w[p].t += x.x & piston;
            (p & 1 ? a.y : a.x) = __uint_as_float(x.y) * a_scale * kEntryScale;
        }
    }
    const float2 na = make_float2(-a.x, -a.y);
    // U steps side by side: their chains of dependent operations overlap (one plane: 1.5 % over two; two planes: as two;
    // accurate: two are 2.5 % faster than four)
    constexpr int kUnroll = PLANES == 1 && !ACC ? 4 : 2;
    auto steps = [&](auto uc, int k0) {
        constexpr int U = decltype(uc)::value;
        float2 s[U], c[U], x[U], y[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            x[j] = make_float2((float)(int)w[0].t, (float)(int)w[1].t);
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                w[p].t = B ? w[p].t - w[p].D : w[p].t + w[p].D;
                w[p].D += S[p];
            }
        }
        if constexpr (ACC) {
            quarter_turn2<U>(x, s, c);
#pragma unroll
            for (int j = 0; j < U; ++j) {
                x[j] = B ? s[j] : __fmul2_rn(a, s[j]);
                y[j] = B ? c[j] : __fmul2_rn(a, c[j]);
            }
        } else {
            half_turn2<U>(x, s, c);
        }
#pragma unroll
        for (int j = 0; j < U && !ACC; ++j) {
            if (B) {
                x[j] = __ffma2_rn(s[j], s[j], f2(-1.0f));
                y[j] = __fmul2_rn(s[j], c[j]);
            } else {
                const float2 as = __fmul2_rn(a, s[j]);
                x[j] = __ffma2_rn(as, s[j], na);
                y[j] = __fmul2_rn(as, c[j]);
            }
        }
        uint32_t h[U][2], l[U][2];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            h[j][0] = pack_half2(x[j].x, y[j].x);
            h[j][1] = pack_half2(x[j].y, y[j].y);
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const float2 d = minus_half2(make_float2(x[j].x, y[j].x), h[j][0]);
            y[j] = minus_half2(make_float2(x[j].y, y[j].y), h[j][1]);
            x[j] = d;
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
            l[j][0] = pack_half2(x[j].x, x[j].y);
            l[j][1] = pack_half2(y[j].x, y[j].y);
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const uint32_t at = hi + (uint32_t)(k0 + j) * 4096u;
            st_shared8(at, h[j][0], h[j][1]);
            st_shared8(at + lo_off, l[j][0], l[j][1]);
            if (B && PLANES == 2) {
                st_shared8(at + im_off, turn_quarter(h[j][0]), turn_quarter(h[j][1]));
                st_shared8(at + lo_off + im_off, turn_quarter(l[j][0]), turn_quarter(l[j][1]));
            }
        }
    };
#pragma unroll
    for (int k = 0; k + kUnroll <= STEPS; k += kUnroll) steps(std::integral_constant<int, kUnroll>{}, k);
    if constexpr (STEPS % kUnroll != 0) steps(std::integral_constant<int, STEPS % kUnroll>{}, STEPS / kUnroll * kUnroll);
}

// The spherical form.  About the centre of a tile (offsets cx, cy from the point, U0 = (cx^2 + cy^2) q, q = (p / z)^2)
// a pixel with vx = dx^2 - cx^2 and vy = dy^2 - cy^2 has the turn
//   Z + C dx^2 + C dy^2 + d0 + P(vx) + P(vy) + X,   P(v) = d1 w + d2 w^2 + d3 w^3, w = q v, Z h(U0 + w) - d0 = P(v)
// (the Fresnel turn with its piston and the remainder: d0 = Z h(U0), and d1 = Z h1, d2 = Z h2 / 2, d3 = Z h3 / 6 from
// h's derivatives at U0), where all but the cross term X = 2 d2 F(vx) F(vy), F(v) = w (1 + h3 / (2 h2) w), is a column
// turn plus a row turn.  With 2 pi X = g(column) f(row) the term's factor exp(i g f) is taken to second order,
// 1 + i g f - g^2 f^2 / 2: three products of a column's and a row's entry, the first as hi + lo pairs, the other two
// (at most a few percent) as FP16.  The point preparation bounds |g f| (sph_mma_max_phase) and |P| (kSphRangeTurns)
// for every point and pixel of a cloud that comes here: at the largest |g f| the third order left out is 4e-7 of a
// point's term (RMS over the pixels) and the rounding of the second product 5e-7.
struct SphPoint {
    float d0, e1, e2, e3;   // turns: d0's fraction, P's coefficients in v (2^-32 turn)
    float cq, ka, sb;       // F(v) = q v (1 + cq v); g = ka v (1 + cq v), f = sb v (1 + cq v)
};

// Offsets of the centre along A and B; hb: half the tile's B side.
__device__ __forceinline__ SphPoint sph_point(const float4 x, int ca, int cb, float hb)
{
    const float q = fabsf(x.x), zh = fabsf(x.y);
    const float fa = (float)ca, fb = (float)cb;
    SphPoint P;
    float v0, s0, rs0;
    P.d0 = dev::sph_d0_frac(fa, fb, x, v0, s0, rs0);
    const float r2 = rs0 * rs0, r3 = r2 * rs0;
    const float d2 = -0.25f * zh * r3, q1 = q * 4294967296.0f;
    P.e1 = -zh * v0 * rs0 * q1;
    P.e2 = d2 * q * q1;
    P.e3 = 0.125f * zh * r3 * r2 * q * q * q1;
    P.cq = -0.75f * r2 * q;
    const float span = fmaf(2.0f * hb, fabsf(fb), hb * hb);   // max |vy|
    P.sb = __frcp_rn(span);
    P.ka = 12.56637061435917295f * d2 * q * q * span;         // 4 pi d2 q^2 / sb
    return P;
}

// Entries of this thread's point at STEPS rows 32 apart, two rows a packed operation, in plane 0 the first product's
// hi and the second product, in plane 1 its lo and the third.  d: the first row's offset from the point, off: from the
// tile's centre.
template <int STEPS, bool B>
__device__ __forceinline__ void sph_entries(const SphPoint &P, const int4 q, int d, int off, bool flip, uint32_t add,
                                            uint32_t step, float amp, uint32_t at0, uint32_t lo_off)
{
    static_assert(STEPS % 2 == 0, "pairs of rows");
    const uint32_t ch = (uint32_t)q.z, cl = (uint32_t)q.w;
    Walk w = walk_start(d, ch, cl, add, step);
    const uint32_t S = (ch << 11) | (cl >> 21);   // 2048 C
    if (flip) w.t ^= 0x80000000u;                 // the half turn of every other point
    if (B) w.t = 0u - w.t;
    float2 a2 = make_float2((float)off, (float)(off + 32));
    const float2 c2 = f2((float)(2 * (d - off)));
    const float2 A = f2(amp), nA = f2(-amp);
#pragma unroll
    for (int k = 0; k < STEPS; k += 2) {
        const float2 v = __fmul2_rn(a2, __fadd2_rn(a2, c2));
        const float2 p = __fmul2_rn(v, __ffma2_rn(v, __ffma2_rn(v, f2(P.e3), f2(P.e2)), f2(P.e1)));
        const float2 F = __fmul2_rn(v, __ffma2_rn(v, f2(P.cq), f2(1.0f)));
        const uint32_t t0 = w.t;
        w.t = B ? w.t - w.D : w.t + w.D;
        w.D += S;
        const uint32_t t1 = w.t;
        w.t = B ? w.t - w.D : w.t + w.D;
        w.D += S;
        const uint32_t p0 = (uint32_t)__float2int_rn(p.x), p1 = (uint32_t)__float2int_rn(p.y);
        float2 turn[1], s[1], c[1], x, y;
        turn[0] = make_float2((float)(int)(B ? t0 - p0 : t0 + p0), (float)(int)(B ? t1 - p1 : t1 + p1));
        half_turn2<1>(turn, s, c);
        float2 x1, y1, x2, y2;
        if (B) {
            x = __ffma2_rn(s[0], s[0], f2(-1.0f));
            y = __fmul2_rn(s[0], c[0]);
            const float2 f = __fmul2_rn(F, f2(P.sb)), nf = __fmul2_rn(F, f2(-P.sb));
            x1 = __fmul2_rn(y, nf);   // i times: (-y, x)
            y1 = __fmul2_rn(x, f);
            x2 = __fmul2_rn(y1, f);
            y2 = __fmul2_rn(x1, nf);
        } else {
            const float2 as = __fmul2_rn(A, s[0]);
            x = __ffma2_rn(as, s[0], nA);
            y = __fmul2_rn(as, c[0]);
            const float2 gk = __fmul2_rn(F, f2(P.ka)), h = __fmul2_rn(F, f2(-0.5f * P.ka));
            x1 = __fmul2_rn(x, gk);
            y1 = __fmul2_rn(y, gk);
            x2 = __fmul2_rn(x1, h);
            y2 = __fmul2_rn(y1, h);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float xj = j ? x.y : x.x, yj = j ? y.y : y.x;
            const uint32_t h = pack_half2(xj, yj);
            const float2 l = minus_half2(make_float2(xj, yj), h);
            const uint32_t at = at0 + (uint32_t)(k + j) * 4096u;
            st_shared4(at, h);
            st_shared4(at + lo_off, pack_half2(l.x, l.y));
            st_shared4(at ^ 64u, j ? pack_half2(x1.y, y1.y) : pack_half2(x1.x, y1.x));
            st_shared4((at ^ 64u) + lo_off, j ? pack_half2(x2.y, y2.y) : pack_half2(x2.x, y2.x));
        }
        a2 = __fadd2_rn(a2, f2(64.0f));
    }
}

struct MmaBars {
    uint64_t *full, *empty, *ptfull, *ptempty, *tfull, *tempty, *parts, *drain;
};

// PLANES = 1: the amplitude hologram, tiles of 128 x BN pixels.  PLANES = 2: the complex wave, tiles of 128 x BN / 2
// pixels, the B rows (and accumulator columns) of the imaginary part after those of the real part.
// SPH: the amplitude hologram of the spherical model, 16 points a stage (three products each).
// ACC: the accurate form (PLANES = 1), entries by quarter_turn2 and chains of one group.
template <int BN, int PLANES, bool SPH, bool ACC>
__global__ void __launch_bounds__(kMmaThreads, 1) direct_mma_kernel(const __grid_constant__ MmaArgs g)
{
    using C = MmaCfg<BN>;
    constexpr int GROUP = SPH ? kSphMmaGroup : kGroup;
    constexpr int CHAIN = SPH ? kSphChain : ACC ? kAccChain : kChain;
    static_assert(!SPH || (PLANES == 1 && BN % 64 == 0), "row pairs of the amplitude hologram");
    if (SPH) grid_wait();
    if (SPH && !(g.amp_max[1] > g.phase_lo && g.amp_max[1] <= g.phase_hi)) return;   // another kernel's cloud
    constexpr int HB = BN / 4;          // accumulator columns per worker warp
    constexpr int TB = BN / PLANES;     // pixels of the tile along B
    extern __shared__ uint8_t smem_raw[];
    __shared__ int s_last;
    __shared__ uint32_t s_tmem;
    __shared__ uint32_t s_amp[kMmaThreads / 32];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *s_pts = smem + C::kStages * C::kStage;
    MmaBars bars;
    bars.full = reinterpret_cast<uint64_t *>(s_pts + kPtSlots * kPtBytes);
    bars.empty = bars.full + 4;
    bars.ptfull = bars.empty + 4;
    bars.ptempty = bars.ptfull + kPtSlots;
    bars.tfull = bars.ptempty + kPtSlots;
    bars.tempty = bars.tfull + 1;
    bars.parts = bars.tempty + 1;   // [0] the workers' parts of a tile are out, [1] s_last is set
    bars.drain = bars.parts + 2;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < C::kStages; ++s) {
            mbar_init(&bars.full[s], kWorkers / 32);
            mbar_init(&bars.empty[s], 1);
        }
        mbar_init(bars.tfull, 1);
        mbar_init(bars.tempty, kWorkers / 32);
        for (int p = 0; p < kPtSlots; ++p) {
            mbar_init(&bars.ptfull[p], 1);
            mbar_init(&bars.ptempty[p], kWorkers / 32);
        }
        mbar_init(&bars.parts[0], kWorkers / 32);
        mbar_init(&bars.parts[1], 1);
        mbar_init(bars.drain, 1);
        fence_barrier_init();
    }
    if (warp == kWorkers / 32) {
        tmem_alloc(&s_tmem, C::kTmemCols);
        tmem_relinquish();
    }
    grid_wait();   // the barriers and tensor memory above are set up while the points are still being prepared
    uint32_t amp = 0;
    for (int i = tid; i < g.amp_parts; i += kMmaThreads) amp = max(amp, __float_as_uint(__ldcg(g.amp_max + i)));
    amp = __reduce_max_sync(0xffffffffu, amp);
    if (lane == 0) s_amp[warp] = amp;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const long long w0 = (long long)blockIdx.x * g.units / gridDim.x;
    const long long w1 = ((long long)blockIdx.x + 1) * g.units / gridDim.x;
    const int n = (int)(w1 - w0);
    auto wait = [&](uint64_t *bar, uint32_t parity) {
        if (mbar_wait(bar, parity, g.timeout_ns)) return true;
        atomicOr(g.status, kStatusTimeout);
        return false;
    };

    if (warp == kWorkers / 32 + 1) {   // the loader
        if (lane == 0) {
            int gl = (int)(w0 % g.groups), i = 0;
            for (; i < n; ++i) {
                if (!wait(&bars.ptempty[i % kPtSlots], ((uint32_t)(i / kPtSlots) & 1u) ^ 1u)) break;
                uint8_t *dst = s_pts + (i % kPtSlots) * kPtBytes;
                uint64_t *bar = &bars.ptfull[i % kPtSlots];
                if (!(blockIdx.x == 0 && i == g.drop)) {
                    constexpr uint32_t GB = GROUP * sizeof(int4), AB = GROUP * sizeof(uint2);
                    mbar_arrive_expect_tx(bar, GB + AB + (SPH ? GB : 0));
                    bulk_copy_g2s(dst, g.geo + (long long)gl * GROUP, GB, bar);
                    bulk_copy_g2s(dst + GB, g.aux + (long long)gl * GROUP, AB, bar);
                    if (SPH) bulk_copy_g2s(dst + GB + AB, g.ext + (long long)gl * GROUP, GB, bar);
                }
                if (++gl == (int)g.groups) gl = 0;
            }
            // every copy issued completes before the CTA ends
            for (int j = i > kPtSlots ? i - kPtSlots : 0; j < i; ++j)
                if (!(blockIdx.x == 0 && j == g.drop))
                    mbar_wait(&bars.ptfull[j % kPtSlots], (uint32_t)(j / kPtSlots) & 1u, g.timeout_ns);
        }
    } else if (warp == kWorkers / 32) {
        if (lane == 0) {
            int g0 = (int)(w0 % g.groups);   // group of stage i
            constexpr uint32_t idesc = umma_idesc_f16(false, kRowsA, BN);
            int in_chain = 0;
            uint32_t chain = 0;
            bool ok = true;
            for (int i = 0; i < n && ok; ++i) {
                const int s = i % C::kStages;
                if (in_chain == 0) {
                    if (!(ok = wait(bars.tempty, (chain & 1u) ^ 1u))) break;
                    tc_fence_after();
                }
                if (!(ok = wait(&bars.full[s], (uint32_t)(i / C::kStages) & 1u))) break;
                tc_fence_after();
                const uint32_t a_hi = smem_addr(smem + s * C::kStage), b_hi = a_hi + 2 * C::kA;
                // products of planes (A, B: 0 = hi, 1 = lo), the large ones last, so the truncation of the small ones
                // is small: lo hi, hi lo, hi hi over the whole row; the spherical form's first product is in the
                // first half of the row (K steps 0 and 1), its third in the second half of the lo planes, its second
                // in that of the hi planes
                bool acc = in_chain != 0;
                auto product = [&](int pa, int pb, int k0, int k1) {
                    const uint64_t ad = sw128_kmajor_desc(a_hi + pa * C::kA), bd = sw128_kmajor_desc(b_hi + pb * C::kB);
#pragma unroll
                    for (int kk = k0; kk < k1; ++kk) {
                        umma_f16(tmem, ad + (uint64_t)(2 * kk), bd + (uint64_t)(2 * kk), idesc, acc ? 1u : 0u);
                        acc = true;
                    }
                };
                constexpr int KH = SPH ? 2 : 4;
                product(1, 0, 0, KH);
                product(0, 1, 0, KH);
                if (SPH) {
                    product(1, 1, 2, 4);
                    product(0, 0, 2, 4);
                }
                product(0, 0, 0, KH);
                umma_commit(&bars.empty[s]);
                const bool tile_end = g0 + 1 == (int)g.groups;
                if (++in_chain == CHAIN || tile_end || i + 1 == n) {
                    umma_commit(bars.tfull);
                    in_chain = 0;
                    ++chain;
                }
                g0 = tile_end ? 0 : g0 + 1;
            }
            // every MMA issued completes before the CTA ends
            umma_commit(bars.drain);
            mbar_wait(bars.drain, 0, g.timeout_ns);
        }
    } else {
        // this thread's two points of a stage (spherical: its point) and its first row; a warp's two rows are 4 apart
        // in the spherical form, whose halves of a row then fall on different banks
        const int pair = tid & 15, rl = SPH ? (warp >> 2) * 8 + (warp & 3) + ((tid >> 4) & 1) * 4 : tid >> 4;
        const uint32_t entry = SPH ? (uint32_t)(rl * 128 + (((pair >> 2) ^ (rl & 7)) << 4) + (pair & 3) * 4)
                                   : (uint32_t)(rl * 128 + (((pair >> 1) ^ (rl & 7)) << 4) + (pair & 1) * 8);
        // amplitudes as multiples of 2^(eb - 126), the power of two above the largest
        const uint32_t amax = __reduce_max_sync(0xffffffffu, s_amp[lane < kMmaThreads / 32 ? lane : 0]);
        const uint32_t eb = min((amax >> 23) & 255u, 252u);
        const float a_scale = __uint_as_float((253u - eb) << 23), unscale = __uint_as_float((eb + 1u) << 23);
        const int quarter = warp & 3, cg = warp >> 2;   // tensor-memory lanes and columns of this warp
        const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(cg * HB), total = acc + C::kTotal;
        int t = (int)(w0 / g.groups), gi = (int)(w0 % g.groups);   // tile and group of stage i
        int ra = t % g.tiles_a * kRowsA + rl, rb = t / g.tiles_a * TB + rl;   // this thread's first rows of the tile
        bool pending = false, pend_first = true, pend_end = false;
        uint32_t folded = 0, sunk = 0;
        int pend_t = 0;
        int in_chain = 0, s = 0;
        uint32_t s_use = 0;   // parity of the ring's round

        // the finished chain to the totals (first: of this CTA's part of the tile)
        auto fold = [&](bool first) -> bool {
            if (!wait(bars.tfull, folded & 1u)) return false;
            ++folded;
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < HB; c += 16) {
                float v[2][8], w[2][8];
                tmem_ld8(acc + (uint32_t)c, v[0]);
                if (c + 8 < HB) tmem_ld8(acc + (uint32_t)c + 8u, v[1]);
                if (!first) {
                    tmem_ld8(total + (uint32_t)c, w[0]);
                    if (c + 8 < HB) tmem_ld8(total + (uint32_t)c + 8u, w[1]);
                }
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    if (c + 8 * j >= HB) break;
                    if (!first)
#pragma unroll
                        for (int k = 0; k < 8; k += 2) {
                            const float2 r =
                                __fadd2_rn(make_float2(w[j][k], w[j][k + 1]), make_float2(v[j][k], v[j][k + 1]));
                            v[j][k] = r.x;
                            v[j][k + 1] = r.y;
                        }
                    tmem_st8(total + (uint32_t)(c + 8 * j), v[j]);
                }
            }
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bars.tempty);
            return true;
        };
        // the end of this CTA's part of tile pt: a whole tile is stored; a part goes to the CTA's slot and is counted on
        // the tile, and the CTA that counts last sums the tile's parts in CTA order (whoever is last) and stores it
        auto sink = [&](const int pt) -> bool {
            if (!CGH_DCHECK(pt >= 0 && pt * g.groups < g.units, g.status)) return false;   // the same for every worker
            const long long Cn = gridDim.x;
            const int lo = (int)(((pt * g.groups + 1) * Cn - 1) / g.units);
            const int hi = (int)((((pt + 1) * g.groups) * Cn - 1) / g.units);
            constexpr int Q4 = HB / 4;
            // slot 0 of a CTA holds its first segment, slot 1 its last: the tile's first CTA may have begun before it
            const int lo_slot = lo * g.units / Cn / g.groups == pt ? 0 : 1;
            auto part = [&](int cs) {
                return g.slots + (2ll * cs + (cs == lo ? lo_slot : 0)) * (Q4 * kWorkers) + tid;
            };
            if (lo != hi) {
                float4 *mine = part((int)blockIdx.x);
#pragma unroll
                for (int q = 0; q < Q4; q += 2) {
                    float v[8];
                    tmem_ld8(total + (uint32_t)(4 * q), v);
                    tmem_ld_wait();
                    mine[q * kWorkers] = make_float4(v[0], v[1], v[2], v[3]);
                    mine[(q + 1) * kWorkers] = make_float4(v[4], v[5], v[6], v[7]);
                }
                __threadfence();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars.parts[0]);
                if (tid == 0) {
                    if (!wait(&bars.parts[0], sunk & 1u)) return false;
                    s_last = atomicAdd(&g.counters[pt], 1) == hi - lo;
                    mbar_arrive(&bars.parts[1]);
                }
                if (!wait(&bars.parts[1], sunk & 1u)) return false;
                ++sunk;
                if (!s_last) return true;
                __threadfence();
            }
            const int a = pt % g.tiles_a * kRowsA + quarter * 32 + lane;
            const int b0 = pt / g.tiles_a * TB + (PLANES == 2 ? (cg & 1) * HB : cg * HB);
            float *out = g.out + (PLANES == 2 ? (long long)(cg >> 1) * g.width * g.height : 0ll);
            const float us = unscale;
#pragma unroll
            for (int q = 0; q < Q4; q += 2) {
                float v[8];
                if (lo == hi) {
                    tmem_ld8(total + (uint32_t)(4 * q), v);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int k = 0; k < 8; ++k) v[k] = 0.0f;
                    for (int cs = lo; cs <= hi; cs += 4) {   // four parts per memory round trip
                        float4 x[4][2];
#pragma unroll
                        for (int j = 0; j < 4; ++j)
#pragma unroll
                            for (int i = 0; i < 2; ++i)
                                x[j][i] = cs + j <= hi ? __ldcg(part(cs + j) + (q + i) * kWorkers)
                                                       : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                v[4 * i] += x[j][i].x;
                                v[4 * i + 1] += x[j][i].y;
                                v[4 * i + 2] += x[j][i].z;
                                v[4 * i + 3] += x[j][i].w;
                            }
                    }
                }
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    v[k] = (ACC ? fmaf(v[k], kAccLoss, v[k]) : v[k]) * (SPH ? kSphUnscale : ACC ? kAccUnscale : kUnscale) * us;
                if (!g.a_rows) {   // lanes are columns: each store writes 32 consecutive pixels of a row
                    if (a < g.width)
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (b0 + 4 * q + k < g.height) {
                                float *o = out + (long long)(b0 + 4 * q + k) * g.width + a;
                                *o = g.add ? *o + v[k] : v[k];
                            }
                } else if (a < g.height) {
                    float *row = out + (long long)a * g.width + b0 + 4 * q;
                    if (g.vec && b0 + 4 * q + 8 <= g.width) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            float4 *o = reinterpret_cast<float4 *>(row) + h;
                            const float4 old = g.add ? *o : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                            *o = make_float4(old.x + v[4 * h], old.y + v[4 * h + 1], old.z + v[4 * h + 2],
                                             old.w + v[4 * h + 3]);
                        }
                    } else {
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (b0 + 4 * q + k < g.width) row[k] = g.add ? row[k] + v[k] : v[k];
                    }
                }
            }
            return true;
        };
        const unsigned long long ka = g.a_rows ? g.ref.ky : g.ref.kx, kb = g.a_rows ? g.ref.kx : g.ref.ky;
        const bool swap = g.a_rows != 0;
        // a finished chain is folded after the next stage is made: its MMAs run meanwhile
        for (int i = 0; i <= n; ++i) {
            bool chain_end = false, tile_end = false;
            if (i < n) {
                const int ps = i % kPtSlots;
                if (!wait(&bars.ptfull[ps], (uint32_t)(i / kPtSlots) & 1u)) break;
                if (!wait(&bars.empty[s], s_use ^ 1u)) break;
                const uint8_t *pts = s_pts + ps * kPtBytes;
                const int4 *geo = reinterpret_cast<const int4 *>(pts) + pair;
                const uint2 *aux = reinterpret_cast<const uint2 *>(pts + GROUP * sizeof(int4)) + pair;
                const uint32_t base = smem_addr(smem + s * C::kStage) + entry;
                const uint32_t add_a = (uint32_t)((ka * (unsigned long long)ra) >> 32) + g.ref.phi0;
                const uint32_t add_b = (uint32_t)((kb * (unsigned long long)rb) >> 32);
                if constexpr (SPH) {
                    const int4 q = *geo;
                    const uint2 x = *aux;
                    const float4 e = *(reinterpret_cast<const float4 *>(pts + GROUP * (sizeof(int4) + sizeof(uint2))) +
                                       pair);
                    const int da = ra - (swap ? q.y : q.x), db = rb - (swap ? q.x : q.y);
                    const int oa = rl - kRowsA / 2, ob = rl - TB / 2;
                    const SphPoint P = sph_point(e, da - oa, db - ob, 0.5f * TB);
                    const uint32_t d0 = (uint32_t)__float2int_rn(P.d0 * 2147483648.0f) << 1;
                    sph_entries<kRowsA / 32, false>(P, q, da, oa, pair & 1, add_a + x.x + d0, ref_step(32 * ka),
                                                    __uint_as_float(x.y) * a_scale * kEntryScale, base, C::kA);
                    sph_entries<TB / 32, true>(P, q, db, ob, pair & 1, add_b, ref_step(32 * kb), 0.0f,
                                               base + 2 * C::kA, C::kB);
                } else {
                    side_entries<kRowsA / 32, false, PLANES, ACC>(geo, aux, swap, ra, add_a, ref_step(32 * ka),
                                                             g.ref.piston ? ~0u : 0u, a_scale, base, C::kA, 0);
                    side_entries<TB / 32, true, PLANES, ACC>(geo, aux, swap, rb, add_b, ref_step(32 * kb), 0u, 0.0f,
                                                        base + 2 * C::kA, C::kB, TB * 128);
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&bars.ptempty[ps]);
                    mbar_arrive(&bars.full[s]);
                }
                if (++s == C::kStages) {
                    s = 0;
                    s_use ^= 1u;
                }
                tile_end = gi + 1 == (int)g.groups || i + 1 == n;
                chain_end = ++in_chain == CHAIN || tile_end;
            }
            if (pending) {
                if (!fold(pend_first)) break;
                pend_first = pend_end;
                if (pend_end && !sink(pend_t)) break;
                pending = false;
            }
            if (chain_end) {
                pending = true;
                pend_end = tile_end;
                pend_t = t;
                in_chain = 0;
            }
            if (++gi == (int)g.groups) {
                gi = 0;
                ++t;
                ra += kRowsA;
                if (t % g.tiles_a == 0) {
                    ra = rl;
                    rb += TB;
                }
            }
        }
    }
    __syncthreads();
    if (warp == kWorkers / 32) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, C::kTmemCols);
    }
}

template <int BN, int PLANES, bool SPH, bool ACC>
cudaError_t launch_as(const MmaArgs &g, int ctas, cudaStream_t s)
{
    static PerDeviceOnce configured;
    const cudaError_t e = configured.run([] {
        return cudaFuncSetAttribute(direct_mma_kernel<BN, PLANES, SPH, ACC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    MmaCfg<BN>::kSmem);
    });
    if (e != cudaSuccess) return e;
    return launch_dependent(direct_mma_kernel<BN, PLANES, SPH, ACC>, dim3(ctas), dim3(kMmaThreads), MmaCfg<BN>::kSmem, s, true, g);
}

template <int PLANES, bool SPH, bool ACC>
cudaError_t launch_bn(int bn, const MmaArgs &g, int ctas, cudaStream_t s)
{
    switch (bn) {
    case 64: return launch_as<64, PLANES, SPH, ACC>(g, ctas, s);
    case 128: return launch_as<128, PLANES, SPH, ACC>(g, ctas, s);
    case 192: return launch_as<192, PLANES, SPH, ACC>(g, ctas, s);
    case 224:
        if constexpr (PLANES == 1 && !SPH) return launch_as<224, PLANES, SPH, ACC>(g, ctas, s);
        else return cudaErrorInvalidValue;
    case 256: return launch_as<256, PLANES, SPH, ACC>(g, ctas, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// The totals take one FP32 addition per chain of 64 points, whose rounding grows with the square root of their number:
// a launch adds at most kMmaLaunchPoints points of a tile in one CTA, and the next launch adds to its output
// (2048x2048, 5 10^5 points: NRMS 4.3e-7; the SIMT kernel's 8.9e-7, one launch about 1.6e-6).  Where the last launch
// would be left with fewer groups than the CTAs need, the groups are cut into equal shares: with L > 1 launches each then
// has at least groups / L > 320 ctas / tiles of them.
int direct_mma_launches(const DirectMmaLayout &lay, int group, int64_t n_points)
{
    const int64_t groups = (n_points + group - 1) / group;
    const int64_t share = (lay.tiles * groups + lay.ctas - 1) / lay.ctas;   // of a CTA; of a tile at most all groups
    return (int)(((share < groups ? share : groups) * group + kMmaLaunchPoints - 1) / kMmaLaunchPoints);
}

cudaError_t launch_direct_mma(const DirectMmaLayout &lay, int planes, const int4 *geo, const uint2 *aux,
                              const float *amp_max, int amp_parts, int n_points, int width, int height, float *out,
                              float *slots, int *counters, int *status, uint64_t timeout_ns, cudaStream_t s, int drop,
                              const PhaseRef &ref, const float4 *ext, float phase_lo, float phase_hi, bool accurate)
{
    const int group = ext != nullptr ? kSphMmaGroup : kGroup;
    if (n_points < 1 || lay.ctas < 1 || (planes != 1 && planes != 2) || (uintptr_t)slots % 16 != 0)
        return cudaErrorInvalidValue;
    MmaArgs g{};
    const int launches = direct_mma_launches(lay, group, n_points);
    const long long all_groups = (n_points + group - 1) / group, per = (all_groups + launches - 1) / launches;
    const int side_a = lay.a_rows ? height : width, side_b = lay.a_rows ? width : height;
    const int tb = lay.bn / planes;
    g.tiles_a = (side_a + kRowsA - 1) / kRowsA;
    const long long tiles = (long long)g.tiles_a * ((side_b + tb - 1) / tb);
    // whole tiles per CTA (one share each) need neither slots nor counters
    if (tiles != lay.tiles || (lay.ctas != tiles && (slots == nullptr || counters == nullptr)))
        return cudaErrorInvalidValue;
    g.phase_lo = phase_lo;
    g.phase_hi = phase_hi;
    g.amp_max = amp_max;
    g.amp_parts = amp_parts;
    g.out = out;
    g.slots = reinterpret_cast<float4 *>(slots);
    g.status = status;
    g.timeout_ns = timeout_ns;
    g.width = width;
    g.height = height;
    g.a_rows = lay.a_rows;
    g.vec = width % 4 == 0 && (uintptr_t)out % 16 == 0 && ((long long)width * height) % 4 == 0;
    g.ref = ref;
    if (ext != nullptr && planes != 1) return cudaErrorInvalidValue;
    const bool even = tiles * ((all_groups - 1) % per + 1) < lay.ctas;
    auto begin = [&](long long k) { return even ? all_groups * k / launches : std::min(all_groups, per * k); };
    for (long long k = 0; begin(k) < all_groups; ++k) {
        const long long first = begin(k);
        g.groups = begin(k + 1) - first;
        g.units = tiles * g.groups;
        if (lay.ctas > g.units || g.units / lay.ctas >= 0x7ffffff0ll) return cudaErrorInvalidValue;
        g.geo = geo + first * group;
        g.aux = aux + first * group;
        g.ext = ext != nullptr ? ext + first * group : nullptr;
        g.counters = counters != nullptr ? counters + k * tiles : nullptr;
        g.drop = k == 0 ? drop : -1;
        g.add = k > 0;
        const cudaError_t e = ext != nullptr ? launch_bn<1, true, false>(lay.bn, g, lay.ctas, s)
                              : planes == 2  ? launch_bn<2, false, false>(lay.bn, g, lay.ctas, s)
                              : accurate     ? launch_bn<1, false, true>(lay.bn, g, lay.ctas, s)
                                             : launch_bn<1, false, false>(lay.bn, g, lay.ctas, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace cgh
