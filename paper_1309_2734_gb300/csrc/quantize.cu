// a6: 8-bit quantisation of an amplitude hologram (min/max rule).
//
// The paper stores its phase-only holograms as unsigned char with
// 255/(2 pi) per radian (Section 4.1).  For the amplitude hologram of Eq. 5
// the range is not known in advance, so it is measured:
//   pass 1: min and max of each block's share of the field, on an
//           order-preserving integer encoding (NaN skipped);
//   pass 2: lo = min, hi = max over the blocks, s = the smallest float >= 255 / ((double)hi - (double)lo),
//           q = floor(fl(fl(v - lo) * s)) clamped to [0, 255], NaN -> 0.
// Each single-precision operation is rounded on its own (no FMA contraction),
// so the output is reproducible bit for bit by any IEEE implementation.
//
// Two dependent launches; each block of the second reduces the parts of the first itself, and starts while the first
// still runs.  A small field is bound by launches, a large one by its two reads.  One call (before, with a third
// launch to clear atomics and 16 pixels a thread): 1920x1080 14.6 us (18.7), 2^24 values 31.5 (35.6), 2^27 215 (214).
#include <algorithm>
#include <cfloat>

#include "device_util.cuh"
#include "host_util.h"
#include "kernels.h"

namespace cgh {

namespace {

__device__ __forceinline__ uint32_t order_key(float f)
{
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__device__ __forceinline__ float from_key(uint32_t k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// The block's minimum and maximum in every thread (256 threads).
__device__ __forceinline__ void block_minmax(uint32_t &lo, uint32_t &hi)
{
    __shared__ uint32_t s_lo[8], s_hi[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
        s_lo[warp] = lo;
        s_hi[warp] = hi;
    }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, s_lo[lane & 7]);
    hi = __reduce_max_sync(0xffffffffu, s_hi[lane & 7]);
}

__global__ void __launch_bounds__(256) minmax_kernel(const float *f, long long n, uint2 *part, bool vec)
{
    grid_wait();
    grid_launch_dependents();
    uint32_t lo = 0xffffffffu, hi = 0u;
    auto take = [&](float v) {
        if (v == v) {
            const uint32_t k = order_key(v);
            lo = min(lo, k);
            hi = max(hi, k);
        }
    };
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long first = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long n4 = vec ? n / 4 : 0;
#pragma unroll 4
    for (long long i = first; i < n4; i += stride) {
        const float4 v = reinterpret_cast<const float4 *>(f)[i];
        take(v.x);
        take(v.y);
        take(v.z);
        take(v.w);
    }
    for (long long i = 4 * n4 + first; i < n; i += stride) take(f[i]);
    block_minmax(lo, hi);
    if (threadIdx.x == 0) part[blockIdx.x] = make_uint2(lo, hi);
}

__device__ __forceinline__ uint8_t quantize_one(float v, float lo, float s)
{
    const float q = floorf(__fmul_rn(__fsub_rn(v, lo), s));
    return (q >= 255.0f) ? (uint8_t)255 : ((q >= 0.0f) ? (uint8_t)q : (uint8_t)0);
}

__global__ void __launch_bounds__(256) map_kernel(const float *f, long long n, const uint2 *part, int parts,
                                                  uint8_t *out, bool vec)
{
    grid_wait();
    uint32_t klo = 0xffffffffu, khi = 0u;
    for (int i = threadIdx.x; i < parts; i += blockDim.x) {
        const uint2 p = __ldcg(part + i);
        klo = min(klo, p.x);
        khi = max(khi, p.y);
    }
    block_minmax(klo, khi);
    const float lo = from_key(klo);
    const float hi = from_key(khi);
    const bool degenerate = !(hi > lo);
    float s = 0.0f;
    if (!degenerate) {
        const double sd = 255.0 / ((double)hi - (double)lo);
        if (sd > (double)FLT_MAX) {
            s = FLT_MAX;
        } else {
            s = __double2float_ru(sd);
            if (isinf(s)) s = FLT_MAX;
        }
    }
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long first = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    long long done = 0;
    if (vec) {
        const long long n4 = n / 4;
#pragma unroll 4
        for (long long i = first; i < n4; i += stride) {
            const float4 v = reinterpret_cast<const float4 *>(f)[i];
            reinterpret_cast<uint32_t *>(out)[i] =
                degenerate ? 0u
                           : quantize_one(v.x, lo, s) | (quantize_one(v.y, lo, s) << 8) |
                                 (quantize_one(v.z, lo, s) << 16) | ((uint32_t)quantize_one(v.w, lo, s) << 24);
        }
        done = n4 * 4;
    }
    for (long long i = done + first; i < n; i += stride) out[i] = degenerate ? (uint8_t)0 : quantize_one(f[i], lo, s);
}

int quant_grid(long long work)
{
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long want = (work + 255) / 256;
    const long long cap = (long long)sms * 8;
    return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

// Phase of the complex wave in [0, 2 pi) (Eq. 3; the listings add 2 pi to
// negative phases), scaled by 255 / (2 pi) and floored, as the listings of
// Section 4.1 store their phase-only holograms (clamped to 255: psi + 2 pi may
// round up to 2 pi in single precision; NaN -> 0).
__device__ __forceinline__ uint8_t kinoform_one(float re, float im)
{
    float psi = atan2f(im, re);
    if (psi < 0.0f) psi = __fadd_rn(psi, 6.28318530717958648f);
    const float x = floorf(__fmul_rn(psi, 40.58451048843331f));   // 255 / (2 pi)
    return (x >= 255.0f) ? (uint8_t)255 : ((x >= 0.0f) ? (uint8_t)x : (uint8_t)0);
}

// VEC: four pixels a thread, 16-byte loads and a 4-byte store (the planes and out aligned), the rest one by one; else, on
// planes of an odd size, one by one with the registers of one (1283x717 6.4 -> 6.0 us).
template <bool VEC>
__global__ void kinoform_kernel(const float *__restrict__ re, const float *__restrict__ im, long long n,
                                uint8_t *__restrict__ out)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long first = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long n4 = VEC ? n / 4 : 0;
    for (long long i = first; VEC && i < n4; i += stride) {
        const float4 r = reinterpret_cast<const float4 *>(re)[i], m = reinterpret_cast<const float4 *>(im)[i];
        reinterpret_cast<uchar4 *>(out)[i] = make_uchar4(kinoform_one(r.x, m.x), kinoform_one(r.y, m.y),
                                                         kinoform_one(r.z, m.z), kinoform_one(r.w, m.w));
    }
    for (long long i = 4 * n4 + first; i < n; i += stride) out[i] = kinoform_one(re[i], im[i]);
}

}  // namespace

cudaError_t launch_kinoform8(const float *re, const float *im, int64_t n, uint8_t *out, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const bool vec = (uintptr_t)re % 16 == 0 && (uintptr_t)im % 16 == 0 && (uintptr_t)out % 4 == 0;
    if (vec) kinoform_kernel<true><<<quant_grid(n / 4), 256, 0, s>>>(re, im, n, out);
    else kinoform_kernel<false><<<quant_grid(n), 256, 0, s>>>(re, im, n, out);
    return cudaGetLastError();
}

cudaError_t launch_quantize8(const float *field, int64_t n, uint8_t *out, uint32_t *scratch, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    uint2 *part = reinterpret_cast<uint2 *>(scratch);
    const bool vec = ((uintptr_t)field % 16 == 0) && ((uintptr_t)out % 16 == 0);
    // 16 values a thread, so that a small field leaves few parts to the mapping blocks
    const int blocks = std::min(quant_grid(n / 16), kQuantParts);
    cudaError_t e = launch_dependent(minmax_kernel, dim3(blocks), dim3(256), 0, s, true, field, (long long)n, part,
                                     (uintptr_t)field % 16 == 0);
    if (e != cudaSuccess) return e;
    return launch_dependent(map_kernel, dim3(quant_grid(vec ? n / 8 : n)), dim3(256), 0, s, true, field, (long long)n, part,
                            blocks, out, vec);
}

}  // namespace cgh
