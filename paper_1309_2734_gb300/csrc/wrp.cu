// f3: step 1 of the wavefront-recording method (Section 2.3): the complex
// amplitude of the point cloud recorded on a virtual plane at distance z_wrp
// from the hologram (same grid), each point summed only over its window.
//
// Window.  The light of point j (distance d_j = z_j - z_wrp > 0 behind the
// plane) that can reach the hologram within the grid's largest diffraction
// angle, sin(theta) = lambda / (2 p), crosses the plane within radius
// d_j tan(theta): in pixels w = d s / sqrt(1 - s^2) / p, s = lambda / (2 p), and
// the window holds the pixels with (m - x_j)^2 + (n - y_j)^2 <= floor(w^2).
// That integer is computed in double with every operation rounded on its own
// (no contraction), so it is the same number on any IEEE machine.
//
// Phase (Eq. 2, at distance d_j): c_j r^2 turns, c_j = p^2 / (2 lambda d_j), in
// 64-bit fixed point as in the point preparation, plus the piston d_j / lambda
// with CGH_PHASE_FRESNEL_PISTON.  r^2 = dx^2 + dy^2 splits into a column turn and
// a row turn, so a term is the product of a column's and a row's
// exp(i 2 pi t), which a tile takes once per point.
//
// Gather, deterministic.  For every band of 64 rows and segment of kSegPoints
// points one CTA lists, in index order (ballot compaction), the points whose
// window reaches the band, with the columns it spans.  One CTA per 32 x 64 pixel
// tile then scans its band's lists for the points whose window's bounding box
// meets the tile and, kBatch of them at a time, makes their 32 column and 64 row
// entries and the squared distance each row leaves to the window's edge in
// shared memory; each warp adds those whose window meets its 16 x 16 block, two
// packed FMAs a pixel inside the window.  No atomics, points in index order, so
// the sums are bit-reproducible.
//
// 2048x2048, 10^5 points 2-10 mm behind the plane (before: a hardware sine and
// cosine per pixel and point, lists counted, scanned by one thread and filled):
// record 0.39 -> 0.25 ms, lists 0.105 -> 0.014 ms, preparation 0.015.  Bound by
// instruction issue (62 % of the slots) and the reads of the entries: about 50
// instructions a warp for a point and block, 56 % of whose pixels are inside the
// window (rows of 32 pixels for a warp: 0.32 ms).
#include <cmath>

#include "device_util.cuh"
#include "half_turn.cuh"
#include "host_util.h"
#include "kernels.h"

namespace cgh {

namespace {

using dev::f2;

constexpr int kTileW = 32, kTileH = 64;   // pixels of a tile
constexpr int kThreads = 256;      // 8 warps, each a block of 16 x 16 pixels
constexpr int kBlock = 16;
constexpr int kSegPoints = 8192;   // points a CTA of the lists walks (10^5 points: 14 us; 16384 points 24 us, most SMs
                                   // with one CTA or two)
constexpr int kScan = 4 * kThreads;   // points a step of the lists takes, four a thread
constexpr int kTileScan = 2 * kThreads;   // list entries a tile's scanning step takes, two a thread
constexpr int kBatch = 32;         // points whose entries are in shared memory at once
static_assert(kSegPoints % kScan == 0 && kPointTile % 4 == 0, "whole steps; four points a thread");

// The grid's constants, each operation rounded on its own (the host's, so the same on any IEEE machine).
struct WrpGrid {
    double pp, l2, s, den, pitch, lambda, z;   // p^2, 2 lambda, sin(theta), cos(theta)
};

WrpGrid wrp_grid(double pitch, double lambda, double z_wrp)
{
    WrpGrid g;
    volatile double two_p = 2.0 * pitch, pp = pitch * pitch, l2 = 2.0 * lambda;
    volatile double s = lambda / two_p;
    volatile double s2 = s * s;
    volatile double c2 = 1.0 - s2;
    g.pp = pp;
    g.l2 = l2;
    g.s = s;
    g.den = std::sqrt(c2);
    g.pitch = pitch;
    g.lambda = lambda;
    g.z = z_wrp;
    return g;
}

// rows[j] = {first row, last row} of the window; of an invalid or padding point an empty range.
__global__ void wrp_prep_kernel(const float *__restrict__ xyz, const float *__restrict__ amp, int n, int n_pad,
                                const WrpGrid g, bool piston, int4 *__restrict__ geo, uint4 *__restrict__ win,
                                int2 *__restrict__ rows, int *status)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_pad) return;
    bool ok = false;
    float fx = 0.0f, fy = 0.0f, a = 0.0f;
    double d = 0.0;
    if (j < n) {
        fx = xyz[3 * j + 0];
        fy = xyz[3 * j + 1];
        const float fz = xyz[3 * j + 2];
        a = amp[j];
        d = __dadd_rn((double)fz, -g.z);
        ok = isfinite(fx) && isfinite(fy) && isfinite(fz) && isfinite(a) && d > 0.0 && fx == rintf(fx) &&
             fy == rintf(fy) && fabsf(fx) <= (float)kMaxCoord && fabsf(fy) <= (float)kMaxCoord;
        if (!ok) atomicOr(status, kStatusInput);
    }
    if (!ok) {
        geo[j] = make_int4(0, 0, 0, 0);
        win[j] = make_uint4(0u, 0u, 0u, 0u);
        rows[j] = make_int2(0x7fffffff, -0x7fffffff);
        return;
    }
    const double c = __ddiv_rn(g.pp, __dmul_rn(g.l2, d));
    const double scaled = (c - floor(c)) * 18446744073709551616.0;   // exact
    const unsigned long long C = (scaled >= 18446744073709551616.0) ? 0ull : __double2ull_rn(scaled);
    geo[j] = make_int4((int)fx, (int)fy, (int)(unsigned)(C >> 32), (int)(unsigned)(C & 0xffffffffull));
    unsigned pist = 0u;
    if (piston) {
        const double zt = d / g.lambda;
        const double pf = (zt - floor(zt)) * 4294967296.0;
        pist = pf >= 4294967295.5 ? 0u : (unsigned)__double2ull_rn(pf);
    }
    // squared window radius, each double operation rounded on its own
    const double w = __ddiv_rn(__ddiv_rn(__dmul_rn(d, g.s), g.den), g.pitch);
    const double w2 = floor(__dmul_rn(w, w));
    const unsigned W2 = w2 >= 2147483647.0 ? 2147483647u : (unsigned)w2;
    unsigned R = (unsigned)sqrtf((float)W2);   // integer radius: R^2 <= W2 < (R + 1)^2
    while ((unsigned long long)(R + 1) * (R + 1) <= W2) ++R;
    while ((unsigned long long)R * R > W2) --R;
    win[j] = make_uint4(pist, __float_as_uint(a), W2, R);
    rows[j] = make_int2((int)fy - (int)R, (int)fy + (int)R);
}

// Ballot compaction of one step, N consecutive items a thread (index order = thread, then item): the position of
// this thread's first hit among the step's hits and their total.  s_wcnt is read before the caller's next barrier.
template <int N>
__device__ __forceinline__ int compact_hits(const bool (&hit)[N], int *s_wcnt, int &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int below = 0, all = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const unsigned mask = __ballot_sync(0xffffffffu, hit[k]);
        below += __popc(mask & ((1u << lane) - 1u));
        all += __popc(mask);
    }
    if (lane == 0) s_wcnt[warp] = all;
    __syncthreads();
    int before = 0;
    total = 0;
#pragma unroll
    for (int k = 0; k < kThreads / 32; ++k) {
        before += k < warp ? s_wcnt[k] : 0;
        total += s_wcnt[k];
    }
    return before + below;
}

__device__ __forceinline__ int clamp16(int v)
{
    return max(-32768, min(32767, v));
}

// One CTA per (band of kTileH rows, segment of kSegPoints points): in index order, the points whose window reaches
// the band, {index, first column | last column << 16}, at list + cell cap (the points of a segment), and their count.
__global__ void __launch_bounds__(kThreads)
    wrp_band_kernel(const int4 *__restrict__ geo, const uint4 *__restrict__ win, const int2 *__restrict__ rows,
                    int n_pad, int cap, int *__restrict__ count, int2 *__restrict__ list)
{
    __shared__ int s_wcnt[2][kThreads / 32];
    const int y0 = blockIdx.x * kTileH;
    const int cell = blockIdx.x * gridDim.y + blockIdx.y;   // band-major, then segment
    const int begin = blockIdx.y * kSegPoints;
    const int end = min(n_pad, begin + kSegPoints);
    int2 *out = list + (long long)cell * cap;
    int written = 0, turn = 0;
    for (int base = begin; base < end; base += kScan, turn ^= 1) {
        const int j = base + 4 * threadIdx.x;
        bool hit[4] = {false, false, false, false};
        if (j < end) {   // n_pad is a multiple of four
            const int4 r01 = *reinterpret_cast<const int4 *>(rows + j), r23 = *reinterpret_cast<const int4 *>(rows + j + 2);
            hit[0] = r01.y >= y0 && r01.x < y0 + kTileH;
            hit[1] = r01.w >= y0 && r01.z < y0 + kTileH;
            hit[2] = r23.y >= y0 && r23.x < y0 + kTileH;
            hit[3] = r23.w >= y0 && r23.z < y0 + kTileH;
        }
        int total;
        int pos = written + compact_hits(hit, s_wcnt[turn], total);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (hit[k]) {
                const int x = geo[j + k].x, R = (int)win[j + k].w;
                out[pos++] = make_int2(j + k, (clamp16(x - R) & 0xffff) | (clamp16(x + R) << 16));
            }
        written += total;
    }
    if (threadIdx.x == 0) count[cell] = written;
}

// A block's rows of equal parity side by side: a lane's eight rows are two 16-byte reads.
__device__ __forceinline__ int left_at(int row)
{
    return (row & ~(kBlock - 1)) + (row & 1) * (kBlock / 2) + ((row >> 1) & (kBlock / 2 - 1));
}

struct WrpShared {
    float4 col[kBatch][kTileW];   // {cos, sin, -sin, cos} of a column's turn
    float4 row[kBatch][kTileH];   // A {cos, cos, sin, sin} of a row's turn
    int left[kBatch][kTileH];     // the row's squared half width W2 - dy^2, at left_at(row)
    int4 geo[kTileScan + kBatch];   // the queue of points that meet the tile
    uint4 win[kTileScan + kBatch];
    int wcnt[2][kThreads / 32];
};

__global__ void __launch_bounds__(kThreads, 3)
    wrp_record_kernel(const int4 *__restrict__ geo, const uint4 *__restrict__ win, int n_pad, int H, int W,
                      int tiles_x, int segs, int cap, const int *__restrict__ count, const int2 *__restrict__ list,
                      float2 *__restrict__ pad, long long pad_ld, float *__restrict__ planes)
{
    extern __shared__ uint8_t s_raw[];
    WrpShared &S = *reinterpret_cast<WrpShared *>(s_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int band = blockIdx.x / tiles_x;
    const int x0 = (blockIdx.x % tiles_x) * kTileW, y0 = band * kTileH;
    // this warp's block, this lane's column of it and rows 2 r + (lane / 16)
    const int bx = (warp & 1) * kBlock, by = (warp >> 1) * kBlock;
    const int cx = bx + (lane & 15), ry = by + (lane >> 4);
    float2 acc[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) acc[r] = make_float2(0.0f, 0.0f);

    // adds np <= kBatch points of the queue from `first` on
    auto batch = [&](int first, int np) {
        // entries: thread t makes entries 2 t and 2 t + 1 of 512 a round (96 a point: its columns, then its rows)
        constexpr int kEntries = kTileW + kTileH;
#pragma unroll 1
        for (int e = 2 * tid; e < np * kEntries; e += 2 * kThreads) {
            const int h = e / kEntries, k = e - h * kEntries;
            const bool is_row = k >= kTileW;
            const int4 g = S.geo[first + h];
            const uint4 v = S.win[first + h];
            const int d0 = is_row ? y0 + (k - kTileW) - g.y : x0 + k - g.x, d1 = d0 + 1;
            const uint32_t q0 = (uint32_t)(d0 * d0), q1 = (uint32_t)(d1 * d1);
            const uint32_t add = is_row ? v.x : 0u;
            const uint32_t t0 = (uint32_t)g.z * q0 + __umulhi((uint32_t)g.w, q0) + add;
            const uint32_t t1 = (uint32_t)g.z * q1 + __umulhi((uint32_t)g.w, q1) + add;
            const float2 turn[1] = {make_float2((float)(int)t0, (float)(int)t1)};
            float2 s[1], c[1];
            dev::half_turn2<1>(turn, s, c);
            float2 co = __ffma2_rn(make_float2(-s[0].x, -s[0].y), s[0], f2(1.0f)), si = __fmul2_rn(s[0], c[0]);
            if (is_row) {
                const int r = k - kTileW;
                const float a = __uint_as_float(v.y);
                co = __fmul2_rn(co, f2(a));
                si = __fmul2_rn(si, f2(a));
                S.row[h][r] = make_float4(co.x, co.x, si.x, si.x);
                S.row[h][r + 1] = make_float4(co.y, co.y, si.y, si.y);
                // a squared distance beyond the window's leaves no pixel (W2 < 2^31, dy^2 < 2^31)
                S.left[h][left_at(r)] = (int)v.z - (int)q0;
                S.left[h][left_at(r + 1)] = (int)v.z - (int)q1;
            } else {
                S.col[h][k] = make_float4(co.x, si.x, -si.x, co.x);
                S.col[h][k + 1] = make_float4(co.y, si.y, -si.y, co.y);
            }
        }
        // the batch's points whose window meets this warp's block
        bool meets = false;
        if (lane < np) {
            const int4 g = S.geo[first + lane];
            const int dx = max(0, max(x0 + bx - g.x, g.x - (x0 + bx + kBlock - 1)));
            const int dy = max(0, max(y0 + by - g.y, g.y - (y0 + by + kBlock - 1)));
            meets = (uint32_t)(dx * dx) + (uint32_t)(dy * dy) <= S.win[first + lane].z;
        }
        unsigned todo = __ballot_sync(0xffffffffu, meets);
        __syncthreads();
        while (todo) {
            const int h = __ffs(todo) - 1;
            todo &= todo - 1;
            const float4 c = S.col[h][cx];
            const int dx = x0 + cx - S.geo[first + h].x;
            const int dx2 = dx * dx;
            const float2 c0 = make_float2(c.x, c.y), c1 = make_float2(c.z, c.w);
            const int4 l0 = *reinterpret_cast<const int4 *>(&S.left[h][left_at(ry)]);
            const int4 l1 = *reinterpret_cast<const int4 *>(&S.left[h][left_at(ry) + 4]);
            const int left[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float4 b = S.row[h][ry + 2 * r];
                if (dx2 <= left[r])   // (re, im) += cos b (cos a, sin a) + sin b (-sin a, cos a)
                    acc[r] = __ffma2_rn(make_float2(b.z, b.w), c1, __ffma2_rn(make_float2(b.x, b.y), c0, acc[r]));
            }
        }
        __syncthreads();   // the tables and the queue are free
    };

    int queued = 0, turn = 0;
    for (int seg = 0; seg < segs; ++seg) {
        const long long cell = (long long)band * segs + seg;
        const int2 *ls = list != nullptr ? list + cell * cap : nullptr;
        const int items = list != nullptr ? count[cell] : min(kSegPoints, n_pad - seg * kSegPoints);
        for (int base = 0; base < items; base += kTileScan, turn ^= 1) {
            const int i = base + 2 * tid;
            bool hit[2] = {false, false};
            int j[2] = {0, 0};
            if (i < items && ls != nullptr) {   // cap and the cells' starts are even
                const int4 e = *reinterpret_cast<const int4 *>(ls + i);
                j[0] = e.x;
                j[1] = e.z;
                hit[0] = (e.y >> 16) >= x0 && (int)(short)e.y < x0 + kTileW;
                hit[1] = i + 1 < items && (e.w >> 16) >= x0 && (int)(short)e.w < x0 + kTileW;
            } else if (i < items) {   // no lists: every point (n_pad and kSegPoints are even)
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    j[k] = seg * kSegPoints + i + k;
                    const int4 g = geo[j[k]];
                    const int R = (int)win[j[k]].w;
                    hit[k] = g.x + R >= x0 && g.x - R < x0 + kTileW && g.y + R >= y0 && g.y - R < y0 + kTileH;
                }
            }
            int total;
            int pos = queued + compact_hits(hit, S.wcnt[turn], total);
#pragma unroll
            for (int k = 0; k < 2; ++k)
                if (hit[k]) {
                    S.geo[pos] = geo[j[k]];
                    S.win[pos++] = win[j[k]];
                }
            queued += total;
            if (queued < kBatch) continue;
            __syncthreads();   // the queue is written
            int done = 0;
            for (; done + kBatch <= queued; done += kBatch) batch(done, kBatch);
            const int rest = queued - done;   // fewer than kBatch: to the front of the queue
            int4 g = make_int4(0, 0, 0, 0);
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (tid < rest) {
                g = S.geo[done + tid];
                v = S.win[done + tid];
            }
            __syncthreads();
            if (tid < rest) {
                S.geo[tid] = g;
                S.win[tid] = v;
            }
            queued = rest;
        }
    }
    __syncthreads();
    if (queued > 0) batch(0, queued);

    const int m = x0 + cx;
    if (m >= W) return;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int n = y0 + ry + 2 * r;
        if (n >= H) continue;
        if (pad != nullptr) {
            pad[(long long)n * pad_ld + m] = acc[r];
        } else {
            planes[(long long)n * W + m] = acc[r].x;
            planes[(long long)H * W + (long long)n * W + m] = acc[r].y;
        }
    }
}

}  // namespace

cudaError_t launch_wrp_prep(const float *d_xyz, const float *d_amp, int n, int n_pad, double pitch, double lambda,
                            double z_wrp, bool piston, int4 *geo, uint4 *win, int2 *rows, int *status, cudaStream_t s)
{
    if (n_pad <= 0) return cudaSuccess;
    wrp_prep_kernel<<<(n_pad + 127) / 128, 128, 0, s>>>(d_xyz, d_amp, n, n_pad, wrp_grid(pitch, lambda, z_wrp), piston,
                                                      geo, win, rows, status);
    return cudaGetLastError();
}

static int wrp_segs(int n_pad)
{
    return n_pad > 0 ? (n_pad - 1) / kSegPoints + 1 : 1;
}

// a segment's list holds at most its points
static int wrp_cap(int n_pad)
{
    return n_pad < kSegPoints ? n_pad : kSegPoints;
}

int64_t wrp_band_cells(int H, int n_pad)
{
    return (int64_t)((H + kTileH - 1) / kTileH) * wrp_segs(n_pad);
}

size_t wrp_list_bytes(int H, int n_pad)
{
    return (size_t)wrp_band_cells(H, n_pad) * wrp_cap(n_pad) * sizeof(int2);
}

cudaError_t launch_wrp_bands(const int4 *geo, const uint4 *win, const int2 *rows, int n_pad, int H, int *count,
                             int2 *list, cudaStream_t s)
{
    const dim3 grid((H + kTileH - 1) / kTileH, wrp_segs(n_pad));
    wrp_band_kernel<<<grid, kThreads, 0, s>>>(geo, win, rows, n_pad, wrp_cap(n_pad), count, list);
    return cudaGetLastError();
}

cudaError_t launch_wrp_record(const int4 *geo, const uint4 *win, int n_pad, int H, int W, const int *count,
                              const int2 *list, float2 *pad, int64_t pad_ld, float *planes, cudaStream_t s)
{
    static PerDeviceOnce configured;   // the queue and the entries exceed the default 48 KB
    const cudaError_t e = configured.run([] {
        return cudaFuncSetAttribute(wrp_record_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sizeof(WrpShared));
    });
    if (e != cudaSuccess) return e;
    const int tiles_x = (W + kTileW - 1) / kTileW, tiles_y = (H + kTileH - 1) / kTileH;
    wrp_record_kernel<<<tiles_x * tiles_y, kThreads, sizeof(WrpShared), s>>>(
        geo, win, n_pad, H, W, tiles_x, wrp_segs(n_pad), wrp_cap(n_pad), count, list, pad, (long long)pad_ld, planes);
    return cudaGetLastError();
}

}  // namespace cgh
