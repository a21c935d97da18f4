// Autotuner and launch-shape selection (host side).
//
// Static rules (no measurement):
//   choose_direct_mma   tile and CTAs of the direct form on the tensor cores;
//   choose_layout       the spherical kernel's CTA shape (less padding) with its split;
//   choose_gemm_bn      GEMM tile width with the least padding of the width;
//   choose_gemm_splits  K splits of the GEMM, to balance tiles over the CTAs.
//
// Measured rules (a context, outside any stream capture):
//   tune_calibrate      times every form on seven synthetic clouds on this
//                       device and fits, per form, the scale of its kernel's
//                       time model and what that leaves out (form_terms);
//   tune_choose_form    the fastest form whose stated NRMS bound is within the
//                       requested tolerance, by that model;
//   tune_choose_bn      the fastest GEMM tile width for a hologram shape and
//                       form, timed on that shape with 4096 points, cached.
// With CGH_TUNE_CACHE=<path> in the environment the measurements are read
// from and written to a small JSON file keyed by the device name.
#include "tuner.h"

#include <algorithm>
#include <array>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "context.h"

namespace cgh {

namespace {
constexpr int kForms = 6;
}  // namespace

// Critical path of a direct launch in point-tile steps of one CTA: rounds of pixel tiles x splits over the
// resident CTA slots, times the longest point chunk (chunks differ by at most one tile); each extra chunk adds a
// plane of partial sums, written and read back by the reduction: 0.2 % per chunk.
static double direct_path(int64_t pixel_tiles, int64_t point_tiles, int64_t s, int64_t slots)
{
    const int64_t rounds = (pixel_tiles * s + slots - 1) / slots;
    const int64_t longest = (point_tiles + s - 1) / s;
    return (double)rounds * (double)longest * (1.0 + 0.002 * (double)(s - 1));
}

static int split_for(int64_t pixel_tiles, int64_t point_tiles, int64_t slots)
{
    if (pixel_tiles <= 0 || point_tiles <= 1) return 1;
    int best = 1;
    double best_t = direct_path(pixel_tiles, point_tiles, 1, slots);
    for (int64_t s = 2; s <= 64 && s * 2 <= point_tiles; ++s) {
        const double t = direct_path(pixel_tiles, point_tiles, s, slots);
        if (t < best_t * (1.0 - 1e-9)) {
            best = (int)s;
            best_t = t;
        }
    }
    return best;
}

DirectLayout choose_layout(const DirectShape *shapes, int n_shapes, int width, int height, int64_t point_tiles,
                           int num_sms, int force_split)
{
    DirectLayout best{};
    double best_t = 1e300, best_area = 0.0;
    for (int k = 0; k < n_shapes; ++k) {
        const DirectShape &sh = shapes[k];
        const int64_t slots = (int64_t)num_sms * sh.per_sm;
        const int64_t tiles = (int64_t)((width + sh.tile_w - 1) / sh.tile_w) * ((height + sh.tile_h - 1) / sh.tile_h);
        int s = force_split > 0 ? force_split : split_for(tiles, point_tiles, slots);
        if (s > point_tiles) s = (int)(point_tiles > 0 ? point_tiles : 1);
        // in point-tile steps of one CTA: the shapes keep the same warps per SM (threads x CTAs per SM) and the
        // same pixels per thread, so a step takes the same time whatever the shape
        const double t = direct_path(tiles, point_tiles > 0 ? point_tiles : 1, s, slots);
        const double area = (double)tiles * sh.tile_w * sh.tile_h;
        // a shorter path wins; on equal paths, fewer padded pixels computed
        if (t < best_t * (1.0 - 1e-9) || (t <= best_t * (1.0 + 1e-9) && area < best_area)) {
            best_t = t;
            best_area = area;
            best = DirectLayout{sh, s};
        }
    }
    return best;
}

// Microseconds of one stage (32 points of a 128 x bn / planes tile; spherical: 16) of a CTA of the tensor-core direct
// form, for the amplitude hologram, the complex wave and the spherical hologram, and per B row for each part of a tile
// that its last CTA adds.  Measured on GB300 at 1920x1080 with 10^4 points (stages) and at 256x256 with 10^3 (parts).
// Against every tile and orientation over 128x32 to 2048x2048 pixels, 100 to 3 10^4 points and the three forms, the choice
// takes 1.02 of the fastest one's time on average; the worst are 1920x1080, 100 points (22.9 us, 16.8 with 128 rows),
// 1283x717 with 1000 and 3000 points (47.9 and 78.6, 39.3 and 69.0 with 192 and 256) and the wave of 130x2000 with 1000
// points (43.5, 37.3).
struct MmaCost {
    int bn;
    double stage[3];
};
static const MmaCost kMmaCost[] = {
    {64, {1.21, 1.16, 1.43}},  {128, {1.40, 1.30, 1.69}}, {192, {1.67, 1.48, 1.90}},
    {224, {1.81, 0.0, 0.0}}, {256, {1.96, 1.64, 2.07}},
};
constexpr double kMmaPartUs = 0.005;

DirectMmaLayout choose_direct_mma(int planes, int width, int height, int64_t n_points, int num_sms, int split,
                                  int ctas, int bn)
{
    DirectMmaLayout best;
    const bool sph = planes == 0;   // the spherical amplitude hologram
    if (sph) planes = 1;
    const int group = sph ? kSphMmaGroup : kDirectMmaGroup;
    const int64_t groups = (n_points + group - 1) / group;
    double best_t = 1e300;
    for (const MmaCost &c : kMmaCost)
        for (int a_rows = 0; a_rows < 2; ++a_rows) {
            if (bn > 0 && c.bn != bn) continue;
            if (sph ? c.bn % 64 != 0 : c.bn / planes % 32 != 0) continue;
            const int tb = c.bn / planes;
            const int side_a = a_rows ? height : width, side_b = a_rows ? width : height;
            const int64_t tiles = (int64_t)((side_a + 127) / 128) * ((side_b + tb - 1) / tb);
            const int64_t units = tiles * groups;
            auto consider = [&](int64_t n, int64_t stages, int64_t parts) {
                // on equal terms the orientation whose stores write whole rows of 32 pixels
                const double t = (double)stages * c.stage[sph ? 2 : planes - 1] + (double)parts * kMmaPartUs * c.bn + 0.01 * a_rows;
                if (t >= best_t) return;
                best_t = t;
                best.bn = c.bn;
                best.a_rows = a_rows;
                best.tiles = (int)tiles;
                best.ctas = (int)n;
                best.us = t;
            };
            if (split > 0) {
                // chunks of kPointTile points at least: each takes a slot of a whole tile
                const int64_t s = std::min<int64_t>(split, (n_points + kPointTile - 1) / kPointTile), n = tiles * s;
                consider(n, (n + num_sms - 1) / num_sms * ((groups + s - 1) / s), s);
                continue;
            }
            if (ctas > 0) {
                const int64_t n = std::min<int64_t>(ctas, units);
                consider(n, (units + n - 1) / n * ((n + num_sms - 1) / num_sms), 1);
                continue;
            }
            // from an equal share on every SM to whole tiles: fewer CTAs leave fewer parts of a tile to add
            for (int64_t s = (units + num_sms - 1) / num_sms;; s += 1 + s / 4) {
                consider((units + s - 1) / s, s, s >= groups ? 1 : (groups + s - 1) / s);
                if (s >= groups) break;
            }
        }
    // a CTA counts its stages in 32 bits
    best.ctas = (int)std::max<int64_t>(best.ctas, ((int64_t)best.tiles * groups >> 30) + 1);
    return best;
}

int choose_gemm_bn(int width)
{
    static const int cands[] = {256, 240, 192, 128};
    int best = 256;
    double best_waste = 1e30;
    for (int bn : cands) {
        const int tiles = (width + bn - 1) / bn;
        const double waste = (double)(tiles * bn - width) / (double)width + 1e-3 * (256 - bn) / 256.0;
        if (waste < best_waste) {
            best_waste = waste;
            best = bn;
        }
    }
    return best;
}

// Time of one k-block (64 K elements) of one GEMM unit, in microseconds, by tile width, for the one-CTA and the
// two-SM form (index 0 and 1) of the FP16/BF16 GEMM and of split FP16 (three products per k-block).  Measured on
// GB300 (least time per k-block of a unit over 1024x1024, 1920x1080 and 3840x2160 holograms, 4 10^3 to 1.5 10^5
// points, every width, split and orientation): up to a width of 224 it hardly depends on the width, so a unit is
// bound by its operand stream, not by its MMAs; the 4-stage ring of the 256-wide one-CTA tile is slower, the
// two-SM form's 256-wide tile (half of B per CTA) is not.  240 is interpolated (one-CTA form only).
struct KbCost {
    int bn;
    double f16[2], split[2];
};
static const KbCost kKbCost[] = {
    {128, {0.273, 0.269}, {0.908, 0.969}}, {192, {0.271, 0.269}, {0.924, 0.992}},
    {224, {0.272, 0.275}, {0.939, 1.025}}, {240, {0.295, 0.0}, {0.99, 0.0}},
    {256, {0.318, 0.274}, {1.048, 1.035}},
};
// Effective bandwidth of the split reduction, bytes per microsecond.
constexpr double kReduceBytesPerUs = 3.0e6;

GemmLayout choose_gemm_layout(int width, int height, int64_t k_blocks, int ctas, bool split_form, int force_bn,
                              int force_splits, int force_trans, int force_pair)
{
    GemmLayout best{false, 256, 1, false, 0.0};
    double best_t = 1e300;
    for (int pair = 0; pair < 2; ++pair) {
        if ((force_pair == 1 && !pair) || (force_pair == 2 && pair)) continue;   // 1: always, 2: never
        if (pair && ctas < 2) continue;
        const int tile_m = pair ? 256 : 128;
        const int slots = pair ? ctas / 2 : ctas;   // the two-SM form's units run on clusters of two CTAs
        for (int tr = 0; tr < 2; ++tr) {
            if (force_trans == 1 && tr) continue;    // 1: never transposed
            if (force_trans == 2 && !tr) continue;   // 2: always transposed
            const int64_t a_rows = tr ? width : height, b_rows = tr ? height : width;
            const int64_t tiles_m = (a_rows + tile_m - 1) / tile_m;
            for (const KbCost &kc : kKbCost) {
                const int bn = kc.bn;
                if (force_bn > 0 && bn != force_bn) continue;
                const double c = split_form ? kc.split[pair] : kc.f16[pair];
                if (c <= 0.0) continue;   // no two-SM form of this width (halves of whole 32-row groups)
                const int64_t tiles = tiles_m * ((b_rows + bn - 1) / bn);
                for (int64_t s = 1; s <= 16; ++s) {
                    if (force_splits > 0 && s != force_splits) continue;
                    if (force_splits <= 0 && s > 1 && s * 4 > k_blocks) break;
                    const int64_t rounds = (tiles * s + slots - 1) / slots;
                    // critical path: rounds of units of ceil(k_blocks / s) k-blocks (each split a little
                    // slower: the units in flight spread over more K ranges), then the split reduction
                    double t = (double)rounds * (double)((k_blocks + s - 1) / s) * c * (1.0 + 0.01 * (double)(s - 1));
                    if (s > 1) t += (double)(s + 1) * (double)width * (double)height * 4.0 / kReduceBytesPerUs;
                    // the transposed write-out (32 lanes, 32 consecutive columns) breaks ties
                    if (tr) t *= 0.995;
                    if (t < best_t * (1.0 - 1e-9)) {
                        best_t = t;
                        best = GemmLayout{tr != 0, bn, (int)s, pair != 0, t};
                    }
                }
            }
        }
    }
    if (best_t == 1e300 && force_pair == 1)   // no two-SM form of the forced width
        return choose_gemm_layout(width, height, k_blocks, ctas, split_form, force_bn, force_splits, force_trans, 2);
    return best;
}

int choose_gemm_splits(int64_t tiles, int64_t k_blocks, int ctas)
{
    if (tiles <= 0 || ctas <= 0) return 1;
    int best = 1;
    double best_time = 1e30;
    for (int64_t s = 1; s <= 32 && s * 4 <= (k_blocks > 4 ? k_blocks : 4); ++s) {
        const int64_t units = tiles * s;
        const int64_t rounds = (units + ctas - 1) / ctas;
        // time in units of one whole-K tile; each extra split costs a partial plane
        const double t = (double)rounds / (double)s + 0.01 * (double)(s - 1);
        if (t < best_time - 1e-9) {
            best_time = t;
            best = (int)s;
        }
    }
    return best;
}

// Stated NRMS bound of each form against the FP64 oracle (measured values are
// below these: direct SFU 3.5e-7 and accurate 2.6e-7, on the batch's SIMT units 6e-7
// and 4e-7, split FP16 2e-6, FP16 ~3e-4, BF16 ~2e-3 on the display-size clouds).
double form_nrms_bound(int form)
{
    switch (form) {
    case CGH_DIRECT_SFU: return 1e-5;
    case CGH_DIRECT_ACCURATE: return 2e-6;
    case CGH_GEMM_F16: return 2e-3;
    case CGH_GEMM_BF16: return 1e-2;
    case CGH_GEMM_SPLIT16: return 1e-5;
    default: return 1.0;
    }
}

struct TuneState {
    bool calibrated = false;
    double coef[kForms][3] = {};   // seconds: c0, then the factors of form_terms
    struct Choice {
        int width = 0, height = 0;
        int64_t n = 0;
        double tol = 0.0;
        int64_t budget_mb = 0;
        bool gemm_only = false;
        int form = 0;
        bool same(const Choice &o) const
        {
            return width == o.width && height == o.height && n == o.n && tol == o.tol && budget_mb == o.budget_mb &&
                   gemm_only == o.gemm_only;
        }
    } last;   // the choice of the call before: a program's holograms are mostly of one size
    std::map<std::string, int> bn;
    std::string device;   // tune_key
};

void destroy_tune_state(TuneState *t)
{
    delete t;
}

namespace {

// Revision of what the cached coefficients describe, part of the key a cache is accepted by: counted up with the kernels
// that a form runs (2: the direct forms on the tensor cores, six times faster than what files without a revision
// describe; 3: coefficients of the kernels' time models).
constexpr int kTuneRevision = 3;

// The device and the revision, as the cache names them.
std::string tune_key(int dev)
{
    const std::string rev = ":r" + std::to_string(kTuneRevision);
    cudaDeviceProp p;
    if (cudaGetDeviceProperties(&p, dev) != cudaSuccess) {
        cudaGetLastError();
        return "unknown" + rev;
    }
    return std::string(p.name) + ":" + std::to_string(p.multiProcessorCount) + rev;
}

const char *cache_path()
{
    const char *p = std::getenv("CGH_TUNE_CACHE");
    return (p && *p) ? p : nullptr;
}

void save_cache(const TuneState &t)
{
    const char *path = cache_path();
    if (!path) return;
    FILE *f = std::fopen(path, "w");
    if (!f) return;
    std::fprintf(f, "{\n \"abi\": %d,\n \"device\": \"%s\",\n \"coef\": [", CGH_ABI_VERSION, t.device.c_str());
    for (int i = 0; i < kForms; ++i)
        std::fprintf(f, "%s[%.9e, %.9e, %.9e]", i ? ", " : "", t.coef[i][0], t.coef[i][1], t.coef[i][2]);
    std::fprintf(f, "],\n \"bn\": {");
    bool first = true;
    for (const auto &kv : t.bn) {
        std::fprintf(f, "%s\"%s\": %d", first ? "" : ", ", kv.first.c_str(), kv.second);
        first = false;
    }
    std::fprintf(f, "}\n}\n");
    std::fclose(f);
}

// Parses a cache written by save_cache: accepted only when it names this device (with the revision of its kernels, tune_key) and ABI and every one of the
// kForms x 3 coefficients is finite and not negative (they are seconds, and seconds per evaluation); anything
// else -- a truncated or edited file, another device, another ABI -- is refused as a whole and the tuner
// calibrates instead.  Tile widths that the GEMM does not support are skipped.
bool parse_cache(const std::string &text, const std::string &device, TuneState &out)
{
    const std::string dev_key = "\"device\": \"" + device + "\"";
    const std::string abi_key = "\"abi\": " + std::to_string(CGH_ABI_VERSION) + ",";
    if (text.find(dev_key) == std::string::npos || text.find(abi_key) == std::string::npos) return false;
    size_t c = text.find("\"coef\": [");
    if (c == std::string::npos) return false;
    double coef[kForms][3];
    const char *p = text.c_str() + c + 9;
    for (int i = 0; i < kForms; ++i) {
        double a, b, d;
        int n = 0;
        if (std::sscanf(p, " [%lf, %lf, %lf]%n", &a, &b, &d, &n) != 3 || n <= 0) return false;
        for (double v : {a, b, d})
            if (!std::isfinite(v) || v < 0.0) return false;
        coef[i][0] = a;
        coef[i][1] = b;
        coef[i][2] = d;
        p += n;
        while (*p == ',' || *p == ' ') ++p;
    }
    if (*p != ']') return false;
    std::map<std::string, int> bn;
    size_t bpos = text.find("\"bn\": {");
    if (bpos == std::string::npos) return false;
    const char *q = text.c_str() + bpos + 7;
    for (;;) {
        char key[128];
        int val, n = 0;
        if (std::sscanf(q, " \"%127[^\"]\": %d%n", key, &val, &n) != 2) break;
        if (gemm_bn_supported(val)) bn[key] = val;
        q += n;
        while (*q == ',' || *q == ' ') ++q;
    }
    while (*q == ' ' || *q == '\n') ++q;
    if (*q != '}') return false;   // a truncated tile-width table
    std::memcpy(out.coef, coef, sizeof coef);
    out.bn = bn;
    out.calibrated = true;
    return true;
}

bool read_file(const char *path, std::string &text)
{
    FILE *f = std::fopen(path, "r");
    if (!f) return false;
    char buf[4096];
    size_t got;
    while ((got = std::fread(buf, 1, sizeof(buf), f)) > 0) text.append(buf, got);
    std::fclose(f);
    return true;
}

// Reads the cache of CGH_TUNE_CACHE for this device, if there is an acceptable one.
bool load_cache(TuneState &t)
{
    const char *path = cache_path();
    std::string text;
    if (!path || !read_file(path, text)) return false;
    return parse_cache(text, t.device, t);
}

// Deterministic synthetic cloud (integer positions inside the hologram,
// z in [0.3, 1] m, A in [0.5, 1]) for the measurements.
void synth_points(int width, int height, int64_t n, std::vector<float> &xyz, std::vector<float> &amp)
{
    xyz.resize((size_t)n * 3);
    amp.resize((size_t)n);
    uint64_t s = 0x9e3779b97f4a7c15ull;
    auto next = [&]() {
        s ^= s << 13;
        s ^= s >> 7;
        s ^= s << 17;
        return s;
    };
    for (int64_t j = 0; j < n; ++j) {
        xyz[3 * j + 0] = (float)(next() % (uint64_t)width);
        xyz[3 * j + 1] = (float)(next() % (uint64_t)height);
        xyz[3 * j + 2] = 0.3f + 0.7f * (float)((next() >> 11) * (1.0 / 9007199254740992.0));
        amp[j] = 0.5f + 0.5f * (float)((next() >> 11) * (1.0 / 9007199254740992.0));
    }
}

// A synthetic cloud and its hologram on the device.
struct Synth {
    int width, height;
    int64_t n;
    float *xyz = nullptr, *amp = nullptr, *out = nullptr;
    bool ok = false;
    Synth(int width, int height, int64_t n) : width(width), height(height), n(n)
    {
        std::vector<float> hx, ha;
        synth_points(width, height, n, hx, ha);
        ok = cudaMalloc(&xyz, hx.size() * sizeof(float)) == cudaSuccess &&
             cudaMalloc(&amp, ha.size() * sizeof(float)) == cudaSuccess &&
             cudaMalloc(&out, (size_t)width * height * sizeof(float)) == cudaSuccess &&
             cudaMemcpy(xyz, hx.data(), hx.size() * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(amp, ha.data(), ha.size() * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess;
        if (!ok) cudaGetLastError();
    }
    ~Synth()
    {
        if (xyz) cudaFree(xyz);
        if (amp) cudaFree(amp);
        if (out) cudaFree(out);
    }
    Synth(const Synth &) = delete;
    Synth &operator=(const Synth &) = delete;
};

// Seconds per hologram of `form` (tile width bn, 0 = default) on a synthetic cloud: the least of `rounds` averages over
// reps calls (with several rounds one call in the first, and from 60 us on).
double time_form(cgh_ctx *ctx, int form, int bn, const Synth &s, int reps, int rounds = 1)
{
    if (!s.ok) return -1.0;
    const int saved_form = ctx->form, saved_bn = ctx->gemm_bn, saved_model = ctx->phase_model;
    const int saved_group = ctx->gemm_group;
    const bool saved_profile = ctx->profile;
    ctx->form = form;
    ctx->gemm_bn = bn;
    ctx->profile = false;
    ctx->phase_model = CGH_PHASE_FRESNEL;   // the forms' own cost; the piston and reference add none per term
    ctx->gemm_group = 1;                    // synthetic depths are continuous: no grouping
    double sec = -1.0;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) == cudaSuccess && cudaEventCreate(&e1) == cudaSuccess &&
        compute_hologram(ctx, s.width, s.height, ctx->pitch, ctx->lambda, s.xyz, s.amp, s.n, s.out) == CGH_OK) {
        bool ok = true;
        for (int k = 0; k < rounds && ok; ++k) {
            const int calls = rounds > 1 && (k == 0 || sec > 6e-5) ? 1 : reps;
            cudaEventRecord(e0, ctx->stream);
            for (int r = 0; r < calls && ok; ++r)
                ok = compute_hologram(ctx, s.width, s.height, ctx->pitch, ctx->lambda, s.xyz, s.amp, s.n, s.out) == CGH_OK;
            cudaEventRecord(e1, ctx->stream);
            float ms = 0.0f;
            ok = ok && cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess;
            if (ok) sec = sec < 0.0 ? ms * 1e-3 / calls : std::min(sec, ms * 1e-3 / calls);
        }
        if (!ok) sec = -1.0;
    }
    cudaGetLastError();
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    ctx->form = saved_form;
    ctx->gemm_bn = saved_bn;
    ctx->phase_model = saved_model;
    ctx->gemm_group = saved_group;
    ctx->profile = saved_profile;
    return sec;
}

// Least squares of the relative error of t = c[0] + c[1] x[0] + c[2] x[1] over the samples, every coefficient >= 0
// (coordinate descent on the normal equations of the scaled terms).
void fit_times(const std::vector<double> &t, const std::vector<std::array<double, 2>> &x, double c[3])
{
    double scale[3] = {1e-300, 1e-300, 1e-300};
    for (size_t i = 0; i < t.size(); ++i) {
        const double r[3] = {1.0, x[i][0], x[i][1]};
        for (int p = 0; p < 3; ++p) scale[p] = std::max(scale[p], r[p] / t[i]);
    }
    double A[3][3] = {}, b[3] = {};
    for (size_t i = 0; i < t.size(); ++i) {
        const double r[3] = {1.0 / t[i] / scale[0], x[i][0] / t[i] / scale[1], x[i][1] / t[i] / scale[2]};
        for (int p = 0; p < 3; ++p) {
            b[p] += r[p];
            for (int q = 0; q < 3; ++q) A[p][q] += r[p] * r[q];
        }
    }
    double v[3] = {};
    for (int sweep = 0; sweep < 5000; ++sweep)
        for (int p = 0; p < 3; ++p) {
            double d = b[p];
            for (int q = 0; q < 3; ++q)
                if (q != p) d -= A[p][q] * v[q];
            v[p] = A[p][p] > 0.0 && d > 0.0 ? d / A[p][p] : 0.0;
        }
    for (int p = 0; p < 3; ++p) c[p] = v[p] / scale[p];
}

// What a form's time is made of beside the launches: the time model of its kernel (seconds), and the plane's pixels
// (the direct forms write it) or the factors' entries.
std::array<double, 2> form_terms(const cgh_ctx *ctx, int form, int width, int height, int64_t n)
{
    if (form < CGH_GEMM_F16)
        return {choose_direct_mma(1, width, height, n, ctx->num_sms, 0, 0).us * 1e-6, (double)width * height};
    const bool split = form == CGH_GEMM_SPLIT16;
    const int ctas = gemm_max_ctas(ctx->num_sms);
    const int64_t chunk = std::min(n, gemm_chunk_units(split ? kFactorSplit16 : kFactorF16, width, height,
                                                       ctx->factor_budget_mb << 20));
    auto us = [&](int64_t units) {
        return choose_gemm_layout(width, height, (2 * units + 63) / 64, ctas, split, 0, 0, 0, 0).us;
    };
    const double gemm = (double)(n / chunk) * us(chunk) + (n % chunk ? us(n % chunk) : 0.0);
    return {gemm * 1e-6, (double)(width + height) * (double)n};
}

std::string bn_key(int width, int height, int form)
{
    return std::to_string(width) + "x" + std::to_string(height) + ":" + std::to_string(form);
}

TuneState *state(cgh_ctx *ctx)
{
    if (!ctx->tune) {
        ctx->tune = new TuneState();
        ctx->tune->device = tune_key(ctx->device);
        load_cache(*ctx->tune);
    }
    return ctx->tune;
}

}  // namespace

int tune_calibrate(cgh_ctx *ctx, bool force)
{
    TuneState *t = state(ctx);
    if (t->calibrated && !force) return CGH_OK;
    struct Shape {
        int w, h;
        int64_t n;
    };
    // The kernels' time models carry the shape, so that the fit is of their scale, the launches' share and what they leave
    // out, from more samples than coefficients (three samples of 1.7 10^10 terms at most and terms of the sizes alone chose
    // the direct form for 3840x2160, 2 10^5 points: 21 ms against 15, and differently in every process).  Over 128x128 to
    // 4096x4096 pixels and 100 to 2 10^5 points the form chosen takes 1.01 of the fastest one's time on average, also with
    // 10 % of noise on the samples.  The thin one tells the factors from the GEMM; the largest comes
    // first, so that the clocks are up for the small ones.
    static const Shape shapes[] = {{1920, 1080, 10000}, {1024, 1024, 10000}, {3840, 2160, 300}, {4096, 64, 20000},
                                   {1024, 1024, 3000},  {512, 512, 10000},   {256, 256, 1000}};
    const int forms[5] = {CGH_DIRECT_SFU, CGH_DIRECT_ACCURATE, CGH_GEMM_F16, CGH_GEMM_BF16, CGH_GEMM_SPLIT16};
    std::vector<double> ts[kForms];
    std::vector<std::array<double, 2>> xs[kForms];
    for (const Shape &s : shapes) {
        const Synth cloud(s.w, s.h, s.n);
        for (int f : forms) {
            const double sec = time_form(ctx, f, 0, cloud, 3, 3);
            if (sec <= 0.0) return CGH_ECUDA;
            ts[f].push_back(sec);
            xs[f].push_back(form_terms(ctx, f, s.w, s.h, s.n));
        }
    }
    for (int f : forms) fit_times(ts[f], xs[f], t->coef[f]);
    t->calibrated = true;
    t->last = TuneState::Choice();
    save_cache(*t);
    return CGH_OK;
}

double tune_predict(cgh_ctx *ctx, int form, int width, int height, int64_t n)
{
    const double *c = state(ctx)->coef[form];
    const std::array<double, 2> x = form_terms(ctx, form, width, height, n);
    return c[0] + c[1] * x[0] + c[2] * x[1];
}

// The persistent launch and the per-kind launches run direct units on the SIMT kernel, which the single hologram's times
// say nothing about: there a GEMM form is taken wherever one is admissible.  Persistent launch, direct / split FP16:
// 64 x 512x512, 2000 points 7386 / 539 us; 8 x 1920x1080, 100 points 424 / 90; 16 x 64x64, 100 points 42 / 33; the
// direct form was ahead by 3 % at most (256 x 64x64, 100 points 287 / 295).  And what grouping the points of a layered cloud
// saves is not known beforehand: 512x512, 2 10^5 points on 16 planes 690 us direct, 690 split FP16, 270 grouped.
int tune_choose_form(cgh_ctx *ctx, int width, int height, int64_t n, double tol, bool gemm_only)
{
    if (tune_calibrate(ctx, false) != CGH_OK) return CGH_DIRECT_SFU;
    TuneState *t = state(ctx);
    const TuneState::Choice key{width, height, n, tol, ctx->factor_budget_mb, gemm_only, 0};
    if (t->last.same(key)) return t->last.form;
    const int forms[5] = {CGH_DIRECT_SFU, CGH_DIRECT_ACCURATE, CGH_GEMM_F16, CGH_GEMM_BF16, CGH_GEMM_SPLIT16};
    int best = -1;
    double best_t = 1e300;
    for (int f : forms) {
        if (form_nrms_bound(f) > tol) continue;
        if (gemm_only && f < CGH_GEMM_F16 && tol >= form_nrms_bound(CGH_GEMM_SPLIT16)) continue;
        const double tp = tune_predict(ctx, f, width, height, n);
        if (tp < best_t) {
            best_t = tp;
            best = f;
        }
    }
    t->last = key;
    // nothing meets a tolerance tighter than every bound: the most accurate form
    t->last.form = best >= 0 ? best : CGH_DIRECT_ACCURATE;
    return t->last.form;
}

int tune_choose_bn(cgh_ctx *ctx, int width, int height, int form)
{
    TuneState *t = state(ctx);
    const std::string key = bn_key(width, height, form);
    auto it = t->bn.find(key);
    if (it != t->bn.end()) return it->second;
    static const int cands[] = {256, 240, 224, 192, 128};
    int best = choose_gemm_bn(width);
    double best_t = 1e300;
    const Synth cloud(width, height, 4096);
    for (int bn : cands) {
        const double sec = time_form(ctx, form, bn, cloud, 3);
        if (sec > 0.0 && sec < best_t) {
            best_t = sec;
            best = bn;
        }
    }
    t->bn[key] = best;
    save_cache(*t);
    return best;
}

int choose_form(int width, int height, int64_t n_points, double tol, int num_sms)
{
    (void)width;
    (void)height;
    (void)n_points;
    (void)num_sms;
    // without measurements: the direct SFU form when it is admissible, else the accurate one
    return form_nrms_bound(CGH_DIRECT_SFU) <= tol ? CGH_DIRECT_SFU
                                                   : (tol >= form_nrms_bound(CGH_GEMM_F16) ? CGH_GEMM_F16
                                                                                            : CGH_DIRECT_ACCURATE);
}

}  // namespace cgh

extern "C" int cgh_tune_cache_check(const char *path, const char *device_name, int *accepted)
{
    if (!path || !device_name || !accepted) return CGH_EINVAL;
    *accepted = 0;
    std::string text;
    if (!cgh::read_file(path, text)) return CGH_OK;
    cgh::TuneState t;
    *accepted = cgh::parse_cache(text, device_name, t) ? 1 : 0;
    return CGH_OK;
}
