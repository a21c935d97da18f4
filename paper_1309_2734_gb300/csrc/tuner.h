// Launch-shape selection and the measured autotuner (host side).
#pragma once

#include <cstdint>

#include "kernels.h"

struct cgh_ctx;

namespace cgh {

// A kernel's CTA shape among n_shapes (each with its threads and CTAs per SM) and its point split: the shortest
// critical path, rounds of (pixel tiles x chunks) over the resident CTAs times the longest chunk, then the least
// padding; force_split > 0 pins the split.
struct DirectLayout {
    DirectShape shape;
    int split;
};
DirectLayout choose_layout(const DirectShape *shapes, int n_shapes, int width, int height, int64_t point_tiles,
                           int num_sms, int force_split);

// The tile and the CTAs of the direct form on the tensor cores (direct_mma.cu) with the shortest predicted time.
// planes = 2: the complex wave, 0: the amplitude hologram of the spherical model.  split > 0: that many equal chunks of the points per tile; ctas > 0: that many CTAs; bn > 0:
// that tile.
DirectMmaLayout choose_direct_mma(int planes, int width, int height, int64_t n_points, int num_sms, int split,
                                  int ctas, int bn = 0);

// GEMM orientation, tile width, K splits and form (one CTA per 128-row tile, or the two-SM form: clusters of two
// CTAs on 256-row tiles) with the shortest predicted time: rounds of units over the ctas CTAs (ctas / 2 clusters)
// times a unit's k-blocks times the measured time of one k-block at that width and form, plus the split
// reduction.  force_* > 0 pin a choice (force_trans: 1 = never transposed, 2 = always; force_pair: 1 = always
// the two-SM form, 2 = never).
struct GemmLayout {
    bool trans;
    int bn;
    int splits;
    bool pair;
    double us;   // predicted time
};
GemmLayout choose_gemm_layout(int width, int height, int64_t k_blocks, int ctas, bool split_form, int force_bn,
                              int force_splits, int force_trans, int force_pair);

// Points (K units) per factor chunk when one chunk's P and Q may take budget bytes (mode: a factor mode).
int64_t gemm_chunk_units(int mode, int width, int height, int64_t budget);

// GEMM tile width (columns of the hologram per tile) with the least padding.
int choose_gemm_bn(int width);

// K splits of the GEMM so that (tiles x splits) units balance over ctas
// persistent CTAs; each split keeps at least 4 k-blocks of 64.
int choose_gemm_splits(int64_t tiles, int64_t k_blocks, int ctas);

// Stated NRMS bound of a form against the FP64 oracle.
double form_nrms_bound(int form);

// Form without measurements (static rule).
int choose_form(int width, int height, int64_t n_points, double tol, int num_sms);

// Measured: calibrate the per-form time model on this device (once; cached).
int tune_calibrate(cgh_ctx *ctx, bool force);
// Predicted seconds per hologram of a form.
double tune_predict(cgh_ctx *ctx, int form, int width, int height, int64_t n);
// Fastest admissible form by the calibrated model.  gemm_only: a GEMM form where one is admissible -- the batch's own
// launches, whose direct units are the SIMT kernel's, and clouds whose points the GEMM forms may group.
int tune_choose_form(cgh_ctx *ctx, int width, int height, int64_t n, double tol, bool gemm_only);
// Fastest GEMM tile width for a shape and form, timed on that shape.
int tune_choose_bn(cgh_ctx *ctx, int width, int height, int form);

}  // namespace cgh
