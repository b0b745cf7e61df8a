// gpfc_detrend.h -- launch parameters of the pre-processing kernels (detrend.cu).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace gpfc {

constexpr int kDetrendMaxSpacings = 8;

struct DetrendParams {
    const double *t;        // [n] sorted times
    const float *f;         // [n] flux
    const uint8_t *mask;    // [n] known transits (nonzero: never used in a fit), or NULL
    int64_t n;
    double time_gap, flux_gap_sigma, clip_sigma, ridge;
    int edge, max_iter, n_sp;
    double sp[kDetrendMaxSpacings];
    int blocks;             // blocks of the moment and segment-start passes
    // workspace (context-owned)
    double *partial;        // [2 * blocks]
    int64_t *blk_count;     // [blocks]
    int64_t *blk_off;       // [blocks + 1]
    int64_t *n_seg;         // [1]
    int64_t *seg_start;     // [n + 1]
    int64_t *seg_keep;      // [n]
    int64_t *seg_off;       // [n]
    // one copy per candidate spacing of a group, [group][n]: a point's four B-splines and its knot
    // interval, the first point of each interval [n + 1], and per interval or coefficient (at its
    // segment's points) the reciprocal knot differences [6], in whose place come the banded matrix
    // [4] and its factor [4], then the segment's BIC and the fit; right side and solution
    int sp0, group;
    double4 *basis;
    int32_t *interval, *first;
    double *band, *rhs, *coef;
    uint8_t *used, *used2;
    double *best[2];        // [n]: smallest BIC of the segments so far, in turn (one group: NULL)
    float *det;             // [n]
    // outputs (caller-owned, device)
    double *t_out;
    float *f_out;
    int32_t *seg_out;       // or NULL
    int64_t *n_out;         // [1]
};

// Scratch of the spacings fitted at the same time: bytes per point of each, and their sum where more
// than one is.
constexpr size_t kDtPointBytes = 122, kDtScratch = (size_t)1 << 30;

cudaError_t launch_detrend(const DetrendParams &p, int num_sms, cudaStream_t st);

}  // namespace gpfc
