// SLIC segmentation (the step before the method's Section III-A): the view
// records and the launch entry of k_slic.cu, kept apart from the hot path's
// declarations.
#pragma once
#include "lfd_internal.cuh"

namespace lfd {

// one view of a SLIC segmentation
struct SlicView {
    int W, H, GW, GH, fmt;
    int stride;                      // entries of `lab` per cell (the largest cell, rounded up to 4)
    long long pitch;                 // bytes per image row
    const void *img;
    float4 *lab;                     // [GW*GH][stride] CIELAB and position of a cell's pixels (scratch)
    long long *sums;                 // [GW*GH][9][6] sums of a cell's pixels per centre of its 3x3 cells (scratch)
    int *labels;                     // [W*H] output
    float *centres, *centres2;       // [GW*GH][5] {L, a, b, x, y} (scratch, ping-pong)
};

// up to SLIC_BATCH views segmented by the same launches (blockIdx.y = view)
constexpr int SLIC_BATCH = 16;
// Scratch of the views that go through the same launches.  A cell takes 432
// bytes of sums, and 16 for each pixel of the largest cell: 41 bytes a pixel
// for 5 x 5 cells, up to 540 for cells of one.  A group of this size is far
// more work than the chip runs at once, so splitting there costs nothing.
constexpr size_t SLIC_SCRATCH = (size_t)2 << 30;
struct SlicBatch {
    SlicView v[SLIC_BATCH];
    float wxy[SLIC_BATCH];                // (m / S)^2 of each view
    int n, max_px, max_cells, max_stride;
};

cudaError_t launch_slic(const SlicBatch &b, const float *const *centres_in, int iterations,
                        float *const *centres_out, cudaStream_t st);

}  // namespace lfd
