// Depth fusion (Section III-D): the launch entries of k_fuse.cu, kept apart
// from the hot path's declarations.
#pragma once
#include "lfd_internal.cuh"

namespace lfd {

// z-buffers of one group of reference views (at least one reference per
// group).  Large groups project a source pixel into more references per depth
// and launch: 9 views of 1280x720 (265 MB in one group) take 383 us with 64 MB
// groups, 324 with 96, 289 with 160, 248 in one.  The bound keeps the
// workspace of large light fields (16 x 1080p: 2 GB) small.
constexpr size_t FUSE_GROUP_BYTES = (size_t)512 << 20;
constexpr int FUSE_MAX_GROUP = 32;       // references per group

// sets bytes (a multiple of 16) of z-buffer to +inf
cudaError_t launch_fuse_clear(unsigned *zbuf, size_t bytes, cudaStream_t st);
// fuses reference views first .. first + count; a.zoff[r]: word offset of
// reference r's planes within its group.  The planes are +inf before and after.
cudaError_t launch_fuse_group(const FuseArgs &a, int first, int count, int max_w, int max_h, int max_px,
                              cudaStream_t st);

}  // namespace lfd
