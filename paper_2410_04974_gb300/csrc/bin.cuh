// The visible queue between the projection and the binning.
#pragma once

#include "common.cuh"

namespace sixdgs {

// Every projection CTA queues the visible pairs of its kStageTile Gaussians at
// a place of its own, so that the queue needs no global counter: entry i of
// segment b is vis[b * kStageTile * n_cams + i], vis_count[b] their number.
//
// A visible pair in the queue (16 bytes): the pair index, the depth bits and
// the tile rectangle; an empty rectangle for a pair that turned out to touch
// no tile.
__device__ __forceinline__ uint4 vis_entry(uint32_t pair, uint32_t depth, uint32_t x0, uint32_t x1, uint32_t y0,
                                           uint32_t y1) {
  return make_uint4(pair, depth, x0 | (x1 << 16), y0 | (y1 << 16));
}

// row = local / w for the small integers of a tile rectangle: a float
// estimate corrected to the exact quotient.
// (64-bit, so that the correction terminates for any 32-bit input; w >= 1).
__device__ __forceinline__ uint32_t rect_row(uint32_t local, uint32_t w) {
  uint64_t row = (uint64_t)__fdividef((float)local, (float)w);
  while (row > 0u && row * w > local) --row;
  while ((row + 1u) * w <= local) ++row;
  return (uint32_t)row;
}

}  // namespace sixdgs
