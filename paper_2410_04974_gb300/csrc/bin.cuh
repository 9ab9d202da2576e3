// The visible queue between the projection and the binning.
#pragma once

#include "common.cuh"
#include "kernels.cuh"
#include "stage.cuh"

namespace sixdgs {

// Every projection CTA queues the visible pairs of its kStageTile Gaussians and
// its views at a place of its own, so that the queue needs no global counter.
// Segment s belongs to Gaussian tile s / parts and to the views from
// (s % parts) * views on; vis_count[s] is its number of entries.
//
// A CTA takes all views of its Gaussians, as it reads their parameters once,
// unless that leaves SMs without one: then the views are divided, down to two
// a CTA, until there are about four CTAs per SM.  6,660 Gaussians at 1408^2 (53
// tiles of Gaussians, cold caches): the projection of 20 views 75 -> 31 us, of 4
// views 36 -> 24 us; 17,133 at 1024^2, 20 views: 57 -> 42 us.
constexpr int kProjFill = 608;   // CTAs
__host__ __device__ inline ViewParts view_parts(int64_t n, int n_cams) {
  const int64_t tiles = (n + kStageTile - 1) / kStageTile;
  int64_t parts = tiles > 0 ? kProjFill / tiles : 1;
  parts = parts < n_cams / 2 ? parts : n_cams / 2;
  if (parts < 1) parts = 1;
  const int64_t views = (n_cams + parts - 1) / parts;
  return {(uint32_t)((n_cams + views - 1) / views), (uint32_t)views};
}
// Words of vis_count.
__host__ __device__ inline int64_t vis_segments_max(int64_t n) { return (n + kStageTile - 1) / kStageTile + kProjFill; }
// First entry of segment s.
__host__ __device__ inline int64_t vis_base(int64_t s, int64_t n, int n_cams, ViewParts vp) {
  const int64_t g0 = s / vp.parts * kStageTile, m = n - g0 < kStageTile ? n - g0 : (int64_t)kStageTile;
  return g0 * n_cams + m * (s % vp.parts * vp.views);
}

// A visible pair in the queue (16 bytes): the pair index, the depth bits and
// the tile rectangle; an empty rectangle for a pair that turned out to touch
// no tile.
__device__ __forceinline__ uint4 vis_entry(uint32_t pair, uint32_t depth, uint32_t x0, uint32_t x1, uint32_t y0,
                                           uint32_t y1) {
  return make_uint4(pair, depth, x0 | (x1 << 16), y0 | (y1 << 16));
}

// Rectangles of more tiles than this are not counted by one thread of the
// projection: by its CTA together, a warp each, or, in a frame whose projection
// leaves most of the chip idle and whose rectangles can be large, by
// bin_count_kernel, which divides them as the scatter does (projection and
// binning together, with the scatter's finer division: 1,000 Gaussians of 5,600
// tiles at 1408^2 1267 -> 164 us, 20,000 of 1,700 at 1920x1080 786 -> 507 us,
// 2,000 of 350 at 4096^2 154 -> 89 us; the frame of 6,660 of 30 at 1408^2 52 -> 48 us).
constexpr uint32_t kBigRect = 16;
__host__ __device__ inline bool defer_big_rects(int64_t n, int n_cams, int64_t total_tiles) {
  return (n + kStageTile - 1) / kStageTile * view_parts(n, n_cams).parts < kProjFill / 2 && total_tiles > 1024 * (int64_t)n_cams;
}

// How the scatter (and the count of large rectangles) divides the visible queue:
// a CTA takes `step` entries of a segment at a time, `split` CTAs share a
// segment's steps in turn.
struct ScatterShare {
  uint32_t grid, split, step;
};
constexpr uint32_t kScatterEntries = 256;   // entries of a step at the most, two a thread
__host__ __device__ inline ScatterShare scatter_share(uint32_t segments, uint32_t segment_size, uint32_t total_tiles,
                                                      int sms) {
  // 16 CTAs per SM: with fewer segments, several CTAs take the steps of one in
  // turn (the binning of 20 views of 6,660 Gaussians at 1408^2, 1.1 M duplicates
  // in 53 segments before: 152 -> 78 us; of 4 views 43 -> 29 us, with the
  // projection's division of the views); a frame of fewer pairs than CTAs gives
  // every CTA one, which may have tens of thousands of tiles (count and binning of
  // 1,000 Gaussians of 22,000 tiles of 8x8 pixels at 1408^2 517 -> 346 us against
  // two a CTA, of 5,600 of 16x16 166 -> 124)
  const uint32_t most_ctas = (uint32_t)sms * 16u;
  // a step's duplicates are counted in 32 bits: at most 2^31 of them
  uint32_t most_step = total_tiles ? (1u << 31) / total_tiles : kScatterEntries;
  if (most_step > kScatterEntries) most_step = kScatterEntries;
  if (most_step < 1u) most_step = 1u;
  ScatterShare s = {0u, 1u, most_step};
  if (segments && 2u * segments <= most_ctas) {
    const uint32_t share = (segment_size * segments + most_ctas - 1) / most_ctas;
    const uint32_t step = share > 1u ? (share + 1u) & ~1u : 1u;
    if (step < s.step) s.step = step;
    const uint32_t steps = (segment_size + s.step - 1) / s.step, ctas = most_ctas / segments;
    s.split = ctas < steps ? ctas : steps;
  }
  s.grid = segments * s.split < most_ctas ? segments * s.split : most_ctas;
  return s;
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
