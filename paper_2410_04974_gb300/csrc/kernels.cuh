// Kernel argument blocks and host launchers of the sixdgs library.
#pragma once

#include "common.cuh"

namespace sixdgs {

// Launch of a kernel that begins with after_previous() (common.cuh).  Outside
// stream capture it may be set up while the kernel before it in the stream
// ends, which hides most of the gap between two small kernels: 59 -> 43 us for
// the seven kernels of a 4,096-Gaussian training step, 67 -> 52 us for the six
// (now seven) of a 6,660-Gaussian frame, 964 -> 945 us at 300k / 8 x 800^2.  A captured
// graph keeps the plain dependency: it hides the gaps itself (no difference
// measured).
template <typename... Params, typename... Args>
cudaError_t launch_after(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, int cluster,
                         cudaStream_t stream, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2] = {};
  cfg.attrs = attr;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(stream, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = (unsigned)cluster;
    attr[cfg.numAttrs].val.clusterDim.y = attr[cfg.numAttrs].val.clusterDim.z = 1;
    ++cfg.numAttrs;
  }
  return cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}

// Counters of one tile, a 32-byte sector of their own: the tiles of a scene's
// silhouette take most of the atomics, and packed counters put them on a few
// L2 slices.
struct __align__(32) TileCounters {
  uint32_t count;    // duplicates, counted by the projection
  uint32_t cursor;   // next free place of the tile's list
  uint32_t pad[6];
};

// Division of a frame's views among the projection's CTAs (bin.cuh).
struct ViewParts {
  uint32_t parts, views;
};

struct ProjectArgs {
  const CamRec* cams;
  int32_t n_cams;
  int64_t n;
  int32_t sh_degree;
  float lambda_opa;
  float inv_tile_w, inv_tile_h;
  int32_t alpha_footprint;   // 1: tile rect within the alpha >= 1/255 box
  const float* mu_p;
  const float* mu_d;
  const float* l_raw;
  const float* opacity_logit;
  const float* sh;
  const float* lambda_raw;   // optional per-Gaussian lambda_opa (pre-sigmoid)
  const float* cond_cache;   // optional cached view-independent state
  PairRec* rec;
  uint32_t* ntiles;
  ushort4* rect;
  uint32_t* depth_key;
  uint4* vis;             // visible queue of the binning (bin.cuh)
  uint32_t* vis_count;
  ViewParts views;        // set by the launch
  bool banded;            // leaves all rectangles to bin_count_kernel
  bool defer_big;         // leaves those of many tiles
  TileCounters* tile;     // their counts are added to
  float* grad_rec;   // zeroed for every visible pair (read by the backward); null: inference plan
  int32_t bulk;      // 1: every parameter plane segment can be staged with bulk copies
  int64_t spin_budget;
  int32_t* status;
};

// Words of the binning's state section (uint32).
enum BinWord {
  kBinClass = 0,         // tiles of every list-length class
  kBinCursor = 64,       // next place of every class in the tile order
  kBinTicket = 128,      // blocks of the list scan that have started (scan_tickets)
  kBinQueue = 129,       // sort work counter
  kBinOver = 130,        // tiles with lists above 16384, 4096, 2048, 1024, 512 and 0 entries
  kBinBase = 136,        // duplicates of the bands so far, two 64-bit words used in turn
  kBinWords = 192
};
constexpr int kBinLevels = 5;   // 16384, 4096, 2048, 1024, 512 entries: what a CTA and its teams sort

// Per-tile lists from the projection's tile counts and visible queue.  A frame
// whose tile state does not fit its workspace is taken in bands of consecutive
// tiles, one after the other (render_banded); any other is one band.
struct BinArgs {
  const CamRec* cams;
  int32_t n_cams;
  uint32_t n;                      // Gaussians per camera
  uint32_t tile_first;             // first tile of the band
  uint32_t total_tiles;            // tiles of the band
  int32_t band;                    // its number; -1: the frame is one band
  TileCounters* tile;
  const uint4* vis;                // visible queue (bin.cuh)
  const uint32_t* vis_count;
  uint32_t segments;               // of the queue
  uint32_t segment_size;           // entries that one can hold
  ViewParts views;
  bool scan_tickets;               // set by the launch: blocks of the scan number themselves
  // set by the launch: CTAs that share the segments, CTAs of one segment, entries of a step
  uint32_t scatter_grid, scatter_split, scatter_step;
  uint32_t* state;                 // kBinWords words
  unsigned long long* scan_state;  // one word per scan block
  uint4* order;                    // TileWork of every tile, longest list class first
  uint2* ranges;
  uint64_t capacity;
  uint64_t* dup;                   // (depth, pair) of every duplicate, grouped by tile
  uint32_t* sorted;                // pair index, by (tile, depth, pair)
  uint32_t* sorted_key;            // global tile id of the same
  uint32_t* counts;                // the public counts section
  int64_t spin_budget;
  int32_t* status;
};

struct BlendArgs {
  const CamRec* cams;
  int32_t n_cams;
  int32_t tile_w, tile_h, batch;
  int32_t short_list;       // set by the launch: lists up to this long are staged by every warp for itself
  const PairRec* rec;
  uint32_t n_pairs;
  const uint32_t* sorted;   // pair index per list entry
  const uint4* order;       // TileWork of every tile, longest lists first
  const uint32_t* n_busy;   // tiles with a list (the others come last)
  float bg[3];
  float* images;
  const float* targets;
  float* grad_images;
  double* loss;
  float inv_count;          // 1 / (3 * total_pixels)
  uint32_t* nwalk;          // optional per-pixel walk length
  unsigned long long* pair_counts;  // optional: evaluated, compositing pairs
  // backward
  const float* images_in;
  const float* grad_in;
  float* grad_rec;          // n_pairs x 12
  int32_t recompute;        // 1: re-derive the stop; 0: use nwalk
  // persistent mode: tiles are taken from this counter (NULL: one CTA per tile)
  uint32_t* tile_queue;
  uint32_t total_tiles;     // of the band (BinArgs)
  uint32_t frame_tiles;     // of the frame
};

struct ProjectBwdArgs {
  const CamRec* cams;
  int32_t n_cams;
  int64_t n;
  int32_t sh_degree;
  float lambda_opa;
  const float* mu_p;
  const float* mu_d;
  const float* l_raw;
  const float* opacity_logit;
  const float* sh;
  const float* lambda_raw;
  const PairRec* rec;
  const uint32_t* ntiles;
  const float* grad_rec;
  float* grad_mu_p;
  float* grad_mu_d;
  float* grad_l_raw;
  float* grad_opacity_logit;
  float* grad_sh;
  float* grad_lambda_raw;
  int32_t accumulate;   // 1: add into the outputs instead of overwriting
  int32_t bulk;         // 1: the parameter planes can be staged with bulk copies
  int64_t spin_budget;
  int32_t* status;
};

struct CondCacheArgs {
  int64_t n;
  const float* l_raw;
  const float* opacity_logit;
  float* cache;      // kCondCachePlanes planes of n floats
};

constexpr int kCondCachePlanes = 25;

struct ScaleRotationArgs {
  int64_t n;
  const float* l_raw;
  float* rotation;   // 9 planes, R row-major
  float* scale;      // 3 planes
  int32_t* status;
};

void launch_project_fwd(ProjectArgs a, cudaStream_t stream);
cudaError_t launch_bin_count(BinArgs a, int sms, cudaStream_t stream);
void launch_scale_rotation(const ScaleRotationArgs& a, cudaStream_t stream);
void launch_cond_cache(const CondCacheArgs& a, cudaStream_t stream);
void launch_peak_probe(int kind, int64_t iters, float* out, int blocks, cudaStream_t stream);
cudaError_t launch_bin(BinArgs a, int sms, cudaStream_t stream);
void launch_blend_fwd(const BlendArgs& a, int64_t total_tiles, cudaStream_t stream);
void launch_blend_fused(const BlendArgs& a, int64_t total_tiles, cudaStream_t stream);
void launch_blend_bwd(const BlendArgs& a, int64_t total_tiles, cudaStream_t stream);
void launch_param_bwd(const ProjectBwdArgs& a, cudaStream_t stream);

// Tiles per block of the list scan.
constexpr int kScanTile = 256;

// A forward frame in bands of tiles, in a workspace whose tile state holds one
// band (api.cu).  plan_bands lays the plan out for at most ws_bytes and returns
// the tiles of a band, 0 if not even one block of the scan fits.  render_banded
// projects once, then counts, bins and blends every band; the duplicates of all
// bands share the capacity, and the images are those of the frame as a whole.
int64_t plan_bands(sixdgs_plan* plan, int64_t ws_bytes);
sixdgs_status render_banded(const sixdgs_plan* plan, int64_t band_tiles, const sixdgs_scene* scene,
                            const sixdgs_camera* cams, void* ws, size_t ws_bytes, float* images_dev,
                            int32_t* status_dev, sixdgs_stream_t stream);

}  // namespace sixdgs
