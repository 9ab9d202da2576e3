// C ABI of the sixdgs library: plan and workspace layout, argument checks
// and the launch sequence of each stage (declared in include/sixdgs.h).
#include <cstring>
#include <initializer_list>

#include "bin.cuh"
#include "common.cuh"
#include "kernels.cuh"
#include "stage.cuh"

using namespace sixdgs;

namespace {

// Internal workspace sections (after the public ones of sixdgs.h).
enum {
  WS_ZERO = 11,        // start of the region condition_project clears
  WS_STATE = 12,       // words of the binning (kernels.cuh, BinWord)
  WS_SCAN = 13,        // look-back words of the list scan
  WS_TILE = 14,        // counters of every tile
  WS_ZERO_END = 15,
  WS_COUNTERS = 16,    // word 32: persistent blend queue
  WS_ORDER = 18,       // TileWork of every tile, longest lists first
  WS_VIS = 19,         // visible queue of the projection (16 bytes an entry)
  WS_DUP = 20,         // (depth, pair) of every duplicate, grouped by tile
  WS_SORT_K = 21,      // SIXDGS_WS_SORTEDKEY
  WS_SORT_V = 22,      // SIXDGS_WS_SORTED
  WS_VIS_COUNT = 23    // entries of every segment of the visible queue
};

constexpr int kMaxCams = 256;

int64_t align_up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

int sm_count() {
  static int cached[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  if (!cached[dev]) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 148;
    cached[dev] = v;
  }
  return cached[dev];
}

template <int kCams>
struct CamUpload {
  CamRec cams[kCams];
  int32_t first, count;
};

// Camera records from the kernel parameters, and the words that the
// projection and the binning count in set to zero (zero_quads 16-byte words;
// grid-stride), and *loss unless it is null.
template <int kCams>
__global__ void upload_cams_kernel(const __grid_constant__ CamUpload<kCams> up, CamRec* dst, uint4* zero,
                                   int64_t zero_quads, double* loss) {
  after_previous();
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i0 < up.count) dst[up.first + i0] = up.cams[i0];
  if (i0 == 0 && loss) *loss = 0.0;
  for (int64_t i = i0; i < zero_quads; i += (int64_t)gridDim.x * blockDim.x) zero[i] = make_uint4(0u, 0u, 0u, 0u);
}

// One launch per kCams cameras; the first also clears.
template <int kCams, typename Make>
void upload_cams(int n_cams, Make make, CamRec* dst, void* zero, int64_t zero_bytes, double* loss, int sms,
                 cudaStream_t stream) {
  for (int first = 0; first < n_cams; first += kCams) {
    CamUpload<kCams> up;
    std::memset(&up, 0, sizeof(up));
    up.first = first;
    up.count = std::min(kCams, n_cams - first);
    for (int i = 0; i < up.count; ++i) up.cams[i] = make(first + i);
    const int64_t quads = first == 0 ? zero_bytes / 16 : 0;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((quads + 1023) / 1024, 2 * sms));
    launch_after(upload_cams_kernel<kCams>, grid, 256, 0, 1, stream, up, dst, static_cast<uint4*>(zero), quads,
                 first == 0 ? loss : nullptr);
  }
}

CamRec make_cam_rec(const sixdgs_camera& c, const sixdgs_settings& st, int32_t tile_offset,
                    int64_t pixel_base) {
  CamRec r;
  std::memset(&r, 0, sizeof(r));
  for (int i = 0; i < 3; ++i) {
    for (int j = 0; j < 3; ++j) r.r[i * 3 + j] = c.world_to_cam[i * 4 + j];
    r.t[i] = c.world_to_cam[i * 4 + 3];
    r.campos[i] = c.campos[i];
  }
  r.fx = c.fx;
  r.fy = c.fy;
  r.cx = c.cx;
  r.cy = c.cy;
  r.znear = c.znear;
  r.limx = kFrustumGuard * (0.5f * (float)c.width) / c.fx;
  r.limy = kFrustumGuard * (0.5f * (float)c.height) / c.fy;
  r.width = c.width;
  r.height = c.height;
  r.tiles_x = (c.width + st.tile_w - 1) / st.tile_w;
  r.tiles_y = (c.height + st.tile_h - 1) / st.tile_h;
  r.tile_offset = tile_offset;
  r.pixel_base = pixel_base;
  return r;
}

template <typename T>
T* ws_ptr(void* ws, const sixdgs_plan* p, int section) {
  return reinterpret_cast<T*>(static_cast<char*>(ws) + p->off[section]);
}

int64_t spin_budget(const sixdgs_plan* p) {
  return p->settings.spin_budget > 0 ? p->settings.spin_budget : (int64_t)1 << 31;
}

sixdgs_status check_ws(const sixdgs_plan* p, void* ws, size_t ws_bytes) {
  if (!p || !ws) return SIXDGS_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(ws) & 255u) != 0) return SIXDGS_ERR_INVALID_ARG;
  if ((int64_t)ws_bytes < p->ws_bytes) return SIXDGS_ERR_WORKSPACE;
  return SIXDGS_OK;
}

// Can every plane segment of a staged tile of Gaussians be copied in bulk
// (16-byte-aligned source, length a multiple of 16 bytes)?  Null pointers
// (absent planes) do not count.
bool bulk_planes(int64_t n, std::initializer_list<const float*> arrays) {
  if (n % 4 != 0) return false;
  for (const float* p : arrays)
    if (p && (reinterpret_cast<uintptr_t>(p) & 15u) != 0) return false;
  return true;
}

sixdgs_status launch_status() {
  return cudaPeekAtLastError() == cudaSuccess ? SIXDGS_OK : SIXDGS_ERR_CUDA;
}

bool valid_scene(const sixdgs_plan* p, const sixdgs_scene* s) {
  return s && s->n == p->n && s->sh_degree == p->sh_degree &&
         (p->n == 0 || (s->mu_p && s->mu_d && s->l_raw && s->opacity_logit && s->sh));
}

// The projection needs l_raw and opacity_logit only without a cached state.
bool valid_fwd_scene(const sixdgs_plan* p, const sixdgs_scene* s) {
  return s && s->n == p->n && s->sh_degree == p->sh_degree &&
         (p->n == 0 || (s->mu_p && s->mu_d && s->sh && (s->cond_cache || (s->l_raw && s->opacity_logit))));
}

BinArgs bin_args(const sixdgs_plan* p, void* ws, int32_t* status_dev) {
  BinArgs a;
  a.cams = ws_ptr<CamRec>(ws, p, SIXDGS_WS_CAMS);
  a.n_cams = p->n_cams;
  a.n = (uint32_t)p->n;
  a.tile_first = 0;
  a.total_tiles = (uint32_t)p->total_tiles;
  a.band = -1;
  a.tile = ws_ptr<TileCounters>(ws, p, WS_TILE);
  a.vis = ws_ptr<uint4>(ws, p, WS_VIS);
  a.vis_count = ws_ptr<uint32_t>(ws, p, WS_VIS_COUNT);
  a.views = view_parts(p->n, p->n_cams);
  a.segments = (uint32_t)((p->n + kStageTile - 1) / kStageTile) * a.views.parts;
  a.segment_size = (uint32_t)kStageTile * a.views.views;
  a.state = ws_ptr<uint32_t>(ws, p, WS_STATE);
  a.scan_state = ws_ptr<unsigned long long>(ws, p, WS_SCAN);
  a.order = ws_ptr<uint4>(ws, p, WS_ORDER);
  a.ranges = ws_ptr<uint2>(ws, p, SIXDGS_WS_RANGES);
  a.capacity = (uint64_t)p->dup_capacity;
  a.dup = ws_ptr<uint64_t>(ws, p, WS_DUP);
  a.sorted = ws_ptr<uint32_t>(ws, p, SIXDGS_WS_SORTED);
  a.sorted_key = ws_ptr<uint32_t>(ws, p, SIXDGS_WS_SORTEDKEY);
  a.counts = ws_ptr<uint32_t>(ws, p, SIXDGS_WS_COUNTS);
  a.scan_tickets = false;
  a.spin_budget = spin_budget(p);
  a.status = status_dev;
  return a;
}

// Byte offsets of the workspace sections, with tile state for tile_slots tiles;
// returns the size.
int64_t lay_out(sixdgs_plan* plan, int64_t tile_slots) {
  const int64_t n_pairs = plan->n_pairs, tiles = tile_slots, dups = plan->dup_capacity;
  const sixdgs_settings& st = plan->settings;
  int64_t o = 0;
  auto take = [&](int section, int64_t bytes) {
    plan->off[section] = o;
    o = align_up(o + bytes, 256);
  };
  take(SIXDGS_WS_CAMS, (int64_t)plan->n_cams * (int64_t)sizeof(CamRec));
  take(SIXDGS_WS_REC, n_pairs * (int64_t)sizeof(PairRec));
  take(SIXDGS_WS_NTILES, align_up(n_pairs, 4) * 4);
  take(SIXDGS_WS_RECT, n_pairs * 8);
  take(SIXDGS_WS_DEPTHKEY, n_pairs * 4);
  take(SIXDGS_WS_GRADREC, st.inference ? 0 : n_pairs * 48);
  take(SIXDGS_WS_RANGES, tiles * 8);
  take(SIXDGS_WS_NWALK, st.store_aux ? plan->total_pixels * 4 : 0);
  take(SIXDGS_WS_COUNTS, 48);
  take(WS_COUNTERS, 64 * 4);
  // cleared by condition_project (the binning leaves its own words clean)
  plan->off[WS_ZERO] = o;
  take(WS_STATE, kBinWords * 4);
  take(WS_SCAN, (tiles + kScanTile - 1) / kScanTile * 8);
  take(WS_TILE, tiles * (int64_t)sizeof(TileCounters));
  plan->off[WS_ZERO_END] = o;
  take(WS_ORDER, tiles * 16);
  take(WS_VIS, n_pairs * 16);
  take(WS_VIS_COUNT, vis_segments_max(plan->n) * 4);
  take(WS_DUP, dups * 8);
  take(WS_SORT_K, dups * 4);
  take(WS_SORT_V, dups * 4);
  plan->off[SIXDGS_WS_SORTED] = plan->off[WS_SORT_V];
  plan->off[SIXDGS_WS_SORTEDKEY] = plan->off[WS_SORT_K];
  return o;
}

// sixdgs_condition_project; loss (may be null) is set to zero on the way.
// banded: the tiles are left uncounted.
sixdgs_status project_frame(const sixdgs_plan* p, const sixdgs_scene* scene, const sixdgs_camera* cams, void* ws,
                            size_t ws_bytes, double* loss, bool banded, int32_t* status_dev,
                            sixdgs_stream_t stream_) {
  sixdgs_status e = check_ws(p, ws, ws_bytes);
  if (e != SIXDGS_OK) return e;
  if (!valid_fwd_scene(p, scene) || !cams) return SIXDGS_ERR_INVALID_ARG;
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  CamRec* dcams = ws_ptr<CamRec>(ws, p, SIXDGS_WS_CAMS);
  int32_t tile_offset = 0;
  int64_t pixel_base = 0;
  for (int i = 0; i < p->n_cams; ++i) {
    const CamRec r = make_cam_rec(cams[i], p->settings, 0, 0);
    tile_offset += r.tiles_x * r.tiles_y;
    pixel_base += (int64_t)r.width * r.height;
  }
  if (tile_offset != p->total_tiles || pixel_base != p->total_pixels) return SIXDGS_ERR_INVALID_ARG;
  tile_offset = 0;
  pixel_base = 0;
  auto next_cam = [&](int i) {
    const CamRec r = make_cam_rec(cams[i], p->settings, tile_offset, pixel_base);
    tile_offset += r.tiles_x * r.tiles_y;
    pixel_base += (int64_t)r.width * r.height;
    return r;
  };
  char* zero = static_cast<char*>(ws) + p->off[WS_ZERO];
  const int64_t zero_bytes = p->off[WS_ZERO_END] - p->off[WS_ZERO];
  // kernel parameters of 128 bytes a camera: the launch copies no more of
  // them than the frame needs
  if (p->n_cams == 1) upload_cams<1>(1, next_cam, dcams, zero, zero_bytes, loss, sm_count(), stream);
  else if (p->n_cams <= 8) upload_cams<8>(p->n_cams, next_cam, dcams, zero, zero_bytes, loss, sm_count(), stream);
  else upload_cams<48>(p->n_cams, next_cam, dcams, zero, zero_bytes, loss, sm_count(), stream);
  ProjectArgs a;
  a.cams = dcams;
  a.n_cams = p->n_cams;
  a.n = p->n;
  a.sh_degree = p->sh_degree;
  a.lambda_opa = p->settings.lambda_opa;
  a.inv_tile_w = 1.f / (float)p->settings.tile_w;
  a.inv_tile_h = 1.f / (float)p->settings.tile_h;
  a.alpha_footprint = p->settings.alpha_footprint;
  a.mu_p = scene->mu_p;
  a.mu_d = scene->mu_d;
  a.l_raw = scene->l_raw;
  a.opacity_logit = scene->opacity_logit;
  a.sh = scene->sh;
  a.lambda_raw = scene->lambda_raw;
  a.cond_cache = scene->cond_cache;
  a.rec = ws_ptr<PairRec>(ws, p, SIXDGS_WS_REC);
  a.ntiles = ws_ptr<uint32_t>(ws, p, SIXDGS_WS_NTILES);
  a.rect = ws_ptr<ushort4>(ws, p, SIXDGS_WS_RECT);
  a.depth_key = ws_ptr<uint32_t>(ws, p, SIXDGS_WS_DEPTHKEY);
  a.vis = ws_ptr<uint4>(ws, p, WS_VIS);
  a.vis_count = ws_ptr<uint32_t>(ws, p, WS_VIS_COUNT);
  a.tile = ws_ptr<TileCounters>(ws, p, WS_TILE);
  a.banded = banded;
  a.grad_rec = p->settings.inference ? nullptr : ws_ptr<float>(ws, p, SIXDGS_WS_GRADREC);
  a.bulk = bulk_planes(p->n, {a.mu_p, a.mu_d, a.sh, a.lambda_raw, a.cond_cache,
                              a.cond_cache ? nullptr : a.l_raw, a.cond_cache ? nullptr : a.opacity_logit});
  a.spin_budget = spin_budget(p);
  a.status = status_dev;
  a.defer_big = defer_big_rects(p->n, p->n_cams, p->total_tiles);
  launch_project_fwd(a, stream);
  if (a.defer_big && !banded && p->n > 0 &&
      launch_bin_count(bin_args(p, ws, status_dev), sm_count(), stream) != cudaSuccess)
    return SIXDGS_ERR_CUDA;
  return launch_status();
}

BlendArgs blend_args(const sixdgs_plan* p, void* ws) {
  BlendArgs a;
  std::memset(&a, 0, sizeof(a));
  a.cams = ws_ptr<CamRec>(ws, p, SIXDGS_WS_CAMS);
  a.n_cams = p->n_cams;
  a.tile_w = p->settings.tile_w;
  a.tile_h = p->settings.tile_h;
  a.batch = p->settings.batch;
  a.rec = ws_ptr<PairRec>(ws, p, SIXDGS_WS_REC);
  a.n_pairs = (uint32_t)p->n_pairs;
  a.sorted = ws_ptr<uint32_t>(ws, p, SIXDGS_WS_SORTED);
  a.order = ws_ptr<uint4>(ws, p, WS_ORDER);
  a.n_busy = ws_ptr<uint32_t>(ws, p, WS_STATE) + kBinOver + kBinLevels;
  for (int i = 0; i < 3; ++i) a.bg[i] = p->settings.bg[i];
  const double norm = p->settings.loss_norm > 0.f ? (double)p->settings.loss_norm
                                                   : 3.0 * (double)p->total_pixels;
  a.inv_count = (float)(1.0 / norm);
  a.nwalk = p->settings.store_aux ? ws_ptr<uint32_t>(ws, p, SIXDGS_WS_NWALK) : nullptr;
  a.pair_counts = p->settings.count_pairs
                      ? reinterpret_cast<unsigned long long*>(ws_ptr<char>(ws, p, SIXDGS_WS_COUNTS) + 16)
                      : nullptr;
  a.tile_queue = p->settings.persistent ? ws_ptr<uint32_t>(ws, p, WS_COUNTERS) + 32 : nullptr;
  a.total_tiles = a.frame_tiles = (uint32_t)p->total_tiles;
  return a;
}

}  // namespace

namespace sixdgs {

int64_t plan_bands(sixdgs_plan* p, int64_t ws_bytes) {
  const int64_t tiles = p->total_tiles;
  // per block of the list scan: its tiles' range, counters and order record, and its look-back word
  constexpr int64_t kPerBlock = kScanTile * (8 + (int64_t)sizeof(TileCounters) + 16) + 8;
  const int64_t fixed = lay_out(p, 0) + 4 * 256;   // four sections' alignment
  const int64_t slots = std::min((ws_bytes - fixed) / kPerBlock * kScanTile, tiles);
  if (slots <= 0) return 0;
  p->ws_bytes = lay_out(p, slots);
  return slots;
}

sixdgs_status render_banded(const sixdgs_plan* p, int64_t slots, const sixdgs_scene* scene, const sixdgs_camera* cams,
                            void* ws, size_t ws_bytes, float* images_dev, int32_t* status_dev,
                            sixdgs_stream_t stream_) {
  sixdgs_status e = project_frame(p, scene, cams, ws, ws_bytes, nullptr, true, status_dev, stream_);
  if (e != SIXDGS_OK) return e;
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  BinArgs b = bin_args(p, ws, status_dev);
  BlendArgs f = blend_args(p, ws);
  f.images = images_dev;
  f.pair_counts = nullptr;   // (nobody could read them)
  b.band = 0;
  for (int64_t first = 0; first < p->total_tiles; first += slots, ++b.band) {
    b.tile_first = (uint32_t)first;
    b.total_tiles = f.total_tiles = (uint32_t)std::min(slots, p->total_tiles - first);
    if (first > 0 && cudaMemsetAsync(b.tile, 0, b.total_tiles * sizeof(TileCounters), stream) != cudaSuccess)
      return SIXDGS_ERR_CUDA;
    if (p->n > 0 && launch_bin_count(b, sm_count(), stream) != cudaSuccess) return SIXDGS_ERR_CUDA;
    if (launch_bin(b, sm_count(), stream) != cudaSuccess) return SIXDGS_ERR_CUDA;
    launch_blend_fwd(f, f.total_tiles, stream);
  }
  return launch_status();
}

}  // namespace sixdgs

extern "C" {

const char* sixdgs_version(void) { return "0.1.0"; }

const char* sixdgs_status_string(int32_t status) {
  switch (status) {
    case SIXDGS_OK: return "ok";
    case SIXDGS_ERR_INVALID_ARG: return "invalid argument";
    case SIXDGS_ERR_CUDA: return "CUDA error";
    case SIXDGS_ERR_CAPACITY: return "duplicate capacity exceeded";
    case SIXDGS_ERR_TIMEOUT: return "device wait timed out";
    case SIXDGS_ERR_NONFINITE: return "non-finite Gaussian";
    case SIXDGS_ERR_WORKSPACE: return "workspace too small";
    default: return "unknown status";
  }
}

sixdgs_status sixdgs_plan_init(int64_t n, int32_t sh_degree, const sixdgs_camera* cams,
                               int32_t n_cams, const sixdgs_settings* st, int64_t dup_capacity,
                               sixdgs_plan* plan) {
  if (!plan || !st || !cams || n < 0 || n_cams < 1 || n_cams > kMaxCams) return SIXDGS_ERR_INVALID_ARG;
  if (sh_degree < 0 || sh_degree > 3) return SIXDGS_ERR_INVALID_ARG;
  if (!(st->tile_w == 8 || st->tile_w == 16 || st->tile_w == 32)) return SIXDGS_ERR_INVALID_ARG;
  if (!(st->tile_h == 8 || st->tile_h == 16)) return SIXDGS_ERR_INVALID_ARG;
  if (st->batch < 32 || st->batch > 1024 || st->batch % 32) return SIXDGS_ERR_INVALID_ARG;
  if (!(st->lambda_opa >= 0.f) || !(st->lambda_opa <= 1.f)) return SIXDGS_ERR_INVALID_ARG;
  if (st->inference != 0 && st->inference != 1) return SIXDGS_ERR_INVALID_ARG;
  if (st->inference && st->store_aux) return SIXDGS_ERR_INVALID_ARG;
  if (st->alpha_footprint != 0 && st->alpha_footprint != 1) return SIXDGS_ERR_INVALID_ARG;
  const int64_t n_pairs = (int64_t)n_cams * n;
  if (n_pairs >= ((int64_t)1 << 31)) return SIXDGS_ERR_INVALID_ARG;
  std::memset(plan, 0, sizeof(*plan));
  int64_t tiles = 0, pixels = 0;
  for (int i = 0; i < n_cams; ++i) {
    const sixdgs_camera& c = cams[i];
    if (c.width <= 0 || c.height <= 0 || !(c.fx > 0.f) || !(c.fy > 0.f)) return SIXDGS_ERR_INVALID_ARG;
    const int64_t tx = (c.width + st->tile_w - 1) / st->tile_w;
    const int64_t ty = (c.height + st->tile_h - 1) / st->tile_h;
    if (tx > 65535 || ty > 65535) return SIXDGS_ERR_INVALID_ARG;
    tiles += tx * ty;
    pixels += (int64_t)c.width * c.height;
  }
  if (tiles >= ((int64_t)1 << 31)) return SIXDGS_ERR_INVALID_ARG;
  if (dup_capacity <= 0) dup_capacity = 4 * n_pairs + 4096;
  if (dup_capacity >= ((int64_t)1 << 30)) return SIXDGS_ERR_INVALID_ARG;

  plan->n = n;
  plan->sh_degree = sh_degree;
  plan->n_cams = n_cams;
  plan->settings = *st;
  plan->n_pairs = n_pairs;
  plan->total_tiles = tiles;
  plan->total_pixels = pixels;
  plan->dup_capacity = dup_capacity;
  plan->depth_passes = 4;
  int bits = 1;
  while (((int64_t)1 << bits) < tiles) ++bits;
  plan->tile_passes = (bits + 7) / 8;

  plan->ws_bytes = lay_out(plan, tiles);
  return SIXDGS_OK;
}

size_t sixdgs_workspace_size(const sixdgs_plan* plan) { return plan ? (size_t)plan->ws_bytes : 0; }

sixdgs_status sixdgs_condition_project(const sixdgs_plan* p, const sixdgs_scene* scene,
                                       const sixdgs_camera* cams, void* ws, size_t ws_bytes,
                                       int32_t* status_dev, sixdgs_stream_t stream) {
  return project_frame(p, scene, cams, ws, ws_bytes, nullptr, false, status_dev, stream);
}

sixdgs_status sixdgs_bin_sort(const sixdgs_plan* p, void* ws, size_t ws_bytes, int32_t* status_dev,
                              sixdgs_stream_t stream_) {
  sixdgs_status e = check_ws(p, ws, ws_bytes);
  if (e != SIXDGS_OK) return e;
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  const BinArgs a = bin_args(p, ws, status_dev);
  if (launch_bin(a, sm_count(), stream) != cudaSuccess) return SIXDGS_ERR_CUDA;
  return launch_status();
}

sixdgs_status sixdgs_raster_fwd(const sixdgs_plan* p, void* ws, size_t ws_bytes, float* images_dev,
                                const float* targets_dev, float* grad_images_dev, double* loss_dev,
                                int32_t* /*status_dev*/, sixdgs_stream_t stream_) {
  sixdgs_status e = check_ws(p, ws, ws_bytes);
  if (e != SIXDGS_OK) return e;
  if (!images_dev) return SIXDGS_ERR_INVALID_ARG;
  const bool any = targets_dev || grad_images_dev || loss_dev;
  const bool all = targets_dev && grad_images_dev && loss_dev;
  if (any && !all) return SIXDGS_ERR_INVALID_ARG;
  BlendArgs a = blend_args(p, ws);
  a.images = images_dev;
  a.targets = targets_dev;
  a.grad_images = grad_images_dev;
  a.loss = loss_dev;
  launch_blend_fwd(a, p->total_tiles, reinterpret_cast<cudaStream_t>(stream_));
  return launch_status();
}

sixdgs_status sixdgs_raster_fwd_bwd(const sixdgs_plan* p, void* ws, size_t ws_bytes, float* images_dev,
                                    const float* targets_dev, float* grad_images_dev, double* loss_dev,
                                    int32_t* /*status_dev*/, sixdgs_stream_t stream_) {
  sixdgs_status e = check_ws(p, ws, ws_bytes);
  if (e != SIXDGS_OK) return e;
  if (p->settings.inference || !images_dev || !targets_dev || !loss_dev) return SIXDGS_ERR_INVALID_ARG;
  BlendArgs a = blend_args(p, ws);
  a.images = images_dev;
  a.targets = targets_dev;
  a.grad_images = grad_images_dev;
  a.loss = loss_dev;
  a.grad_rec = ws_ptr<float>(ws, p, SIXDGS_WS_GRADREC);
  launch_blend_fused(a, p->total_tiles, reinterpret_cast<cudaStream_t>(stream_));
  return launch_status();
}

sixdgs_status sixdgs_blend_bwd(const sixdgs_plan* p, void* ws, size_t ws_bytes, const float* images_dev,
                               const float* grad_images_dev, int32_t* /*status_dev*/, sixdgs_stream_t stream_) {
  sixdgs_status e = check_ws(p, ws, ws_bytes);
  if (e != SIXDGS_OK) return e;
  if (p->settings.inference) return SIXDGS_ERR_INVALID_ARG;
  if (!images_dev || !grad_images_dev) return SIXDGS_ERR_INVALID_ARG;
  BlendArgs a = blend_args(p, ws);
  a.images_in = images_dev;
  a.grad_in = grad_images_dev;
  a.grad_rec = ws_ptr<float>(ws, p, SIXDGS_WS_GRADREC);
  a.recompute = p->settings.store_aux ? 0 : 1;
  launch_blend_bwd(a, p->total_tiles, reinterpret_cast<cudaStream_t>(stream_));
  return launch_status();
}

sixdgs_status sixdgs_project_bwd(const sixdgs_plan* p, const sixdgs_scene* scene, void* ws,
                                 size_t ws_bytes, float* grad_mu_p, float* grad_mu_d, float* grad_l_raw,
                                 float* grad_opacity_logit, float* grad_sh, float* grad_lambda_raw,
                                 int32_t accumulate, int32_t* status_dev, sixdgs_stream_t stream_) {
  sixdgs_status e = check_ws(p, ws, ws_bytes);
  if (e != SIXDGS_OK) return e;
  if (p->settings.inference) return SIXDGS_ERR_INVALID_ARG;
  if (!valid_scene(p, scene)) return SIXDGS_ERR_INVALID_ARG;
  if (p->n > 0 && (!grad_mu_p || !grad_mu_d || !grad_l_raw || !grad_opacity_logit || !grad_sh))
    return SIXDGS_ERR_INVALID_ARG;
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  ProjectBwdArgs b;
  b.cams = ws_ptr<CamRec>(ws, p, SIXDGS_WS_CAMS);
  b.n_cams = p->n_cams;
  b.n = p->n;
  b.sh_degree = p->sh_degree;
  b.lambda_opa = p->settings.lambda_opa;
  b.mu_p = scene->mu_p;
  b.mu_d = scene->mu_d;
  b.l_raw = scene->l_raw;
  b.opacity_logit = scene->opacity_logit;
  b.sh = scene->sh;
  b.lambda_raw = scene->lambda_raw;
  b.rec = ws_ptr<PairRec>(ws, p, SIXDGS_WS_REC);
  b.ntiles = ws_ptr<uint32_t>(ws, p, SIXDGS_WS_NTILES);
  b.grad_rec = ws_ptr<float>(ws, p, SIXDGS_WS_GRADREC);
  b.grad_mu_p = grad_mu_p;
  b.grad_mu_d = grad_mu_d;
  b.grad_l_raw = grad_l_raw;
  b.grad_opacity_logit = grad_opacity_logit;
  b.grad_sh = grad_sh;
  b.grad_lambda_raw = grad_lambda_raw;
  b.accumulate = accumulate;
  b.bulk = bulk_planes(p->n, {b.mu_p, b.mu_d, b.l_raw, b.opacity_logit, b.sh, b.lambda_raw});
  b.spin_budget = spin_budget(p);
  b.status = status_dev;
  launch_param_bwd(b, stream);
  return launch_status();
}

sixdgs_status sixdgs_raster_bwd(const sixdgs_plan* p, const sixdgs_scene* scene, void* ws,
                                size_t ws_bytes, const float* images_dev,
                                const float* grad_images_dev, float* grad_mu_p, float* grad_mu_d,
                                float* grad_l_raw, float* grad_opacity_logit, float* grad_sh,
                                float* grad_lambda_raw, int32_t accumulate, int32_t* status_dev,
                                sixdgs_stream_t stream) {
  sixdgs_status e = check_ws(p, ws, ws_bytes);
  if (e != SIXDGS_OK) return e;
  if (p->settings.inference) return SIXDGS_ERR_INVALID_ARG;
  if (!valid_scene(p, scene)) return SIXDGS_ERR_INVALID_ARG;
  if (p->n > 0 && (!grad_mu_p || !grad_mu_d || !grad_l_raw || !grad_opacity_logit || !grad_sh))
    return SIXDGS_ERR_INVALID_ARG;
  e = sixdgs_blend_bwd(p, ws, ws_bytes, images_dev, grad_images_dev, status_dev, stream);
  if (e != SIXDGS_OK) return e;
  return sixdgs_project_bwd(p, scene, ws, ws_bytes, grad_mu_p, grad_mu_d, grad_l_raw, grad_opacity_logit,
                            grad_sh, grad_lambda_raw, accumulate, status_dev, stream);
}

sixdgs_status sixdgs_render_batched(const sixdgs_plan* p, const sixdgs_scene* scene,
                                    const sixdgs_camera* cams_host, void* ws, size_t ws_bytes,
                                    float* images_dev, const float* targets_dev, float* grad_images_dev,
                                    double* loss_dev, float* grad_mu_p, float* grad_mu_d, float* grad_l_raw,
                                    float* grad_opacity_logit, float* grad_sh, float* grad_lambda_raw,
                                    int32_t* status_dev, sixdgs_stream_t stream) {
  sixdgs_status e = check_ws(p, ws, ws_bytes);
  if (e != SIXDGS_OK) return e;
  const bool train = targets_dev != nullptr;
  if (train) {
    if (p->settings.inference || !loss_dev || !valid_scene(p, scene)) return SIXDGS_ERR_INVALID_ARG;
    if (p->n > 0 && (!grad_mu_p || !grad_mu_d || !grad_l_raw || !grad_opacity_logit || !grad_sh))
      return SIXDGS_ERR_INVALID_ARG;
  }
  e = project_frame(p, scene, cams_host, ws, ws_bytes, train ? loss_dev : nullptr, false, status_dev, stream);
  if (e != SIXDGS_OK) return e;
  e = sixdgs_bin_sort(p, ws, ws_bytes, status_dev, stream);
  if (e != SIXDGS_OK) return e;
  if (!train) return sixdgs_raster_fwd(p, ws, ws_bytes, images_dev, nullptr, nullptr, nullptr, status_dev, stream);
  e = sixdgs_raster_fwd_bwd(p, ws, ws_bytes, images_dev, targets_dev, grad_images_dev, loss_dev, status_dev,
                            stream);
  if (e != SIXDGS_OK) return e;
  return sixdgs_project_bwd(p, scene, ws, ws_bytes, grad_mu_p, grad_mu_d, grad_l_raw, grad_opacity_logit,
                            grad_sh, grad_lambda_raw, 0, status_dev, stream);
}

sixdgs_status sixdgs_peak_probe(int32_t kind, int64_t iters, float* out_dev, int32_t blocks,
                                sixdgs_stream_t stream) {
  if ((kind != 0 && kind != 1) || iters < 0 || blocks < 1 || !out_dev) return SIXDGS_ERR_INVALID_ARG;
  launch_peak_probe(kind, iters, out_dev, blocks, reinterpret_cast<cudaStream_t>(stream));
  return launch_status();
}

sixdgs_status sixdgs_condition_cache(int64_t n, const float* l_raw_dev, const float* opacity_logit_dev,
                                     float* cache_dev, sixdgs_stream_t stream) {
  if (n < 0 || (n > 0 && (!l_raw_dev || !opacity_logit_dev || !cache_dev))) return SIXDGS_ERR_INVALID_ARG;
  CondCacheArgs a;
  a.n = n;
  a.l_raw = l_raw_dev;
  a.opacity_logit = opacity_logit_dev;
  a.cache = cache_dev;
  launch_cond_cache(a, reinterpret_cast<cudaStream_t>(stream));
  return launch_status();
}

sixdgs_status sixdgs_scale_rotation(int64_t n, const float* l_raw_dev, float* rotation_dev, float* scale_dev,
                                    int32_t* status_dev, sixdgs_stream_t stream) {
  if (n < 0 || (n > 0 && (!l_raw_dev || !rotation_dev || !scale_dev))) return SIXDGS_ERR_INVALID_ARG;
  ScaleRotationArgs a;
  a.n = n;
  a.l_raw = l_raw_dev;
  a.rotation = rotation_dev;
  a.scale = scale_dev;
  a.status = status_dev;
  launch_scale_rotation(a, reinterpret_cast<cudaStream_t>(stream));
  return launch_status();
}

}  // extern "C"
