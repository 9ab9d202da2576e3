// Shared device-side definitions of the sixdgs library (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sixdgs.h"

namespace sixdgs {

// ---- constants of the inherited 3DGS rasteriser (6DGS section 4.4) --------
constexpr float kDilation = 0.3f;       // px^2 added to the 2D covariance diagonal
constexpr float kRadiusSigmas = 3.0f;   // screen extent in standard deviations
constexpr float kAlphaMin = 1.0f / 255.0f;
constexpr float kAlphaMax = 0.99f;
constexpr float kTMin = 1e-4f;
constexpr float kFrustumGuard = 1.3f;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
// log2(1/255): an entry is skipped when its log2-alpha q is below this
constexpr float kQMin = -7.994353436858858f;
// log2(0.99): alpha is clamped to 0.99 above this
constexpr float kQMax = -0.014499569695115089f;

constexpr int kMaxShCoeffs = 16;

// Per-camera record stored in the workspace (128 bytes).
struct __align__(16) CamRec {
  float r[9];        // world-to-camera rotation, row-major
  float t[3];        // world-to-camera translation
  float campos[3];
  float fx, fy, cx, cy;
  float znear;
  float limx, limy;  // frustum guard on x/z, y/z for the Jacobian
  int32_t width, height;
  int32_t tiles_x, tiles_y;
  int32_t tile_offset;   // first global tile id of this camera
  int64_t pixel_base;    // pixels of all earlier cameras; image floats start at 3 * pixel_base
  int32_t pad[2];
};
static_assert(sizeof(CamRec) == 128, "CamRec must stay 128 bytes");

// Record of one (view, Gaussian) pair, consumed by the blend (48 bytes).
//  a = (u, v, qa, qb), b = (qc, lo, r, g), c = (b, hx, hy, depth)
// with q(dx, dy) = qa dx^2 + qb dx dy + qc dy^2 + lo = log2(alpha_cond) +
// log2(e) * (-1/2 Delta^T conic Delta), Delta = (u - px, v - py), and
// (hx, hy) the half-extents of the box around (u, v) outside which
// q < log2(1/255) (the entry is skipped at every pixel there).
struct __align__(16) PairRec {
  float4 a, b, c;
};

// What the sort and the blend need to know of a tile, in one 16-byte load:
// (global tile id, list start, list end, camera).
__device__ __forceinline__ uint4 tile_work(uint32_t tile, uint2 range, uint32_t cam) {
  return make_uint4(tile, range.x, range.y, cam);
}

// Camera of global tile gt.
__device__ __forceinline__ int find_camera(const CamRec* cams, int n_cams, uint32_t gt) {
  int lo = 0, hi = n_cams - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if ((uint32_t)cams[mid].tile_offset <= gt) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// First statement of every kernel of a frame: waits until the kernel before it
// in the stream is done and its writes are visible.  A no-op for a plain
// launch.  (No kernel lets its successor start earlier than at its own end:
// waiting CTAs beside a running kernel slowed large frames, 764 -> 822 us for 20
// views of 183k Gaussians at 1024^2, and gained nothing for small ones.)
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void raise_status(int32_t* status, int code) {
  if (status) atomicOr(status, 1 << code);
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float sigmoidf_(float x) { return 1.0f / (1.0f + __expf(-x)); }

// q of one list entry (a, b) at the pixel centre whose negation is npix
// = (-px, -py); d = (u - px, v - py) comes out as one packed subtraction.
// Explicit rounding intrinsics keep the forward and backward walks
// bit-identical.
__device__ __forceinline__ float entry_q(const float4& a, const float4& b, float2 npix, float2& d) {
  d = __fadd2_rn(make_float2(a.x, a.y), npix);
  const float t1 = __fmaf_rn(a.z, d.x, __fmul_rn(a.w, d.y));   // qa dx + qb dy
  const float t2 = __fmaf_rn(__fmul_rn(b.x, d.y), d.y, b.y);   // qc dy^2 + lo
  return __fmaf_rn(t1, d.x, t2);
}

}  // namespace sixdgs
