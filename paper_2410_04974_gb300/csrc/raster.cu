// Stages 3 and 4a: front-to-back blending of every screen tile and its
// reverse (the 3DGS rasteriser that 6DGS section 4.4 keeps after slicing).
//
// One CTA per global tile (all cameras' tiles in one grid, so cameras of
// different resolutions share a launch); each warp owns an 8x4 sub-block of
// the tile, each half-warp a 4x4 block of it, one pixel per lane.  The tile's
// sorted list is walked in batches: each batch of pair records is gathered
// into shared memory by the whole CTA, each thread testing its entries' alpha
// >= 1/255 ellipses against all blocks of the tile (ballots: a bit per block
// and entry); then every warp turns its two blocks' ballots into lists and
// composites each pixel against its block's list, in list order.  An entry a
// block passes over would be skipped at every pixel of it (q < log2(1/255)),
// so the result is the same as walking every entry at every pixel.  A CTA
// leaves as soon as __syncthreads_count reports every pixel saturated; a warp
// leaves a batch as soon as all its lanes are done.
//
// The walks are bound by instructions, most of them spent at pixels that an
// entry does not reach and on finding the next entry.  Hence the 4x4 blocks
// (a Gaussian of 5 pixels radius reaches 11 of them, 174 pixels, against 230
// pixels of 8x4 blocks; a warp's two lists are nearly equally long), and the
// lists: a walk takes four entries' addresses with one load instead of
// scanning a ballot bit by bit.  Against 8x4 blocks tested by their own warps
// (fused kernel / warp instructions): 858 -> 722 us, 755 -> 618 M at 300k /
// 8 x 800^2; 1487 -> 1244 us at 2M / 4 x 1920x1080; forward 663 -> 599 us for
// 20 views of 183k Gaussians at 1024^2.
//
// Per entry and pixel:  q = qa dx^2 + qb dx dy + qc dy^2 + lo  (log2 alpha),
// skipped when q < log2(1/255); alpha = min(0.99, 2^q); stop (excluding the
// entry) when T (1 - alpha) < 1e-4; C += c alpha T; T *= (1 - alpha).
// Explicit rounding intrinsics make the backward replay bit-identical.
// Pairs of values that take the same
// operation (the pixel offset, T (1 - alpha) and alpha T, two colour
// channels) use the packed two-wide FP32 instructions, with the same
// rounding as the scalar ones.
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace sixdgs {

constexpr int kSubW = 8;   // warp sub-block: 8 x 4 pixels
constexpr int kSubH = 4;
constexpr int kBlkW = 4;   // half-warp block: 4 x 4 pixels

// Pixel of this thread in sub-block `warp` (row-major) of tile (tx, ty).
__device__ __forceinline__ int2 map_pixel(const BlendArgs& a, int tx, int ty, int warp) {
  const int lane = threadIdx.x & 31;
  const int sub_per_row = a.tile_w / kSubW;
  const int sx = (warp % sub_per_row) * kSubW, sy = (warp / sub_per_row) * kSubH;
  return make_int2(tx * a.tile_w + sx + (lane >> 4) * kBlkW + (lane & 3), ty * a.tile_h + sy + ((lane >> 2) & 3));
}
// The negated centre of a pixel, which is what the walks carry.
__device__ __forceinline__ float2 neg_centre(int2 p) { return make_float2(-((float)p.x + 0.5f), -((float)p.y + 0.5f)); }

// The 4x4 blocks of a tile of kTileW x 4 kNby pixels that the entry (u, v, qa,
// qb), (qc, lo), (hx, hy) can reach, bit y * kTileW / 4 + x: those where q >=
// log2(1/255) at some point of the block's pixel-centre rectangle.  (x0, y0):
// the tile's first pixel centre.  For every row of blocks (a band of four
// pixel rows) the ellipse {q >= log2(1/255) - m} meets the band in a convex
// set, whose columns reach from the leftmost to the rightmost point: the
// ellipse's own extreme points (+-hx) if the band holds them, else the
// boundary at the band's row nearest to them.  The margin m (in log2 units)
// covers the FP32 rounding of a pixel's q, at most a few ulp of S = |qa| dx^2 +
// |qc| dy^2 at the tile's far corner, and of the boundary's square root; so no
// pixel that would composite the entry is ever passed over.  One thread tests
// an entry against all blocks: a quarter of the instructions of every warp
// testing every entry against its own blocks.  (Compiled for every tile shape:
// 651 -> 646 us for the fused kernel at 300k / 8 x 800^2.)
template <int kTileW, int kNby>
__device__ __forceinline__ uint32_t block_mask(float4 a, float4 b, float4 c, float x0, float y0) {
  constexpr int kNbx = kTileW / kBlkW;
  constexpr float fw = (float)(kTileW - 1), fh = (float)(kNby * kSubH - 1);
  const float ux = a.x - x0, vy = a.y - y0, hx = c.y, hy = c.z;
  if (!(ux + hx >= 0.f && ux - hx <= fw && vy + hy >= 0.f && vy - hy <= fh)) return 0u;
  const float A = -a.z, B = -a.w, C = -b.x;   // A dx^2 + B dx dy + C dy^2 <= L
  const float dxm = fmaxf(fabsf(ux), fabsf(ux - fw)), dym = fmaxf(fabsf(vy), fabsf(vy - fh));
  const float S = A * dxm * dxm + C * dym * dym;
  if (!(A > 1e-30f && C > 1e-30f && S < 1e30f)) return ~0u >> (32 - kNbx * kNby);
  const float L = b.y - kQMin + (1e-3f + 1e-6f * S);
  const float ia = rcp_approx(A);
  const float k = 0.5f * B * ia;                    // middle of the columns of a row: dx = -k dy
  const float E = L * ia, F = k * k - C * ia;       // their half-length: sqrt(E + F dy^2)
  const float dyr = -0.5f * B * rcp_approx(C) * hx;   // row of the rightmost point (leftmost: -dyr)
  // the columns ux - dxr - pad .. ux - dxl + pad of a band, in blocks
  const float pad = 2e-3f + 1e-6f * dxm;
  const float x_first = (ux - pad - (float)(kBlkW - 1)) * (1.f / kBlkW), x_last = (ux + pad) * (1.f / kBlkW);
  uint32_t mask = 0u;
#pragma unroll
  for (int r = 0; r < kNby; ++r) {
    const float d1 = vy - (float)(r * kSubH), d0 = d1 - (float)(kSubH - 1);
    const float cr = fminf(fmaxf(dyr, d0), d1), cl = fminf(fmaxf(-dyr, d0), d1);
    const float sr = fmaf(F, cr * cr, E), sl = fmaf(F, cl * cl, E);
    const bool in_r = cr == dyr, in_l = cl == -dyr;
    const float dxr = in_r ? hx : fmaf(-k, cr, sqrt_approx(fmaxf(sr, 0.f)));
    const float dxl = in_l ? -hx : fmaf(-k, cl, -sqrt_approx(fmaxf(sl, 0.f)));
    if (in_r || in_l || fmaxf(sr, sl) >= 0.f) {
      // block x spans 4 x .. 4 x + 3
      const int first = max(__float2int_ru(fmaf(dxr, -1.f / kBlkW, x_first)), 0);
      const int last = min(__float2int_rd(fmaf(dxl, -1.f / kBlkW, x_last)), kNbx - 1);
      if (first <= last) mask |= ((2u << last) - (1u << first)) << (r * kNbx);
    }
  }
  return mask;
}

__device__ __forceinline__ uint32_t block_mask(const BlendArgs& t, float4 a, float4 b, float4 c, float x0, float y0) {
  if (t.tile_w == 16) return t.tile_h == 16 ? block_mask<16, 4>(a, b, c, x0, y0) : block_mask<16, 2>(a, b, c, x0, y0);
  if (t.tile_w == 8) return t.tile_h == 16 ? block_mask<8, 4>(a, b, c, x0, y0) : block_mask<8, 2>(a, b, c, x0, y0);
  return t.tile_h == 16 ? block_mask<32, 4>(a, b, c, x0, y0) : block_mask<32, 2>(a, b, c, x0, y0);
}

// A list entry as staged in shared memory: its blend record (u, v, qa, qb),
// (qc, lo, r, g), b and its pair index (bits of c.w).  One struct
// per entry, so a walk addresses all three parts from one index.
struct __align__(16) Entry {
  float4 a, b, c;
};

__device__ __forceinline__ void null_entry(Entry& e, uint32_t p) {   // reaches no pixel
  e.a = make_float4(-1e30f, -1e30f, 0.f, 0.f);
  e.b = make_float4(0.f, -1e30f, 0.f, 0.f);
  e.c = make_float4(0.f, 0.f, 0.f, __uint_as_float(p));
}

// Shared memory of a CTA: the batch's entries and a null entry, which pads the
// lists (entry a.batch), the ballots of every block over the batch (word
// block * cull_stride(batch) + g: entries 32 g to 32 g + 31), then each warp's
// scratch.
__host__ __device__ constexpr int cull_stride(int batch) { return (batch / 32 + 3) & ~3; }
__host__ __device__ constexpr int stage_bytes(int batch, int blocks) {
  return (batch + 1) * (int)sizeof(Entry) + blocks * cull_stride(batch) * 4;
}
__device__ __forceinline__ int blocks_of(const BlendArgs& a) { return a.tile_w * a.tile_h / (kBlkW * kSubH); }
__device__ __forceinline__ uint32_t* cull_of(const BlendArgs& a, Entry* s_e) {
  return reinterpret_cast<uint32_t*>(s_e + a.batch + 1);
}
// The ballots of the warp's left block (its sub-blocks and their blocks are
// both row-major; its right block's follow).
__device__ __forceinline__ const uint32_t* warp_cull(const BlendArgs& a, Entry* s_e) {
  return cull_of(a, s_e) + 2 * (threadIdx.x >> 5) * cull_stride(a.batch);
}
__device__ __forceinline__ char* scratch_of(const BlendArgs& a, void* s_mem) {
  return reinterpret_cast<char*>(s_mem) + stage_bytes(a.batch, blocks_of(a));
}

__device__ __forceinline__ void copy_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Stages list entries [start, start + cnt) and their blocks' ballots.
// npix: neg_centre of a pixel of the tile (whose sides are powers of two).
__device__ __forceinline__ void load_batch(const BlendArgs& a, uint32_t start, int cnt, float2 npix, Entry* s_e) {
  if (threadIdx.x == 0) null_entry(s_e[a.batch], 0u);
  const int lane = threadIdx.x & 31, blocks = blocks_of(a);
  uint32_t* cull = cull_of(a, s_e);
  // the records go to shared memory by asynchronous copies, which hold no
  // registers, all of a thread's in flight together
  for (int i0 = threadIdx.x; i0 < cnt; i0 += 2 * blockDim.x) {
    uint32_t p[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int i = i0 + u * blockDim.x;
      p[u] = i < cnt ? a.sorted[start + i] : 0xffffffffu;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (p[u] < a.n_pairs) {
        Entry* e = s_e + i0 + u * blockDim.x;
        const PairRec* r = a.rec + p[u];
        copy_async16(&e->a, &r->a);
        copy_async16(&e->b, &r->b);
        copy_async16(&e->c, &r->c);
      }
  }
  const float x0 = (float)((int)-npix.x & ~(a.tile_w - 1)) + 0.5f;   // first pixel centre of the tile
  const float y0 = (float)((int)-npix.y & ~(a.tile_h - 1)) + 0.5f;
  copy_async_wait();
  for (int i0 = threadIdx.x & ~31; i0 < cnt; i0 += blockDim.x) {
    const int i = i0 + lane;
    uint32_t mask = 0u;
    if (i < cnt) {
      const uint32_t p = a.sorted[start + i];
      Entry& e = s_e[i];
      if (p < a.n_pairs) {
        mask = block_mask(a, e.a, e.b, e.c, x0, y0);
        e.c.w = __uint_as_float(p);
      } else {  // unreachable for a consistent sort
        null_entry(e, 0u);
      }
    }
    uint32_t word = 0u;   // of block `lane`
#pragma unroll 4
    for (int b = 0; b < blocks; ++b) {
      const uint32_t w = __ballot_sync(0xffffffffu, (mask >> b) & 1u);
      if (lane == b) word = w;
    }
    if (lane < blocks) cull[lane * cull_stride(a.batch) + (i0 >> 5)] = word;
  }
}

// Sparse frames (below, sparse()): a list of at most a.short_list (32 or fewer)
// entries is staged by every warp for itself, in places of its own and tested
// against its own 8x4 sub-block, and walked by the bits of one ballot.  Such a
// tile is bound by the instructions around its few steps, and waits for the one
// warp that tests entries against all blocks: no CTA barrier, no ballots and no
// lists of every block, no padded steps.  2,000 Gaussians of 350 tiles at 4096^2
// (6.7 entries a tile with a list), against staging by the CTA: forward 208 -> 146
// us, fused 535 -> 394; tiles of 8x8 pixels 407 -> 204 and 949 -> 521.  (With the
// walk over the blocks' lists kept, each warp testing its own: forward 220.)
__host__ __device__ constexpr int short_list(int batch, int warps) {
  return batch / warps < 32 ? batch / warps : 32;
}
// The calling warp's places.
__device__ __forceinline__ Entry* short_entries(const BlendArgs& a, Entry* s_e) {
  return s_e + (threadIdx.x >> 5) * a.short_list;
}

// Stages the short list [range.x, range.y) for the calling warp; returns the
// entries whose alpha >= 1/255 boxes meet its sub-block, or (kExact, where a
// backward walk follows) whose ellipses do.
template <bool kExact>
__device__ __forceinline__ uint32_t load_short(const BlendArgs& a, uint2 range, float2 npix, Entry* s_e) {
  const int lane = threadIdx.x & 31;
  bool reach = false;
  if (lane < (int)(range.y - range.x)) {
    const uint32_t p = a.sorted[range.x + lane];
    Entry& e = short_entries(a, s_e)[lane];
    if (p < a.n_pairs) {
      const PairRec& r = a.rec[p];
      const float4 ra = r.a, rb = r.b, rc = r.c;
      e.a = ra;
      e.b = rb;
      e.c = make_float4(rc.x, rc.y, rc.z, __uint_as_float(p));
      // first pixel centre of the warp's sub-block
      const float x0 = -npix.x - (float)((lane >> 4) * kBlkW + (lane & 3)), y0 = -npix.y - (float)((lane >> 2) & 3);
      reach = kExact ? block_mask<kSubW, 1>(ra, rb, rc, x0, y0) != 0u
                     : ra.x + rc.y >= x0 && ra.x - rc.y <= x0 + (float)(kSubW - 1) && ra.y + rc.z >= y0 &&
                           ra.y - rc.z <= y0 + (float)(kSubH - 1);
    }   // (else unreachable for a consistent sort)
  }
  const uint32_t mask = __ballot_sync(0xffffffffu, reach);
  __syncwarp();
  return mask;
}

// The backward walk runs in two passes per warp so that no value has to be
// summed across the lanes of a warp for every list entry:
//  1. pixel-parallel (lane = pixel), front to back like the forward: the
//     transmittance T and the running dL/dC . (colour prefix) Q are carried
//     per pixel, and each pixel's dL/dq and blend weight w for the entry are
//     written to the warp's shared-memory slots (kSlots = 8 entries of each
//     half-warp at a time);
//  2. entry-parallel, once the slots are full (or the batch ends): lane
//     16 h + 8 r + s takes slot s of half h over two rows of its 4 x 4 block
//     and sums, over their 8 pixels, dq, c dq, c^2 dq and dL/dC . w (c the
//     column relative to the block's centre); the two halves of the block are
//     added with a shuffle, and lane 16 h + s turns the sums into the entry's
//     nine record gradients (moments of dq in dx = u - px, dy = v - py) and
//     adds them to the record gradients in global memory.
// A slot's 32 pixel values are stored with a stride of 33 (one float2 of
// padding per slot), so the row writes of pass 1 and the column reads of
// pass 2 are both free of shared-memory bank conflicts.
constexpr int kSlots = 8;
constexpr int kChunk = 128;   // list entries whose ballots are turned into lists at a time
constexpr int kStep = 4;      // entries walked between two looks at the lists

// A block's list: byte offsets of its entries in the staging area (at most
// 1,024 x 48), padded with the null entry to a multiple of kStep.
struct __align__(16) WalkLists {
  uint16_t off[2][kChunk + 8];
};
struct __align__(16) WarpScratch {
  WalkLists lists;
  float2 dqw[kSlots][33];   // (dL/dq / ln 2, w) of slot s at pixel p, at [s][p]
  float4 pix[35];           // dL/dC of pixel p at p + (p >> 3) (rows in other banks)
  uint2 slot[2][kSlots / kStep];   // offsets of the entries in the slots, four to a word pair
};

// Fills a warp's lists with the batch's entries [c0, c0 + kChunk) (cnt in the
// batch); returns the number of steps of the longer one, a multiple of kStep.
// cull: the ballots of the warp's left block (its right one's follow).
// kTwin: both lists get the entries of either block (which change nothing at the
// other).
template <bool kTwin>
__device__ __forceinline__ int fill_lists(const uint32_t* cull, int batch, int c0, int cnt, WalkLists& lists,
                                          uint32_t* n_warp = nullptr) {
  const int lane = threadIdx.x & 31;
  const uint32_t below = (1u << lane) - 1u;
  uint32_t n0 = 0u, n1 = 0u;
  __syncwarp();   // the lists are no longer read
  cull += c0 >> 5;
#pragma unroll
  for (int g = 0; g < kChunk / 32; ++g) {
    const int base = c0 + 32 * g;
    if (base < cnt) {
      uint32_t m0 = cull[g], m1 = cull[cull_stride(batch) + g];
      if (kTwin) m0 = m1 = m0 | m1;
      const uint16_t off = (uint16_t)((base + lane) * (int)sizeof(Entry));
      if ((m0 >> lane) & 1u) lists.off[0][n0 + __popc(m0 & below)] = off;
      if ((m1 >> lane) & 1u) lists.off[1][n1 + __popc(m1 & below)] = off;
      n0 += __popc(m0);
      n1 += __popc(m1);
      if (n_warp) *n_warp += __popc(m0 | m1);
    }
  }
  const int steps = (int)(max(n0, n1) + (kStep - 1)) & ~(kStep - 1);
  const int h = lane >> 4;
  for (int i = (int)(h ? n1 : n0) + (lane & 15); i < steps; i += 16)
    lists.off[h][i] = (uint16_t)(batch * (int)sizeof(Entry));
  __syncwarp();
  return steps;
}

// Offsets of four consecutive list entries (i a multiple of kStep).
__device__ __forceinline__ uint2 list_quad(const WalkLists& lists, int i) {
  return *reinterpret_cast<const uint2*>(&lists.off[(threadIdx.x >> 4) & 1][i]);
}
__device__ __forceinline__ uint32_t quad_off(uint2 q, int k) {
  const uint32_t w = k < 2 ? q.x : q.y;
  return (k & 1) ? w >> 16 : w & 0xffffu;
}
__device__ __forceinline__ const Entry& entry_at(const Entry* s_e, uint32_t off) {
  return *reinterpret_cast<const Entry*>(reinterpret_cast<const char*>(s_e) + off);
}

// Per-pixel front-to-back walk of a tile's list (the forward blend): T and
// C accumulate over the entries that reach the pixel's block; walked is
// the number of list entries before the stop (the list length if none).
struct FwdPixel {
  float T, C0, C1, C2;
  uint32_t walked;
  bool staged;   // the whole list was loaded as one batch (CTA-uniform)
};

template <bool kCount>
__device__ __forceinline__ FwdPixel fwd_walk(const BlendArgs& a, float2 npix, uint2 range, bool inside, Entry* s_e,
                                             WalkLists& lists, uint32_t& n_eval, uint32_t& n_comp,
                                             uint32_t& n_warp) {
  const int B = a.batch;
  float T = 1.f, C2 = 0.f;
  float2 C01 = make_float2(0.f, 0.f);
  bool done = !inside;
  uint32_t walked = range.y - range.x;
  bool staged = false;
  for (uint32_t start = range.x; start < range.y; start += B) {
    if (__syncthreads_count(done) == (int)blockDim.x) break;
    const int cnt = (int)min((uint32_t)B, range.y - start);
    load_batch(a, start, cnt, npix, s_e);
    staged = start == range.x && start + cnt == range.y;
    __syncthreads();
    if (__all_sync(0xffffffffu, done)) continue;
    uint32_t stop_off = 0xffffffffu;   // of the entry this pixel stopped at in this batch
    for (int c0 = 0; c0 < cnt; c0 += kChunk) {
      const int steps = fill_lists<false>(warp_cull(a, s_e), B, c0, cnt, lists, kCount ? &n_warp : nullptr);
      bool all = false;
#pragma unroll 1
      for (int i = 0; i < steps && !all; i += kStep) {
        const uint2 quad = list_quad(lists, i);
#pragma unroll
        for (int k = 0; k < kStep; ++k) {
          // Branch-free: a skipped (or finished) pixel takes alpha = 0, which
          // leaves T and C bit-for-bit unchanged.
          const uint32_t off = quad_off(quad, k);
          const Entry& en = entry_at(s_e, off);
          const float4 ra = en.a, rb = en.b;
          const float blue = en.c.x;
          float2 d;
          const float q = entry_q(ra, rb, npix, d);
          const bool vis = !done && q >= kQMin;
          const float alpha = vis ? fminf(kAlphaMax, ex2_approx(q)) : 0.f;
          // (T (1 - alpha), alpha T) in one packed multiply
          const float2 tw = __fmul2_rn(make_float2(T, T), make_float2(__fsub_rn(1.f, alpha), alpha));
          const bool stop = tw.x < kTMin;   // (never for alpha = 0: T is not below kTMin)
          const float w = stop ? 0.f : tw.y;
          C01 = __ffma2_rn(make_float2(rb.z, rb.w), make_float2(w, w), C01);
          C2 = __fmaf_rn(blue, w, C2);
          T = stop ? T : tw.x;
          stop_off = stop ? off : stop_off;
          if (kCount) {
            n_eval += (done || off == (uint32_t)(B * (int)sizeof(Entry))) ? 0u : 1u;
            n_comp += (vis && !stop) ? 1u : 0u;
          }
          done = done || stop;
        }
        all = __all_sync(0xffffffffu, done);
      }
      if (all) break;
    }
    if (stop_off != 0xffffffffu) walked = start - range.x + stop_off / (uint32_t)sizeof(Entry);
  }
  return FwdPixel{T, C01.x, C01.y, C2, walked, staged};
}

// The same for a short list, whose entries in `mask` the warp takes one by one.
__device__ __forceinline__ FwdPixel fwd_walk_short(const BlendArgs& a, float2 npix, uint2 range, bool inside,
                                                   Entry* s_e, uint32_t mask) {
  float T = 1.f, C2 = 0.f;
  float2 C01 = make_float2(0.f, 0.f);
  uint32_t walked = range.y - range.x;
  bool done = !inside;
  const Entry* e = short_entries(a, s_e);
  while (mask) {
    const int j = __ffs(mask) - 1;
    mask &= mask - 1u;
    const float4 ra = e[j].a, rb = e[j].b;
    const float blue = e[j].c.x;
    float2 d;
    const float q = entry_q(ra, rb, npix, d);
    const bool vis = !done && q >= kQMin;
    const float alpha = vis ? fminf(kAlphaMax, ex2_approx(q)) : 0.f;
    const float2 tw = __fmul2_rn(make_float2(T, T), make_float2(__fsub_rn(1.f, alpha), alpha));
    const bool stop = tw.x < kTMin;
    const float w = stop ? 0.f : tw.y;
    C01 = __ffma2_rn(make_float2(rb.z, rb.w), make_float2(w, w), C01);
    C2 = __fmaf_rn(blue, w, C2);
    T = stop ? T : tw.x;
    if (stop) walked = (uint32_t)j;
    done = done || stop;
  }
  return FwdPixel{T, C01.x, C01.y, C2, walked, true};
}

// Sum over the 32 pixels of a sub-block, rows first, then columns from the
// outermost bit in (an order that does not depend on how the pixels are dealt
// to the lanes; lane bits: half, row, row, column, column).
__device__ __forceinline__ float sub_block_sum(float v) {
#pragma unroll
  for (int o : {8, 4, 16, 2, 1}) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Forward blend of tile tw (tile_work) by the calling CTA.
template <bool kCount, bool kStore, bool kShort>
__device__ __forceinline__ void blend_fwd_tile(const BlendArgs& a, uint4 tw, float4* s_mem) {
  Entry* s_e = reinterpret_cast<Entry*>(s_mem);
  WalkLists* lists = reinterpret_cast<WalkLists*>(scratch_of(a, s_mem));
  __shared__ float s_red[16];

  const CamRec& cam = a.cams[tw.w];
  const uint32_t local = tw.x - (uint32_t)cam.tile_offset;
  const int2 pm = map_pixel(a, local % cam.tiles_x, local / cam.tiles_x, threadIdx.x >> 5);
  const bool inside = pm.x < cam.width && pm.y < cam.height;
  const float2 npix = neg_centre(pm);
  const uint2 range = make_uint2(tw.y, tw.z);
  const int lane = threadIdx.x & 31;

  uint32_t n_eval = 0, n_comp = 0, n_warp = 0;
  FwdPixel fp;
  if constexpr (kShort) fp = fwd_walk_short(a, npix, range, inside, s_e, load_short<false>(a, range, npix, s_e));
  else fp = fwd_walk<kCount>(a, npix, range, inside, s_e, lists[threadIdx.x >> 5], n_eval, n_comp, n_warp);
  float T = fp.T, C0 = fp.C0, C1 = fp.C1, C2 = fp.C2;
  const uint32_t walked = fp.walked;

  float l1 = 0.f;
  if (inside) {
    C0 = __fmaf_rn(T, a.bg[0], C0);
    C1 = __fmaf_rn(T, a.bg[1], C1);
    C2 = __fmaf_rn(T, a.bg[2], C2);
    const int64_t hw = (int64_t)cam.width * cam.height;
    const int64_t pix = (int64_t)pm.y * cam.width + pm.x;
    float* img = a.images + 3 * cam.pixel_base;
    img[pix] = C0;
    img[hw + pix] = C1;
    img[2 * hw + pix] = C2;
    if (kStore) a.nwalk[cam.pixel_base + pix] = walked;
    if (a.targets) {
      const float* tg = a.targets + 3 * cam.pixel_base + pix;
      float* gi = a.grad_images + 3 * cam.pixel_base + pix;
      const float d0 = C0 - tg[0], d1 = C1 - tg[hw], d2 = C2 - tg[2 * hw];
      gi[0] = d0 > 0.f ? a.inv_count : (d0 < 0.f ? -a.inv_count : 0.f);
      gi[hw] = d1 > 0.f ? a.inv_count : (d1 < 0.f ? -a.inv_count : 0.f);
      gi[2 * hw] = d2 > 0.f ? a.inv_count : (d2 < 0.f ? -a.inv_count : 0.f);
      l1 = fabsf(d0) + fabsf(d1) + fabsf(d2);
    }
  }
  if (kCount) {
    unsigned long long e = n_eval, c = n_comp;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, o);
      c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if (lane == 0) {
      atomicAdd(a.pair_counts, e);
      atomicAdd(a.pair_counts + 1, c);
      atomicAdd(a.pair_counts + 2, (unsigned long long)n_warp);
    }
  }
  if (a.targets) {
    l1 = sub_block_sum(l1);
    if (lane == 0) s_red[threadIdx.x >> 5] = l1;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) s += s_red[w];
      atomicAdd(a.loss, s * (double)a.inv_count);
    }
  }
}

__device__ __forceinline__ void red_add(float* addr, float x) {
  asm volatile("red.global.add.f32 [%0], %1;" ::"l"(addr), "f"(x) : "memory");
}

// Four consecutive floats (16-byte aligned) added in one vector reduction.
__device__ __forceinline__ void red_add4(float* addr, float x, float y, float z, float w) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(x), "f"(y), "f"(z), "f"(w)
               : "memory");
}

// Pass 2 over slots [0, k) of both halves.  null_off: offset of the null entry.
// kTwins: both halves' slots hold the same entries, whose sums are added before
// they go to global memory.
template <bool kTwins>
__device__ __forceinline__ void flush_slots(const BlendArgs& a, WarpScratch& ws, int k, const Entry* s_e, float2 npix,
                                            uint32_t null_off) {
  static_assert(kSlots == 8 && kBlkW == 4 && kSubH == 4, "two rows of a block per lane");
  __syncwarp();
  const int lane = threadIdx.x & 31;
  const int s = lane & (kSlots - 1);
  const int r = (lane >> 3) & 1;           // rows 2 r and 2 r + 1 of the block
  const int h = lane >> 4;
  const float2* row = ws.dqw[s] + (lane & ~7);
  const float4* pix = ws.pix + (lane & ~7) + (lane >> 3);
  float R1[2] = {0.f, 0.f}, R2[2] = {0.f, 0.f};
  float2 RG[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};   // (sum dq, sum dC2 w)
  float2 G01 = make_float2(0.f, 0.f);                              // (sum dC0 w, sum dC1 w)
#pragma unroll
  for (int p = 0; p < 2 * kBlkW; ++p) {
    const int y = p / kBlkW;
    const float2 v = row[p];
    const float4 dc = pix[p];   // (dC0, dC1, 1, dC2)
    const float cc = (float)(p % kBlkW) - 0.5f * (float)(kBlkW - 1);   // column about the centre
    R1[y] = fmaf(cc, v.x, R1[y]);
    R2[y] = fmaf(cc * cc, v.x, R2[y]);
    RG[y] = __ffma2_rn(make_float2(dc.z, dc.w), v, RG[y]);
    G01 = __ffma2_rn(make_float2(dc.x, dc.y), make_float2(v.y, v.y), G01);
  }
  const float ra = 2.f * (float)r - 0.5f * (float)(kSubH - 1), rb = ra + 1.f;   // rows about the centre
  // moments of dq in (c, r) about the centre: 1, c, r, c^2, c r, r^2; then dL/dC . w
  float m[9] = {RG[0].x + RG[1].x,
                R1[0] + R1[1],
                fmaf(ra, RG[0].x, rb * RG[1].x),
                R2[0] + R2[1],
                fmaf(ra, R1[0], rb * R1[1]),
                fmaf(ra * ra, RG[0].x, rb * rb * RG[1].x),
                G01.x,
                G01.y,
                RG[0].y + RG[1].y};
#pragma unroll
  for (int q = 0; q < 9; ++q) m[q] += __shfl_xor_sync(0xffffffffu, m[q], kSlots);
  const uint32_t off = reinterpret_cast<const uint16_t*>(ws.slot[h])[s];
  const bool mine = r == 0 && s < k && off != null_off;
  const uint32_t lanes = kTwins ? __ballot_sync(0xffffffffu, mine) : 0u;
  if (mine) {
    const Entry& en = entry_at(s_e, off);
    // dx = U - c, dy = V - r; the block's centre from this lane's pixel
    const float U = en.a.x + (npix.x + ((float)(lane & 3) - 0.5f * (float)(kBlkW - 1)));
    const float V = en.a.y + (npix.y + ((float)((lane >> 2) & 3) - 0.5f * (float)(kSubH - 1)));
    float g[9];
    g[0] = fmaf(U, m[0], -m[1]);                          // sum dq dx
    g[1] = fmaf(V, m[0], -m[2]);                          // sum dq dy
    g[2] = fmaf(U, fmaf(U, m[0], -2.f * m[1]), m[3]);     // sum dq dx^2
    g[3] = fmaf(U, fmaf(V, m[0], -m[2]), fmaf(-V, m[1], m[4]));   // sum dq dx dy
    g[4] = fmaf(V, fmaf(V, m[0], -2.f * m[2]), m[5]);     // sum dq dy^2
    g[5] = m[0];
    g[6] = m[6];
    g[7] = m[7];
    g[8] = m[8];
    if (kTwins) {
#pragma unroll
      for (int q = 0; q < 9; ++q) g[q] += __shfl_xor_sync(lanes, g[q], 16);
    }
    if (!kTwins || h == 0) {
      float* dst = a.grad_rec + (size_t)__float_as_uint(en.c.w) * 12;
      // a record is 48 bytes, 16-byte aligned: floats 0-3 and 4-7 as vectors
      red_add4(dst, g[0], g[1], g[2], g[3]);
      red_add4(dst + 4, g[4], g[5], g[6], g[7]);
      if (g[8] != 0.f) red_add(dst + 8, g[8]);
    }
  }
  __syncwarp();
}

// Backward replay of a tile's list for the calling thread's pixel, front to
// back (as the forward), accumulating the record gradients of every entry.
// kRecompute: re-derive the stop from the transmittance; otherwise the pixel
// walks `bound` entries.  staged (CTA-uniform): the whole list is already in
// shared memory (a single batch that the forward of the same CTA staged).
// kTwins (the kernels for sparse frames): a warp's two blocks walk the same list,
// and their sums go to global memory together.  In frames of few Gaussians over
// many tiles a warp's blocks reach much the same entries, and every record takes
// the sums of thousands of blocks, which bounds the kernel: 1,000 Gaussians of
// 5,600 tiles at 1408^2 blend_bwd 1,117 -> 597 us, fused 1,135 -> 813.  (Deciding
// it list by list gained nothing: 611 and 812.)
template <bool kRecompute, bool kTwins>
__device__ __forceinline__ void bwd_walk(const BlendArgs& a, float2 npix, uint2 range, bool inside, const float* Cf,
                                         const float* dC, uint32_t bound, bool staged, Entry* s_e, WarpScratch& ws) {
  const int B = a.batch;
  const int lane = threadIdx.x & 31;
  const uint32_t null_off = (uint32_t)(B * (int)sizeof(Entry));
  // dL/dalpha_i = sum_c dC_c (c_i T_i - S_c / (1 - alpha_i)) with S the colour
  // behind entry i, S_c = C_c - P_c (P the running front-to-back sum), so
  // sum_c dC_c S_c = D0 - Q with D0 = dC . C and Q = dC . P kept as a scalar.
  // (Carrying D0 - Q itself saves an instruction and a register, but its error
  // is larger: Q rounds much as C did, and the difference cancels that.)
  const float D0 = dC[0] * Cf[0] + dC[1] * Cf[1] + dC[2] * Cf[2];
  float T = 1.f, Q = 0.f;
  bool done = !inside;
  if (kRecompute || !inside) bound = inside ? 0xffffffffu : 0u;   // outside the image: an empty walk
  // (dC0, dC1, 1, dC2): pass 2 pairs the 1 with dq and dC2 with w
  ws.pix[lane + (lane >> 3)] = make_float4(dC[0], dC[1], 1.f, dC[2]);
  int k0 = 0;         // slots filled (warp-uniform, a multiple of kStep)

  for (uint32_t start = range.x; start < range.y; start += B) {
    // a staged list is already in shared memory (read-only): no CTA barrier
    if (!staged && __syncthreads_count(done) == (int)blockDim.x) break;
    const int cnt = (int)min((uint32_t)B, range.y - start);
    if (!staged) {
      load_batch(a, start, cnt, npix, s_e);
      __syncthreads();
    }
    if (__all_sync(0xffffffffu, done)) continue;
    // entries at offsets below lim of this batch lie within the pixel's walk
    const uint32_t lim = min((uint32_t)cnt, bound - min(bound, start - range.x)) * (uint32_t)sizeof(Entry);
    for (int c0 = 0; c0 < cnt; c0 += kChunk) {
      const int steps = fill_lists<kTwins>(warp_cull(a, s_e), B, c0, cnt, ws.lists);
      bool all = false;
#pragma unroll 1
      for (int i = 0; i < steps && !all; i += kStep) {
        const uint2 quad = list_quad(ws.lists, i);
        if ((lane & 15) == 0) ws.slot[lane >> 4][k0 / kStep] = quad;
        float2* slot = &ws.dqw[k0][lane];
        // the results wait in registers until all four are there: a store would
        // keep the next entry's loads from starting (668 -> 651 us at 300k / 8 x
        // 800^2)
        float2 res[kStep];
        uint32_t off = 0;
#pragma unroll
        for (int k = 0; k < kStep; ++k) {
          // Branch-free, as in the forward: alpha = 0 for a pixel that skips
          // the entry or is finished, which leaves T and Q unchanged and gives
          // zero dq and w.
          off = quad_off(quad, k);
          const Entry& en = entry_at(s_e, off);
          const float4 ra = en.a, rb = en.b;
          const float blue = en.c.x;
          float2 d;
          const float q = entry_q(ra, rb, npix, d);
          const bool vis = (kRecompute ? !done : off < lim) && q >= kQMin;
          const float e = ex2_approx(q);
          const float alpha = vis ? fminf(kAlphaMax, e) : 0.f;
          const float om = __fsub_rn(1.f, alpha);
          const float2 tw = __fmul2_rn(make_float2(T, T), make_float2(om, alpha));   // (T (1 - alpha), alpha T)
          const float test_T = tw.x;
          // stored walk: never a stop inside it, and alpha = 0 past it
          const bool stop = kRecompute && test_T < kTMin;
          const float w = stop ? 0.f : tw.y;
          const float G = dC[0] * rb.z + dC[1] * rb.w + dC[2] * blue;
          Q = fmaf(w, G, Q);   // now includes this entry: D0 - Q is behind it
          const float dLda = T * G - (D0 - Q) * rcp_approx(om);
          // dL/dq / ln 2 (the factor ln 2 of d 2^q / dq is applied by the
          // per-Gaussian backward); no gradient through the 0.99 clamp; alpha = 0
          // (skipped, off the walk) gives dq = 0
          const float dq = (!stop && e <= kAlphaMax) ? dLda * alpha : 0.f;
          T = stop ? T : test_T;
          if (kRecompute) done = done || stop;
          res[k] = make_float2(dq, w);
        }
#pragma unroll
        for (int k = 0; k < kStep; ++k) slot[k * 33] = res[k];
        k0 += kStep;
        if (k0 == kSlots) {
          flush_slots<kTwins>(a, ws, kSlots, s_e, npix, null_off);
          k0 = 0;
        }
        // (a padded list says nothing about the walk's end)
        all = __all_sync(0xffffffffu, kRecompute ? done : off >= lim && off != null_off);
      }
      if (all || __all_sync(0xffffffffu, kRecompute ? done : (uint32_t)(c0 + kChunk) * (uint32_t)sizeof(Entry) >= lim))
        break;
    }
    if (!kRecompute) done = done || start - range.x + cnt >= bound;
    if (k0) {   // the slots refer to this batch's shared-memory records
      flush_slots<kTwins>(a, ws, k0, s_e, npix, null_off);
      k0 = 0;
    }
  }
}

// The same for a short list, whose entries in `mask` the warp takes one by one,
// both of its blocks the same.
template <bool kRecompute>
__device__ __forceinline__ void bwd_walk_short(const BlendArgs& a, float2 npix, bool inside, const float* Cf,
                                               const float* dC, uint32_t bound, uint32_t mask, Entry* s_e,
                                               WarpScratch& ws) {
  const int lane = threadIdx.x & 31;
  const uint32_t first = (uint32_t)(short_entries(a, s_e) - s_e) * (uint32_t)sizeof(Entry);
  const float D0 = dC[0] * Cf[0] + dC[1] * Cf[1] + dC[2] * Cf[2];
  float T = 1.f, Q = 0.f;
  if (kRecompute || !inside) bound = inside ? 0xffffffffu : 0u;
  ws.pix[lane + (lane >> 3)] = make_float4(dC[0], dC[1], 1.f, dC[2]);
  int k = 0;   // slots filled
  while (mask) {
    const uint32_t j = (uint32_t)__ffs(mask) - 1u, off = first + j * (uint32_t)sizeof(Entry);
    mask &= mask - 1u;
    const Entry& en = entry_at(s_e, off);
    const float4 ra = en.a, rb = en.b;
    const float blue = en.c.x;
    float2 d;
    const float q = entry_q(ra, rb, npix, d);
    const bool vis = j < bound && q >= kQMin;
    const float e = ex2_approx(q);
    const float alpha = vis ? fminf(kAlphaMax, e) : 0.f;
    const float om = __fsub_rn(1.f, alpha);
    const float2 tw = __fmul2_rn(make_float2(T, T), make_float2(om, alpha));
    const bool stop = kRecompute && tw.x < kTMin;
    const float w = stop ? 0.f : tw.y;
    const float G = dC[0] * rb.z + dC[1] * rb.w + dC[2] * blue;
    Q = fmaf(w, G, Q);
    const float dLda = T * G - (D0 - Q) * rcp_approx(om);
    const float dq = (!stop && e <= kAlphaMax) ? dLda * alpha : 0.f;
    T = stop ? T : tw.x;
    if (stop) bound = 0u;
    ws.dqw[k][lane] = make_float2(dq, w);
    if ((lane & 15) == 0) reinterpret_cast<uint16_t*>(ws.slot[lane >> 4])[k] = (uint16_t)off;
    if (++k == kSlots) {
      flush_slots<true>(a, ws, kSlots, s_e, npix, 0xffffffffu);
      k = 0;
    }
  }
  if (k) flush_slots<true>(a, ws, k, s_e, npix, 0xffffffffu);
}

// Backward blend of tile tw by the calling CTA.  kRecompute: re-derive
// the stop from the transmittance (no per-pixel state); otherwise walk each
// pixel's stored number of entries.
template <bool kRecompute, bool kShort, bool kShorts>
__device__ __forceinline__ void blend_bwd_tile(const BlendArgs& a, uint4 tw, float4* s_mem) {
  const CamRec& cam = a.cams[tw.w];
  const uint32_t local = tw.x - (uint32_t)cam.tile_offset;
  const int2 pm = map_pixel(a, local % cam.tiles_x, local / cam.tiles_x, threadIdx.x >> 5);
  const bool inside = pm.x < cam.width && pm.y < cam.height;
  const float2 npix = neg_centre(pm);
  const uint2 range = make_uint2(tw.y, tw.z);

  float Cf[3] = {0.f, 0.f, 0.f}, dC[3] = {0.f, 0.f, 0.f};
  uint32_t bound = range.y - range.x;
  if (inside) {
    const int64_t hw = (int64_t)cam.width * cam.height;
    const int64_t pix = (int64_t)pm.y * cam.width + pm.x;
    const float* img = a.images_in + 3 * cam.pixel_base;
    const float* gi = a.grad_in + 3 * cam.pixel_base;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      Cf[ch] = img[ch * hw + pix];
      dC[ch] = gi[ch * hw + pix];
    }
    if (!kRecompute) bound = a.nwalk[cam.pixel_base + pix];
  }
  WarpScratch* ws = reinterpret_cast<WarpScratch*>(scratch_of(a, s_mem));
  Entry* s_e = reinterpret_cast<Entry*>(s_mem);
  if constexpr (kShort) {
    const uint32_t mask = load_short<true>(a, range, npix, s_e);
    bwd_walk_short<kRecompute>(a, npix, inside, Cf, dC, bound, mask, s_e, ws[threadIdx.x >> 5]);
  } else {
    bwd_walk<kRecompute, kShorts>(a, npix, range, inside, Cf, dC, bound, false, s_e, ws[threadIdx.x >> 5]);
  }
}

// Forward blend, fused L1 loss and backward blend of tile tw by the calling
// CTA, for the training step whose loss is the L1 term (section
// 4.4): each pixel's dL/dC = sign(C - target) / M is known as soon as its
// forward walk ends, so the backward replay follows in the same CTA with C,
// dL/dC and the walk length in registers, and a list that fitted in one
// batch is replayed from the shared memory the forward filled, each warp
// starting its backward as soon as its own forward ends (the loss partials
// are summed after the backward, at the CTA's only barrier past the load).
// Images,
// dL/dC, loss and record gradients equal those of raster_fwd followed by
// blend_bwd in stored-walk mode, bit for bit up to the order of the atomic
// additions.
template <bool kShort, bool kShorts>
__device__ __forceinline__ void blend_fused_tile(const BlendArgs& a, uint4 tw, float4* s_mem) {
  Entry* s_e = reinterpret_cast<Entry*>(s_mem);
  __shared__ float s_red[16];

  const CamRec& cam = a.cams[tw.w];
  const uint32_t local = tw.x - (uint32_t)cam.tile_offset;
  const int2 pm = map_pixel(a, local % cam.tiles_x, local / cam.tiles_x, threadIdx.x >> 5);
  const bool inside = pm.x < cam.width && pm.y < cam.height;
  const float2 npix = neg_centre(pm);
  const uint2 range = make_uint2(tw.y, tw.z);
  const int lane = threadIdx.x & 31;

  WarpScratch& ws = reinterpret_cast<WarpScratch*>(scratch_of(a, s_mem))[threadIdx.x >> 5];
  uint32_t n_eval = 0, n_comp = 0, n_warp = 0;
  FwdPixel fp;
  uint32_t mask = 0u;
  if constexpr (kShort) {
    mask = load_short<true>(a, range, npix, s_e);
    fp = fwd_walk_short(a, npix, range, inside, s_e, mask);
  } else {
    fp = fwd_walk<false>(a, npix, range, inside, s_e, ws.lists, n_eval, n_comp, n_warp);
  }
  float Cf[3] = {0.f, 0.f, 0.f}, dC[3] = {0.f, 0.f, 0.f};
  float l1 = 0.f;
  if (inside) {
    Cf[0] = __fmaf_rn(fp.T, a.bg[0], fp.C0);
    Cf[1] = __fmaf_rn(fp.T, a.bg[1], fp.C1);
    Cf[2] = __fmaf_rn(fp.T, a.bg[2], fp.C2);
    const int64_t hw = (int64_t)cam.width * cam.height;
    const int64_t pix = (int64_t)pm.y * cam.width + pm.x;
    float* img = a.images + 3 * cam.pixel_base;
    const float* tg = a.targets + 3 * cam.pixel_base + pix;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      img[ch * hw + pix] = Cf[ch];
      const float d = Cf[ch] - tg[ch * hw];
      dC[ch] = d > 0.f ? a.inv_count : (d < 0.f ? -a.inv_count : 0.f);
      l1 += fabsf(d);
    }
    if (a.grad_images) {
      float* gi = a.grad_images + 3 * cam.pixel_base + pix;
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) gi[ch * hw] = dC[ch];
    }
    if (a.nwalk) a.nwalk[cam.pixel_base + pix] = fp.walked;
  }
  l1 = sub_block_sum(l1);
  if (lane == 0) s_red[threadIdx.x >> 5] = l1;
  __syncwarp();
  if constexpr (kShort) bwd_walk_short<false>(a, npix, inside, Cf, dC, fp.walked, mask, s_e, ws);
  else bwd_walk<false, kShorts>(a, npix, range, inside, Cf, dC, fp.walked, fp.staged, s_e, ws);
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) sum += s_red[w];
    atomicAdd(a.loss, sum * (double)a.inv_count);
  }
}

// Register budgets of the kernels that run the backward walk (swept on the
// 300k / 8 x 800^2 frame).
#ifndef SIXDGS_FUSED_MAXNREG
#define SIXDGS_FUSED_MAXNREG 64
#endif
#ifndef SIXDGS_BWD_MAXNREG
#define SIXDGS_BWD_MAXNREG 64
#endif
// Tiles without a list, one per warp from order[first] on: the background, and
// with targets its loss and dL/dC (the same sums as the blends' own).
template <bool kStore>
__device__ __forceinline__ void blend_empty(const BlendArgs& a, uint32_t first) {
  __shared__ double s_loss[16];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double loss = 0.0;
  if (first + warp < a.total_tiles) {
    const uint4 tw = a.order[first + warp];
    const CamRec& cam = a.cams[tw.w];
    const uint32_t local = tw.x - (uint32_t)cam.tile_offset;
    const int tx = local % cam.tiles_x, ty = local / cam.tiles_x;
    const int64_t hw = (int64_t)cam.width * cam.height;
    float* img = a.images + 3 * cam.pixel_base;
#pragma unroll 4
    for (int b = 0; b < (int)blockDim.x / 32; ++b) {
      const int2 pm = map_pixel(a, tx, ty, b);
      const int64_t pix = (int64_t)pm.y * cam.width + pm.x;
      float l1 = 0.f;
      if (pm.x < cam.width && pm.y < cam.height) {
        if (kStore) a.nwalk[cam.pixel_base + pix] = 0u;
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
          img[ch * hw + pix] = a.bg[ch];
          if (a.targets) {
            const float d = a.bg[ch] - a.targets[3 * cam.pixel_base + ch * hw + pix];
            if (a.grad_images)
              a.grad_images[3 * cam.pixel_base + ch * hw + pix] =
                  d > 0.f ? a.inv_count : (d < 0.f ? -a.inv_count : 0.f);
            l1 += fabsf(d);
          }
        }
      }
      if (a.targets) loss += sub_block_sum(l1);
    }
  }
  if (!a.targets) return;
  if (lane == 0) s_loss[warp] = loss * (double)a.inv_count;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) sum += s_loss[w];
    atomicAdd(a.loss, sum);
  }
}

template <bool kValue>
struct Bool {
  static constexpr bool value = kValue;
};

// Work unit u of a blend launch.  Tiles are taken in the binning's order,
// longest lists first, so that the launch does not end on a few CTAs that
// started a long list late (917 -> 858 us for the fused kernel at 300k / 8 x
// 800^2, 68 -> 52 us for the forward of one 1408^2 view of 175k Gaussians).
// The tiles without a list, 70% of that frame's, come last, one per warp of a
// CTA: a CTA each spent most of its time waiting for a handful of loads.  With
// that, the one-load tile record and the asynchronous staging of a batch
// (load_batch): fused kernel 722 -> 663 us at 300k / 8 x 800^2, forward 600 ->
// 536 us for 20 views of 183k Gaussians at 1024^2.
// tile(tw, short): a tile with a list, which is a short one or not.
template <bool kShorts, typename Tile, typename Empty>
__device__ __forceinline__ bool blend_unit(const BlendArgs& a, uint32_t u, Tile tile, Empty empty) {
  const uint4 tw = a.order[min(u, a.total_tiles - 1)];
  const uint32_t busy = min(*a.n_busy, a.total_tiles);
  if (u < busy) {
    if (tw.x < (kShorts ? a.frame_tiles : a.total_tiles)) {
      if constexpr (kShorts) {
        if (tw.z - tw.y > (uint32_t)a.short_list) tile(tw, Bool<false>{});
        else tile(tw, Bool<true>{});
      } else {
        tile(tw, Bool<false>{});
      }
    }
    return true;
  }
  const uint32_t first = busy + (u - busy) * (blockDim.x / 32);
  if (first >= a.total_tiles) return false;
  empty(first);
  return true;
}

template <bool kShorts, typename Tile, typename Empty>
__device__ __forceinline__ void for_each_blend_tile(const BlendArgs& a, Tile tile, Empty empty) {
  after_previous();
  if (!a.tile_queue) {
    blend_unit<kShorts>(a, blockIdx.x, tile, empty);
    return;
  }
  __shared__ uint32_t s_next;
  while (true) {
    if (threadIdx.x == 0) s_next = atomicAdd(a.tile_queue, 1u);
    __syncthreads();
    const uint32_t next = s_next;
    if (!blend_unit<kShorts>(a, next, tile, empty)) break;
    __syncthreads();
  }
}

template <bool kShorts>
__global__ void __maxnreg__(SIXDGS_FUSED_MAXNREG) blend_fused_kernel(BlendArgs a) {
  extern __shared__ float4 s_mem[];
  for_each_blend_tile<kShorts>(
      a, [&](uint4 tw, auto s) { blend_fused_tile<decltype(s)::value, kShorts>(a, tw, s_mem); },
      [&](uint32_t first) {
        if (a.nwalk) blend_empty<true>(a, first);
        else blend_empty<false>(a, first);
      });
}

// One CTA per tile (grid = tiles), or persistent: a grid of as many CTAs as
// fit on the GPU at once, each taking tiles from a device counter until all
// cameras' tiles are done.
template <bool kCount, bool kStore, bool kShorts>
// (the forward's registers: 64 / 48 / 40 give 617 / 599 / 606 us for 20 views of
// 183k Gaussians at 1024^2)
#ifndef SIXDGS_FWD_MAXNREG
#define SIXDGS_FWD_MAXNREG 48
#endif
__global__ void __maxnreg__(SIXDGS_FWD_MAXNREG) blend_fwd_kernel(BlendArgs a) {
  extern __shared__ float4 s_mem[];
  for_each_blend_tile<kShorts>(
      a, [&](uint4 tw, auto s) { blend_fwd_tile<kCount, kStore, decltype(s)::value>(a, tw, s_mem); },
      [&](uint32_t first) { blend_empty<kStore>(a, first); });
}

template <bool kRecompute, bool kShorts>
__global__ void __maxnreg__(SIXDGS_BWD_MAXNREG) blend_bwd_kernel(BlendArgs a) {
  extern __shared__ float4 s_mem[];
  for_each_blend_tile<kShorts>(
      a, [&](uint4 tw, auto s) { blend_bwd_tile<kRecompute, decltype(s)::value, kShorts>(a, tw, s_mem); }, [](uint32_t) {});
}

// Batches near or above 48 KB of shared memory (with the kernels' static
// shared memory) need the opt-in limit.
static void allow_smem(const void* fn, int bytes) {
  if (bytes > 40 * 1024) cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

// CTAs of `fn` resident on the whole GPU at once (the persistent grid).
static int resident_grid(const void* fn, int threads, int smem, int64_t tiles) {
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
  const int64_t g = (int64_t)std::max(per_sm, 1) * std::max(sms, 1);
  return (int)std::min<int64_t>(g, tiles);
}

// Frames with fewer (view, Gaussian) pairs a tile than this, whose lists are
// short or their records few, take kernels compiled with the two paths for them
// (kShorts); the other kernels are compiled without, as the paths cost registers
// (fused 652 instead of 648 us at 300k / 8 x 800^2).  With / without them, fused and
// forward us: 2.4 pairs a tile (4 views of 10,000 volume Gaussians at 1024^2) 136 /
// 146 and 53 / 57; 4.9: 153 / 161 and 59 / 64; 7.7 (60,000 of a shell at 1408^2):
// 70.3 / 70.6 and 28.6 / 30.7; 15.5: 93.8 / 92.8 and 38.9 / 38.9; 24: 240 / 241 and
// 90 / 92; 52: 213 / 211 and 80 / 80.
constexpr uint32_t kSparsePairs = 8;
static bool sparse(const BlendArgs& a) {
  return a.n_pairs / kSparsePairs < a.total_tiles || a.total_tiles != a.frame_tiles;   // (a band of a frame: always)
}

// scratch: the backward walk's per-warp shared memory (the forward: lists only)
template <typename K>
static void launch_blend(K kernel, BlendArgs a, int64_t total_tiles, bool scratch, cudaStream_t stream) {
  const int threads = a.tile_w * a.tile_h;
  // two warps a CTA: the staging area bounds the CTAs per SM (8 at a batch of 512),
  // and short lists need little of it
  if (threads == 64 && sparse(a)) a.batch = std::min(a.batch, 256);
  a.short_list = short_list(a.batch, threads / 32);
  const int smem = stage_bytes(a.batch, threads / (kBlkW * kSubH)) + threads / 32 * (int)(scratch ? sizeof(WarpScratch) : sizeof(WalkLists));
  allow_smem((const void*)kernel, smem);
  if (a.tile_queue) {
    cudaMemsetAsync(a.tile_queue, 0, sizeof(uint32_t), stream);
    const int grid = resident_grid((const void*)kernel, threads, smem, total_tiles);
    launch_after(kernel, grid, threads, smem, 1, stream, a);
  } else {
    launch_after(kernel, (unsigned)total_tiles, threads, smem, 1, stream, a);
  }
}

void launch_blend_fwd(const BlendArgs& a, int64_t total_tiles, cudaStream_t stream) {
  if (total_tiles == 0) return;
  if (a.pair_counts) {   // counts the general walk's pairs in any frame
    if (a.nwalk) launch_blend(blend_fwd_kernel<true, true, false>, a, total_tiles, false, stream);
    else launch_blend(blend_fwd_kernel<true, false, false>, a, total_tiles, false, stream);
  } else if (sparse(a)) {
    if (a.nwalk) launch_blend(blend_fwd_kernel<false, true, true>, a, total_tiles, false, stream);
    else launch_blend(blend_fwd_kernel<false, false, true>, a, total_tiles, false, stream);
  } else {
    if (a.nwalk) launch_blend(blend_fwd_kernel<false, true, false>, a, total_tiles, false, stream);
    else launch_blend(blend_fwd_kernel<false, false, false>, a, total_tiles, false, stream);
  }
}

void launch_blend_fused(const BlendArgs& a, int64_t total_tiles, cudaStream_t stream) {
  if (total_tiles == 0) return;
  if (sparse(a)) launch_blend(blend_fused_kernel<true>, a, total_tiles, true, stream);
  else launch_blend(blend_fused_kernel<false>, a, total_tiles, true, stream);
}

void launch_blend_bwd(const BlendArgs& a, int64_t total_tiles, cudaStream_t stream) {
  if (total_tiles == 0) return;
  if (sparse(a)) {
    if (a.recompute) launch_blend(blend_bwd_kernel<true, true>, a, total_tiles, true, stream);
    else launch_blend(blend_bwd_kernel<false, true>, a, total_tiles, true, stream);
  } else {
    if (a.recompute) launch_blend(blend_bwd_kernel<true, false>, a, total_tiles, true, stream);
    else launch_blend(blend_bwd_kernel<false, false>, a, total_tiles, true, stream);
  }
}

}  // namespace sixdgs
