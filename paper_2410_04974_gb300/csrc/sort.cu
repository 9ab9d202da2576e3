// Stage 2: per-tile lists of (view, Gaussian) pairs ordered by depth (the
// 3DGS duplicate/sort step kept by 6DGS section 4.4).
//
// The composite order (global tile, depth, Gaussian id) is built tile first:
//   1. the projection counts every tile's duplicates and queues its visible
//      pairs (project.cu);
//   2. bin_scan_kernel    -- exclusive scan of the counts: every tile's range
//                            (single pass, decoupled look-back) and the
//                            number of tiles of every list-length class;
//   3. bin_scatter_kernel -- every duplicate (depth, pair) to the next free
//                            place of its tile's range, and the order of the
//                            tiles, longest lists first;
//   4. bin_sort_kernel    -- every tile's entries sorted on chip by (depth,
//                            pair).
// The entries of a tile are distinct and all of one view, whose pair index
// grows with the Gaussian id, so sorting (depth, pair) gives the stable
// (depth, id) order whatever order the scatter's atomics left.
//
// Why not radix passes over all duplicates: those moved every duplicate once
// per digit and needed a dozen dependent launches (compaction, four depth
// passes, two scans and an expansion, two or three tile passes, ranges).
// Tile first, a duplicate is written once, read once and written sorted, in
// three launches.  Measured (sum of the kernels; radix -> tile first):
//   300k / 8 x 800^2 (2.5 M duplicates)     206 -> 85 us
//   2M / 4 x 1920x1080 (3.4 M)              236 -> 96 us
//   500k / 64 mixed views (29 M)           1907 -> 900 us
//   one view, 54 k duplicates                74 -> 28 us
// (the projection, which counts the tiles, takes 83 -> 99 us at 300k).
#include <algorithm>

#include "bin.cuh"
#include "common.cuh"
#include "kernels.cuh"
#include "stage.cuh"

namespace sixdgs {

constexpr int kBinThreads = 256;
constexpr int kBinWarps = kBinThreads / 32;
constexpr int kCluster = 8;               // CTAs that share one very long list
constexpr int kClasses = 64;

constexpr unsigned long long kScanAgg = 1ull << 62;
constexpr unsigned long long kScanInc = 2ull << 62;
constexpr unsigned long long kScanValMask = (1ull << 62) - 1;

__device__ __forceinline__ unsigned long long ld_volatile64(const unsigned long long* p) {
  return *reinterpret_cast<const volatile unsigned long long*>(p);
}
__device__ __forceinline__ void st_volatile64(unsigned long long* p, unsigned long long v) {
  *reinterpret_cast<volatile unsigned long long*>(p) = v;
}

// Exclusive block scan of one value per thread; returns the thread's prefix
// and the block total through `total`.  s_warp needs THREADS/32 + 1 words.
// T: wide enough for the total.
template <int THREADS, typename T>
__device__ __forceinline__ T block_excl_scan(T v, T& total, T* s_warp) {
  constexpr int WARPS = THREADS / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    T w = lane < WARPS ? s_warp[lane] : (T)0;
    T wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T y = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += y;
    }
    if (lane < WARPS) s_warp[lane] = wi - w;
    if (lane == WARPS - 1) s_warp[WARPS] = wi;
  }
  __syncthreads();
  total = s_warp[WARPS];
  T r = s_warp[warp] + incl - v;
  __syncthreads();
  return r;
}

// Decoupled look-back over 64-bit scan state (Merrill and Garland, 2016), run
// by one full warp.  Publishes this block's aggregate, waits for the
// predecessors and publishes the inclusive prefix.  Returns the exclusive
// prefix.  The wait is bounded by a clock budget; on expiry the status word
// gets SIXDGS_ERR_TIMEOUT and the callers carry on with clamped ranges.
// first: the words of the 32 blocks before, one per lane, as scan_ahead read
// them before the block's own counts, so that a block whose predecessors are
// long done does not wait for them a second time.
__device__ __forceinline__ unsigned long long scan_ahead(const unsigned long long* state, uint32_t tile) {
  const long long idx = (long long)tile - 1 - (threadIdx.x & 31);
  return idx >= 0 ? ld_volatile64(&state[idx]) : kScanInc;
}
__device__ unsigned long long scan_lookback(unsigned long long* state, uint32_t tile,
                                            unsigned long long block_total, unsigned long long first,
                                            int64_t budget, int32_t* status) {
  const int lane = threadIdx.x & 31;
  if (tile == 0) {
    if (lane == 0) st_volatile64(&state[0], kScanInc | block_total);
    return 0;
  }
  if (lane == 0) st_volatile64(&state[tile], kScanAgg | block_total);
  unsigned long long excl = 0;
  long long p = (long long)tile - 1;
  const long long t0 = clock64();
  bool timed_out = false;
  unsigned long long w = first;
  while (true) {
    uint32_t flag = (uint32_t)(w >> 62);
    uint32_t inc = __ballot_sync(0xffffffffu, flag == 2u);
    uint32_t not_ready = __ballot_sync(0xffffffffu, flag == 0u);
    int i_inc = inc ? __ffs(inc) - 1 : 32;
    uint32_t need = i_inc >= 31 ? 0xffffffffu : ((2u << i_inc) - 1u);
    if (not_ready & need) {
      bool expired = __shfl_sync(0xffffffffu, (clock64() - t0) > budget, 0);
      if (expired) {
        timed_out = true;
        break;
      }
      const long long idx = p - lane;
      w = idx >= 0 ? ld_volatile64(&state[idx]) : kScanInc;
      continue;
    }
    unsigned long long val = (lane <= i_inc) ? (w & kScanValMask) : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) val += __shfl_xor_sync(0xffffffffu, val, o);
    excl += val;
    if (i_inc < 32) break;
    p -= 32;
    const long long idx = p - lane;
    w = idx >= 0 ? ld_volatile64(&state[idx]) : kScanInc;
  }
  if (lane == 0) {
    if (timed_out) raise_status(status, SIXDGS_ERR_TIMEOUT);
    st_volatile64(&state[tile], kScanInc | ((excl + block_total) & kScanValMask));
  }
  return excl;
}

// Class of a list length: 0 for an empty list, else four classes per power of
// two of len - 1: lists of up to 2^p entries (p >= 1) have classes up to 4 p,
// longer ones classes from 4 p + 1 (the last class takes the rest).
__device__ __forceinline__ uint32_t length_class(uint32_t len) {
  if (len == 0u) return 0u;
  const uint32_t m = len - 1u;
  const uint32_t l = m ? 31u - __clz(m) : 0u;
  const uint32_t frac = l >= 2u ? (m >> (l - 2u)) & 3u : (l == 1u ? (m & 1u) * 2u : 0u);
  return min(1u + 4u * l + frac, (uint32_t)kClasses - 1u);
}

// Adds this block's tiles to per-class counters in shared memory; returns the
// tile's rank within its class and block.  Called by the whole block, tiles
// past the end with valid = false.  Empty lists (most of a frame that shows
// an object) are counted by ballot, not by colliding atomics.
__device__ __forceinline__ uint32_t count_class(uint32_t cls, bool valid, uint32_t* s_class) {
  const int lane = threadIdx.x & 31;
  const uint32_t empty = __ballot_sync(0xffffffffu, valid && cls == 0u);
  uint32_t base = 0;
  if (lane == 0 && empty) base = atomicAdd(&s_class[0], (uint32_t)__popc(empty));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (!valid) return 0u;
  if (cls == 0u) return base + __popc(empty & ((1u << lane) - 1u));
  return atomicAdd(&s_class[cls], 1u);
}

// --------------------------------------------------------------------------
// Ranges of the tiles' lists
// --------------------------------------------------------------------------
// Latency-bound (T x 4 bytes in, T x 12 out).  One tile per thread, so that a
// frame of a few thousand tiles is spread over several SMs.
// A block waits for those of lower numbers.  A grid of at most one block per SM
// (eight fit) is on the chip as a whole, also beside the scans of other streams,
// so that no block waits for one that cannot start, whatever order the hardware
// starts them in; a larger grid takes its numbers as tickets, so that the blocks
// waited for have started.  (Tickets for every frame: the round trip of one
// atomic, 0.8 us of 90 for 175k Gaussians at 1408^2, 1.2 of 47 for 6,660.)
__global__ void __launch_bounds__(kBinThreads) bin_scan_kernel(BinArgs a) {
  after_previous();
  __shared__ unsigned long long s_warp[kBinWarps + 1];
  __shared__ uint32_t s_class[kClasses];
  __shared__ unsigned long long s_excl;
  __shared__ uint32_t s_block;
  const int tid = threadIdx.x;
  if (tid < kClasses) s_class[tid] = 0u;
  uint32_t block = blockIdx.x;
  if (a.scan_tickets) {
    if (tid == 0) s_block = atomicAdd(&a.state[kBinTicket], 1u);
    __syncthreads();
    block = s_block;
    if (block >= gridDim.x) return;   // never after a projection, which clears the ticket
  }
  const uint32_t t = block * kScanTile + tid;
  const bool valid = t < a.total_tiles;
  const unsigned long long ahead = tid < 32 ? scan_ahead(a.scan_state, block) : 0ull;
  const uint32_t cnt = valid ? a.tile[t].count : 0u;
  // duplicates of the bands before, whose lists come first
  unsigned long long* base = reinterpret_cast<unsigned long long*>(a.state + kBinBase);
  const unsigned long long before = a.band > 0 ? base[a.band & 1] : 0ull;
  // 64 bits: a block's tiles may hold 2^32 duplicates or more (16.8 million
  // Gaussians on each), which the capacity check has to see
  unsigned long long total;
  const unsigned long long excl = block_excl_scan<kBinThreads>((unsigned long long)cnt, total, s_warp);
  if (tid < 32) {
    const unsigned long long e = scan_lookback(a.scan_state, block, total, ahead, a.spin_budget, a.status);
    if (tid == 0) s_excl = e;
  }
  // counters of the kernels that follow; the pair counters behind the first two
  // public words are the blend's
  if (block == 0 && tid < 10) a.counts[2 + tid] = 0u;
  if (block == 0 && tid == 10) a.counts[0] = 0u;
  if (block == 0 && tid == 11) a.state[kBinQueue] = 0u;
  __syncthreads();
  // lists beyond the duplicate capacity are cut there (and reported below)
  const unsigned long long off = before + s_excl + excl;
  const uint32_t start = (uint32_t)min(off, (unsigned long long)a.capacity);
  const uint32_t end = (uint32_t)min(off + cnt, (unsigned long long)a.capacity);
  if (valid) {
    a.tile[t].cursor = start;
    a.ranges[t] = end > start ? make_uint2(start, end) : make_uint2(0u, 0u);
  }
  count_class(length_class(end - start), valid, s_class);
  __syncthreads();
  if (tid < kClasses && s_class[tid]) atomicAdd(&a.state[kBinClass + tid], s_class[tid]);
  if (block == gridDim.x - 1 && tid == 0) {
    const unsigned long long k = before + s_excl + total;
    if (a.band >= 0) base[(a.band + 1) & 1] = k;
    a.counts[1] = (uint32_t)min(k, 0xffffffffull);
    if (k > a.capacity) raise_status(a.status, SIXDGS_ERR_CAPACITY);
  }
}

// --------------------------------------------------------------------------
// Duplicates to their tiles, and the tile order
// --------------------------------------------------------------------------
// A CTA takes a segment of the visible queue, 256 entries at a time (where there
// are fewer segments than CTAs, a part of one), and
// spreads their duplicates over its threads whatever the rectangles' sizes:
// duplicate o goes to thread o % 128, which finds its entry by a binary search
// of the entries' prefix sums in shared memory.  Bound by L2 requests (one
// atomic and one 8-byte store a duplicate, at random places), so the atomics
// are issued by full warps, kScatterBatch a thread in flight.  (A thread that
// walks its own entry's duplicates needs neither search nor barrier, but more
// and emptier atomic instructions: 60 instead of 51 us at 300k / 8 x 800^2.)
constexpr int kScatterThreads = 128;
static_assert(kScatterEntries == 2 * kScatterThreads, "two entries a thread");
constexpr int kScatterBatch = 4;
template <bool kCount>
__device__ __forceinline__ void scatter(const BinArgs& a) {
  after_previous();
  constexpr int kWarps = kScatterThreads / 32;
  __shared__ uint32_t s_class[kClasses], s_base[kClasses], s_longer[kClasses];
  __shared__ uint32_t s_warp[kWarps + 1];
  __shared__ uint32_t s_incl[kScatterEntries];   // inclusive prefix of the entries' tile counts
  __shared__ uint4 s_entry[kScatterEntries];     // (first tile, tiles_x << 16 | width, pair, depth)
  __shared__ uint32_t s_vis;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_vis = 0u;
  if (!kCount && blockIdx.x >= a.scatter_grid) {
    // these CTAs build the tile order: longest class first, any order within a
    // class (it decides when a tile is worked on, never a result)
    if (warp == 0) {   // tiles of longer classes: a suffix sum over the 64 classes
      const uint32_t c0 = a.state[kBinClass + lane], c1 = a.state[kBinClass + 32 + lane];
      uint32_t x0 = c0, x1 = c1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y0 = __shfl_down_sync(0xffffffffu, x0, o), y1 = __shfl_down_sync(0xffffffffu, x1, o);
        if (lane + o < 32) {
          x0 += y0;
          x1 += y1;
        }
      }
      const uint32_t high = __shfl_sync(0xffffffffu, x1, 0);
      s_longer[lane] = x0 - c0 + high;
      s_longer[32 + lane] = x1 - c1;
    }
    if (tid < kClasses) s_class[tid] = 0u;
    const uint32_t t = (blockIdx.x - a.scatter_grid) * kScatterThreads + tid;
    const bool valid = t < a.total_tiles;
    const uint2 r = valid ? a.ranges[t] : make_uint2(0u, 0u);
    const uint32_t cam = valid ? (uint32_t)find_camera(a.cams, a.n_cams, a.tile_first + t) : 0u;
    __syncthreads();
    const uint32_t cls = length_class(r.y - r.x);
    const uint32_t rank = count_class(cls, valid, s_class);
    __syncthreads();
    if (tid < kClasses && s_class[tid])
      s_base[tid] = s_longer[tid] + atomicAdd(&a.state[kBinCursor + tid], s_class[tid]);
    __syncthreads();
    if (valid) {
      const uint32_t at = s_base[cls] + rank;
      if (at < a.total_tiles) a.order[at] = tile_work(a.tile_first + t, r, cam);
    }
    if (blockIdx.x == a.scatter_grid) {
      // tiles with lists above the sort's limits: those of the classes beyond
      if (tid <= kBinLevels) a.state[kBinOver + tid] = s_longer[tid == 0 ? 4 * 14 : tid < kBinLevels ? 4 * (13 - tid) : 0];
    }
    // the scan is over: its words are clean for the next call
    if (tid == 0 && t % kScanTile == 0) a.scan_state[t / kScanTile] = 0ull;
    if (t == 0) a.state[kBinTicket] = 0u;
    return;
  }

  uint32_t visible = 0;
  const uint32_t step = a.scatter_step, stride = step * a.scatter_split;
  for (uint32_t w = blockIdx.x; w < a.segments * a.scatter_split; w += a.scatter_grid) {
    const uint32_t seg = w / a.scatter_split;
    const uint32_t count = min(a.vis_count[seg], a.segment_size);
    const uint4* vis = a.vis + vis_base(seg, a.n, a.n_cams, a.views);
    for (uint32_t c0 = (w - seg * a.scatter_split) * step; c0 < count; c0 += stride) {
      uint4 e[2];
      uint32_t nt[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t i = c0 + 2 * tid + h;
        e[h] = 2 * tid + h < step && i < count ? vis[i] : make_uint4(0u, 0u, 0u, 0u);
        nt[h] = ((e[h].z >> 16) - (e[h].z & 0xffffu)) * ((e[h].w >> 16) - (e[h].w & 0xffffu));
        if (kCount && a.band < 0 && nt[h] <= kBigRect) nt[h] = 0u;   // the projection counted them
      }
      uint32_t total;
      const uint32_t excl = block_excl_scan<kScatterThreads>(nt[0] + nt[1], total, s_warp);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        s_incl[2 * tid + h] = excl + nt[0] + (h ? nt[1] : 0u);
        if (nt[h]) {
          ++visible;
          const CamRec& cam = a.cams[e[h].x / a.n];
          const uint32_t x0 = e[h].z & 0xffffu, y0 = e[h].w & 0xffffu;
          s_entry[2 * tid + h] = make_uint4((uint32_t)cam.tile_offset + y0 * (uint32_t)cam.tiles_x + x0,
                                            ((uint32_t)cam.tiles_x << 16) | ((e[h].z >> 16) - x0), e[h].x, e[h].y);
        }
      }
      __syncthreads();
      for (uint32_t o0 = tid; o0 < total; o0 += kScatterThreads * kScatterBatch) {
        uint32_t pos[kScatterBatch];
        uint64_t key[kScatterBatch];
#pragma unroll
        for (int k = 0; k < kScatterBatch; ++k) {
          const uint32_t o = o0 + k * kScatterThreads;
          pos[k] = 0xffffffffu;
          if (o < total) {
            uint32_t l = 0;   // entries whose duplicates all come before o
#pragma unroll
            for (uint32_t s = kScatterEntries / 2; s > 0; s >>= 1)
              if (s_incl[l + s - 1] <= o) l += s;
            const uint4 en = s_entry[l];
            const uint32_t w = en.y & 0xffffu;
            const uint32_t local = o - (l ? s_incl[l - 1] : 0u);
            const uint32_t row = rect_row(local, w);
            const uint32_t tile = en.x + row * (en.y >> 16) + (local - row * w) - a.tile_first;
            key[k] = ((uint64_t)en.w << 32) | en.z;
            if (tile < a.total_tiles) {
              if constexpr (kCount) atomicAdd(&a.tile[tile].count, 1u);
              else pos[k] = atomicAdd(&a.tile[tile].cursor, 1u);
            }
          }
        }
#pragma unroll
        for (int k = 0; k < kScatterBatch; ++k)
          if (!kCount && pos[k] < a.capacity) a.dup[pos[k]] = key[k];
      }
      __syncthreads();
    }
  }
  if (kCount) return;
  visible = __reduce_add_sync(0xffffffffu, visible);
  if (lane == 0 && visible) atomicAdd(&s_vis, visible);
  __syncthreads();
  if (tid == 0 && s_vis) atomicAdd(&a.counts[0], s_vis);
}

__global__ void __launch_bounds__(kScatterThreads) bin_scatter_kernel(BinArgs a) { scatter<false>(a); }
// The counts of the rectangles that the projection left: large ones
// (defer_big_rects), or, for a band of a frame, all.
__global__ void __launch_bounds__(kScatterThreads) bin_count_kernel(BinArgs a) { scatter<true>(a); }

// --------------------------------------------------------------------------
// Sort of one tile's entries
// --------------------------------------------------------------------------
// A team of kWarps warps sorts up to 32 kItems kWarps entries, kItems (2 to 16)
// a thread, with bitonic networks (Batcher, 1968) in registers: element i of
// the network is item i % kItems of thread i / kItems, so that strides below
// kItems stay in a thread, strides below 32 kItems are shuffles and only
// longer ones go through shared memory.  What bounds it is integer
// instructions, so
//   * the network runs on 32-bit keys: the depth above the list's smallest,
//     without the low bits that do not fit, over the entry's place in the
//     unsorted list;
//   * the keys of a thread whose run is to descend are complemented, so that
//     every comparison of a run is ascending (two instructions, no selects).
// Entries that agree in that much depth (equal depths, or neighbours in a long
// list) may come out in the wrong order.  Then, and only then, the full
// (depth, pair) keys are laid out in that order in shared memory and odd-even
// transposition rounds put the few displaced neighbours right; a list with
// many equal depths, still not in order after kFixRounds, is sorted by its
// 64-bit keys.
constexpr int kFixRounds = 8;
constexpr int kMaxItems = 16;

template <int kWarps>
__device__ __forceinline__ void team_sync(uint32_t team) {
  __syncwarp();
  if (kWarps > 1) asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(32 * kWarps) : "memory");
}

// Is `flag` set in any thread of the team?  (Also a team barrier.)
template <int kWarps>
__device__ __forceinline__ bool team_any(uint32_t team, bool flag) {
  __syncwarp();
  if (kWarps == 1) return __any_sync(0xffffffffu, flag);
  uint32_t any;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %3, 0;\n barrier.cta.red.or.pred.aligned q, %1, %2, p;\n"
      " selp.u32 %0, 1, 0, q;\n}"
      : "=r"(any)
      : "r"(team + 1), "r"(32 * kWarps), "r"((uint32_t)flag)
      : "memory");
  return any != 0u;
}

__device__ __forceinline__ void order_pair(uint32_t& x, uint32_t& y) {
  const uint32_t lo = min(x, y);
  y = max(x, y);
  x = lo;
}
__device__ __forceinline__ void order_pair(uint64_t& x, uint64_t& y) {
  const bool swap = x > y;
  const uint64_t lo = swap ? y : x;
  y = swap ? x : y;
  x = lo;
}

template <int kItems, typename Key>
__device__ __forceinline__ void flip(Key (&key)[kItems], bool on) {
  const Key m = on ? ~(Key)0 : (Key)0;
#pragma unroll
  for (int i = 0; i < kItems; ++i) key[i] ^= m;
}

template <int kItems, typename Key>
__device__ __forceinline__ void merge_in_thread(Key (&key)[kItems]) {
#pragma unroll
  for (int j = kItems / 2; j > 0; j >>= 1)
#pragma unroll
    for (int i = 0; i < kItems; ++i)
      if (!(i & j)) order_pair(key[i], key[i | j]);
}

// Sorts the team's 32 kItems kWarps keys.  tid: thread of the team; s_x: 4
// keys a thread for the strides across warps (unused by one warp).
template <int kItems, int kWarps, typename Key>
__device__ __forceinline__ void bitonic_sort(Key (&key)[kItems], uint32_t team, uint32_t tid, Key* s_x) {
  constexpr uint32_t kThreads = 32 * kWarps;
#pragma unroll
  for (int k = 2; k < kItems; k <<= 1)
#pragma unroll
    for (int j = k / 2; j > 0; j >>= 1)
#pragma unroll
      for (int i = 0; i < kItems; ++i)
        if (!(i & j)) {
          if ((i & k) == 0) order_pair(key[i], key[i | j]);
          else order_pair(key[i | j], key[i]);
        }
  bool down = (tid & 1u) != 0u;   // the thread's run descends: its keys are complemented
  flip(key, down);
  merge_in_thread(key);
#pragma unroll 1
  for (uint32_t k = 2; k <= kThreads; k <<= 1) {   // in threads: runs of k kItems elements
    const bool next = (tid & k) != 0u;
    flip(key, down != next);
    down = next;
#pragma unroll 1
    for (uint32_t m = k >> 1; m > 0u; m >>= 1) {
      const bool lower = (tid & m) == 0u;   // of the two threads, the one that keeps the smaller keys
      if (kWarps > 1 && m >= 32u) {
#pragma unroll
        for (int i0 = 0; i0 < kItems; i0 += 4) {
          team_sync<kWarps>(team);
#pragma unroll
          for (int i = 0; i < 4; ++i) s_x[i * kThreads + tid] = key[i0 + i];
          team_sync<kWarps>(team);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const Key other = s_x[i * kThreads + (tid ^ m)];
            key[i0 + i] = ((key[i0 + i] < other) == lower) ? key[i0 + i] : other;
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
          const Key other = __shfl_xor_sync(0xffffffffu, key[i], m);
          key[i] = ((key[i] < other) == lower) ? key[i] : other;
        }
      }
    }
    merge_in_thread(key);
  }
  team_sync<kWarps>(team);
}

// Place of element e in a team's shared memory: one word of padding a thread,
// so that neither thread-order writes nor consecutive reads collide.
template <int kItems>
__device__ __forceinline__ uint32_t padded(uint32_t e) {
  return e + e / kItems;
}
constexpr uint32_t kTeamWords = 512 + 512 / kMaxItems;   // 64-bit words of shared memory per warp

// The list src[0, len) in order in s (padded()).
template <int kItems, int kWarps>
__device__ __noinline__ void sort_full(const uint64_t* src, uint32_t len, uint32_t team, uint32_t tid, uint64_t* s) {
  constexpr uint32_t kThreads = 32 * kWarps;
  uint64_t key[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i) key[i] = i * kThreads + tid < len ? src[i * kThreads + tid] : ~0ull;
  team_sync<kWarps>(team);
  bitonic_sort<kItems, kWarps>(key, team, tid, s);
#pragma unroll
  for (int i = 0; i < kItems; ++i) s[padded<kItems>(tid * kItems + i)] = key[i];
  team_sync<kWarps>(team);
}

// The same for a list almost in order: place e holds entry at[e] of src.
template <int kItems, int kWarps>
__device__ __noinline__ void fix_order(const uint64_t* src, uint32_t len, uint32_t team, uint32_t tid, uint64_t* s,
                                       const uint32_t* s_at) {
  constexpr uint32_t kThreads = 32 * kWarps;
  uint32_t at[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i) at[i] = s_at[padded<kItems>(tid * kItems + i)];
  team_sync<kWarps>(team);
#pragma unroll
  for (int i = 0; i < kItems; ++i)
    if (tid * kItems + i < len) s[padded<kItems>(tid * kItems + i)] = src[at[i]];
  for (int round = 0;; ++round) {
    bool moved = false;
#pragma unroll
    for (uint32_t odd = 0; odd < 2; ++odd) {   // e and e + 1 of even, then of odd e
      team_sync<kWarps>(team);
      for (uint32_t e = 2 * tid + odd; e + 1 < len; e += 2 * kThreads) {
        const uint64_t x = s[padded<kItems>(e)], y = s[padded<kItems>(e + 1)];
        if (x > y) {
          s[padded<kItems>(e)] = y;
          s[padded<kItems>(e + 1)] = x;
          moved = true;
        }
      }
    }
    if (!team_any<kWarps>(team, moved)) break;
    if (round == kFixRounds) {
      sort_full<kItems, kWarps>(src, len, team, tid, s);
      break;
    }
  }
}

// Sorts src[0, len), len <= 32 kItems kWarps, and calls store(e, full) for
// the team's elements e < len in order, consecutive threads for consecutive
// e: full() gives the element's (depth, pair) key.
template <int kItems, int kWarps, typename Store>
__device__ __forceinline__ void sort_team(const uint64_t* src, uint32_t len, uint32_t team, uint32_t tid, uint64_t* s,
                                          Store store) {
  constexpr uint32_t kThreads = 32 * kWarps, kCap = kThreads * kItems;
  constexpr int kBits = 5 + (kItems >= 2) + (kItems >= 4) + (kItems >= 8) + (kItems >= 16) + (kWarps >= 2) +
                        (kWarps >= 4) + (kWarps >= 8);   // log2(kCap)
  uint32_t key[kItems];
  uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t e = i * kThreads + tid;
    key[i] = e < len ? (uint32_t)(src[e] >> 32) : 0u;
    if (e < len) {
      lo = min(lo, key[i]);
      hi = max(hi, key[i]);
    }
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  uint32_t* s_w = reinterpret_cast<uint32_t*>(s);
  if (kWarps > 1) {
    if ((tid & 31u) == 0u) {
      s_w[tid >> 4] = lo;
      s_w[(tid >> 4) + 1] = hi;
    }
    team_sync<kWarps>(team);
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      lo = min(lo, s_w[2 * w]);
      hi = max(hi, s_w[2 * w + 1]);
    }
  }
  const int shift = max(kBits - __clz(hi - lo), 0);   // __clz(0) = 32
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t e = i * kThreads + tid;
    key[i] = e < len ? (((key[i] - lo) >> shift) << kBits) | e : 0xffffffffu;
  }
  bitonic_sort<kItems, kWarps>(key, team, tid, s_w);
  bool tie = false;
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t e = tid * kItems + i;
    s_w[padded<kItems>(e)] = key[i] & (kCap - 1u);
    if (i > 0) tie = tie || ((key[i] ^ key[i - 1]) < kCap && e < len);
  }
  // a tie across two threads: the neighbour's last key
  uint32_t last = __shfl_up_sync(0xffffffffu, key[kItems - 1], 1);
  if (kWarps > 1) {
    uint32_t* s_last = s_w + kCap + kCap / kItems;
    if ((tid & 31u) == 31u) s_last[tid >> 5] = key[kItems - 1];
    team_sync<kWarps>(team);
    if ((tid & 31u) == 0u && tid) last = s_last[(tid >> 5) - 1];
  }
  tie = tie || (tid && (key[0] ^ last) < kCap && tid * kItems < len);
  if (team_any<kWarps>(team, tie)) {
    fix_order<kItems, kWarps>(src, len, team, tid, s, s_w);
    for (uint32_t e = tid; e < len; e += kThreads) store(e, [&]() { return s[padded<kItems>(e)]; });
  } else {
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const uint32_t e = i * kThreads + tid;
      if (e < len) store(e, [&]() { return src[s_w[padded<kItems>(e)]]; });
    }
  }
}

// Sorted lists of the CTA's teams: one tile each.
template <int kItems, int kWarps>
__device__ __forceinline__ void sort_tile(const BinArgs& a, uint32_t tile, uint32_t start, uint32_t len,
                                          uint64_t* s_key) {
  const uint32_t team = threadIdx.x / (32 * kWarps), tid = threadIdx.x % (32 * kWarps);
  sort_team<kItems, kWarps>(a.dup + start, len, team, tid, s_key + team * kWarps * kTeamWords,
                            [&](uint32_t e, auto full) {
                              a.sorted[start + e] = (uint32_t)full();
                              a.sorted_key[start + e] = tile;
                            });
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// A list of more than kRun entries: runs of kRun sorted on chip, then merged
// pairwise, each entry finding its rank in the sibling run by a binary search
// (kMergeBatch of them in flight per thread).  The merges go back and forth
// between dup and the (sorted_key, sorted) arrays, which hold a key in two
// words.  By one CTA for up to kAlone entries, so that as many lists are worked
// on as CTAs fit; above, where few lists hold a frame up, by a cluster.  (All
// of them by clusters, of whose eight CTAs two had a run to sort: the kernel
// took 775 instead of 458 us at 500k / 64 mixed views.)
constexpr uint32_t kRun = kMaxItems * kBinThreads;
constexpr uint32_t kAlone = 4 * kRun;
constexpr int kMergeBatch = 4;

template <bool kByCluster>
__device__ __noinline__ void sort_long(const BinArgs& a, uint32_t start, uint32_t len, uint32_t tile, uint64_t* s) {
  const uint32_t rank = kByCluster ? cluster_rank() : 0u;
  constexpr uint32_t kRanks = kByCluster ? kCluster : 1;
  constexpr uint32_t kStride = kRanks * kBinThreads;
  auto sync = [&]() {
    if (kByCluster) cluster_sync();
    else __syncthreads();
  };
  uint64_t* A = a.dup + start;
  uint32_t* hi = a.sorted_key + start;
  uint32_t* lo = a.sorted + start;
  for (uint32_t r = rank * kRun; r < len; r += kRanks * kRun) {
    const uint32_t m = min(kRun, len - r);
    // (the run goes to the other arrays: its entries are still read here)
    sort_team<kMaxItems, kBinWarps>(A + r, m, 0u, threadIdx.x, s, [&](uint32_t e, auto full) {
      const uint64_t k = full();
      hi[r + e] = (uint32_t)(k >> 32);
      lo[r + e] = (uint32_t)k;
    });
    __syncthreads();
  }
  sync();
  bool in_a = false;
  for (uint32_t w = kRun; w < len; w *= 2) {
    const bool last = w >= (len + 1) / 2;
    auto load = [&](uint32_t i) -> uint64_t {
      return in_a ? __ldcg(A + i) : ((uint64_t)__ldcg(hi + i) << 32) | __ldcg(lo + i);
    };
    for (uint32_t i0 = rank * kBinThreads + threadIdx.x; i0 < len; i0 += kMergeBatch * kStride) {
      uint64_t x[kMergeBatch];
      uint32_t s0[kMergeBatch], n[kMergeBatch], l[kMergeBatch];   // sibling run, entries of it below x
#pragma unroll
      for (int k = 0; k < kMergeBatch; ++k) {
        const uint32_t i = min(i0 + k * kStride, len - 1u);
        x[k] = load(i);
        s0[k] = min((i / w ^ 1u) * w, len);
        n[k] = min(w, len - s0[k]);
        l[k] = 0u;
      }
      for (uint32_t step = w; step > 0u; step >>= 1) {
#pragma unroll
        for (int k = 0; k < kMergeBatch; ++k)
          if (l[k] + step <= n[k] && load(s0[k] + l[k] + step - 1u) < x[k]) l[k] += step;
      }
#pragma unroll
      for (int k = 0; k < kMergeBatch; ++k) {
        const uint32_t i = i0 + k * kStride;
        if (i < len) {
          const uint32_t run = i / w;
          const uint32_t out = min((run & ~1u) * w + (i - run * w) + l[k], len - 1u);
          if (in_a) {
            hi[out] = last ? tile : (uint32_t)(x[k] >> 32);
            lo[out] = (uint32_t)x[k];
          } else {
            A[out] = x[k];
          }
        }
      }
    }
    in_a = !in_a;
    sync();
  }
  if (in_a) {
    for (uint32_t i = rank * kBinThreads + threadIdx.x; i < len; i += kStride) {
      lo[i] = (uint32_t)__ldcg(A + i);
      hi[i] = tile;
    }
  }
}

__global__ void __launch_bounds__(kBinThreads, 4) bin_sort_kernel(BinArgs a) {
  after_previous();
  __shared__ uint64_t s_key[kBinWarps * kTeamWords];
  __shared__ uint32_t s_unit;
  const int tid = threadIdx.x;
  // order: over[0] tiles with lists above kAlone entries, up to over[1] those
  // above 4096, over[2] 2048, over[3] 1024, over[4] 512, over[5] the rest that
  // are not empty
  uint32_t over[kBinLevels + 1];
  over[kBinLevels] = min(a.state[kBinOver + kBinLevels], a.total_tiles);
#pragma unroll
  for (int l = kBinLevels - 1; l >= 0; --l) over[l] = min(a.state[kBinOver + l], over[l + 1]);
  if (blockIdx.x == 0 && tid < 2 * kClasses) a.state[kBinClass + tid] = 0u;   // clean for the next call
  for (uint32_t u = blockIdx.x / kCluster; u < over[0]; u += gridDim.x / kCluster) {
    const uint4 w = a.order[u];
    sort_long<true>(a, w.y, w.z - w.y, w.x, s_key);
    cluster_sync();
  }
  // units of the rest: one, two, four or eight tiles a CTA
  const uint32_t u1 = over[2] - over[0], u2 = u1 + (over[3] - over[2] + 1) / 2, u4 = u2 + (over[4] - over[3] + 3) / 4;
  const uint32_t units = u4 + (over[5] - over[4] + 7) / 8;
  while (true) {
    __syncthreads();
    if (tid == 0) s_unit = atomicAdd(&a.state[kBinQueue], 1u);
    __syncthreads();
    const uint32_t u = s_unit;
    if (u >= units) break;
    uint32_t at, end, teams;
    if (u < u1) at = over[0] + u, end = over[2], teams = 1;
    else if (u < u2) at = over[2] + 2 * (u - u1), end = over[3], teams = 2;
    else if (u < u4) at = over[3] + 4 * (u - u2), end = over[4], teams = 4;
    else at = over[4] + 8 * (u - u4), end = over[5], teams = 8;
    at += threadIdx.x / (kBinThreads / teams);
    const uint4 w = at < end ? a.order[at] : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t len = teams == 1 ? min(w.z - w.y, kAlone) : min(w.z - w.y, kRun / teams);
    if (len == 0u) continue;   // (the whole team)
    if (len > kRun) sort_long<false>(a, w.y, len, w.x, s_key);
    else if (teams == 1) sort_tile<16, 8>(a, w.x, w.y, len, s_key);
    else if (teams == 2) sort_tile<16, 4>(a, w.x, w.y, len, s_key);
    else if (teams == 4) sort_tile<16, 2>(a, w.x, w.y, len, s_key);
    else if (len > 256u) sort_tile<16, 1>(a, w.x, w.y, len, s_key);
    else if (len > 128u) sort_tile<8, 1>(a, w.x, w.y, len, s_key);
    else if (len > 64u) sort_tile<4, 1>(a, w.x, w.y, len, s_key);
    else sort_tile<2, 1>(a, w.x, w.y, len, s_key);
  }
}

// Grids: the scan has one block per 256 tiles; the scatter at most 16 CTAs per
// SM, each with the segments of its stride, and one per 128 tiles for the order;
// the sort, which takes its tiles from a queue, a whole number of clusters, at
// most 4 CTAs per SM.
static void share_segments(BinArgs& a, int sms) {
  const ScatterShare s = scatter_share(a.segments, a.segment_size, a.total_tiles, sms);
  a.scatter_grid = s.grid;
  a.scatter_split = s.split;
  a.scatter_step = s.step;
}

cudaError_t launch_bin_count(BinArgs a, int sms, cudaStream_t stream) {
  share_segments(a, sms);
  return launch_after(bin_count_kernel, a.scatter_grid, kScatterThreads, 0, 1, stream, a);
}

cudaError_t launch_bin(BinArgs a, int sms, cudaStream_t stream) {
  const uint32_t blocks = std::max(1u, (a.total_tiles + kScanTile - 1) / kScanTile);
  a.scan_tickets = blocks > (uint32_t)sms;
  cudaError_t e = launch_after(bin_scan_kernel, blocks, kBinThreads, 0, 1, stream, a);
  if (e != cudaSuccess) return e;
  share_segments(a, sms);
  const uint32_t order = std::max(1u, (a.total_tiles + kScatterThreads - 1) / kScatterThreads);
  e = launch_after(bin_scatter_kernel, a.scatter_grid + order, kScatterThreads, 0, 1, stream, a);
  if (e != cudaSuccess) return e;
  const uint32_t most = std::max(1u, (uint32_t)sms * 4u / kCluster);
  const uint32_t clusters = std::min(most, (std::max(a.total_tiles, 1u) + kCluster - 1) / kCluster);
  return launch_after(bin_sort_kernel, clusters * kCluster, kBinThreads, 0, kCluster, stream, a);
}

}  // namespace sixdgs
