// hist_batch.cu -- many histograms in one launch (Sec. III.B: small slices or
// packets batched into one call that returns many histograms).
//
// Two ways, for up to kBatchMaxImages images a launch.  With every image in the
// lane-private layout (the default), two chained launches (batch_few_kernel or
// batch_lane_kernel<true>, then batch_lane_kernel<false>): small images whole,
// by warps and groups of warps, the others in pieces.  With other layouts a
// memset of the outputs and batch_images_kernel, whose CTAs each count a
// contiguous range of the concatenated bytes, an equal share of the batch's
// cost (the bytes plus a fixed cost per image), and add what falls in it into
// the images' outputs at the image boundaries.  Neither needs scratch memory,
// so a batch captures into a CUDA graph as it is.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <chrono>
#include <vector>

#include "hist.h"
#include "hist_device.cuh"
#include "hist_internal.h"

using namespace histdev;
using namespace histlib;

namespace {

constexpr uint32_t kBatchMaxImages = HIST_BATCH_MAX_IMAGES;
// dynamic shared memory: the table, then the size prefix (u64 per image + 1)
constexpr size_t kBatchSmem = (size_t)kTableWords * 4 + (size_t)(kBatchMaxImages + 1) * 8;

constexpr uint32_t kPerWarp = HIST_LAYOUT_PER_WARP;

// The layout of an image: per regime (index 0 for every image when the
// launch has no regimes) a layout, and a second one below a size.
struct RegimeLayouts {
  uint32_t layout[HIST_REGIMES];
  uint32_t small_bytes[HIST_REGIMES];
  uint32_t small_layout[HIST_REGIMES];
};

struct BatchImgArgs {
  const uint8_t* const* ptrs;
  const size_t* sizes;
  uint32_t* out;
  const uint8_t* regime;  // per image, or null: every image takes entry 0
  uint32_t count;
  RegimeLayouts lay;
};

// Exclusive prefix of the image sizes into pre[0..count] (all threads).
__device__ void size_prefix(const size_t* sizes, uint32_t count, unsigned long long* pre) {
  __shared__ unsigned long long wsum[kWarps];
  const int t = threadIdx.x, nt = blockDim.x;
  const uint32_t per = (count + nt - 1) / nt;  // images per thread, consecutive
  const uint32_t b0 = t * per;
  unsigned long long local = 0;
  for (uint32_t i = 0; i < per && b0 + i < count; ++i) local += sizes[b0 + i];
  // inclusive scan of `local` over the block
  unsigned long long x = local;
  const int lane = t & 31, w = t >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  unsigned long long before = 0;
  for (int i = 0; i < w; ++i) before += wsum[i];
  unsigned long long run = before + x - local;  // exclusive start of this thread's images
  for (uint32_t i = 0; i < per && b0 + i < count; ++i) {
    pre[b0 + i] = run;
    run += sizes[b0 + i];
  }
  if (t == nt - 1) pre[count] = before + x;
  __syncthreads();
}

// The CTAs split the batch by cost: an image costs kImageCost before its
// bytes (its table reduction and output adds) plus one per byte, so a CTA
// whose range holds many small images takes fewer bytes.  The 4096-image
// batch (9.83 GB, one graph launch): 6.51 TB/s with no fixed cost, 6.63 at
// 32 KiB, 6.64 - 6.69 at 64 KiB, 6.65 at 128 KiB, 6.49 at 256 KiB.
constexpr unsigned long long kImageCost = 64ull << 10;

// The cut at cost position x, as a position in the concatenated bytes: the
// start of the image whose fixed cost holds x, else x's byte moved to a 32
// KiB boundary of its image's memory (split_point; not past the image's
// end).  Both CTAs of the cut compute it from the same x.
__device__ unsigned long long batch_cut(const BatchImgArgs& a, const unsigned long long* pre, unsigned long long x) {
  const unsigned long long W = pre[a.count] + (unsigned long long)a.count * kImageCost;
  if (x >= W) return pre[a.count];
  uint32_t i = 0, hi = a.count;  // the last image whose cost starts at or before x
  while (i + 1 < hi) {
    const uint32_t mid = (i + hi) >> 1;
    if (pre[mid] + (unsigned long long)mid * kImageCost <= x) i = mid;
    else hi = mid;
  }
  const unsigned long long c0 = pre[i] + (unsigned long long)i * kImageCost + kImageCost;
  const unsigned long long n = pre[i + 1] - pre[i];
  if (x <= c0) return pre[i];
  const unsigned long long c = split_point(a.ptrs[i], x - c0);
  return pre[i] + (c < n ? c : n);
}

template <int UNROLL, int MINB>
__global__ void __launch_bounds__(kThreads, MINB) batch_images_kernel(BatchImgArgs a) {
  extern __shared__ __align__(16) uint32_t smem[];
  uint32_t* table = smem;
  unsigned long long* pre = reinterpret_cast<unsigned long long*>(smem + kTableWords);
  __shared__ CtaShared cs;
  __shared__ uint32_t part[kThreads];

  zero_table(table);
  size_prefix(a.sizes, a.count, pre);
  const unsigned long long W = pre[a.count] + (unsigned long long)a.count * kImageCost;
  const unsigned long long lo0 = batch_cut(a, pre, W * blockIdx.x / gridDim.x);
  const unsigned long long hi = batch_cut(a, pre, W * (blockIdx.x + 1) / gridDim.x);
  if (lo0 >= hi) return;
  // first image whose bytes reach past lo0
  uint32_t lo_i = 0, hi_i = a.count;
  while (lo_i + 1 < hi_i) {
    const uint32_t mid = (lo_i + hi_i) >> 1;
    if (pre[mid] <= lo0) lo_i = mid;
    else hi_i = mid;
  }
  uint32_t i = lo_i;
  unsigned long long lo = lo0;
  while (lo < hi && i < a.count) {
    const unsigned long long img_end = pre[i + 1];
    if (img_end <= lo) {
      ++i;
      continue;
    }
    const unsigned long long seg_end = img_end < hi ? img_end : hi;
    const size_t off = (size_t)(lo - pre[i]);
    const size_t len = (size_t)(seg_end - lo);
    const uint8_t* base = a.ptrs[i] + off;
    const uint32_t r = a.regime ? a.regime[i] : 0u;
    // selects rather than an index, so the parameters stay out of local memory
    const uint32_t big = r == 0 ? a.lay.layout[0] : (r == 1 ? a.lay.layout[1] : a.lay.layout[2]);
    const uint32_t cut = r == 0 ? a.lay.small_bytes[0] : (r == 1 ? a.lay.small_bytes[1] : a.lay.small_bytes[2]);
    const uint32_t sml = r == 0 ? a.lay.small_layout[0] : (r == 1 ? a.lay.small_layout[1] : a.lay.small_layout[2]);
    const uint32_t lay = a.sizes[i] < cut ? sml : big;
    const int path = lay == kPerWarp ? PATH_PLAIN : PATH_SHIFT;
    const int lk = lay == kPerWarp ? 0 : (int)(lay > 5u ? 5u : lay);
    const Split sp = split_bytes(base, len);
    count_range_dispatch<UNROLL>(path, lk, reinterpret_cast<const uint4*>(base + sp.head), 0, sp.nvec, table,
                                 part, threadIdx.x, blockDim.x);
    // the pattern is not read for SHIFT or PLAIN
    const bool cleared = flush_table(path, lk, table, cs.pat, part, cs, true);
    count_edges(base, sp, cs);
    __syncthreads();
    if (threadIdx.x < HIST_BINS && cs.res[threadIdx.x])
      atomicAdd(a.out + (size_t)i * HIST_BINS + threadIdx.x, cs.res[threadIdx.x]);
    if (!cleared) {
      // clear the slots this layout used (the per-warp tables fill the table)
      const int words = path == PATH_PLAIN ? kTableWords : (HIST_BINS << lk);
      uint4* t4 = reinterpret_cast<uint4*>(table);
      for (int w = threadIdx.x; w < (words >> 2); w += blockDim.x) t4[w] = make_uint4(0, 0, 0, 0);
    }
    __syncthreads();
    lo = seg_end;
    ++i;
  }
}

// ------------------------------------------------ the lane-private kernels --
//
// A batch whose images are all counted in the lane-private table (layout 5,
// the default) is two launches of batch_lane_kernel, each of one CTA of 1024
// threads per SM, each CTA taking an equal share of the cost of the launch's
// images, a contiguous range of them placed end to end.
//
// The first launch counts whole images of at most kLaneSmall bytes: those of
// at most kLaneTiny by a warp each, in a 256-bin table of its own, the others
// by four groups of eight warps, an image at a time each, a thread per bin,
// in a lane-private table each.  It also clears the outputs of the other
// images.  The second launch counts those, piece by piece, the whole CTA on
// each, which has the start of the next piece fetched into L2 while it
// reduces the table; its CTAs start on the SMs that the first's leave and
// wait for it before they write.  With at most kBatchFew images the first
// launch is a light one (batch_few_kernel: a warp per image counts the tiny
// ones and clears the others' outputs) and the second counts all the rest:
// the groups' tables and ranges cost more than they bring for few images, and
// the second launch's CTAs find free SMs at once.  Two launches because the groups' tables
// (128 KiB) would take the L1 cache from the large images' loads (64 stream
// chunks of 16 MiB: 161 us with 80 KiB of shared memory, 176 with 146), and
// because one kernel with both loops spills registers.
//
// Bound by the HBM read on large images, by the prologue (sizes, two scans,
// the window's list: 3.5 us) and latency on small ones.  On the GPU, replayed
// from a graph, before (one CTA-wide loop over all images, two CTAs per SM)
// and now: 4096 images of 64 .. 4096 a side (9.97 GB) 1491 -> 1406 us (7.09
// TB/s), 464 of 314 .. 2303 (0.68 GB) 123 -> 112, 2048 of 16 .. 256 (29 MB)
// 38.8 -> 18.8, 4096 of 8 .. 22 51 -> 7.5 us.  Both launches are chained: the
// first clears its tables while the work before the call ends.

constexpr uint32_t kLaneGroups = 4;
constexpr int kLaneGroupThreads = kThreads / (int)kLaneGroups;
static_assert(kLaneGroupThreads == HIST_BINS, "one bin per thread of a group");
constexpr int kLaneWindow = 64;  // images of the range taken at a time
constexpr uint32_t kLanePer = kBatchMaxImages / kThreads;  // images per thread in the cost prefix
template <bool SMALL>
__host__ __device__ constexpr size_t lane_smem() {
  return (size_t)(SMALL ? kLaneGroups : 1u) * kTableWords * 4;
}

// Largest image a group counts whole.
constexpr uint32_t kLaneSmall = 128u << 10;
// Largest image a warp counts alone.  Its increments meet in banks (3.5
// wavefronts per 32 uniform pixels), but a lane-private table takes 512
// wavefronts to sum and clear: as many as 6.5 KB of uniform pixels, or more
// of peaked ones, lose to conflicts.
constexpr uint32_t kLaneTiny = 4u << 10;
constexpr int kTinyLoads = 2;  // vectors in flight per lane
// Fixed cost of an image beside its bytes: what a group or a CTA counts in
// the time of an image's reduction.
constexpr unsigned long long kLaneSmallCost = 24ull << 10;
template <bool SMALL>
__device__ __forceinline__ unsigned long long lane_cost(unsigned long long n) {
  return n + (SMALL ? kLaneSmallCost : kImageCost);
}

// Batches of at most so many images are of few images (batch_few_kernel).
// Both ways, us: 1 image of 8 .. 22 a side 2.7 (with the group launch 4.7),
// 26 of 36 .. 249 5.8 (8.1), 100 of 180 .. 948 12.2 (18.1), 300 of 20 .. 1686
// 24.3 (30.3), 1000 of 16 .. 256 14.0 (16.3), 1000 of 180 .. 948 58.6 (60.2);
// but 1500 of 36 .. 249 20.1 (19.7), 2048 of 16 .. 256 20.6 (19.1).
constexpr uint32_t kBatchFew = 1024;

struct LanePiece {
  const uint8_t* base;
  uint32_t len;
  uint32_t image;  // bit 31: the whole image
};
struct alignas(16) LaneItem {
  const uint4* body;
  uint32_t nvec;
  uint32_t image;
  uint32_t head, tail;
};

struct LaneArgs {
  const uint8_t* const* ptrs;
  const size_t* sizes;
  uint32_t* out;
  unsigned long long inv;  // floor((2^64 - 1) / grid)
  uint32_t count;
  bool few;  // every image that is not tiny is the second launch's
};

template <bool SMALL>
struct LaneShared {
  unsigned long long wsum[kWarps];
  unsigned long long lo, hi;    // the CTA's cost range
  unsigned long long share;     // the batch's bytes / grid
  unsigned long long next_pos;  // cost position of the next window's first image
  uint32_t i0;                  // the range's first image
  uint32_t n;                   // entries of the window's list, the tiny images' first
  uint32_t tiny;                // of them the tiny ones
  uint32_t wcount[2][2];
  LanePiece piece[SMALL ? 1 : kLaneWindow];
  LaneItem item[SMALL ? kLaneWindow : 1];
  uint32_t res[SMALL ? 1 : HIST_BINS];
  uint32_t eh[SMALL ? kLaneGroups : 1][HIST_BINS];  // edge bytes
};

// Whether an image of n bytes is the SMALL launch's: tiny, or at most
// kLaneSmall bytes and half of a CTA's share of the batch (with fewer bytes
// the images are better spread over the SMs in pieces: 26 images of 61 ..
// 2615 a side 16.6 us, 18.8 if each of at most a share is counted whole, and
// 2048 thumbnails 22.5 us if only those of a quarter are, 19.5 at half).
__device__ __forceinline__ bool lane_small(unsigned long long n, unsigned long long share) {
  return n <= kLaneTiny || (n <= kLaneSmall && n * 2 <= share);
}

// Inclusive block scan of v; the block's sum in `total` (one barrier; the
// caller puts one before wsum is written again).
__device__ __forceinline__ unsigned long long warp_scan(unsigned long long v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}
__device__ __forceinline__ unsigned long long block_scan(unsigned long long v, unsigned long long* wsum,
                                                         unsigned long long& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned long long x = warp_scan(v);
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  const unsigned long long s = warp_scan(wsum[lane]);  // kWarps == 32
  total = __shfl_sync(0xffffffffu, s, 31);
  const unsigned long long before = __shfl_sync(0xffffffffu, s, (w + 31) & 31);
  return (w ? before : 0ull) + x;
}
static_assert(kWarps == 32, "a lane per warp in block_scan");

// floor(x / grid) or a little less, for inv = floor((2^64 - 1) / grid): every
// CTA takes the same cuts from it, without the 64-bit division's 150
// instructions in 32 warps (2 us).
__device__ __forceinline__ unsigned long long grid_share(unsigned long long x, unsigned long long inv) {
  return __umul64hi(x, inv);
}

// The window of images from i0 on, whose first has cost position
// ls.next_pos: warps 0 and 1 (an image per lane) list what this CTA counts of
// them.  All threads call (barriers before and after are the caller's).
template <bool SMALL>
__device__ __forceinline__ void lane_window(const LaneArgs& a, uint32_t i0, LaneShared<SMALL>& ls) {
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  if (t >= kLaneWindow) return;
  const GroupBar<kLaneWindow> bar = {15};
  const uint32_t i = i0 + (uint32_t)t;
  const bool in = i < a.count;
  const unsigned long long n = in ? (unsigned long long)a.sizes[i] : 0ull;
  const uint8_t* p = in ? a.ptrs[i] : nullptr;
  const bool mine = n && lane_small(n, ls.share) == SMALL;
  const unsigned long long c = mine ? lane_cost<SMALL>(n) : 0ull;
  const unsigned long long x = warp_scan(c);
  const unsigned long long pos = ls.next_pos;
  if (lane == 31) ls.wsum[w] = x;
  bar.sync();
  const unsigned long long p0 = pos + (w ? ls.wsum[0] : 0ull) + x - c;
  unsigned long long b0 = 0, e0 = 0;
  if (mine && p0 < ls.hi) {
    if (SMALL) {
      // the range holding its first cost position counts it
      if (p0 >= ls.lo) e0 = n;
    } else {
      b0 = ls.lo > p0 ? split_point(p, ls.lo - p0) : 0ull;
      e0 = split_point(p, ls.hi - p0);
      if (e0 > n) e0 = n;
    }
  }
  const bool tiny = SMALL && b0 < e0 && n <= kLaneTiny, other = b0 < e0 && !tiny;
  const unsigned mt = __ballot_sync(0xffffffffu, tiny), mo = __ballot_sync(0xffffffffu, other);
  if (lane == 0) {
    ls.wcount[w][0] = __popc(mt);
    ls.wcount[w][1] = __popc(mo);
  }
  bar.sync();
  const uint32_t ntiny = ls.wcount[0][0] + ls.wcount[1][0];
  if (tiny || other) {
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t k = tiny ? (w ? ls.wcount[0][0] : 0u) + __popc(mt & lt)
                            : ntiny + (w ? ls.wcount[0][1] : 0u) + __popc(mo & lt);
    if (SMALL) {
      // (a warp's vectors need no whole lines)
      const Split sp = split_bytes_at(p, (size_t)n, tiny ? 16 : kLineBytes);
      LaneItem& q = ls.item[k];
      q.body = reinterpret_cast<const uint4*>(p + sp.head);
      q.nvec = (uint32_t)sp.nvec;
      q.image = i;
      q.head = (uint32_t)sp.head;
      q.tail = (uint32_t)sp.tail;
    } else {
      LanePiece& q = ls.piece[k];
      q.base = p + b0;
      q.len = (uint32_t)(e0 - b0);
      q.image = i | (b0 == 0 && e0 == n ? 1u << 31 : 0u);
    }
  }
  if (t == kLaneWindow - 1) {
    ls.next_pos = p0 + c;
    ls.tiny = ntiny;
    ls.n = ntiny + ls.wcount[0][1] + ls.wcount[1][1];
  }
}

// Count the window's pieces, the whole CTA, into the table (clear before and
// after).
__device__ __forceinline__ void lane_pieces(const LaneArgs& a, uint32_t* table, LaneShared<false>& ls) {
  const int t = threadIdx.x;
  for (uint32_t k = 0; k < ls.n; ++k) {
    piece_count(ls.piece[k].base, ls.piece[k].len, table, ls.eh[0], nullptr, nullptr);
    if (k + 1 < ls.n) {
      const uint32_t at = (uint32_t)t * kLineBytes;
      if (at < ls.piece[k + 1].len) asm volatile("prefetch.global.L2 [%0];" ::"l"(ls.piece[k + 1].base + at));
    }
    __syncthreads();
    lane_reduce<kThreads, true>(table, ls.res, t);
    __syncthreads();
    if (t < HIST_BINS) {
      const uint32_t h = ls.res[t] + ls.eh[0][t];
      ls.eh[0][t] = 0;
      if (k == 0) pdl_wait();  // the output is clear
      const uint32_t image = ls.piece[k].image;
      uint32_t* o = a.out + (size_t)(image & 0x7fffffffu) * HIST_BINS + t;
      if (image >> 31) *o = h;
      else if (h) atomicAdd(o, h);
    }
    __syncthreads();
  }
}

// Count an image of head bytes, nvec vectors and tail bytes with one warp, U
// vectors in flight per lane, into its 256 words h.
template <int U>
__device__ __forceinline__ void tiny_image(const uint4* body, uint32_t head, uint32_t nvec, uint32_t tail,
                                           uint32_t* h) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t edge = 0x100u;
  if (lane < head) edge = (reinterpret_cast<const uint8_t*>(body) - head)[lane];
  else if (lane - head < tail) edge = reinterpret_cast<const uint8_t*>(body + nvec)[lane - head];
  LaneRange r = lane_range(body, 0, nvec, (int)lane);
  uint4 v[U];
  lane_load<U, 32>(v, r);
  if (edge < 0x100u) atomicAdd(&h[edge], 1u);
  while (r.left) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      if ((uint32_t)(u * 32) < r.left) vec_count(v[u], h);
    r.q += U * 32;
    r.left = r.left > U * 32 ? r.left - U * 32 : 0u;
    lane_load<U, 32>(v, r);
  }
  __syncwarp();
}

// Count the window's tiny images, a warp each, in the warp's 256 words of the
// first table (clear before and after).
__device__ __forceinline__ void lane_tiny(const LaneArgs& a, uint32_t* tables, const LaneShared<true>& ls) {
  const uint32_t w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t* h = tables + w * HIST_BINS;
  for (uint32_t i = w; i < ls.tiny; i += kWarps) {
    const LaneItem& it = ls.item[i];
    tiny_image<kTinyLoads>(it.body, it.head, it.nvec, it.tail, h);
    uint32_t* out = a.out + (size_t)it.image * HIST_BINS;
#pragma unroll
    for (int k = 0; k < HIST_BINS / 32; ++k) {
      out[lane + 32 * k] = h[lane + 32 * k];
      h[lane + 32 * k] = 0;
    }
    __syncwarp();
  }
}

// Count the window's other images, a group each at a time (the tables clear
// before and after).
__device__ __forceinline__ void lane_items(const LaneArgs& a, uint32_t* tables, LaneShared<true>& ls) {
  const uint32_t g = threadIdx.x / kLaneGroupThreads;
  const int t = threadIdx.x % kLaneGroupThreads;
  const GroupBar<kLaneGroupThreads> bar = {1 + (int)g};
  uint32_t* table = tables + g * kTableWords;
  const uint32_t base = smem_addr(table) + ((t & 31) << 2);
  const uint32_t n = ls.n;
  uint32_t i = ls.tiny + g;
  if (i >= n) return;
  uint4 v[kLaneLoads];
  lane_load<kLaneLoads, kLaneGroupThreads>(v, lane_range(ls.item[i].body, 0, ls.item[i].nvec, t));
  auto edge_of = [&](const LaneItem& it) -> uint32_t {
    if ((uint32_t)t >= it.head + it.tail) return 0x100u;
    return (uint32_t)t < it.head ? *(reinterpret_cast<const uint8_t*>(it.body) - it.head + t)
                                 : reinterpret_cast<const uint8_t*>(it.body + it.nvec)[t - it.head];
  };
  uint32_t edge = edge_of(ls.item[i]);
  for (; i < n; i += kLaneGroups) {
    const LaneItem& it = ls.item[i];
    if (edge < 0x100u) atomicAdd(&ls.eh[g][edge], 1u);
    edge = 0x100u;
    LaneRange next = {nullptr, 0};
    if (i + kLaneGroups < n) {
      const LaneItem& it2 = ls.item[i + kLaneGroups];
      edge = edge_of(it2);
      next = lane_range(it2.body, 0, it2.nvec, t);
    }
    lane_count<kLaneLoads, kLaneGroupThreads>(v, lane_range(it.body, 0, it.nvec, t), base, next);
    bar.sync();
    uint32_t h = lane_row(table, t);
    if (it.head + it.tail) {
      h += ls.eh[g][t];
      ls.eh[g][t] = 0;
    }
    a.out[(size_t)it.image * HIST_BINS + t] = h;
    bar.sync();
  }
}

// The first launch of a batch of few images: a warp each, which counts a tiny
// one, all its vectors in flight, and clears the output of any other.  Bound
// by the chain of three reads (sizes, pointers, pixels).
constexpr int kFewWarps = 8;
__global__ void __launch_bounds__(kFewWarps * 32) batch_few_kernel(const __grid_constant__ LaneArgs a) {
  __shared__ uint32_t tables[kFewWarps][HIST_BINS];
  const uint32_t w = threadIdx.x >> 5, lane = threadIdx.x & 31, i = blockIdx.x * kFewWarps + w;
  uint32_t* h = tables[w];
#pragma unroll
  for (int k = 0; k < HIST_BINS / 32; ++k) h[lane + 32 * k] = 0;
  __syncwarp();
  pdl_wait();
  pdl_launch_dependents();
  if (i >= a.count) return;
  const unsigned long long n = a.sizes[i];
  if (n != 0 && n <= kLaneTiny) {
    const uint8_t* p = a.ptrs[i];
    const Split sp = split_bytes_at(p, (size_t)n, 16);
    tiny_image<kLaneTiny / (32 * 16)>(reinterpret_cast<const uint4*>(p + sp.head), (uint32_t)sp.head,
                                      (uint32_t)sp.nvec, (uint32_t)sp.tail, h);
  }
  uint32_t* out = a.out + (size_t)i * HIST_BINS;
#pragma unroll
  for (int k = 0; k < HIST_BINS / 32; ++k) out[lane + 32 * k] = h[lane + 32 * k];
}

template <bool SMALL>
__global__ void __launch_bounds__(kThreads, 1) batch_lane_kernel(const __grid_constant__ LaneArgs a) {
  extern __shared__ __align__(16) uint32_t tables[];
  __shared__ LaneShared<SMALL> ls;
  const int t = threadIdx.x;
  {
    uint4* t4 = reinterpret_cast<uint4*>(tables);
    for (int i = t; i < (int)(lane_smem<SMALL>() / 16); i += kThreads) t4[i] = make_uint4(0, 0, 0, 0);
  }
  if (t < (int)(sizeof(ls.eh) / 4)) (&ls.eh[0][0])[t] = 0;
  if (t == 0) ls.i0 = a.count;
  // the work before the call is complete from here on: it may have written
  // the arrays and the images, and the second launch reads both
  if (SMALL) pdl_wait();
  pdl_launch_dependents();
  // the batch's bytes: thread t holds images kLanePer t ...
  unsigned long long n[kLanePer], local = 0, total;
#pragma unroll
  for (uint32_t k = 0; k < kLanePer; ++k) {
    const uint32_t i = (uint32_t)t * kLanePer + k;
    n[k] = i < a.count ? (unsigned long long)a.sizes[i] : 0ull;
    local += n[k];
  }
  // one image per warp of the grid (the grid has at least kBatchMaxImages
  // warps: launch_batch_lane)
  const uint32_t zi = blockIdx.x * kWarps + ((uint32_t)t >> 5);
  const unsigned long long zsize = SMALL && zi < a.count ? (unsigned long long)a.sizes[zi] : 0ull;
  block_scan(local, ls.wsum, total);
  const unsigned long long share = a.few ? 0 : grid_share(total, a.inv);
  if (SMALL && zi < a.count && !(zsize && lane_small(zsize, share))) {
    // an output that is not this launch's to write
#pragma unroll
    for (int k = 0; k < HIST_BINS / 32; ++k) a.out[(size_t)zi * HIST_BINS + (t & 31) + 32 * k] = 0;
  }
  // this launch's images' costs, and the one that holds cost position lo
  local = 0;
#pragma unroll
  for (uint32_t k = 0; k < kLanePer; ++k) {
    n[k] = n[k] && lane_small(n[k], share) == SMALL ? lane_cost<SMALL>(n[k]) : 0ull;
    local += n[k];
  }
  if (!__syncthreads_or(local != 0)) {  // (and wsum is read)
    if (!SMALL) pdl_wait();  // the launch ends after the first
    return;
  }
  unsigned long long pos = block_scan(local, ls.wsum, total) - local;
  const unsigned long long lo = grid_share(total * blockIdx.x, a.inv);
  if (t == 0) {
    ls.lo = lo;
    ls.hi = blockIdx.x + 1 == gridDim.x ? total : grid_share(total * (blockIdx.x + 1), a.inv);
    ls.share = share;
  }
#pragma unroll
  for (uint32_t k = 0; k < kLanePer; ++k) {
    if (n[k] && pos <= lo && lo < pos + n[k]) {
      ls.i0 = (uint32_t)t * kLanePer + k;
      ls.next_pos = pos;
    }
    pos += n[k];
  }
  __syncthreads();
  for (uint32_t i0 = ls.i0; i0 < a.count; i0 += kLaneWindow) {
    lane_window<SMALL>(a, i0, ls);
    __syncthreads();
    const bool last = ls.next_pos >= ls.hi;
    if constexpr (SMALL) {
      if (ls.tiny) {
        lane_tiny(a, tables, ls);
        __syncthreads();
      }
      lane_items(a, tables, ls);
    } else {
      lane_pieces(a, tables, ls);
    }
    __syncthreads();  // the window's list is read
    if (last) break;
  }
  if (!SMALL) pdl_wait();  // (a CTA with nothing to write)
}

// The regime of image blockIdx.x (rule in hist.h): 256 threads; thread t
// takes run t of the sample (16 consecutive pixels from floor(t n / 256)), or
// pixels 16 t .. 16 t + 15 of an image of at most 4096 pixels, as the five
// words that hold them (byte by byte where one of the words is not all the
// image's), counts them in shared memory; then the largest bin and the sum of
// squares (below 2^25: m <= 4096).  With `after` the launch follows the
// batch's counting launches and fills the SMs as their CTAs end: they started
// after the work before the call was complete, and this one ends after them.
// Bound by latency (the arrays, the pixels, three barriers) and the shared
// atomics' conflicts.  With a byte load per pixel, before the counting
// launches, and now: the regimes call on 2227 images of 17 .. 375 a side 38.0
// -> 33.0 us (28.8 without regimes), on 300 of 64 .. 2000 45.0 -> 41.1 (41.1);
// words, but before the counting launches, 35.0 and 43.2.
__global__ void __launch_bounds__(HIST_BINS) regime_kernel(const uint8_t* const* ptrs, const size_t* sizes,
                                                           uint32_t theta, uint8_t* regime, bool after) {
  __shared__ uint32_t h[HIST_BINS];
  __shared__ uint32_t wmax[HIST_BINS / 32], wsq[HIST_BINS / 32];
  const int t = threadIdx.x;
  const uint32_t i = blockIdx.x;
  if (!after) pdl_wait();
  pdl_launch_dependents();
  const unsigned long long n = sizes[i];
  const uint8_t* x = ptrs[i];
  h[t] = 0;
  const bool runs = n > HIST_REGIME_SAMPLE;
  const unsigned long long start = runs ? ((unsigned long long)t * n) >> 8 : 16ull * (unsigned long long)t;
  const int len = start >= n ? 0 : n - start < 16 ? (int)(n - start) : 16;
  const uint8_t* p = x + start;
  const uint32_t off = (uint32_t)((uintptr_t)p & 3u);
  const bool whole = len == 16 && start >= off && start - off + 20 <= n;
  uint32_t v[5];
  if (whole) {
    const uint32_t* q = reinterpret_cast<const uint32_t*>(p - off);
#pragma unroll
    for (int u = 0; u < 5; ++u) v[u] = __ldg(q + u);
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = __funnelshift_r(v[u], v[u + 1], 8 * off);
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      v[u] = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (4 * u + k < len) v[u] |= (uint32_t)__ldg(p + 4 * u + k) << (8 * k);
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 16; ++u)
    if (u < len) atomicAdd(&h[(v[u >> 2] >> (8 * (u & 3))) & 0xffu], 1u);
  __syncthreads();
  const uint32_t c = h[t];
  const uint32_t mx = __reduce_max_sync(0xffffffffu, c);
  const uint32_t sq = __reduce_add_sync(0xffffffffu, c * c);
  if ((t & 31) == 0) {
    wmax[t >> 5] = mx;
    wsq[t >> 5] = sq;
  }
  __syncthreads();
  if (t == 0) {
    const unsigned long long m = n < HIST_REGIME_SAMPLE ? n : HIST_REGIME_SAMPLE;
    uint32_t M = 0, S = 0;
    for (int w = 0; w < HIST_BINS / 32; ++w) {
      M = wmax[w] > M ? wmax[w] : M;
      S += wsq[w];
    }
    uint8_t r = (uint8_t)HIST_REGIME_WIDE;
    if (m == 0) r = (uint8_t)HIST_REGIME_WIDE;
    else if ((unsigned long long)M * 1000ull >= (unsigned long long)theta * m) r = (uint8_t)HIST_REGIME_DEGENERATE;
    else if (64ull * S >= m * m) r = (uint8_t)HIST_REGIME_PEAKED;
    regime[i] = r;
  }
  if (after) pdl_wait();
}

// `after`: the launches before on the stream are this batch's counting ones,
// which read no regime (else they are any work, which it waits for).
int launch_regimes(const uint8_t* const* d_ptrs, const size_t* d_sizes, uint32_t count, uint32_t theta,
                   uint8_t* d_regime, bool after, cudaStream_t s) {
  for (uint32_t first = 0; first < count; first += 65535u) {
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute at[1];
    lc.gridDim = dim3(count - first < 65535u ? count - first : 65535u);
    lc.blockDim = dim3(HIST_BINS);
    lc.stream = s;
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    const cudaError_t e =
        cudaLaunchKernelEx(&lc, regime_kernel, d_ptrs + first, d_sizes + first, theta, d_regime + first, after);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  return HIST_OK;
}

RegimeLayouts layouts_of(const hist_batch_tuning& tu) {
  RegimeLayouts l;
  for (uint32_t r = 0; r < HIST_REGIMES; ++r) {
    l.layout[r] = 5;
    l.small_bytes[r] = tu.small_bytes;
    l.small_layout[r] = tu.small_log2k;
  }
  return l;
}

RegimeLayouts layouts_of(const hist_batch_table& tb) {
  RegimeLayouts l;
  for (uint32_t r = 0; r < HIST_REGIMES; ++r) {
    l.layout[r] = tb.regime[r].layout;
    l.small_bytes[r] = tb.regime[r].small_bytes;
    l.small_layout[r] = tb.regime[r].small_layout;
  }
  return l;
}

// Whether a batch counts every image in the lane-private table.
bool lane_layouts(const RegimeLayouts& l) {
  for (uint32_t r = 0; r < HIST_REGIMES; ++r)
    if (l.layout[r] != 5 || (l.small_bytes[r] && l.small_layout[r] != 5)) return false;
  return true;
}

// The launches of batch_lane_kernel.  The first waits for the work before it
// before it reads; the second starts after that, reads nothing that the first
// writes, and writes after it.
int launch_batch_lane(const uint8_t* const* d_ptrs, const size_t* d_sizes, uint32_t count, uint32_t* d_out,
                      cudaStream_t s) {
  static int attr[kMaxDevices];
  const int rc = ensure_smem_attr_bytes((const void*)batch_lane_kernel<true>, attr, lane_smem<true>());
  if (rc) return rc;
  for (uint32_t first = 0; first < count; first += kBatchMaxImages) {
    LaneArgs a;
    a.ptrs = d_ptrs + first;
    a.sizes = d_sizes + first;
    a.out = d_out + (size_t)first * HIST_BINS;
    a.count = count - first < kBatchMaxImages ? count - first : kBatchMaxImages;
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute at[1];
    // (at least kBatchMaxImages warps in all)
    const int sms = sm_count(), least = (int)kBatchMaxImages / kWarps;
    lc.gridDim = dim3((unsigned)(sms > least ? sms : least));
    lc.blockDim = dim3(kThreads);
    lc.stream = s;
    a.inv = ~0ull / lc.gridDim.x;
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    a.few = a.count <= kBatchFew;
    cudaError_t e;
    if (a.few) {
      cudaLaunchConfig_t cc = lc;
      cc.gridDim = dim3((a.count + kFewWarps - 1) / kFewWarps);
      cc.blockDim = dim3(kFewWarps * 32);
      e = cudaLaunchKernelEx(&cc, batch_few_kernel, a);
    } else {
      lc.dynamicSmemBytes = lane_smem<true>();
      e = cudaLaunchKernelEx(&lc, batch_lane_kernel<true>, a);
    }
    if (e != cudaSuccess) return cuda_fail(e);
    lc.dynamicSmemBytes = lane_smem<false>();
    e = cudaLaunchKernelEx(&lc, batch_lane_kernel<false>, a);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  return HIST_OK;
}

int launch_batch_images(const hist_batch_tuning& tu, const RegimeLayouts& lay, const uint8_t* regime,
                        const uint8_t* const* d_ptrs, const size_t* d_sizes, uint32_t count, uint32_t* d_out,
                        cudaStream_t s) {
  if (lane_layouts(lay)) return launch_batch_lane(d_ptrs, d_sizes, count, d_out, s);
  if (count) {  // (no images: only the kernel's attributes are set up)
    const cudaError_t e = cudaMemsetAsync(d_out, 0, (size_t)count * HIST_BINS * sizeof(uint32_t), s);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  // one CTA per SM with 64 registers (2 or 4 loads in flight), or two with 32
  // registers (2 loads in flight)
  static int attr21[kMaxDevices], attr41[kMaxDevices], attr22[kMaxDevices];
  const void* fn;
  int* done;
  if (tu.ctas_per_sm == 2) {
    fn = (const void*)batch_images_kernel<2, 2>;
    done = attr22;
  } else if (tu.unroll == 4) {
    fn = (const void*)batch_images_kernel<4, 1>;
    done = attr41;
  } else {
    fn = (const void*)batch_images_kernel<2, 1>;
    done = attr21;
  }
  int rc = ensure_smem_attr_bytes(fn, done, kBatchSmem);
  if (rc) return rc;
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, kBatchSmem);
  if (e != cudaSuccess) return cuda_fail(e);
  if (per_sm < 1) per_sm = 1;
  const int want = (int)(tu.ctas_per_sm ? tu.ctas_per_sm : 1);
  const int grid = sm_count() * (want < per_sm ? want : per_sm);
  for (uint32_t first = 0; first < count; first += kBatchMaxImages) {
    BatchImgArgs a;
    a.ptrs = d_ptrs + first;
    a.sizes = d_sizes + first;
    a.out = d_out + (size_t)first * HIST_BINS;
    a.regime = regime ? regime + first : nullptr;
    a.count = count - first < kBatchMaxImages ? count - first : kBatchMaxImages;
    a.lay = lay;
    void* params[] = {&a};
    e = cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(kThreads), params, kBatchSmem, s);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  return HIST_OK;
}

bool tuning_ok(const hist_batch_tuning* t) {
  return t && (t->unroll == 2 || t->unroll == 4) && t->ctas_per_sm >= 1 && t->ctas_per_sm <= 2 &&
         !(t->ctas_per_sm == 2 && t->unroll == 4) && t->small_log2k <= 5;
}

bool layout_ok(uint32_t l) { return l <= 5 || l == kPerWarp; }

bool table_ok(const hist_batch_table* t) {
  if (!t || !(t->unroll == 2 || t->unroll == 4) || t->ctas_per_sm < 1 || t->ctas_per_sm > 2 ||
      (t->ctas_per_sm == 2 && t->unroll == 4) || t->theta_milli > 1000)
    return false;
  for (uint32_t r = 0; r < HIST_REGIMES; ++r)
    if (!layout_ok(t->regime[r].layout) || !layout_ok(t->regime[r].small_layout)) return false;
  return true;
}

hist_batch_tuning shape_of(const hist_batch_table& t) {
  hist_batch_tuning tu;
  memset(&tu, 0, sizeof(tu));
  tu.ctas_per_sm = t.ctas_per_sm;
  tu.unroll = t.unroll;
  return tu;
}

// The regimes call.  The lane-private launches count every image alike, so
// they come first and the classification fills their tail.
int batch_regimes(const uint8_t* const* d_ptrs, const size_t* d_sizes, uint32_t count, uint32_t* d_out,
                  uint8_t* d_regime, const hist_batch_table& tb, cudaStream_t s) {
  if (count == 0) return HIST_OK;
  const RegimeLayouts lay = layouts_of(tb);
  const bool after = lane_layouts(lay);
  int rc = HIST_OK;
  if (!after) rc = launch_regimes(d_ptrs, d_sizes, count, tb.theta_milli, d_regime, false, s);
  if (rc == HIST_OK) rc = launch_batch_images(shape_of(tb), lay, d_regime, d_ptrs, d_sizes, count, d_out, s);
  if (rc == HIST_OK && after) rc = launch_regimes(d_ptrs, d_sizes, count, tb.theta_milli, d_regime, true, s);
  return rc;
}

// Capture `enqueue` (which enqueues on the stream it is given) into an
// instantiated graph; the kernels' attributes are set up by `prepare`
// outside the capture.
template <class Prep, class Enq>
int capture_graph(Prep prepare, Enq enqueue, hist_batch_graph** out) {
  cudaStream_t cs;
  cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
  if (e != cudaSuccess) return cuda_fail(e);
  int rc = prepare(cs);
  cudaGraph_t g = nullptr;
  cudaGraphExec_t ge = nullptr;
  if (rc == HIST_OK) {
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      rc = enqueue(cs);
      cudaError_t e2 = cudaStreamEndCapture(cs, &g);
      if (rc == HIST_OK && e2 != cudaSuccess) rc = cuda_fail(e2);
    } else {
      rc = cuda_fail(e);
    }
  }
  if (rc == HIST_OK) {
    e = cudaGraphInstantiate(&ge, g, 0);
    if (e != cudaSuccess) rc = cuda_fail(e);
  }
  if (g) cudaGraphDestroy(g);
  cudaStreamDestroy(cs);
  if (rc) return rc;
  *out = reinterpret_cast<hist_batch_graph*>(ge);
  return HIST_OK;
}

}  // namespace

extern "C" {

void hist_batch_tuning_init(hist_batch_tuning* t) {
  if (!t) return;
  memset(t, 0, sizeof(*t));
  // the lane-private layout for every image (its launches have a shape of
  // their own; this one is the other layouts')
  t->ctas_per_sm = 2;
  t->unroll = 2;
  t->small_bytes = 0;
  t->small_log2k = 5;
}

int hist_batch(const uint8_t* const* d_ptrs, const size_t* d_sizes, uint32_t count, uint32_t* d_out,
               const hist_batch_tuning* tuning, hist_cuda_stream s) {
  hist_batch_tuning tu;
  if (tuning) tu = *tuning;
  else hist_batch_tuning_init(&tu);
  if (!tuning_ok(&tu) || (count && (!d_ptrs || !d_sizes || !d_out))) return HIST_EINVAL;
  if (count == 0) return HIST_OK;
  return launch_batch_images(tu, layouts_of(tu), nullptr, d_ptrs, d_sizes, count, d_out, (cudaStream_t)s);
}

int hist_batch_capture(const uint8_t* const* d_ptrs, const size_t* d_sizes, uint32_t count, uint32_t* d_out,
                       const hist_batch_tuning* tuning, hist_batch_graph** out) {
  if (!out) return HIST_EINVAL;
  *out = nullptr;
  hist_batch_tuning tu;
  if (tuning) tu = *tuning;
  else hist_batch_tuning_init(&tu);
  if (!tuning_ok(&tu) || count == 0 || !d_ptrs || !d_sizes || !d_out) return HIST_EINVAL;
  // attributes and occupancy are set up outside the capture (a launch of no images)
  return capture_graph(
      [&](cudaStream_t cs) { return launch_batch_images(tu, layouts_of(tu), nullptr, d_ptrs, d_sizes, 0, d_out, cs); },
      [&](cudaStream_t cs) { return hist_batch(d_ptrs, d_sizes, count, d_out, &tu, (hist_cuda_stream)cs); }, out);
}

void hist_batch_table_init(hist_batch_table* t) {
  if (!t) return;
  memset(t, 0, sizeof(*t));
  t->ctas_per_sm = 2;
  t->unroll = 2;
  t->theta_milli = HIST_THETA_MILLI_DEFAULT;
  for (uint32_t r = 0; r < HIST_REGIMES; ++r) {
    t->regime[r].layout = 5;
    t->regime[r].small_bytes = 0;
    t->regime[r].small_layout = 5;
  }
}

int hist_batch_classify(const uint8_t* const* d_ptrs, const size_t* d_sizes, uint32_t count, uint32_t theta_milli,
                        uint8_t* d_regime, hist_cuda_stream s) {
  if (theta_milli > 1000 || (count && (!d_ptrs || !d_sizes || !d_regime))) return HIST_EINVAL;
  return launch_regimes(d_ptrs, d_sizes, count, theta_milli, d_regime, false, (cudaStream_t)s);
}

int hist_batch_regimes(const uint8_t* const* d_ptrs, const size_t* d_sizes, uint32_t count, uint32_t* d_out,
                       uint8_t* d_regime, const hist_batch_table* table, hist_cuda_stream s) {
  hist_batch_table tb;
  if (table) tb = *table;
  else hist_batch_table_init(&tb);
  if (!table_ok(&tb) || (count && (!d_ptrs || !d_sizes || !d_out || !d_regime))) return HIST_EINVAL;
  return batch_regimes(d_ptrs, d_sizes, count, d_out, d_regime, tb, (cudaStream_t)s);
}

int hist_batch_regimes_capture(const uint8_t* const* d_ptrs, const size_t* d_sizes, uint32_t count,
                               uint32_t* d_out, uint8_t* d_regime, const hist_batch_table* table,
                               hist_batch_graph** out) {
  if (!out) return HIST_EINVAL;
  *out = nullptr;
  hist_batch_table tb;
  if (table) tb = *table;
  else hist_batch_table_init(&tb);
  if (!table_ok(&tb) || count == 0 || !d_ptrs || !d_sizes || !d_out || !d_regime) return HIST_EINVAL;
  return capture_graph(
      [&](cudaStream_t cs) {
        return launch_batch_images(shape_of(tb), layouts_of(tb), d_regime, d_ptrs, d_sizes, 0, d_out, cs);
      },
      [&](cudaStream_t cs) { return batch_regimes(d_ptrs, d_sizes, count, d_out, d_regime, tb, cs); }, out);
}

int hist_batch_graph_launch(hist_batch_graph* g, hist_cuda_stream s) {
  if (!g) return HIST_EINVAL;
  cudaError_t e = cudaGraphLaunch(reinterpret_cast<cudaGraphExec_t>(g), (cudaStream_t)s);
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

int hist_batch_graph_destroy(hist_batch_graph* g) {
  if (!g) return HIST_EINVAL;
  cudaError_t e = cudaGraphExecDestroy(reinterpret_cast<cudaGraphExec_t>(g));
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

int hist_batch_autotune(const uint8_t* const* d_ptrs, const size_t* d_sizes, uint32_t count, uint32_t* d_out,
                        uint32_t repeats, hist_batch_tuning* best, float* best_ms) {
  if (!best || count == 0 || !d_ptrs || !d_sizes || !d_out) return HIST_EINVAL;
  if (repeats == 0) repeats = 3;
  cudaStream_t s;
  cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  if (e != cudaSuccess) return cuda_fail(e);
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  // candidates: the sub-bins of small images, and CTAs per SM and loads in
  // flight where they shape the launch (the lane-private launches are the same
  // for all: timed once, with the default's)
  std::vector<hist_batch_tuning> cands;
  const uint32_t smalls[][2] = {{0, 5}, {1u << 16, 2}, {1u << 16, 3}, {1u << 18, 3}, {1u << 20, 4}};
  for (uint32_t cps = 1; cps <= 2; ++cps)
    for (uint32_t un : {2u, 4u})
      for (const auto& sm : smalls) {
        if (cps == 2 && un == 4) continue;
        hist_batch_tuning t;
        hist_batch_tuning_init(&t);
        const bool shape = cps != t.ctas_per_sm || un != t.unroll;
        t.ctas_per_sm = cps;
        t.unroll = un;
        t.small_bytes = sm[0];
        t.small_log2k = sm[1];
        if (shape && lane_layouts(layouts_of(t))) continue;
        cands.push_back(t);
      }
  float bms = 1e30f;
  int rc = HIST_OK;
  for (const auto& t : cands) {
    rc = hist_batch(d_ptrs, d_sizes, count, d_out, &t, (hist_cuda_stream)s);  // warm-up
    if (rc) break;
    float tot = 0;
    for (uint32_t r = 0; r < repeats && rc == HIST_OK; ++r) {
      cudaEventRecord(e0, s);
      rc = hist_batch(d_ptrs, d_sizes, count, d_out, &t, (hist_cuda_stream)s);
      cudaEventRecord(e1, s);
      cudaEventSynchronize(e1);
      float ms = 0;
      cudaEventElapsedTime(&ms, e0, e1);
      tot += ms;
    }
    if (rc) break;
    const float avg = tot / repeats;
    if (avg < bms) {
      bms = avg;
      *best = t;
    }
  }
  e = cudaStreamSynchronize(s);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaStreamDestroy(s);
  if (rc) return rc;
  if (e != cudaSuccess) return cuda_fail(e);
  if (best_ms) *best_ms = bms;
  return HIST_OK;
}

}  // extern "C"

namespace {

// Mean time of `enqueue` on `s` over `repeats` runs after one warm-up run
// (CUDA events), or a negative HIST_E* code.
template <class Enq>
float time_runs(Enq enqueue, cudaStream_t s, cudaEvent_t e0, cudaEvent_t e1, uint32_t repeats, int* rc) {
  *rc = enqueue();
  if (*rc) return 0.0f;
  float tot = 0.0f;
  for (uint32_t r = 0; r < repeats; ++r) {
    cudaEventRecord(e0, s);
    *rc = enqueue();
    cudaEventRecord(e1, s);
    if (*rc) return 0.0f;
    cudaError_t e = cudaEventSynchronize(e1);
    if (e != cudaSuccess) {
      *rc = cuda_fail(e);
      return 0.0f;
    }
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, e0, e1);
    tot += ms;
  }
  return tot / (float)repeats;
}

}  // namespace

extern "C" int hist_batch_autotune_regimes(const uint8_t* const* d_ptrs, const size_t* d_sizes, uint32_t count,
                                           uint32_t* d_out, uint8_t* d_regime, uint32_t repeats,
                                           hist_batch_table* best, hist_regime_report* report) {
  if (!best || count == 0 || !d_ptrs || !d_sizes || !d_out || !d_regime) return HIST_EINVAL;
  if (repeats == 0) repeats = 3;
  hist_batch_table tb;
  hist_batch_table_init(&tb);
  tb.theta_milli = best->theta_milli <= 1000 && best->theta_milli ? best->theta_milli : HIST_THETA_MILLI_DEFAULT;
  hist_regime_report rep;
  memset(&rep, 0, sizeof(rep));
  cudaStream_t s;
  cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  if (e != cudaSuccess) return cuda_fail(e);
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  // the images' regimes, pointers and sizes on the host
  std::vector<uint8_t> reg(count);
  std::vector<const uint8_t*> ptrs(count);
  std::vector<size_t> sizes(count);
  int rc = launch_regimes(d_ptrs, d_sizes, count, tb.theta_milli, d_regime, false, s);
  if (rc == HIST_OK) {
    e = cudaMemcpyAsync(reg.data(), d_regime, count, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(ptrs.data(), d_ptrs, count * sizeof(void*), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(sizes.data(), d_sizes, count * sizeof(size_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) rc = cuda_fail(e);
  }
  // candidate settings: a layout, and none or one smaller layout for small images
  std::vector<hist_regime_setting> cands;
  const uint32_t layouts[] = {kPerWarp, 0, 1, 2, 3, 4, 5};
  const uint32_t smalls[][2] = {{0, 5}, {64u << 10, 0}, {64u << 10, kPerWarp}, {1u << 20, 2}};
  for (uint32_t l : layouts)
    for (const auto& sm : smalls) {
      if (sm[0] && sm[1] == l) continue;
      hist_regime_setting c;
      memset(&c, 0, sizeof(c));
      c.layout = l;
      c.small_bytes = sm[0];
      c.small_layout = sm[0] ? sm[1] : l;
      cands.push_back(c);
    }
  rep.candidates = (uint32_t)cands.size();
  // per regime: its images alone, every candidate (each image counted with
  // the setting in entry 0: no regime array)
  const hist_batch_tuning shape = shape_of(tb);
  for (uint32_t r = 0; r < HIST_REGIMES && rc == HIST_OK; ++r) {
    std::vector<const uint8_t*> rp;
    std::vector<size_t> rz;
    for (uint32_t i = 0; i < count; ++i)
      if (reg[i] == r) {
        rp.push_back(ptrs[i]);
        rz.push_back(sizes[i]);
        rep.bytes[r] += sizes[i];
      }
    rep.images[r] = (uint32_t)rp.size();
    if (rp.empty()) continue;
    const uint32_t rc_n = (uint32_t)rp.size();
    const uint8_t** dp = nullptr;
    size_t* dz = nullptr;
    uint32_t* dout = nullptr;
    e = cudaMalloc((void**)&dp, rc_n * sizeof(void*));
    if (e == cudaSuccess) e = cudaMalloc((void**)&dz, rc_n * sizeof(size_t));
    if (e == cudaSuccess) e = cudaMalloc((void**)&dout, (size_t)rc_n * HIST_BINS * sizeof(uint32_t));
    if (e == cudaSuccess) e = cudaMemcpy(dp, rp.data(), rc_n * sizeof(void*), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dz, rz.data(), rc_n * sizeof(size_t), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) rc = e == cudaErrorMemoryAllocation ? HIST_ENOMEM : cuda_fail(e);
    float bms = 1e30f;
    for (size_t k = 0; k < cands.size() && rc == HIST_OK; ++k) {
      RegimeLayouts lay;
      for (uint32_t q = 0; q < HIST_REGIMES; ++q) {
        lay.layout[q] = cands[k].layout;
        lay.small_bytes[q] = cands[k].small_bytes;
        lay.small_layout[q] = cands[k].small_layout;
      }
      const float ms = time_runs(
          [&]() {
            return launch_batch_images(shape, lay, nullptr, dp, dz, rc_n, dout, s);
          },
          s, e0, e1, repeats, &rc);
      if (rc) break;
      if (cands[k].layout == 5 && cands[k].small_bytes == 0) rep.ms_default[r] = ms;
      if (ms < bms) {
        bms = ms;
        tb.regime[r] = cands[k];
      }
    }
    rep.ms[r] = bms < 1e30f ? bms : 0.0f;
    cudaFree(dp);
    cudaFree(dz);
    cudaFree(dout);
  }
  // the launch shape of the whole batch with the chosen settings (the
  // lane-private launches have one: the default's is kept)
  const uint32_t shapes[][2] = {{2, 2}, {1, 2}, {1, 4}};
  const bool one_shape = lane_layouts(layouts_of(tb));
  float bms = 1e30f;
  hist_batch_table chosen = tb;
  for (const auto& sh : shapes) {
    if (rc) break;
    hist_batch_table t = tb;
    if (one_shape && (sh[0] != tb.ctas_per_sm || sh[1] != tb.unroll)) continue;
    t.ctas_per_sm = sh[0];
    t.unroll = sh[1];
    const float ms = time_runs([&]() { return batch_regimes(d_ptrs, d_sizes, count, d_out, d_regime, t, s); }, s, e0,
                               e1, repeats, &rc);
    if (rc) break;
    if (ms < bms) {
      bms = ms;
      chosen = t;
    }
  }
  if (rc == HIST_OK) {
    rep.batch_ms = bms;
    hist_batch_table def;
    hist_batch_table_init(&def);
    def.theta_milli = tb.theta_milli;
    rep.batch_default_ms =
        time_runs([&]() { return batch_regimes(d_ptrs, d_sizes, count, d_out, d_regime, def, s); }, s, e0, e1,
                  repeats, &rc);
  }
  // leave d_out holding the batch under the chosen table
  if (rc == HIST_OK) rc = batch_regimes(d_ptrs, d_sizes, count, d_out, d_regime, chosen, s);
  e = cudaStreamSynchronize(s);
  if (rc == HIST_OK && e != cudaSuccess) rc = cuda_fail(e);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaStreamDestroy(s);
  if (rc) return rc;
  *best = chosen;
  if (report) *report = rep;
  return HIST_OK;
}
