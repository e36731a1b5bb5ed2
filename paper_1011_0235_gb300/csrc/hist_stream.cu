// hist_stream.cu -- the chunked stream of Sec. III.B with the kernel switch of
// Sec. III.C, all on the device.
//
// Every batch of chunks a stream is given (hist_stream_push / push_many) is
// counted by one launch of batch_flat_kernel, which needs no device-wide
// waits: a chunk's counts do not depend on the kernel or the pattern that
// count it (every kernel counts in the lane-private table, which refines
// every pattern), and the chunks' epilogues record the exact switches and
// patterns (see the comments above the kernels).
#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <mutex>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include "hist.h"
#include "hist_device.cuh"
#include "hist_internal.h"
#include "hist_plan.h"

using namespace histdev;
using namespace histlib;

namespace {

constexpr uint32_t kMaxBatch = 1024;   // chunks per launch
constexpr uint32_t kSmallBatch = 128;  // chunks per launch of the smaller parameter block
constexpr uint32_t kChunkRing = 4 * kMaxBatch;  // scratch: chunk accumulators
constexpr uint32_t kLaunchRing = 8;             // scratch: per-launch records
constexpr uint32_t kPollLimit = 1u << 22;  // bounded wait: about a second
constexpr uint32_t kStatusTimeout = 4;     // device status: a wait ran out

// The stream's state proper, at the front of StreamDev.
struct StreamHead {
  unsigned long long totals[HIST_BINS];
  uint32_t last_hist[HIST_BINS];
  // pat[cur]: the pattern for the next chunk; pat[cur ^ 1]: the one the last
  // completed chunk was given.  A launch writes the new ones over the two
  // and flips cur, so no pattern is copied.
  hist_pattern pat[2];
  // the last launch known to be complete, and which of pat is the current
  // one (one 16-byte cp.async)
  alignas(16) unsigned long long launches_done;
  uint32_t cur;
  uint32_t flag;              // switch computed from the last completed chunk
  unsigned long long chunks;  // completed chunks
  uint32_t last_kernel;       // kernel the last completed chunk ran
  uint32_t status;            // 0, or kStatusTimeout
  uint32_t recounted;         // AUTO: chunks whose switch the sample of the chunk before misjudged
  uint32_t pad;
};

// Device-resident stream state.
struct StreamDev {
  StreamHead h;
  // Launches of one stream overlap, so their scratch is in rings: chunk g
  // (counted from the stream's first chunk) sums into slot g mod kChunkRing,
  // which returns to zero in the chunk's epilogue; launch L (from 1) counts
  // its epilogues in slot L mod kLaunchRing.
  unsigned long long racc[kChunkRing][HIST_BINS];  // chunks counted by several CTAs (see acc_word)
  uint32_t rbins[kChunkRing];                      // bins of the chunk complete, where several CTAs completed it
  // a window of more than one chunk: every chunk's histogram (a window of up
  // to 256 chunks plus a batch of 1024 fit), its sample histogram and sample
  // size (AUTO), and the window histogram after the last launch's last chunk
  uint32_t whist[kChunkRing][HIST_BINS];
  uint32_t wsamp[kChunkRing][HIST_BINS];
  uint32_t wsn[kChunkRing];                    // pixels in chunk g's sample
  uint32_t wn[kChunkRing];                     // chunk g's size
  unsigned long long wmw[HIST_BINS];
  uint32_t lepis[kLaunchRing];                 // by launch number mod kLaunchRing
};

struct ChunkDesc {
  const uint8_t* in;
  uint32_t* out;
  uint32_t n;
  uint32_t pad;
};

// What every kernel of a push is given.
struct PushHead {
  StreamDev* st;
  uint32_t count;
  uint32_t budget;
  uint32_t theta;
  uint32_t mode;
  uint32_t window;                  // chunks in the moving window
  uint32_t early;                   // chunks may be read before the work before the launch completes (kHostChunk:
                                    // over the host link, one chunk; kReplayed: a captured launch)
  unsigned long long first_chunk;   // number of this batch's first chunk among the stream's chunks
  unsigned long long launch;        // number of this launch among the stream's launches (from 1)
  unsigned long long prev;          // number of the launch before it (0: none)
};

constexpr uint32_t kHostChunk = 2;
constexpr uint32_t kReplayed = 3;

// The counting launch's parameters: the header and the chunk table.  Two
// capacities, so that a launch of a few chunks does not carry (and the driver
// does not copy) a 24 KiB table; the kernel is instantiated for both.
template <uint32_t CAP>
struct BatchArgs : PushHead {
  static constexpr uint32_t kCap = CAP;
  uint32_t trace_first;             // index of this batch's first chunk in the trace
  uint32_t trace_cap;               // chunks the trace holds
  unsigned long long* trace;        // optional phase timestamps (see hist_stream_trace)
  RangePlan plan;  // the host's split of the batch's cost
  ChunkDesc c[CAP];
};
using SmallArgs = BatchArgs<kSmallBatch>;
using LargeArgs = BatchArgs<kMaxBatch>;
static_assert(sizeof(LargeArgs) <= 32764, "kernel parameters are limited to 32764 bytes");
static_assert(offsetof(StreamHead, launches_done) % 16 == 0 && alignof(StreamDev) >= 16 &&
                  offsetof(StreamHead, cur) == offsetof(StreamHead, launches_done) + 8,
              "one 16-byte cp.async");

// Phase timestamps (%globaltimer, ns) of chunk j by CTA slot k (0: the first
// CTA, 1: the middle one, 2: the last one), eight slots per chunk and CTA, of
// which the flat launch records phase 0 (start of the CTA's piece of the
// chunk), 5 (table reduced) and 7 (end).
constexpr int kTracePhases = 8;
constexpr int kTraceCtas = 3;

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// ------------------------------------------------------------ flat batches --
//
// A chunk's counts do not depend on the kernel or the pattern that count it,
// so the chunks of a batch need not be counted one after the other.
// batch_flat_kernel splits the batch's chunks, placed end to end, into one
// contiguous range per CTA by a cost model (a chunk costs its bytes plus
// kFlatChunkCost, flat_cost; the host computes the split), so a CTA counts
// one or two pieces of chunks and reduces its table only where its range
// crosses a chunk boundary.  A CTA adds a piece's per-bin sums and the memory
// blocks it counted into the chunk's accumulator (acc_word); the CTA whose
// add completes a chunk runs the chunk's epilogue (output, totals, and the
// switch and pattern of the launch's last two chunks, which the state
// keeps).  No CTA waits for another, so the launch is not cooperative, and a
// chunk's accumulator returns to zero in its epilogue.
//
// The plain and the adaptive kernel of the switch count in the same
// lane-private table (hist_device.cuh).  While the plain kernel had one table
// per warp and the adaptive one the pattern's own slots below the full
// budget, AUTO launches predicted each chunk's kernel from a sample of the
// chunk before, weighed and laid out the chunks by it and counted the
// mispredicted ones again: 64 chunks of 16 MiB took 208 us a push of N(128,
// 8) and 287 us on the degenerate workload, in a 960-slot adaptive stream 435
// us; all now take what the full table takes, 159 us.

// Cost of a chunk beyond its bytes.  Launches of 1024 x 16 KiB, 100 x 64 KiB
// and 512 x 256 KiB chunks: 12.1, 10.8 and 38.6 us with 32 KiB, 10.7, 8.1 and
// 28.9 with 64 KiB, 10.7, 8.8 and 29.0 with 96 KiB.
constexpr unsigned long long kFlatChunkCost = 64ull << 10;
// Largest chunk a group counts (flat_groups).  512 x 256 KiB: 28.9 us, 40.6 if
// the whole CTA counts them; 512 KiB gains nothing more.
constexpr uint32_t kGroupChunkMax = 256u << 10;
// The batch's last two chunks, when small, also cost kFlatTailCost, placed
// before their bytes: their epilogues derive the patterns the stream keeps
// (1000 x 4 KiB chunks: 10.0 us without it, 7.6 us).  Beside 16 MiB chunks
// the epilogues are noise and the extra cost would only shift the split.
constexpr unsigned long long kFlatTailCost = 128ull << 10;
__host__ __device__ __forceinline__ unsigned long long flat_tail(unsigned long long n, uint32_t j, uint32_t count) {
  return j + 2 >= count && n <= kGroupChunkMax ? kFlatTailCost : 0ull;
}
// chunk j's cost: the fixed cost and the tail cost, then one per byte
__host__ __device__ __forceinline__ unsigned long long flat_cost(unsigned long long n, uint32_t j, uint32_t count) {
  return n + kFlatChunkCost + flat_tail(n, j, count);
}

// Whole small chunks are counted by groups of warps (flat_groups), each with
// a table of its own.
constexpr int kGroups = 4;
constexpr int kGroupThreads = kThreads / kGroups;
static_assert(kGroupThreads == HIST_BINS, "one bin per thread of a group");
constexpr int kEpiBar = 1 + kGroups;  // named barrier of a group's (or the CTA's) epilogue threads: kEpiBar + group

// Dynamic shared memory: the groups' tables in a launch with groups, else the
// one table that pieces are counted in.  The L1 cache gets what shared memory
// leaves, and the loads in flight need it: 64 chunks of 16 MiB take 161 us
// with 80 KiB of shared memory in all, 176 us with 146 KiB.
constexpr size_t kFlatSmem = (size_t)kTableWords * 4;
constexpr size_t kFlatGroupSmem = kGroups * kFlatSmem;

// A chunk as the CTAs keep it in shared memory: the chunk table sits in the
// kernel's parameters, which are read through the constant cache, 0.5 - 1 us
// a miss (a group that read each chunk's entry as it came to it took 2.5 us
// a chunk of 4 KiB).
struct FlatDesc {
  const uint8_t* in;
  uint32_t* out;
  uint32_t n;
  uint32_t j;
};
// A piece of a chunk: bytes [b0, e0) (e0 = 0: an empty chunk).
struct FlatPiece {
  FlatDesc d;
  uint32_t b0, e0;
};
constexpr uint32_t kListItems = 2 * kWarps;  // chunks the groups take at a time

// CTA-wide state of batch_flat_kernel (shared memory).
template <uint32_t CAP>
struct FlatShared {
  alignas(16) unsigned long long ring_seen[2];  // launches_done as the launch started (cp.async)
  EpiShared es[kGroups];
  uint32_t res[HIST_BINS];      // sums of the piece in the table
  uint32_t eh[2][HIST_BINS];    // unaligned edge bytes of the CTA's pieces, in turn
  uint32_t samp[2][HIST_BINS];  // AUTO: the sample's pixels in them
  int last;
  int released;  // this CTA has waited for the previous launch
  uint32_t epis; // chunk epilogues this CTA ran
  FlatDesc win[kWarps];         // the chunks of the range the CTA is at
  FlatPiece piece[kWarps];      // its pieces of them
  uint32_t npiece, nwl;
  unsigned long long pos;       // cost position of the chunk after them
  uint16_t wl[CAP];             // whole chunks left to the groups, in batch order
  GroupItem items[kListItems];  // the chunks the groups are at
  uint32_t gmax[kGroups][2][HIST_BINS / 32];  // each group's largest bins per warp: chunk, sample
  uint32_t geh[kGroups][HIST_BINS];    // each group's edge bytes
  uint32_t gsamp[kGroups][HIST_BINS];  // and sample
  // the launch's last two chunks, where the groups counted them: histogram,
  // sample and chunk, for their epilogues after the groups
  uint32_t lhist[2][HIST_BINS], lsamp[2][HIST_BINS];
  FlatDesc ldesc[2];
  int lhave[2];
};

template <class A>
__device__ __forceinline__ void flat_mark(const A& a, uint32_t j, int phase, bool lead) {
  const int tslot = blockIdx.x == 0 ? 0 : (blockIdx.x == gridDim.x / 2 ? 1 : (blockIdx.x == gridDim.x - 1 ? 2 : -1));
  if (a.trace && tslot >= 0 && lead && a.trace_first + j < a.trace_cap)
    a.trace[((size_t)(a.trace_first + j) * kTraceCtas + tslot) * kTracePhases + phase] = globaltimer();
}
template <class A>
__device__ __forceinline__ void flat_mark(const A& a, uint32_t j, int phase) {
  flat_mark(a, j, phase, threadIdx.x == 0);
}

// ---- samples (AUTO)
//
// hist_stream_state.recounted counts the chunks of AUTO pushes whose kernel
// a sample of the chunk before would have chosen wrongly: 4096 pixels of it
// (256 evenly spaced 16-byte vectors from its first 16-byte boundary; a
// smaller chunk whole) against the switch of the whole chunk.  With a window
// of more than one chunk the samples, scaled by chunk size, are summed over
// the window and compared with the window's exact switch
// (window_flat_kernel).  The CTAs take the sample's vectors while they count
// the pieces that hold them: a launch of its own after the count cost 9 us a
// push.
constexpr uint32_t kSampleVecs = HIST_BINS;  // 16-byte vectors per sample: 4096 pixels

// Whether chunk j of the launch is sampled.
__device__ __forceinline__ bool flat_sampled(const PushHead& a, uint32_t j) {
  return a.mode == HIST_MODE_AUTO && (a.window > 1 || j + 1 < a.count);
}
// Sample vector k of the n bytes at `in`: its offset, or 0xffffffff when the
// sample is the whole chunk.
__device__ __forceinline__ bool sample_whole(const uint8_t* in, uint32_t n) {
  return split_bytes_at(in, n, 16).nvec < kSampleVecs;
}
__device__ __forceinline__ uint32_t sample_at(const uint8_t* in, uint32_t n, uint32_t k) {
  const Split sp = split_bytes_at(in, n, 16);
  if (sp.nvec < kSampleVecs) return 0xffffffffu;
  return (uint32_t)(sp.head + 16 * ((size_t)k * sp.nvec / kSampleVecs));
}
// The larger of the warps' maxima m[0..7].
__device__ __forceinline__ uint32_t max8(const uint32_t* m) {
  uint32_t mx = m[0];
#pragma unroll
  for (int i = 1; i < HIST_BINS / 32; ++i) mx = m[i] > mx ? m[i] : mx;
  return mx;
}

// A chunk (n pixels, largest bin mx) whose sample (4096 pixels, largest bin
// ms) gives another switch is counted.
__device__ __forceinline__ void flat_compare(const PushHead& a, uint32_t n, uint32_t mx, uint32_t ms) {
  if (reaches_theta(mx, n, a.theta) != reaches_theta(ms, 16 * kSampleVecs, a.theta))
    atomicAdd(&a.st->h.recounted, 1u);
}

// Chunk d is complete; threads t = 0..255, which share named barrier `id`, hold
// its histogram (h) and its sample's (s), a bin each: its output, totals and
// window entries, its switch against the sample's, and if it is one of the
// launch's last two, the pattern and the switch the state keeps (a window's
// switch: window_flat_kernel).  The threads have waited for the previous
// launch; a barrier of theirs stands between two calls.
static __device__ __noinline__ void flat_epilogue(const PushHead& a, const FlatDesc& d, uint32_t h, uint32_t s,
                                                  EpiShared& es, int t, int id) {
  StreamDev* st = a.st;
  const uint32_t n = d.n, j = d.j;
  const bool whole = sample_whole(d.in, n);
  if (d.out) d.out[t] = h;
  if (h) atomicAdd(&st->h.totals[t], (unsigned long long)h);
  if (a.window > 1) {
    const uint32_t rs = (uint32_t)((a.first_chunk + j) % kChunkRing);
    st->whist[rs][t] = h;
    if (a.mode == HIST_MODE_AUTO) {
      st->wsamp[rs][t] = whole ? h : s;
      if (t == 0) {
        st->wsn[rs] = whole ? n : 16 * kSampleVecs;
        st->wn[rs] = n;
      }
    }
  }
  const GroupBar<HIST_BINS> bar = {id};
  if (a.window == 1 && flat_sampled(a, j) && !whole) {
    const uint32_t mh = __reduce_max_sync(0xffffffffu, h), ms = __reduce_max_sync(0xffffffffu, s);
    if ((t & 31) == 0) {
      es.wmax[t >> 5] = mh;
      es.warg[t >> 5] = ms;
    }
    bar.sync();
    if (t == 0) flat_compare(a, n, max8(es.wmax), max8(es.warg));
    bar.sync();
  }
  if (j + 2 < a.count) return;
  if (j + 1 == a.count) st->h.last_hist[t] = h;
  // the last chunk's pattern goes into the slot that becomes the current one
  const uint32_t cur = __ldcg(&st->h.cur) & 1u;
  BinPlace place;
  const hist_degeneracy_result r = block_pattern(h, n, a.budget, a.theta, es, t, bar, place);
  store_place(st->h.pat[j + 1 == a.count ? cur ^ 1u : cur], t, a.budget, place);
  if (t != 0 || a.window > 1) return;
  if (j + 1 < a.count) {
    if (a.mode == HIST_MODE_AUTO) st->h.last_kernel = r.flag;
  } else {
    if (a.mode != HIST_MODE_AUTO)
      st->h.last_kernel = a.mode == HIST_MODE_ADAPTIVE ? HIST_FLAG_ADAPTIVE : HIST_FLAG_PLAIN;
    else if (a.count == 1) st->h.last_kernel = __ldcg(&st->h.flag);
    st->h.flag = r.flag;
  }
}

// A CTA that ran chunk epilogues adds them to the launch's count once it is
// done; the CTA whose add completes the launch's chunks flips the stream's
// current pattern (every epilogue has read which it was) and counts the
// chunks.  A CTA that ran them all needs no count.
template <class A>
__device__ __forceinline__ void flat_finish(const A& a, uint32_t epis) {
  StreamDev* st = a.st;
  uint32_t* done = &st->lepis[a.launch % kLaunchRing];
  if (epis != a.count) {
    if (atomicAdd(done, epis) + epis != a.count) return;
    *done = 0;
  }
  atomicXor(&st->h.cur, 1u);
  atomicAdd(&st->h.chunks, (unsigned long long)a.count);
}

// Launches of one stream overlap (programmatic dependent launch): every
// CTA lets the next launch start as soon as it starts, so the next launch's
// CTAs take the SM slots that this launch's CTAs free as they finish, clear
// their tables and read their ranges.  Unless the caller has declared every
// chunk complete when it was pushed (a.early, HIST_OVERLAP_PUSHES), a CTA
// then waits for the work before the launch on the CUDA stream to complete
// before it reads a chunk byte: that work may be the kernel that wrote the
// chunk, and only the wait makes its writes visible.  A CTA waits for it in
// any case before its first epilogue, which reads and writes the stream
// state, and before it first adds into a chunk ring slot, whose last user -- a
// launch at least kChunkRing / kMaxBatch - 1 launches back -- must be complete
// (flat_ring_ready: by launches_done, the number that each launch writes once
// it knows the launch before it to be complete, or by the wait).
__device__ __forceinline__ void flat_prev_done(const PushHead& a) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(&a.st->h.launches_done), "l"(a.prev) : "memory");
}

// Thread 0, before its CTA first adds into a ring slot.  A launch that waited at
// its start has its slots.  An early one has them when launches_done says so,
// which in a queue of small pinned chunks it does some microseconds later; but
// that number may be too old -- a replayed graph sets it back to what it was
// when its pushes were captured, and captured pushes advance the launches'
// numbers without running -- so after kRingPolls polls the launch waits for the
// one before it instead, as a captured launch does at once (the replay before
// leaves the number ahead of it).  Only hist_stream_test_hold_ring holds the
// slots for longer (a bounded wait).  1 GiB overlapping 152.0 us a push, 153.5
// if every early launch waits; 64 x 1 MiB from pinned memory 403 us, 643 if a
// launch waits where the number is not there at once.
constexpr uint32_t kRingPolls = 64;  // about 60 us
template <class A>
__device__ __noinline__ void flat_ring_ready(const A& a, FlatShared<A::kCap>& fs) {
  constexpr unsigned long long back = kChunkRing / kMaxBatch - 1;
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (!a.early && fs.ring_seen[0] + back >= a.launch) return;
  uint32_t it = 0;
  if (a.early) {
    for (; a.early != kReplayed && it < kRingPolls; ++it) {
      if (ld_acquire(&a.st->h.launches_done) + back >= a.launch) return;
      __nanosleep(256);
    }
    pdl_wait();
    if (!fs.released) {
      fs.released = 1;
      flat_prev_done(a);
    }
  }
  while (ld_acquire(&a.st->h.launches_done) + back < a.launch) {
    if (++it >= kPollLimit) {
      atomicOr(&a.st->h.status, kStatusTimeout);
      break;
    }
    __nanosleep(256);
  }
}

// A launch that reads over the host link lets the next one start only when
// CTA 0 has half of its piece, and at most 64 KiB, left: the next chunk's
// first reads come before this one's last, and however many chunks are queued
// two launches of kHostGrid CTAs hold SMs while they wait for the link (if all
// did, eight one-shots of 64 MiB on another stream beside 16 x 16 MiB would
// take 1145 us; so 251, alone 117).  With chunks of 512 KiB and 1 MiB, whose
// epilogues take longer than their bytes over the link, up to five launches
// (80 CTAs) are resident.  The launches of one CTA (push_one_kernel) let the
// next one start at once: seven to nine of them are resident at most, whether
// the link is busy with other copies or not, and the same eight one-shots take
// 183 us beside 400 chunks of 64 KiB (1.12 ms).  Let in after the loads they
// would take 143, but the chunks 1.59 ms, those of 128 KiB 2.13 for 1.23.
template <class A>
__device__ __forceinline__ bool host_late(const A& a) {
  return a.early == kHostChunk && blockIdx.x == 0;
}
__device__ __forceinline__ uint32_t host_mid(const uint8_t* in, uint32_t b, uint32_t e) {
  uint32_t left = (e - b) / 2;
  if (left > 65536u) left = 65536u;
  const uint32_t m = e - left, over = (uint32_t)(((uintptr_t)in + m) & (kLineBytes - 1));
  return m - b > over && left ? m - over : e;
}

// Count piece k of the window's (the CTA's number `turn`; `ring`: whether the
// ring check is behind) into the table, which is clear before and after, and
// publish it: into the chunk's accumulator, or, when it is the whole chunk,
// straight into the chunk's epilogue.  The CTA that completes a chunk runs
// its epilogue, by the first 256 threads while the others go on to the CTA's
// next piece, whose first 128 KiB are fetched into L2 while this one's table
// is reduced.  All threads call.
template <class A>
__device__ __forceinline__ void flat_piece(const A& a, uint32_t k, uint32_t turn, bool& ring, uint32_t* table,
                                           FlatShared<A::kCap>& fs) {
  StreamDev* st = a.st;
  const int t = threadIdx.x;
  const FlatPiece& p = fs.piece[k];
  uint32_t h = 0, s = 0;
  flat_mark(a, p.d.j, 0);
  if (p.e0) {
    const uint8_t* vec = nullptr;
    if (flat_sampled(a, p.d.j) && t < (int)kSampleVecs) {
      // (every cut between pieces is a multiple of 16 bytes in memory)
      const uint32_t at = sample_at(p.d.in, p.d.n, t);
      if (at != 0xffffffffu && at >= p.b0 && at < p.e0) vec = p.d.in + at;
    }
    const bool late = host_late(a);
    uint32_t b = p.b0, e = late ? host_mid(p.d.in, b, p.e0) : p.e0;
    for (;;) {
      piece_count(p.d.in + b, e - b, table, fs.eh[turn & 1], vec, fs.samp[turn & 1]);
      if (!late) break;
      pdl_launch_dependents();
      if (e == p.e0) break;
      b = e;
      e = p.e0;
      vec = nullptr;
    }
    if (k + 1 < fs.npiece) {
      const FlatPiece& q = fs.piece[k + 1];
      const uint32_t at = (uint32_t)t * kLineBytes;
      if (at < q.e0 - q.b0) asm volatile("prefetch.global.L2 [%0];" ::"l"(q.d.in + q.b0 + at));
    }
    __syncthreads();
    lane_reduce<kThreads, true>(table, fs.res, t);
    __syncthreads();
    if (t < HIST_BINS) {
      h = fs.res[t] + fs.eh[turn & 1][t];
      s = fs.samp[turn & 1][t];
      fs.eh[turn & 1][t] = fs.samp[turn & 1][t] = 0;
    }
    flat_mark(a, p.d.j, 5);
  }
  bool complete = p.e0 - p.b0 == p.d.n;
  if (!complete) {
    if (!ring) {
      if (t == 0) flat_ring_ready(a, fs);
      if (a.early) __syncthreads();
      ring = true;
    }
    const uint32_t slot = (uint32_t)((a.first_chunk + p.d.j) % kChunkRing);
    unsigned long long* acc = &st->racc[slot][t & (HIST_BINS - 1)];
    bool done = false;
    if (t < HIST_BINS) {
      const unsigned long long add = acc_word(h, acc_blocks(p.d.in, p.b0, p.e0), s);
      const unsigned long long sum = atomicAdd(acc, add) + add;
      done = ((uint32_t)(sum >> 32) & kAccBlockMask) == acc_blocks(p.d.in, 0, p.d.n);
      h = (uint32_t)sum;
      s = (uint32_t)(sum >> 50);
    }
    const int bins = __syncthreads_count(done);
    if (bins == HIST_BINS) {
      // this CTA's adds were the last to every bin
      complete = true;
      if (t < HIST_BINS) *acc = 0;
    } else if (bins > 0) {
      // two CTAs' adds crossed: the one that brings the completed bins to 256
      // reads them all
      if (t == 0) {
        __threadfence();
        fs.last = atomicAdd(&st->rbins[slot], (uint32_t)bins) + (uint32_t)bins == HIST_BINS;
        __threadfence();
      }
      __syncthreads();
      complete = fs.last != 0;
      if (complete) {
        if (t < HIST_BINS) {
          const unsigned long long sum = __ldcg(acc);
          h = (uint32_t)sum;
          s = (uint32_t)(sum >> 50);
          *acc = 0;
        }
        if (t == 0) st->rbins[slot] = 0;
      }
    }
  }
  if (t < HIST_BINS) {
    if (complete) {
      if (a.early) {
        pdl_wait();
        if (t == 0 && !fs.released) {
          fs.released = 1;
          flat_prev_done(a);
        }
      }
      flat_epilogue(a, p.d, h, s, fs.es[0], t, kEpiBar);
      if (t == 0) fs.epis += 1;
    }
    flat_mark(a, p.d.j, 7);
  }
}

// Chunks [j0, j0 + kWarps), the first at cost position fs.pos: into fs.win, a
// warp each with a warp-uniform index (their constant-cache misses overlap),
// then warp 0, a chunk per lane, lists the CTA's pieces of them and, in fs.wl,
// the whole ones left to the groups.  Chunk j's byte b sits at its cost
// position + b (after the tail cost for the last two chunks); a range takes
// the bytes whose cost position it holds.  All threads call (begins and ends
// with a barrier).
template <class A>
__device__ __forceinline__ void flat_window(const A& a, uint32_t j0, FlatShared<A::kCap>& fs) {
  const uint32_t w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (j0 + w < a.count) {
    const FlatDesc d = {a.c[j0 + w].in, a.c[j0 + w].out, a.c[j0 + w].n, j0 + w};
    if (lane == 0) fs.win[w] = d;
  }
  __syncthreads();
  if (w == 0) {
    const unsigned long long lo = a.plan.lo[blockIdx.x], hi = a.plan.lo[blockIdx.x + 1];
    const bool in = j0 + lane < a.count;
    const FlatDesc d = in ? fs.win[lane] : FlatDesc{nullptr, nullptr, 0, 0};
    const uint32_t n = d.n;
    const unsigned long long c = in ? flat_cost(n, d.j, a.count) : 0ull;
    unsigned long long x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if ((int)lane >= o) x += y;
    }
    const unsigned long long p0 = fs.pos + x - c;
    // a chunk of at most a quarter of a CTA's range is not split: the range
    // holding its first cost position counts it whole, so it needs no
    // accumulator or ring; a small one is left to the groups
    bool piece = false, item = false;
    unsigned long long b0 = 0, e0 = 0;
    if (in && p0 < hi) {
      if (n == 0 || plan_whole(n, a.plan.range)) {
        item = p0 >= lo && n != 0 && n <= a.plan.group_max;
        piece = p0 >= lo && !item;
        e0 = n;
      } else {
        // byte b sits at cost q0 + b, after the chunk's tail cost
        const unsigned long long q0 = p0 + flat_tail(n, d.j, a.count);
        if (hi > q0) {
          b0 = lo > q0 ? split_point(d.in, lo - q0) : 0ull;
          e0 = split_point(d.in, hi - q0);
          if (e0 > (unsigned long long)n) e0 = n;
          piece = b0 < e0;
        }
      }
    }
    const unsigned mp = __ballot_sync(0xffffffffu, piece), mi = __ballot_sync(0xffffffffu, item);
    const unsigned lt = (1u << lane) - 1u;
    if (piece) fs.piece[__popc(mp & lt)] = FlatPiece{d, (uint32_t)b0, (uint32_t)e0};
    if (item) fs.wl[fs.nwl + __popc(mi & lt)] = (uint16_t)d.j;
    __syncwarp();
    if (lane == 31) {
      fs.pos = p0 + c;
      fs.npiece = __popc(mp);
      fs.nwl += __popc(mi);
    }
  }
  __syncthreads();
}

__device__ __forceinline__ GroupItem group_item(const PushHead& a, const FlatDesc& d) {
  const Split sp = split_bytes(d.in, d.n);
  GroupItem it;
  it.body = reinterpret_cast<const uint4*>(d.in + sp.head);
  it.out = d.out;
  it.nvec = (uint32_t)sp.nvec;
  it.n = d.n;
  it.j = d.j;
  it.edges = (uint32_t)sp.head | ((uint32_t)sp.tail << 8) |
             (flat_sampled(a, d.j) && !sample_whole(d.in, d.n) ? 1u << 16 : 0u);
  return it;
}

// ------------------------------------------------ whole small chunks --
//
// A CTA that counts a small chunk whole spends little of its time loading
// it: a 64 KiB chunk is one round of four loads per thread, after which the
// table is reduced and the epilogue run.  So the CTA leaves such chunks to
// the end of its range and counts them with kGroups groups of warps, each
// with its own table and named barrier, entry g, g + kGroups, ... of the list
// for group g.  What a chunk costs beyond its pixels is mostly instructions
// that every warp of its group executes, so a group is 8 warps, one thread
// per bin, and a chunk's addresses are computed once (GroupItem); a thread
// sums its bin's row of the table itself and clears it, with a barrier before
// and one after, and keeps the bin in a register through the epilogue.  A
// group loads the first vectors of its next chunk before it counts the last
// ones of the current one.  Bound by the HBM read at 64 KiB, by instructions
// and latency below: on the GPU, pushes in a row, 1000 x 4 KiB 18.4 -> 7.6 us,
// 1024 x 16 KiB 20.7 -> 10.7, 1024 x 64 KiB 29.2 -> 18.2 (AUTO 40.9 -> 20.9),
// 512 x 256 KiB 37.2 -> 28.9 us (two groups of 16 warps, per-warp tables in
// AUTO mode, addresses computed by every warp before).

// The list's chunks [i0, i0 + kListItems) into fs.items (first >= 0: the list
// is first, first + 1, ...; else fs.wl), a warp per chunk.  All threads call;
// the caller's barriers stand before and after.
template <class A>
__device__ __forceinline__ void group_items(const A& a, uint32_t nwl, int first, uint32_t i0,
                                            FlatShared<A::kCap>& fs) {
  for (uint32_t k = threadIdx.x >> 5; k < kListItems && i0 + k < nwl; k += kWarps) {
    const uint32_t j = first >= 0 ? (uint32_t)first + i0 + k : fs.wl[i0 + k];
    const FlatDesc d = {a.c[j].in, a.c[j].out, a.c[j].n, j};
    if ((threadIdx.x & 31) == 0) fs.items[k] = group_item(a, d);
  }
}

// This group's chunks g, g + kGroups, ... of the first `count` in fs.items,
// its table clear, geh and gsamp too (a barrier of the group's stands
// before).  Their epilogues but those of the launch's last two chunks, which
// are left in fs.lhist.  All of the group's threads call.
template <class A>
__device__ __noinline__ void group_count(const A& a, uint32_t count, bool released, uint32_t* tables,
                                         FlatShared<A::kCap>& fs) {
  StreamDev* st = a.st;
  const int g = threadIdx.x / kGroupThreads, t = threadIdx.x % kGroupThreads;
  const GroupBar<kGroupThreads> bar = {g + 1};
  uint32_t* table = tables + (size_t)g * kTableWords;
  const uint32_t base = smem_addr(table) + ((t & 31) << 2);
  uint32_t total = 0;
  uint32_t prev_n = 0;  // size of a chunk still to be compared with its sample
  uint32_t i = (uint32_t)g;
  if (i >= count) return;
  uint4 v[kLaneLoads];
  lane_load<kLaneLoads, kGroupThreads>(v, lane_range(fs.items[i].body, 0, fs.items[i].nvec, t));
  uint32_t edge = group_edge(fs.items[i], t);
  for (; i < count; i += kGroups) {
    const GroupItem& it = fs.items[i];
    const bool more = i + kGroups < count;
    flat_mark(a, it.j, 0, t == 0);
    if (edge < 0x100u) atomicAdd(&fs.geh[g][edge], 1u);
    edge = 0x100u;
    LaneRange next = {nullptr, 0};
    if (more) {
      const GroupItem& it2 = fs.items[i + kGroups];
      edge = group_edge(it2, t);
      next = lane_range(it2.body, 0, it2.nvec, t);
    }
    lane_count<kLaneLoads, kGroupThreads>(v, lane_range(it.body, 0, it.nvec, t), base, next);
    if (it.edges >> 16) {
      // read after the chunk, so that its lines are in L2: ahead of it each
      // 16-byte vector is a DRAM access of its own
      const uint8_t* in = reinterpret_cast<const uint8_t*>(it.body) - (it.edges & 0xffu);
      vec_count(ldg_stream(reinterpret_cast<const uint4*>(in + sample_at(in, it.n, t))), fs.gsamp[g]);
    }
    bar.sync();
    if (prev_n && t == 0) flat_compare(a, prev_n, max8(fs.gmax[g][0]), max8(fs.gmax[g][1]));
    prev_n = 0;
    uint32_t h = lane_row(table, t), s = 0;
    if (it.edges) {
      h += fs.geh[g][t];
      s = fs.gsamp[g][t];
      fs.geh[g][t] = fs.gsamp[g][t] = 0;
    }
    if (!released) {
      // the previous launch writes the stream state and may write the
      // same outputs
      pdl_wait();
      released = true;
      if (t == 0) flat_prev_done(a);
    }
    bar.sync();
    flat_mark(a, it.j, 5, t == 0);
    const uint32_t left = a.count - it.j;  // 1, 2: one of the launch's last two chunks
    if (left <= 2) {
      fs.lhist[left - 1][t] = h;
      fs.lsamp[left - 1][t] = s;
      if (t == 0) {
        fs.ldesc[left - 1] = FlatDesc{reinterpret_cast<const uint8_t*>(it.body) - (it.edges & 0xffu), it.out, it.n, it.j};
        fs.lhave[left - 1] = 1;
      }
    } else {
      if (it.out) it.out[t] = h;
      total += h;  // a group's small chunks: below 2^32 pixels
      if (a.window > 1) {
        const uint32_t rs = (uint32_t)((a.first_chunk + it.j) % kChunkRing);
        st->whist[rs][t] = h;
        if (a.mode == HIST_MODE_AUTO) {
          const bool whole = !(it.edges >> 16);
          st->wsamp[rs][t] = whole ? h : s;
          if (t == 0) {
            st->wsn[rs] = whole ? it.n : 16 * kSampleVecs;
            st->wn[rs] = it.n;
          }
        }
      } else if (it.edges >> 16) {
        const uint32_t mh = __reduce_max_sync(0xffffffffu, h), ms = __reduce_max_sync(0xffffffffu, s);
        if ((t & 31) == 0) {
          fs.gmax[g][0][t >> 5] = mh;
          fs.gmax[g][1][t >> 5] = ms;
        }
        prev_n = it.n;
      }
    }
    flat_mark(a, it.j, 7, t == 0);
  }
  if (total) atomicAdd(&st->h.totals[t], (unsigned long long)total);
  if (a.window == 1 && a.mode == HIST_MODE_AUTO) {
    bar.sync();
    if (prev_n && t == 0) flat_compare(a, prev_n, max8(fs.gmax[g][0]), max8(fs.gmax[g][1]));
  }
}

// All threads call (after a barrier); returns after the CTA's groups have
// counted the nwl chunks of the list (first >= 0: chunks first, first + 1,
// ...) and run their epilogues.  `wait`: the work before the launch has still
// to be waited for.
template <class A>
__device__ __forceinline__ void flat_groups(const A& a, uint32_t nwl, int first, bool wait, uint32_t* tables,
                                            FlatShared<A::kCap>& fs) {
  if (nwl == 0) {
    if (wait) pdl_wait();
    return;
  }
  const int g = threadIdx.x / kGroupThreads, t = threadIdx.x % kGroupThreads;
  {
    uint4* t4 = reinterpret_cast<uint4*>(tables + (size_t)g * kTableWords);
#pragma unroll
    for (int k = 0; k < kTableWords / 4 / kGroupThreads; ++k) t4[t + k * kGroupThreads] = make_uint4(0, 0, 0, 0);
  }
  fs.geh[g][t] = fs.gsamp[g][t] = 0;
  if (threadIdx.x < 2) fs.lhave[threadIdx.x] = 0;
  bool released = wait || fs.released != 0;
  for (uint32_t i0 = 0; i0 < nwl; i0 += kListItems) {
    if (i0) __syncthreads();
    group_items(a, nwl, first, i0, fs);
    __syncthreads();
    if (wait && i0 == 0) pdl_wait();
    group_count(a, nwl - i0 < kListItems ? nwl - i0 : kListItems, released, tables, fs);
  }
  __syncthreads();
  if (threadIdx.x == 0) fs.epis += nwl;
  // the last chunk's epilogue by the first 256 threads, the one before by the
  // next
  if (g < 2 && fs.lhave[g]) {
    if (!released) pdl_wait();
    flat_epilogue(a, fs.ldesc[g], fs.lhist[g][t], fs.lsamp[g][t], fs.es[g], t, kEpiBar + g);
  }
}

// One CTA of 1024 threads per SM, each thread with four 16-byte loads in
// flight (64 registers).  Two CTAs per SM with two loads each keep as many
// bytes in flight, but the SM's two CTAs do not progress alike (the
// scheduler favours the older one), so one of them finishes its range well
// before the other and the SM then runs a single CTA at half its loads in
// flight; one CTA per SM has no such pair.  Bound by the HBM read on large
// chunks, by a chain of round trips to L2 on one small one: on the GPU,
// pushes in a row, 64 x 16 MiB 166.6 -> 158.4 us (6.8 TB/s; overlapping
// 162 -> 155.6 us from a graph, 152.0 called one by one), 128 x 1 MiB 39.2 ->
// 28.0 us (AUTO 28.9), one chunk of 1 MiB 15.6 -> 7.5 us.
template <class A>
__global__ void __launch_bounds__(kThreads, 1) batch_flat_kernel(const __grid_constant__ A a) {
  extern __shared__ __align__(16) uint32_t tables[];
  __shared__ FlatShared<A::kCap> fs;
  const int t = threadIdx.x;

  // what the range needs of the parameters is read before the wait
  const bool groups = a.plan.groups[blockIdx.x >> 5] >> (blockIdx.x & 31) & 1u;
  if (groups || !host_late(a)) pdl_launch_dependents();
  if (t == 0) {
    fs.released = a.early ? 0 : 1;
    fs.epis = 0;
  }
  if (groups) {
    // the range holds whole chunks for the groups only
    const uint32_t s0 = a.plan.s[blockIdx.x], s1 = a.plan.s[blockIdx.x + 1];
    __syncthreads();
    flat_groups(a, s1 - s0, (int)s0, !a.early, tables, fs);
    if (!a.early && blockIdx.x == 0 && t == kThreads - 1) flat_prev_done(a);
  } else {
    const uint32_t j0 = a.plan.j[blockIdx.x];
    if (t == 0) {
      fs.pos = a.plan.pre[blockIdx.x];
      fs.nwl = 0;
    }
    zero_table(tables);
    if (t < HIST_BINS) fs.eh[0][t] = fs.eh[1][t] = fs.samp[0][t] = fs.samp[1][t] = 0;
    flat_window(a, j0, fs);
    if (!a.early) {
      pdl_wait();
      if (blockIdx.x == 0 && t == kThreads - 1) flat_prev_done(a);
      if (t == 0)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(fs.ring_seen)),
                     "l"(&a.st->h.launches_done)
                     : "memory");
    }
    bool ring = false;
    uint32_t turn = 0;
    for (uint32_t j = j0;;) {
      for (uint32_t k = 0; k < fs.npiece; ++k) flat_piece(a, k, turn++, ring, tables, fs);
      j += kWarps;
      if (fs.pos >= a.plan.lo[blockIdx.x + 1] || j >= a.count) break;
      flat_window(a, j, fs);
    }
    __syncthreads();
    if (fs.nwl) flat_groups(a, fs.nwl, -1, false, tables, fs);
  }
  __syncthreads();
  if (t == 0) {
    if (fs.epis) flat_finish(a, fs.epis);
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
}

// A push of one short chunk: one CTA, without a plan, a chunk table or
// accumulators.  Bound by the chain of the wait, one or two rounds of loads,
// the reduction, the epilogue's pattern and the launch itself; batch_flat_kernel
// reads its ranges and its chunk's entry from 6.6 KB of parameters first (two
// constant misses) and clears the groups' tables.  A chunk of 9001 bytes in AUTO
// mode, pushes in a row: 5.1 -> 3.5 us (declared complete 3.8 -> 2.2).
__global__ void __launch_bounds__(kThreads, 1) push_one_kernel(const PushHead a, const FlatDesc d) {
  __shared__ __align__(16) uint32_t table[kTableWords];
  __shared__ uint32_t res[HIST_BINS], eh[HIST_BINS];
  __shared__ EpiShared es;
  const int t = threadIdx.x;
  pdl_launch_dependents();
  zero_table(table);
  if (t < HIST_BINS) eh[t] = 0;
  if (!a.early) pdl_wait();
  __syncthreads();
  if (d.n) piece_count(d.in, d.n, table, eh, nullptr, nullptr);
  __syncthreads();
  lane_reduce<kThreads, false>(table, res, t);
  __syncthreads();
  if (t >= HIST_BINS) return;
  if (a.early) pdl_wait();
  if (t == 0) flat_prev_done(a);
  flat_epilogue(a, d, res[t] + eh[t], 0u, es, t, kEpiBar);
  const GroupBar<HIST_BINS> bar = {kEpiBar};
  bar.sync();
  if (t == 0) flat_finish(a, 1);
}

// A window of W > 1 chunks.  The window histogram after chunk g is the sum
// of the histograms of chunks g-W+1 .. g (chunks before number 0 count as
// empty; a resumed stream restarts at 0).  The histograms of the last
// kChunkRing chunks stay in rings, so every window is summed on its own:
// thread b + 256 q takes bin b of every fourth run of eight chunks, so that a
// window of 32 is one round of loads.
constexpr int kWindowThreads = 4 * HIST_BINS;
constexpr uint32_t kWindowRun = 8;                              // chunks per thread and round
constexpr uint32_t kWindowRound = kWindowRun * kWindowThreads / HIST_BINS;  // chunks per round

// Largest bin and total of a 256-bin window held one bin per thread (256
// threads on barrier `id` call; two barriers); returned to every thread.
template <class T>
__device__ __forceinline__ void window_max_sum(T v, T* smax, T* ssum, int id, T& mx, T& sm) {
  const GroupBar<HIST_BINS> bar = {id};
  const int b = threadIdx.x & (HIST_BINS - 1), w = b >> 5;
  T m = v, s = v;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const T m2 = __shfl_xor_sync(0xffffffffu, m, o);
    m = m2 > m ? m2 : m;
    s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  if ((b & 31) == 0) {
    smax[w] = m;
    ssum[w] = s;
  }
  bar.sync();
  mx = smax[0];
  sm = ssum[0];
#pragma unroll
  for (int i = 1; i < HIST_BINS / 32; ++i) {
    mx = smax[i] > mx ? smax[i] : mx;
    sm += ssum[i];
  }
  bar.sync();
}

// The end of the window after the launch's chunk c, a bin per thread in x and
// its samples' sum in f (256 threads on barrier `id`): the switch and what
// depends on it.
__device__ __forceinline__ void window_end(const PushHead& a, uint32_t c, unsigned long long x, float f,
                                           unsigned long long* smax, unsigned long long* ssum, float* fmax,
                                           float* fsum, int id) {
  StreamDev* st = a.st;
  const int b = threadIdx.x & (HIST_BINS - 1);
  unsigned long long mx, sm;
  window_max_sum(x, smax, ssum, id, mx, sm);
  const uint32_t flag = reaches_theta(mx, sm, a.theta) ? HIST_FLAG_ADAPTIVE : HIST_FLAG_PLAIN;
  if (a.mode == HIST_MODE_AUTO && c + 1 < a.count) {
    float fm, fs;
    window_max_sum(f, fmax, fsum, id, fm, fs);
    const uint32_t pred = (fs > 0.0f && fm * 1000.0f >= fs * (float)a.theta) ? HIST_FLAG_ADAPTIVE : HIST_FLAG_PLAIN;
    if (b == 0 && pred != flag) atomicAdd(&st->h.recounted, 1u);
  }
  const uint32_t fixed = a.mode == HIST_MODE_ADAPTIVE ? HIST_FLAG_ADAPTIVE : HIST_FLAG_PLAIN;
  if (c + 1 == a.count) {
    st->wmw[b] = x;
    if (b == 0) {
      if (a.count == 1) st->h.last_kernel = a.mode == HIST_MODE_AUTO ? __ldcg(&st->h.flag) : fixed;
      st->h.flag = flag;
    }
  } else if (c + 2 == a.count && b == 0) {
    st->h.last_kernel = a.mode == HIST_MODE_AUTO ? flag : fixed;
  }
}

// The window switches of a launch's chunks, chained after the counting launch.
// The last chunk's window and the stream's switch after it are kept, and the
// switch of the chunk before it, which is the kernel the last chunk ran.  In
// AUTO mode every window but the last also takes its switch from the samples,
// in FP32 and in the chunks' order (FP64 is slow on this part and the samples
// are estimates), and a chunk whose two switches differ is counted; in the
// other modes only the last two windows are asked for.
//
// Two kernels.  window_runs_kernel: M windows of consecutive chunks a CTA,
// which share their rows' loads, the next round's in flight while one is
// summed (64 registers, one CTA per SM).  window_flat_kernel: a window a CTA
// in 32 registers, two CTAs per SM.  Bound by L2 latency with few windows, by
// the rows read (count x W KiB, twice in AUTO mode) with many.  A push with
// its window, us, with window_flat_kernel for every chunk and now:
//   128 x 1 MiB W 32         33.7   31.8   (28.9 without a window)
//   81 x 570 KB W 161        29.6   24.8   (15.9)
//   152 x 5 KB W 256         25.4   18.5   (6.4)
//   500 x 5 KB W 100, 256    27.9, 44.6   22.6, 31.4   (9.1)
//   1000 x 5 KB W 100, 256   42.9, 71.7   34.6, 46.1   (11.4)
//   639 x 5 KB W 203, plain  35.6   16.0   (10.0)
// One wave of CTAs is a window each (M = 1; with M = 2 128 x 1 MiB take 34.9);
// up to two waves, and short windows, stay with window_flat_kernel (300 x 5 KB
// W 32 11.1, with M = 2 12.9; 1000 x 5 KB W 32 24.2, with M = 8 27.9).
__global__ void __launch_bounds__(kWindowThreads) window_flat_kernel(const PushHead a) {
  __shared__ unsigned long long part[kWindowThreads / HIST_BINS - 1][HIST_BINS];
  __shared__ uint32_t samp[kWindowRound][HIST_BINS];
  __shared__ unsigned long long smax[HIST_BINS / 32], ssum[HIST_BINS / 32];
  __shared__ float fmax[HIST_BINS / 32], fsum[HIST_BINS / 32];
  __shared__ float scale[HIST_WINDOW_MAX];
  StreamDev* st = a.st;
  const int b = threadIdx.x & (HIST_BINS - 1), q = threadIdx.x / HIST_BINS;
  pdl_launch_dependents();
  pdl_wait();
  const unsigned long long W = a.window, c = blockIdx.x, g = a.first_chunk + c;
  const unsigned long long first = g >= W - 1 ? g - (W - 1) : 0ull;
  const uint32_t len = (uint32_t)(g - first + 1);
  const bool sampled = a.mode == HIST_MODE_AUTO && c + 1 < a.count;
  // each window chunk's scale, one thread per chunk
  if (sampled && threadIdx.x < len) {
    const uint32_t slot = (uint32_t)((first + threadIdx.x) % kChunkRing);
    const uint32_t sn = __ldcg(&st->wsn[slot]);
    scale[threadIdx.x] = sn ? (float)__ldcg(&st->wn[slot]) / (float)sn : 0.0f;
  }
  unsigned long long v = 0;
  float f = 0.0f;
  for (uint32_t k0 = 0; k0 < len; k0 += kWindowRound) {
    uint32_t h[kWindowRun], s[kWindowRun];
#pragma unroll
    for (uint32_t i = 0; i < kWindowRun; ++i) {
      const uint32_t k = k0 + q * kWindowRun + i;
      const uint32_t slot = (uint32_t)((first + k) % kChunkRing);
      h[i] = k < len ? __ldcg(&st->whist[slot][b]) : 0u;
      s[i] = sampled && k < len ? __ldcg(&st->wsamp[slot][b]) : 0u;
    }
#pragma unroll
    for (uint32_t i = 0; i < kWindowRun; ++i) v += h[i];
    if (sampled) {
#pragma unroll
      for (uint32_t i = 0; i < kWindowRun; ++i) samp[q * kWindowRun + i][b] = s[i];
      __syncthreads();
      if (q == 0) {
        const uint32_t m = len - k0 < kWindowRound ? len - k0 : kWindowRound;
#pragma unroll 8
        for (uint32_t i = 0; i < m; ++i) f += (float)samp[i][b] * scale[k0 + i];
      }
      __syncthreads();
    }
  }
  if (q > 0) part[q - 1][b] = v;
  __syncthreads();
  if (q > 0) return;
#pragma unroll
  for (int i = 0; i < kWindowThreads / HIST_BINS - 1; ++i) v += part[i][b];
  window_end(a, (uint32_t)c, v, f, smax, ssum, fmax, fsum, 1);
}

// Windows skip + M blockIdx.x .. + M - 1 of the launch's.  Rows that all of
// them hold are added once for all, the others window by window.
template <int M>
__global__ void __launch_bounds__(kWindowThreads) window_runs_kernel(const PushHead a, uint32_t skip) {
  constexpr int Q = kWindowThreads / HIST_BINS, E = M < Q ? 1 : M / Q, P = M < Q ? M : Q;
  // (Q groups of threads; group q < P ends windows q, q + Q, .. of E)
  __shared__ union {
    float samp[kWindowRound][HIST_BINS];
    unsigned long long part[Q][P][HIST_BINS];
  } u;
  __shared__ unsigned long long smax[Q][HIST_BINS / 32], ssum[Q][HIST_BINS / 32];
  __shared__ float fmax[Q][HIST_BINS / 32], fsum[Q][HIST_BINS / 32];
  __shared__ __align__(16) float scale[(HIST_WINDOW_MAX + M - 2) / kWindowRound * kWindowRound + kWindowRound];
  StreamDev* st = a.st;
  const int b = threadIdx.x & (HIST_BINS - 1), q = threadIdx.x / HIST_BINS;
  pdl_launch_dependents();
  pdl_wait();
  const uint32_t c0 = skip + blockIdx.x * M, nw = a.count - c0 < M ? a.count - c0 : M;
  // row 0 is the first window's first chunk, row r in slot base + r of the
  // rings; window w's rows are [from(w), to(w))
  const unsigned long long g0 = a.first_chunk + c0;
  const uint32_t back = g0 < a.window - 1 ? (uint32_t)g0 : a.window - 1;
  const uint32_t base = (uint32_t)((g0 - back) % kChunkRing), rows = back + nw;
  auto from = [&](uint32_t w) { return back + w + 1 > a.window ? back + w + 1 - a.window : 0u; };
  auto to = [&](uint32_t w) { return back + w + 1; };
  const bool sampled = a.mode == HIST_MODE_AUTO && c0 + 1 < a.count;
  // each row's scale, one thread per row
  if (sampled && threadIdx.x < sizeof(scale) / sizeof(scale[0])) {
    float x = 0.0f;
    if (threadIdx.x < rows) {
      const uint32_t slot = (base + threadIdx.x) % kChunkRing;
      const uint32_t sn = __ldcg(&st->wsn[slot]);
      x = sn ? (float)__ldcg(&st->wn[slot]) / (float)sn : 0.0f;
    }
    scale[threadIdx.x] = x;
  }
  unsigned long long all = 0, v[M] = {};  // rows of every window, and of window w beside them
  float f[E] = {};
  uint32_t h[kWindowRun], s[kWindowRun];
  auto load = [&](uint32_t k0) {
#pragma unroll
    for (uint32_t i = 0; i < kWindowRun; ++i) {
      const uint32_t k = k0 + q * kWindowRun + i;
      const uint32_t slot = (base + k) % kChunkRing;
      h[i] = k < rows ? __ldcg(&st->whist[slot][b]) : 0u;
      s[i] = sampled && k < rows ? __ldcg(&st->wsamp[slot][b]) : 0u;
    }
  };
  load(0);
  for (uint32_t k0 = 0; k0 < rows; k0 += kWindowRound) {
    // (rows past the last are zeros: they change no sum of one window)
    const bool common = M == 1 || (k0 >= from(M - 1) && k0 + kWindowRound <= to(0));
#pragma unroll
    for (uint32_t i = 0; i < kWindowRun; ++i) {
      if (common) {
        all += h[i];
      } else {
        const uint32_t k = k0 + q * kWindowRun + i;
#pragma unroll
        for (int w = 0; w < M; ++w)
          if (k >= from(w) && k < to(w)) v[w] += h[i];
      }
      if (sampled) u.samp[q * kWindowRun + i][b] = (float)s[i];
    }
    if (k0 + kWindowRound < rows) load(k0 + kWindowRound);
    if (sampled) {
      __syncthreads();
      if (q < P) {
        if (common) {
#pragma unroll 2
          for (uint32_t i = 0; i < kWindowRound; i += 4) {
            const float4 sc = *reinterpret_cast<const float4*>(&scale[k0 + i]);
            const float x[4] = {sc.x, sc.y, sc.z, sc.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float y = u.samp[i + j][b];
#pragma unroll
              for (int e = 0; e < E; ++e) f[e] = fmaf(y, x[j], f[e]);
            }
          }
        } else {
#pragma unroll 4
          for (uint32_t i = 0; i < kWindowRound; ++i) {
            const float y = u.samp[i][b], x = scale[k0 + i];
#pragma unroll
            for (int e = 0; e < E; ++e)
              if (k0 + i >= from(e * Q + q) && k0 + i < to(e * Q + q)) f[e] = fmaf(y, x, f[e]);
          }
        }
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int e = 0; e < E; ++e) {
    if (e) __syncthreads();
#pragma unroll
    for (int w = 0; w < P; ++w) u.part[q][w][b] = v[e * Q + w] + all;
    __syncthreads();
    if (q < P && (uint32_t)(e * Q + q) < nw) {
      unsigned long long x = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) x += u.part[i][q][b];
      window_end(a, c0 + e * Q + q, x, f[e], smax[q], ssum[q], fmax[q], fsum[q], 1 + q);
    }
  }
}

// The queries of a stream's state are launches chained to the push before
// them (they wait for it before they read), and let a push behind them start:
// a device-to-device copy of the totals between two pushes kept the second
// one's CTAs from the SMs that the first one's free (64 x 16 MiB overlapping,
// totals after each push: 166.4 -> 154.3 us; 1024 ragged chunks of at most 64
// KiB: 24.6 -> 19.4).

// The moving-window histogram after the last chunk (none: zeros): the last
// chunk's histogram for a window of one, else the window kept by
// window_flat_kernel.  At L2: the work before may have written it while this
// launch was waiting.
__device__ __forceinline__ unsigned long long window_bin(const StreamDev* st, uint32_t window, bool any, int b) {
  if (!any) return 0ull;
  return window == 1 ? (unsigned long long)__ldcg(&st->h.last_hist[b]) : __ldcg(&st->wmw[b]);
}

__global__ void __launch_bounds__(HIST_BINS) window_copy_kernel(const StreamDev* st, uint32_t window, bool any,
                                                                unsigned long long* out) {
  pdl_launch_dependents();
  pdl_wait();
  out[threadIdx.x] = window_bin(st, window, any, threadIdx.x);
}

__global__ void __launch_bounds__(HIST_BINS) totals_copy_kernel(const StreamDev* st, unsigned long long* out) {
  pdl_launch_dependents();
  pdl_wait();
  out[threadIdx.x] = __ldcg(&st->h.totals[threadIdx.x]);
}

// Change detection between the stream's totals and its moving-window
// histogram after the last chunk (256 threads).
__global__ void __launch_bounds__(HIST_BINS) stream_change_kernel(const StreamDev* st, uint32_t window, bool any,
                                                                  uint32_t tau_milli, hist_change_result* res) {
  __shared__ ChangeShared sh;
  const int b = threadIdx.x;
  pdl_launch_dependents();
  pdl_wait();
  const unsigned long long m = window_bin(st, window, any, b);
  const hist_change_result r = change_eval(__ldcg(&st->h.totals[b]), m, tau_milli, sh);
  if (b == 0) *res = r;
}

// The stream state of hist_stream_run_noalloc: one fixed array of the
// library (file scope, 256-byte aligned, sizeof(StreamDev) bytes), so that
// the call allocates no device memory.  Host code reaches it only through
// the address cudaGetSymbolAddress returns (noalloc_setup).
static __device__ __align__(256) StreamDev g_noalloc_state;

// The totals and status of a no-alloc run, to the caller's buffers.
__global__ void noalloc_out_kernel(const StreamDev* st, unsigned long long* totals, uint32_t* status) {
  const int b = threadIdx.x;
  if (b < HIST_BINS) totals[b] = st->h.totals[b];
  if (b == 0 && status) *status = st->h.status;
}

__global__ void __launch_bounds__(HIST_BINS) init_kernel(StreamDev* st, uint32_t budget) {
  __shared__ hist_pattern pat;
  __shared__ EpiShared es;
  __shared__ uint32_t zero[HIST_BINS];
  zero[threadIdx.x] = 0;
  __syncthreads();
  block_epilogue(zero, 0, budget, HIST_THETA_MILLI_DEFAULT, pat, es);
  __syncthreads();
  const uint32_t* src = reinterpret_cast<const uint32_t*>(&pat);
  for (int k = 0; k < 2; ++k) {
    uint32_t* dst = reinterpret_cast<uint32_t*>(&st->h.pat[k]);
    if (threadIdx.x < sizeof(hist_pattern) / 4) dst[threadIdx.x] = src[threadIdx.x];
  }
}

}  // namespace

constexpr uint32_t kMaxStaging = 4;

struct hist_stream {
  hist_config cfg;
  StreamDev* d;
  int sms;
  int grid;
  unsigned long long chunks_launched;  // chunks pushed
  unsigned long long flat_launches;  // counting launches so far (scratch ring positions)
  unsigned long long prev_launch;    // number of the last one that ran (hist_stream_test_hold_ring skips numbers)
  unsigned long long flat_chunks;    // chunks of those launches
  unsigned long long resume_chunk;   // first chunk after the last set_state
  // tracing (optional)
  unsigned long long* trace;
  uint32_t trace_cap;
  uint32_t trace_next;
  // host-fed staging (optional)
  uint32_t depth;
  size_t max_chunk;
  uint8_t* staging[kMaxStaging];
  cudaEvent_t copied[kMaxStaging];
  cudaEvent_t consumed[kMaxStaging];
  cudaStream_t copy_stream;
  unsigned long long host_pushes;
  // the caller's device allocator (alloc null: cudaMalloc / cudaFree)
  hist_allocator alloc;
  // host buffer of a launch's parameters (null: one is allocated per launch)
  void* args;
};

namespace {

// Device memory of a stream: from the caller's allocator if it gave one.
int dev_alloc(hist_stream* st, void** p, size_t bytes) {
  *p = nullptr;
  if (!st->alloc.alloc) {
    const cudaError_t e = cudaMalloc(p, bytes);
    return e == cudaSuccess ? HIST_OK : (e == cudaErrorMemoryAllocation ? HIST_ENOMEM : cuda_fail(e));
  }
  void* q = st->alloc.alloc(bytes, st->alloc.ctx);
  if (!q) return HIST_ENOMEM;
  if ((uintptr_t)q % 256u) {
    st->alloc.free(q, bytes, st->alloc.ctx);
    return HIST_EINVAL;
  }
  *p = q;
  return HIST_OK;
}

void dev_free(hist_stream* st, void* p, size_t bytes) {
  if (!p) return;
  if (st->alloc.alloc) st->alloc.free(p, bytes, st->alloc.ctx);
  else cudaFree(p);
}

// A launch that may start while the work before it on `s` ends
// (programmatic dependent launch); the kernel waits (griddepcontrol.wait)
// before it reads what that work writes.
cudaError_t launch_chained(const void* fn, dim3 grid, dim3 block, void** params, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = block;
  lc.dynamicSmemBytes = smem;
  lc.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  return cudaLaunchKernelExC(&lc, fn, params);
}

// The grid of a launch and its CTAs' ranges (plan_ranges): at most `grid`
// CTAs, and no more than kCtaCost bytes, or a chunk, each needs.
constexpr unsigned long long kCtaCost = 32ull << 10;
uint32_t flat_plan(RangePlan* p, uint32_t count, const size_t* ns, uint32_t grid) {
  PlanCosts<kMaxBatch> c;
  auto size = [&](uint32_t i) { return (unsigned long long)ns[i]; };
  plan_costs(&c, count, size, [&](uint32_t i) { return flat_cost(ns[i], i, count); });
  unsigned long long want = (c.bytes + kCtaCost - 1) / kCtaCost;
  if (want < count) want = count;
  if (want < grid) grid = (uint32_t)want;
  plan_ranges(p, c, count, grid, kGroupChunkMax, size);
  return grid;
}

// The grid of a launch that reads over the host link: 1 MiB of loads in
// flight.  16 x 16 MiB take 1272 us with 8 CTAs as with 152, 64 x 1 MiB 394
// with 8, 388 with 16, 402 with 24 to 152; the other SMs are left to other
// streams.
constexpr uint32_t kHostGrid = 16;

// Whether launches on `s` are captured (or may be: the question failed).
bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusActive;
  if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) {
    cudaGetLastError();
    return true;
  }
  return capture != cudaStreamCaptureStatusNone;
}

// What every kernel of the next push of `count` chunks is given, and the
// stream's counters after it.
void push_head(const hist_stream* st, uint32_t count, bool host, cudaStream_t s, PushHead* a) {
  a->st = st->d;
  a->count = count;
  a->first_chunk = st->flat_chunks;
  a->window = st->cfg.window;
  a->launch = st->flat_launches + 1;
  a->prev = st->prev_launch;
  a->budget = st->cfg.budget;
  a->theta = st->cfg.theta_milli;
  a->mode = st->cfg.mode;
  a->early = host ? kHostChunk : 0u;
  if (!host && (st->cfg.flags & HIST_OVERLAP_PUSHES)) a->early = capturing(s) ? kReplayed : 1u;
}
void pushed(hist_stream* st, uint32_t count) {
  st->flat_launches += 1;
  st->prev_launch = st->flat_launches;
  st->flat_chunks += count;
  st->chunks_launched += count;
}

// A push of one chunk of at most kOneMax bytes (window of one chunk, no trace)
// is one CTA's (push_one_kernel); pushes in a row, with batch_flat_kernel and so:
// 16 bytes 4.6 and 3.2 us, 16 KiB 5.4 and 3.6, 64 KiB 6.3 and 4.8, 128 KiB 8.0
// and 6.5.
constexpr size_t kOneMax = 128u << 10;
int launch_one(hist_stream* st, const uint8_t* in, size_t n, uint32_t* out, bool host, cudaStream_t s) {
  PushHead a;
  push_head(st, 1, host, s, &a);
  FlatDesc d;
  d.in = in;
  d.out = out;
  d.n = (uint32_t)n;
  d.j = 0;
  void* params[] = {&a, &d};
  const cudaError_t e = launch_chained((const void*)push_one_kernel, dim3(1), dim3(kThreads), params, 0, s);
  if (e != cudaSuccess) return cuda_fail(e);
  pushed(st, 1);
  return HIST_OK;
}

// The launches of one batch: the counting launch, and with a window of more
// than one chunk the window's switches.  Each may start while the one before
// ends and waits for it before it reads what that one writes.  `host`: the
// chunks are in host memory that the kernels can read, and were complete when
// they were pushed.
template <class A>
int launch_batch(hist_stream* st, uint32_t count, const uint8_t* const* ins, const size_t* ns, uint32_t* const* outs,
                 bool host, cudaStream_t s) {
  // the stream's parameter buffer: the header and the plan are cleared, the
  // chunk entries written (the launch copies the parameters)
  static_assert(sizeof(A) <= sizeof(LargeArgs), "one buffer for both parameter blocks");
  const bool own = st->args == nullptr;
  A* a = own ? (A*)calloc(1, sizeof(A)) : (A*)st->args;
  if (!a) return HIST_ENOMEM;
  if (!own) memset((void*)a, 0, (size_t)((char*)a->c - (char*)a));
  push_head(st, count, host, s, a);
  a->trace = st->trace;
  a->trace_cap = st->trace_cap;
  a->trace_first = st->trace_next;
  for (uint32_t i = 0; i < count; ++i) {
    a->c[i].in = ins[i];
    a->c[i].n = (uint32_t)ns[i];
    a->c[i].out = outs ? outs[i] : nullptr;
  }
  const bool windowed = st->cfg.window > 1;
  uint32_t most = (uint32_t)st->grid;
  if (host && most > kHostGrid) most = kHostGrid;
  const uint32_t grid = flat_plan(&a->plan, count, ns, most);
  void* params[] = {a};
  cudaError_t e =
      launch_chained((const void*)batch_flat_kernel<A>, dim3(grid), dim3(kThreads), params,
                     a->plan.group_max ? kFlatGroupSmem : kFlatSmem, s);
  PushHead head = *a;
  if (e == cudaSuccess && windowed) {
    // (window_flat_kernel's comment: which kernel, with M = m)
    uint32_t skip = st->cfg.mode != HIST_MODE_AUTO && count > 2 ? count - 2 : 0;
    const uint32_t windows = count - skip;
    void* hparams[] = {&head, &skip};
    const uint32_t sms = (uint32_t)st->sms;
    const uint32_t m = windows <= sms ? 1u : windows <= 4 * sms ? 4u : 8u;
    const bool runs = m == 1 || (m == 4 ? windows > 2 * sms && st->cfg.window >= 100 : windows * st->cfg.window >= 100000);
    const void* fn = !runs    ? (const void*)window_flat_kernel
                     : m == 1 ? (const void*)window_runs_kernel<1>
                     : m == 4 ? (const void*)window_runs_kernel<4>
                              : (const void*)window_runs_kernel<8>;
    e = launch_chained(fn, dim3(runs ? (windows + m - 1) / m : windows), dim3(kWindowThreads), hparams, 0, s);
  }
  if (own) free(a);
  if (e != cudaSuccess) return cuda_fail(e);
  pushed(st, count);
  if (st->trace) st->trace_next += count;
  return HIST_OK;
}

int push_chunks(hist_stream* st, uint32_t count, const uint8_t* const* ins, const size_t* ns, uint32_t* const* outs,
                cudaStream_t s, bool host = false) {
  if (count == 1 && ns[0] <= kOneMax && st->cfg.window == 1 && !st->trace)
    return launch_one(st, ins[0], ns[0], outs ? outs[0] : nullptr, host, s);
  for (uint32_t i = 0; i < count; i += kMaxBatch) {
    const uint32_t c = count - i < kMaxBatch ? count - i : kMaxBatch;
    int rc = c <= kSmallBatch ? launch_batch<SmallArgs>(st, c, ins + i, ns + i, outs ? outs + i : nullptr, host, s)
                              : launch_batch<LargeArgs>(st, c, ins + i, ns + i, outs ? outs + i : nullptr, host, s);
    if (rc) return rc;
  }
  return HIST_OK;
}

// The address at which kernels launched on `s` read the n bytes of host memory
// at p, or null: the bytes must lie in one range of memory that CUDA has
// pinned, and `s` must not be capturing (a push from the host is no part of a
// graph: the staged path's error says so).  About 0.1 us.
const uint8_t* host_readable(const uint8_t* p, size_t n, cudaStream_t s) {
  typedef CUresult (*Ask)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);
  static const Ask ask = []() -> Ask {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult found;
    const cudaError_t e =
        cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 12000, cudaEnableDefault, &found);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess && found == cudaDriverEntryPointSuccess ? (Ask)f : nullptr;
  }();
  if (!ask) return nullptr;
  if (capturing(s)) return nullptr;
  unsigned int type = 0, managed = 1;
  CUdeviceptr d = 0, start = 0;
  size_t size = 0;
  CUpointer_attribute at[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED,
                              CU_POINTER_ATTRIBUTE_DEVICE_POINTER, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                              CU_POINTER_ATTRIBUTE_RANGE_SIZE};
  void* data[] = {&type, &managed, &d, &start, &size};
  if (ask(5, at, data, (CUdeviceptr)(uintptr_t)p) != CUDA_SUCCESS) return nullptr;
  const uint64_t at0 = (uint64_t)(uintptr_t)p - (uint64_t)start;
  if (type != CU_MEMORYTYPE_HOST || managed || !d || (uint64_t)(uintptr_t)p < (uint64_t)start || at0 > size ||
      n > size - at0)
    return nullptr;
  return reinterpret_cast<const uint8_t*>((uintptr_t)d);
}

bool config_ok(const hist_config* c) {
  return c && c->budget >= HIST_BUDGET_MIN && c->budget <= HIST_BUDGET_MAX && c->theta_milli <= 1000 &&
         c->mode <= HIST_MODE_ADAPTIVE && c->window >= 1 && c->window <= HIST_WINDOW_MAX &&
         (c->flags & ~HIST_OVERLAP_PUSHES) == 0;
}

int grid_for(const hist_config* cfg, int sms, const void* fn, size_t smem) {
  // every CTA that can be resident at once, or fewer if the caller asks
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, smem) != cudaSuccess || per_sm < 1)
    per_sm = 1;
  const int cap = per_sm * sms;
  const int g = cfg->grid ? (int)cfg->grid : cap;
  return g > cap ? cap : g;
}

// The counting kernels' shared-memory opt-in, once per (kernel, device).
int flat_kernels_setup() {
  static std::mutex mu;
  static int attr[2][kMaxDevices];
  std::lock_guard<std::mutex> lock(mu);
  int rc = ensure_smem_attr_bytes((const void*)batch_flat_kernel<SmallArgs>, attr[0], kFlatGroupSmem);
  if (rc == HIST_OK) rc = ensure_smem_attr_bytes((const void*)batch_flat_kernel<LargeArgs>, attr[1], kFlatGroupSmem);
  return rc;
}

// The grid of the counting launches (the larger variant's occupancy: the
// smaller one needs less shared memory).
int flat_grid(const hist_config* cfg, int sms) {
  const int g = grid_for(cfg, sms, (const void*)batch_flat_kernel<LargeArgs>, kFlatGroupSmem);
  return g < (int)kPlanCtas ? g : (int)kPlanCtas;
}

// Once per device, with that device current: the no-alloc state's device
// address and the counting kernels' shared-memory opt-in (none of it
// allocates).
int noalloc_setup(void** state) {
  static std::mutex mu;
  static void* ptr[kMaxDevices];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e);
  if (dev < 0 || dev >= kMaxDevices) return HIST_EINVAL;
  std::lock_guard<std::mutex> lock(mu);
  if (!ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_state);
    if (e != cudaSuccess || !p) return cuda_fail(e != cudaSuccess ? e : cudaErrorInvalidSymbol);
    const int rc = flat_kernels_setup();
    if (rc) return rc;
    ptr[dev] = p;
  }
  *state = ptr[dev];
  return HIST_OK;
}

void release_staging(hist_stream* st) {
  for (uint32_t i = 0; i < kMaxStaging; ++i) {
    dev_free(st, st->staging[i], st->max_chunk);
    if (st->copied[i]) cudaEventDestroy(st->copied[i]);
    if (st->consumed[i]) cudaEventDestroy(st->consumed[i]);
    st->staging[i] = nullptr;
    st->copied[i] = st->consumed[i] = nullptr;
  }
  if (st->copy_stream) cudaStreamDestroy(st->copy_stream);
  st->copy_stream = nullptr;
  st->depth = 0;
  st->max_chunk = 0;
}

}  // namespace

extern "C" {

void hist_config_init(hist_config* c) {
  if (!c) return;
  memset(c, 0, sizeof(*c));
  c->budget = HIST_BUDGET_MAX;
  c->theta_milli = HIST_THETA_MILLI_DEFAULT;
  c->mode = HIST_MODE_AUTO;
  c->grid = 0;
  c->window = 1;
}

int hist_stream_create(const hist_config* cfg, hist_stream** out) {
  return hist_stream_create_with_allocator(cfg, nullptr, out);
}

int hist_stream_create_with_allocator(const hist_config* cfg, const hist_allocator* alloc, hist_stream** out) {
  if (!out || !config_ok(cfg)) return HIST_EINVAL;
  *out = nullptr;
  if (alloc && (!alloc->alloc) != (!alloc->free)) return HIST_EINVAL;
  hist_stream* st = (hist_stream*)calloc(1, sizeof(hist_stream));
  if (!st) return HIST_ENOMEM;
  st->cfg = *cfg;
  if (alloc) st->alloc = *alloc;
  st->sms = sm_count();
  int rc = flat_kernels_setup();
  if (rc) {
    free(st);
    return rc;
  }
  st->grid = flat_grid(cfg, st->sms);
  rc = dev_alloc(st, (void**)&st->d, sizeof(StreamDev));
  if (rc) {
    free(st);
    return rc;
  }
  cudaError_t e = cudaMemset(st->d, 0, sizeof(StreamDev));
  if (e == cudaSuccess) {
    init_kernel<<<1, HIST_BINS>>>(st->d, cfg->budget);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    dev_free(st, st->d, sizeof(StreamDev));
    free(st);
    return cuda_fail(e);
  }
  st->args = malloc(sizeof(LargeArgs));  // null: launches allocate their own
  *out = st;
  return HIST_OK;
}

int hist_stream_destroy(hist_stream* st) {
  if (!st) return HIST_EINVAL;
  cudaError_t e = cudaDeviceSynchronize();
  release_staging(st);
  dev_free(st, st->d, sizeof(StreamDev));
  free(st->args);
  free(st);
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

int hist_stream_push(hist_stream* st, const uint8_t* d_chunk, size_t n, uint32_t* d_chunk_out,
                     hist_cuda_stream s) {
  if (!st || (!d_chunk && n) || n >= ((size_t)1 << 32)) return HIST_EINVAL;
  return push_chunks(st, 1, &d_chunk, &n, d_chunk_out ? &d_chunk_out : nullptr, (cudaStream_t)s);
}

int hist_stream_push_many(hist_stream* st, uint32_t count, const uint8_t* const* d_chunks, const size_t* sizes,
                          uint32_t* const* d_chunk_outs, hist_cuda_stream s) {
  if (!st || (count && (!d_chunks || !sizes))) return HIST_EINVAL;
  for (uint32_t i = 0; i < count; ++i)
    if ((!d_chunks[i] && sizes[i]) || sizes[i] >= ((size_t)1 << 32)) return HIST_EINVAL;
  if (count == 0) return HIST_OK;
  return push_chunks(st, count, d_chunks, sizes, d_chunk_outs, (cudaStream_t)s);
}

int hist_stream_attach_staging(hist_stream* st, size_t max_chunk, uint32_t depth) {
  if (!st || max_chunk == 0 || max_chunk >= ((size_t)1 << 32) || depth < 2 || depth > kMaxStaging)
    return HIST_EINVAL;
  if (st->depth) return HIST_ESTATE;
  st->max_chunk = max_chunk;  // the staging buffers' size, also when they are freed
  int rc = HIST_OK;
  cudaError_t e = cudaStreamCreateWithFlags(&st->copy_stream, cudaStreamNonBlocking);
  for (uint32_t i = 0; e == cudaSuccess && rc == HIST_OK && i < depth; ++i) {
    rc = dev_alloc(st, (void**)&st->staging[i], max_chunk);
    if (rc == HIST_OK) e = cudaEventCreateWithFlags(&st->copied[i], cudaEventDisableTiming);
    if (e == cudaSuccess && rc == HIST_OK) e = cudaEventCreateWithFlags(&st->consumed[i], cudaEventDisableTiming);
  }
  if (e != cudaSuccess || rc != HIST_OK) {
    release_staging(st);
    return rc != HIST_OK ? rc : (e == cudaErrorMemoryAllocation ? HIST_ENOMEM : cuda_fail(e));
  }
  st->depth = depth;
  st->host_pushes = 0;
  return HIST_OK;
}

int hist_stream_push_host(hist_stream* st, const uint8_t* h_chunk, size_t n, uint32_t* d_chunk_out,
                          hist_cuda_stream s) {
  if (!st || (!h_chunk && n)) return HIST_EINVAL;
  if (!st->depth) return HIST_ESTATE;
  if (n > st->max_chunk) return HIST_EINVAL;
  // Pinned memory is counted in place, a chunk's reads beside the launch
  // before it, as with HIST_OVERLAP_PUSHES (the caller's bytes are complete by
  // contract).  Copied into staging, with the events between copy and count,
  // and so: 64 x 64 KiB 729 and 195 us, 64 x 1 MiB 860 and 403, 16 x 4 MiB 404
  // and 347; 16 x 16 MiB take the link's time both ways (1310 and 1271 in a row).
  if (const uint8_t* d = n ? host_readable(h_chunk, n, (cudaStream_t)s) : nullptr)
    return push_chunks(st, 1, &d, &n, d_chunk_out ? &d_chunk_out : nullptr, (cudaStream_t)s, true);
  const uint32_t b = (uint32_t)(st->host_pushes % st->depth);
  cudaStream_t cs = st->copy_stream;
  // the buffer's previous chunk kernel must be done before it is overwritten
  cudaError_t e = cudaStreamWaitEvent(cs, st->consumed[b], 0);
  if (e == cudaSuccess && n) e = cudaMemcpyAsync(st->staging[b], h_chunk, n, cudaMemcpyHostToDevice, cs);
  if (e == cudaSuccess) e = cudaEventRecord(st->copied[b], cs);
  if (e == cudaSuccess) e = cudaStreamWaitEvent((cudaStream_t)s, st->copied[b], 0);
  if (e != cudaSuccess) return cuda_fail(e);
  const uint8_t* in = st->staging[b];
  int rc = push_chunks(st, 1, &in, &n, d_chunk_out ? &d_chunk_out : nullptr, (cudaStream_t)s);
  if (rc) return rc;
  e = cudaEventRecord(st->consumed[b], (cudaStream_t)s);
  if (e != cudaSuccess) return cuda_fail(e);
  st->host_pushes += 1;
  return HIST_OK;
}

int hist_stream_test_hold_ring(hist_stream* st, uint32_t launches) {
  if (!st || launches == 0 || launches > 1024) return HIST_EINVAL;
  // the next launch's number runs ahead of the launches the device has seen
  // complete, so its ring check waits for launches that never ran
  st->flat_launches += launches;
  return HIST_OK;
}

int hist_stream_trace(hist_stream* st, uint64_t* d_trace, uint32_t capacity_chunks) {
  if (!st || (d_trace && capacity_chunks == 0)) return HIST_EINVAL;
  st->trace = reinterpret_cast<unsigned long long*>(d_trace);
  st->trace_cap = d_trace ? capacity_chunks : 0;
  st->trace_next = 0;
  return HIST_OK;
}

int hist_stream_flush(hist_stream* st, hist_cuda_stream s) {
  (void)s;  // every push completes its chunks' epilogues in its own launches
  return st ? HIST_OK : HIST_EINVAL;
}

int hist_stream_totals(hist_stream* st, uint64_t* d_totals, hist_cuda_stream s) {
  if (!st || !d_totals) return HIST_EINVAL;
  cudaError_t e;
  if ((uintptr_t)d_totals % sizeof(uint64_t) == 0) {
    const StreamDev* d = st->d;
    unsigned long long* out = reinterpret_cast<unsigned long long*>(d_totals);
    void* params[] = {&d, &out};
    e = launch_chained((const void*)totals_copy_kernel, dim3(1), dim3(HIST_BINS), params, 0, (cudaStream_t)s);
  } else {
    e = cudaMemcpyAsync(d_totals, st->d->h.totals, HIST_BINS * sizeof(uint64_t), cudaMemcpyDeviceToDevice,
                        (cudaStream_t)s);
  }
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

int hist_stream_window(hist_stream* st, uint64_t* d_window, hist_cuda_stream s) {
  if (!st || !d_window) return HIST_EINVAL;
  const StreamDev* d = st->d;
  uint32_t window = st->cfg.window;
  bool any = st->chunks_launched > st->resume_chunk;
  unsigned long long* out = reinterpret_cast<unsigned long long*>(d_window);
  void* params[] = {&d, &window, &any, &out};
  const cudaError_t e =
      launch_chained((const void*)window_copy_kernel, dim3(1), dim3(HIST_BINS), params, 0, (cudaStream_t)s);
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

int hist_stream_change(hist_stream* st, uint32_t tau_milli, hist_change_result* d_res, hist_cuda_stream s) {
  if (!st || !d_res || tau_milli > 1000) return HIST_EINVAL;
  const StreamDev* d = st->d;
  uint32_t window = st->cfg.window;
  bool any = st->chunks_launched > st->resume_chunk;
  void* params[] = {&d, &window, &any, &tau_milli, &d_res};
  const cudaError_t e =
      launch_chained((const void*)stream_change_kernel, dim3(1), dim3(HIST_BINS), params, 0, (cudaStream_t)s);
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

int hist_stream_get_state(hist_stream* st, hist_stream_state* h, hist_cuda_stream s) {
  if (!st || !h) return HIST_EINVAL;
  StreamHead tmp;
  cudaError_t e = cudaMemcpyAsync(&tmp, &st->d->h, sizeof(StreamHead), cudaMemcpyDeviceToHost, (cudaStream_t)s);
  if (e == cudaSuccess) e = cudaStreamSynchronize((cudaStream_t)s);
  if (e != cudaSuccess) return cuda_fail(e);
  memset(h, 0, sizeof(*h));
  memcpy(h->totals, tmp.totals, sizeof(h->totals));
  memcpy(h->last_hist, tmp.last_hist, sizeof(h->last_hist));
  h->pattern = tmp.pat[tmp.cur & 1u];
  h->last_pattern = tmp.pat[(tmp.cur & 1u) ^ 1u];
  h->chunks = tmp.chunks;
  h->flag = tmp.flag;
  h->last_kernel = tmp.last_kernel;
  h->status = tmp.status;
  h->recounted = tmp.recounted;
  return HIST_OK;
}

int hist_stream_set_state(hist_stream* st, const hist_stream_state* h, hist_cuda_stream s) {
  if (!st || !h) return HIST_EINVAL;
  if (hist_pattern_check(&h->pattern) != HIST_OK || hist_pattern_check(&h->last_pattern) != HIST_OK ||
      h->pattern.budget != st->cfg.budget || h->flag > HIST_FLAG_ADAPTIVE)
    return HIST_EINVAL;
  StreamHead tmp;
  memset(&tmp, 0, sizeof(tmp));
  memcpy(tmp.totals, h->totals, sizeof(tmp.totals));
  memcpy(tmp.last_hist, h->last_hist, sizeof(tmp.last_hist));
  tmp.pat[0] = h->pattern;
  tmp.pat[1] = h->last_pattern;
  tmp.chunks = h->chunks;
  tmp.flag = h->flag;
  tmp.last_kernel = h->last_kernel;
  // launches go on to be numbered (a graph captured before may write its own
  // numbers), none before them is running; the scratch is zero again
  tmp.launches_done = st->prev_launch = st->flat_launches;
  cudaError_t e = cudaMemsetAsync(st->d, 0, sizeof(StreamDev), (cudaStream_t)s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(&st->d->h, &tmp, sizeof(StreamHead), cudaMemcpyHostToDevice, (cudaStream_t)s);
  if (e == cudaSuccess) e = cudaStreamSynchronize((cudaStream_t)s);
  st->flat_chunks = 0;  // the rings restart with the zeroed scratch
  st->resume_chunk = st->chunks_launched;  // and so does the moving window
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

int hist_stream_run_noalloc(const uint8_t* const* d_chunks, const size_t* sizes, uint32_t count,
                            const hist_config* cfg, uint32_t* d_chunk_outs, uint64_t* d_totals, uint32_t* d_status,
                            hist_cuda_stream s) {
  if (!cfg || !d_totals || count == 0 || count > HIST_NOALLOC_MAX_CHUNKS || !d_chunks || !sizes) return HIST_EINVAL;
  hist_config c = *cfg;
  c.grid = 0;  // ignored: the counting launch takes every resident CTA
  if (!config_ok(&c)) return HIST_EINVAL;
  for (uint32_t i = 0; i < count; ++i)
    if ((!d_chunks[i] && sizes[i]) || sizes[i] >= ((size_t)1 << 32)) return HIST_EINVAL;
  void* state = nullptr;
  int rc = noalloc_setup(&state);
  if (rc) return rc;
  // a fresh stream on the fixed state: the same launches as hist_stream_push_many
  hist_stream st;
  memset(&st, 0, sizeof(st));
  st.cfg = c;
  st.d = static_cast<StreamDev*>(state);
  st.sms = sm_count();
  st.grid = flat_grid(&c, st.sms);
  uint32_t* outs[HIST_NOALLOC_MAX_CHUNKS];
  for (uint32_t i = 0; i < count; ++i) outs[i] = d_chunk_outs ? d_chunk_outs + (size_t)i * HIST_BINS : nullptr;
  cudaError_t e = cudaMemsetAsync(state, 0, sizeof(StreamDev), (cudaStream_t)s);
  if (e != cudaSuccess) return cuda_fail(e);
  init_kernel<<<1, HIST_BINS, 0, (cudaStream_t)s>>>(st.d, c.budget);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e);
  rc = push_chunks(&st, count, d_chunks, sizes, outs, (cudaStream_t)s);
  if (rc) return rc;
  noalloc_out_kernel<<<1, HIST_BINS, 0, (cudaStream_t)s>>>(st.d, reinterpret_cast<unsigned long long*>(d_totals),
                                                           d_status);
  e = cudaGetLastError();
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

}  // extern "C"
