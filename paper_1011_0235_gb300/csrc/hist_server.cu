// hist_server.cu -- a serving loop for histogram requests on many streams.
//
// Each request is the next chunk of one of `streams` independent streams; a
// stream's adaptive state (the switch flag, the binning pattern and the
// layout derived from it, the totals and the last histogram) stays on the
// device, as hist_stream_push would leave it (Sec. III.B / III.C).
//
// Continuous batching on the host: submitted requests wait in a FIFO queue;
// whenever a batch slot is free, the queued requests that fit the HBM byte
// budget and whose stream's last request has completed form a batch, launched
// on the slot's own CUDA stream, so batches overlap on the device.  A batch
// is one kernel with no device-side waits: the host splits the requests among
// the CTAs by a cost model (bytes plus a fixed cost per request), each CTA
// counts its pieces and adds them into the requests' accumulators; the CTA
// that completes a request runs its epilogue.  Small requests are counted
// whole by groups of warps, each of which runs its requests' epilogues itself.
// A request counted whole by one CTA skips the accumulator.
//
// Once a request's output is written, its epilogue writes the batch's sequence
// number into the request's completion word in pinned host memory, so the
// host sees each request complete without waiting for the rest of its batch,
// and the stream's next request may run in a batch that fills the SMs while
// this one drains.  Every kernel and pattern counts in the lane-private table,
// so nothing that the epilogue does after that has to be waited for: the
// totals are added to, and the rest of the stream's state follows from its
// last two requests' histograms alone, each of which writes a record of its
// own (SrvRec), then the request's state word.  A batch whose words are all
// there is done: its slot (its scratch and its bytes of the budget) is
// released without a driver call.
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>
#include <time.h>

#include <list>
#include <new>
#include <vector>

#include "hist.h"
#include "hist_device.cuh"
#include "hist_internal.h"
#include "hist_plan.h"

using namespace histdev;
using namespace histlib;

namespace {

constexpr uint32_t kSrvMaxBatch = HIST_SERVER_MAX_BATCH;
constexpr uint32_t kSrvMaxSlots = HIST_SERVER_MAX_INFLIGHT;
// cost of a request beyond its bytes, in bytes: about what one CTA counts
// while it reduces its table, publishes its piece and runs a request's
// epilogue and completion
constexpr unsigned long long kReqCost = 256ull << 10;
// the same for a small request, counted beside three others (64 to 160 KiB,
// and 128 KiB instead of 256 above, measured within 2 % of these on a burst)
constexpr unsigned long long kSmallReqCost = 96ull << 10;
constexpr uint32_t kSmallReq = 256u << 10;  // largest request a group counts
// cost units per CTA of a batch (the grid is at most every resident CTA);
// from launch to completion a request takes 10.9 us at the median with 32
// KiB, 11.4 with 64, 12.4 with 128 (50k requests/s)
constexpr unsigned long long kCtaCost = 32ull << 10;
constexpr int kGroups = 4;
constexpr int kGroupThreads = kThreads / kGroups;
static_assert(kGroupThreads == HIST_BINS, "one bin per thread of a group");
constexpr int kEpiBar = 1 + kGroups;  // named barrier of the threads of a CTA's epilogue
// dynamic shared memory: the groups' tables in a batch with groups, else one
constexpr size_t kSrvSmem = (size_t)kTableWords * 4;
constexpr size_t kSrvGroupSmem = kGroups * kSrvSmem;
// request-table capacities of the kernel variants (the table travels in the
// launch's parameters, 24 bytes per request; from the launch call to a word
// seen on the host, an empty kernel takes 7.6 us with few parameters, 8.7 with
// 9.6 KB, 10.2 with 28 KB)
constexpr uint32_t kSmallCap = 32, kMidCap = 256;

__host__ __device__ __forceinline__ unsigned long long srv_cost(unsigned long long n) {
  return n + (n <= kSmallReq ? kSmallReqCost : kReqCost);
}

// Per-stream state on the device: the totals, and the records of the stream's
// last two requests, request c's (from 0) in rec[c & 1].  The state is the
// last record's, with the pattern and the kernel choice of the one before.
// Admission of request c waits for request c - 2's state word, so a record is
// never written by two requests at a time.
struct SrvRec {
  uint32_t hist[HIST_BINS];
  hist_pattern pat;  // derived from it
  uint32_t flag;     // the switch after it
};
struct SrvStream {
  unsigned long long totals[HIST_BINS];
  SrvRec rec[2];
};

struct SrvReq {
  const uint8_t* in;
  uint32_t* out;
  uint32_t n;
  uint32_t stream;  // 2 stream + the request's record
};

// Per batch slot, on the device.  Both return to zero when a request's
// epilogue has read them, so a slot needs clearing only once.
struct SrvSlot {
  unsigned long long acc[kSrvMaxBatch][HIST_BINS];  // requests counted by several CTAs (acc_word)
  uint32_t rbins[kSrvMaxBatch];                     // bins complete, where several CTAs completed a request
};

struct SrvCommon {
  SrvStream* streams;
  SrvSlot* slot;
  // the slot's words in pinned, mapped host memory: request r's completion
  // word in done[r], its state word in done[kSrvMaxBatch + r]
  uint32_t* done;
  uint32_t seq;  // the batch's sequence number, written into both words of request r
  uint32_t count;
  uint32_t budget;
  uint32_t theta;
};

template <uint32_t CAP>
struct SrvArgs {
  SrvCommon c;
  RangePlan plan;
  SrvReq req[CAP];
};

// A piece of a request, bytes [b0, e0) (e0 = 0: an empty request), as the CTAs
// keep it in shared memory (the table sits in the kernel's parameters, read
// through the constant cache: 0.5 - 1 us a miss).
struct SrvPiece {
  SrvReq q;
  uint32_t r;  // the request's number in the batch
  uint32_t b0, e0;
};

constexpr uint32_t kSrvItems = 2 * kWarps;  // requests the groups take at a time

struct SrvShared {
  EpiShared es[kGroups];
  uint32_t res[HIST_BINS];
  uint32_t eh[2][HIST_BINS];  // edge bytes of the CTA's pieces, in turn
  int last;
  uint16_t wl[kSrvMaxBatch];  // whole requests left to the groups
  GroupItem items[kSrvItems]; // the ones the groups are at (j: the stream)
  uint32_t item_r[kSrvItems]; // their numbers in the batch
  SrvReq win[kWarps];         // the requests of the range the CTA is at
  SrvPiece piece[kWarps];     // its pieces of them
  uint32_t npiece, nwl;
  unsigned long long pos;     // cost position of the request after them
  uint32_t geh[kGroups][HIST_BINS];
};

// Request r (n bytes) is complete, threads t = 0..255 (which share named
// barrier `id`) hold a bin each in h: write its output and publish the
// request's completion word, then add to its stream's totals, write its record
// (`sr`: SrvReq::stream) and publish its state word.
__device__ __noinline__ void srv_epilogue(const SrvCommon& a, uint32_t r, uint32_t sr, uint32_t n, uint32_t* out,
                                          uint32_t h, EpiShared& es, int t, int id) {
  SrvStream* st = a.streams + (sr >> 1);
  const GroupBar<HIST_BINS> bar = {id};
  if (out) out[t] = h;
  // the output precedes the completion word: the barrier orders the threads'
  // writes before thread 0's system-scope release store, whose release is
  // cumulative (an explicit system fence before it measured 1.5 % slower on
  // a burst of 4000 requests and orders nothing more)
  bar.sync();
  if (t == 0)
    asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(a.done + r), "r"(a.seq) : "memory");
  if (h) atomicAdd(&st->totals[t], (unsigned long long)h);
  SrvRec* rec = st->rec + (sr & 1u);
  rec->hist[t] = h;
  BinPlace place;
  const hist_degeneracy_result d = block_pattern(h, n, a.budget, a.theta, es, t, bar, place);
  store_place(rec->pat, t, a.budget, place);
  if (t == 0) rec->flag = d.flag;
  // (the same release argument as for the completion word)
  bar.sync();
  if (t == 0)
    asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(a.done + kSrvMaxBatch + r), "r"(a.seq) : "memory");
}

// Count piece d (the CTA's k-th) into the table, which is clear before and
// after, and publish it: into the request's accumulator, or, when it is the
// whole request, straight into the request's epilogue.  Epilogues are run by
// the first 256 threads while the others go on to the CTA's next piece.  All
// threads call.
__device__ __forceinline__ void srv_piece(const SrvCommon& a, const SrvPiece& d, uint32_t k, uint32_t* table,
                                          SrvShared& ss) {
  const int t = threadIdx.x;
  uint32_t h = 0;
  if (d.e0) {
    piece_count(d.q.in + d.b0, d.e0 - d.b0, table, ss.eh[k & 1], nullptr, nullptr);
    __syncthreads();
    lane_reduce<kThreads, true>(table, ss.res, t);
    __syncthreads();
    if (t < HIST_BINS) {
      h = ss.res[t] + ss.eh[k & 1][t];
      ss.eh[k & 1][t] = 0;
    }
  }
  bool complete = d.e0 - d.b0 == d.q.n;
  if (!complete) {
    unsigned long long* acc = &a.slot->acc[d.r][t & (HIST_BINS - 1)];
    bool done = false;
    if (t < HIST_BINS) {
      const unsigned long long add = acc_word(h, acc_blocks(d.q.in, d.b0, d.e0), 0);
      const unsigned long long sum = atomicAdd(acc, add) + add;
      done = ((uint32_t)(sum >> 32) & kAccBlockMask) == acc_blocks(d.q.in, 0, d.q.n);
      h = (uint32_t)sum;
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
        ss.last = atomicAdd(&a.slot->rbins[d.r], (uint32_t)bins) + (uint32_t)bins == HIST_BINS;
        __threadfence();
      }
      __syncthreads();
      complete = ss.last != 0;
      if (complete) {
        if (t < HIST_BINS) {
          h = (uint32_t)__ldcg(acc);
          *acc = 0;
        }
        if (t == 0) a.slot->rbins[d.r] = 0;
      }
    }
  }
  if (complete && t < HIST_BINS) srv_epilogue(a, d.r, d.q.stream, d.q.n, d.q.out, h, ss.es[0], t, kEpiBar);
}

// Requests [r0, r0 + kWarps), the first at cost position ss.pos: into ss.win,
// a warp each (their constant-cache misses overlap), then warp 0, a request
// per lane, lists the CTA's pieces of them and, in ss.wl, the whole ones left
// to the groups.  All threads call (begins and ends with a barrier).
template <uint32_t CAP>
__device__ __forceinline__ void srv_window(const SrvArgs<CAP>& args, uint32_t r0, SrvShared& ss) {
  const uint32_t w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const RangePlan& p = args.plan;
  __syncthreads();
  if (r0 + w < args.c.count) {
    const SrvReq q = args.req[r0 + w];
    if (lane == 0) ss.win[w] = q;
  }
  __syncthreads();
  if (w == 0) {
    const unsigned long long lo = p.lo[blockIdx.x], hi = p.lo[blockIdx.x + 1];
    const bool in = r0 + lane < args.c.count;
    const SrvReq q = in ? ss.win[lane] : SrvReq{nullptr, nullptr, 0, 0};
    const uint32_t n = q.n;
    const unsigned long long c = in ? srv_cost(n) : 0ull;
    unsigned long long x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if ((int)lane >= o) x += y;
    }
    const unsigned long long p0 = ss.pos + x - c;
    // this CTA's bytes of the request: its cost range cut to [0, n), each
    // cut moved to a 32 KiB boundary of the request's memory; a request of
    // at most a quarter of a CTA's range is not split (the range holding its
    // first cost position counts it whole, with no accumulator), and a small
    // one of those is left to the groups
    bool piece = false, item = false;
    unsigned long long b0 = 0, e0 = 0;
    if (in && p0 < hi) {
      if (n == 0 || plan_whole(n, p.range)) {
        item = p0 >= lo && n != 0 && n <= p.group_max;
        piece = p0 >= lo && !item;
        e0 = n;
      } else {
        b0 = lo > p0 ? split_point(q.in, lo - p0) : 0ull;
        e0 = split_point(q.in, hi - p0);
        if (e0 > (unsigned long long)n) e0 = n;
        piece = b0 < e0;
      }
    }
    const unsigned mp = __ballot_sync(0xffffffffu, piece), mi = __ballot_sync(0xffffffffu, item);
    const unsigned lt = (1u << lane) - 1u;
    if (piece) ss.piece[__popc(mp & lt)] = SrvPiece{q, r0 + lane, (uint32_t)b0, (uint32_t)e0};
    if (item) ss.wl[ss.nwl + __popc(mi & lt)] = (uint16_t)(r0 + lane);
    __syncwarp();
    if (lane == 31) {
      ss.pos = p0 + c;
      ss.npiece = __popc(mp);
      ss.nwl += __popc(mi);
    }
  }
  __syncthreads();
}

// Request r of the batch as the groups' k-th item.  A warp calls.
__device__ __forceinline__ void srv_item(const SrvReq& q, uint32_t r, uint32_t k, SrvShared& ss) {
  if ((threadIdx.x & 31) == 0) {
    const Split sp = split_bytes(q.in, q.n);
    GroupItem it;
    it.body = reinterpret_cast<const uint4*>(q.in + sp.head);
    it.out = q.out;
    it.nvec = (uint32_t)sp.nvec;
    it.n = q.n;
    it.j = q.stream;
    it.edges = (uint32_t)sp.head | ((uint32_t)sp.tail << 8);
    ss.items[k] = it;
    ss.item_r[k] = r;
  }
}

// This group's requests g, g + kGroups, ... of the first `count` in ss.items
// (its table and edge histogram clear).  All of the group's threads call.
__device__ __forceinline__ void srv_group(const SrvCommon& a, uint32_t count, uint32_t* tables, SrvShared& ss) {
  const int g = threadIdx.x / kGroupThreads, t = threadIdx.x % kGroupThreads;
  const GroupBar<kGroupThreads> bar = {g + 1};
  uint32_t* table = tables + (size_t)g * kTableWords;
  const uint32_t base = smem_addr(table) + ((t & 31) << 2);
  uint32_t i = (uint32_t)g;
  if (i >= count) return;
  for (; i < count; i += kGroups) {
    const GroupItem& it = ss.items[i];
    const uint32_t edge = group_edge(it, t);
    uint4 v[kLaneLoads];
    const LaneRange r = lane_range(it.body, 0, it.nvec, t);
    lane_load<kLaneLoads, kGroupThreads>(v, r);
    if (edge < 0x100u) atomicAdd(&ss.geh[g][edge], 1u);
    lane_count<kLaneLoads, kGroupThreads>(v, r, base);
    bar.sync();
    uint32_t h = lane_row(table, t);
    if (it.edges) {
      h += ss.geh[g][t];
      ss.geh[g][t] = 0;
    }
    // (its barriers also keep the next request's increments from this one's
    // reduction)
    srv_epilogue(a, ss.item_r[i], it.j, it.n, it.out, h, ss.es[g], t, g + 1);
  }
}

// One CTA of 1024 threads per SM, four loads in flight per thread (as the
// stream's counting kernel).  Bound by the HBM read in a burst and by latency
// (launch, one round of loads, an accumulator's and an epilogue's round trips)
// on single requests.  Before -- per-warp tables for the streams the switch
// called plain, the default pattern's slot lookup for first requests, a cost
// prefix with 64-bit divisions in every CTA -- and now: a burst of 600
// requests of 4 KiB .. 64 MiB on 256 streams 1320 -> 740 us, one of 4000 3.48
// -> 6.1 TB/s; at 50k requests/s p50 18.3 -> 13.5 us, p99 40.7 -> 25.8.  Where
// streams have many requests waiting, the chain of a stream's requests bounds,
// 12 us a request: 600 of 1 .. 8 KiB on 16 streams 788 us with the stream held
// until its state was written and an event per batch, 665 without, 636 with
// the tables of only the groups that have a request cleared.
template <uint32_t CAP>
__global__ void __launch_bounds__(kThreads, 1) server_batch_kernel(const __grid_constant__ SrvArgs<CAP> args) {
  extern __shared__ __align__(16) uint32_t tables[];
  __shared__ SrvShared ss;
  const SrvCommon& a = args.c;
  const RangePlan& p = args.plan;
  const int t = threadIdx.x;
  const bool groups = p.groups[blockIdx.x >> 5] >> (blockIdx.x & 31) & 1u;
  const uint32_t s0 = p.s[blockIdx.x], s1 = p.s[blockIdx.x + 1];
  uint32_t nwl = s1 - s0;
  int first = (int)s0;
  if (!groups) {
    zero_table(tables);
    if (t < HIST_BINS) ss.eh[0][t] = ss.eh[1][t] = 0;
    if (t == 0) {
      ss.pos = p.pre[blockIdx.x];
      ss.nwl = 0;
    }
    uint32_t k = 0;
    for (uint32_t r0 = p.j[blockIdx.x]; r0 < a.count; r0 += kWarps) {
      srv_window(args, r0, ss);
      for (uint32_t i = 0; i < ss.npiece; ++i) srv_piece(a, ss.piece[i], k++, tables, ss);
      if (ss.pos >= p.lo[blockIdx.x + 1]) break;
    }
    __syncthreads();
    nwl = ss.nwl;
    first = -1;
  }
  if (nwl == 0) return;
  const uint32_t w = (uint32_t)t >> 5;
  auto number = [&](uint32_t k) { return first >= 0 ? (uint32_t)first + k : (uint32_t)ss.wl[k]; };
  // (a request's parameters arrive while the groups that have one clear their
  // tables)
  const uint32_t r = w < nwl ? number(w) : 0;
  const SrvReq q = w < nwl ? args.req[r] : SrvReq{nullptr, nullptr, 0, 0};
  if (!groups) __syncthreads();
  {
    const int g = t / kGroupThreads, gt = t % kGroupThreads;
    uint4* t4 = reinterpret_cast<uint4*>(tables + (size_t)g * kTableWords);
    if ((uint32_t)g < nwl) {
#pragma unroll
      for (int i = 0; i < kTableWords / 4 / kGroupThreads; ++i) t4[gt + i * kGroupThreads] = make_uint4(0, 0, 0, 0);
    }
    ss.geh[g][gt] = 0;
  }
  if (w < nwl) srv_item(q, r, w, ss);
  for (uint32_t i0 = 0; i0 < nwl; i0 += kSrvItems) {
    if (i0) __syncthreads();
    for (uint32_t k = w; k < kSrvItems && i0 + k < nwl; k += kWarps)
      if (i0 || k >= kWarps) srv_item(args.req[number(i0 + k)], number(i0 + k), k, ss);
    __syncthreads();
    srv_group(a, nwl - i0 < kSrvItems ? nwl - i0 : kSrvItems, tables, ss);
  }
}

// Every stream starts with the plain kernel and the default pattern, in both
// records (one CTA).
__global__ void __launch_bounds__(HIST_BINS) server_init_kernel(SrvStream* s, uint32_t streams, uint32_t budget) {
  __shared__ EpiShared es;
  const int t = threadIdx.x;
  BinPlace place;
  block_pattern(0u, 0ull, budget, HIST_THETA_MILLI_DEFAULT, es, t, CtaBar(), place);
  for (uint32_t i = 0; i < streams; ++i)
    for (int k = 0; k < 2; ++k) {
      store_place(s[i].rec[k].pat, t, budget, place);
      if (t == 0) s[i].rec[k].flag = HIST_FLAG_PLAIN;
    }
}

uint64_t now_ns() {
  timespec ts;
  clock_gettime(CLOCK_MONOTONIC, &ts);
  return (uint64_t)ts.tv_sec * 1000000000ull + (uint64_t)ts.tv_nsec;
}

struct PendingReq {
  uint32_t stream;
  const uint8_t* in;
  size_t n;
  uint32_t* out;
  uint64_t tag;
  uint64_t submit_ns;
};

// A stream as the host sees it.
struct HostStream {
  uint64_t admitted = 0;   // requests put on the GPU
  uint64_t scan = 0;       // the last admission scan that met the stream
  bool busy = false;       // the last one's completion has not been returned
  bool owed[2] = {false, false};  // a request that writes record k has not published its state word
};

struct BatchSlot {
  bool busy = false;
  cudaStream_t cs = nullptr;
  SrvSlot* d_slot = nullptr;
  // completion words of the batch's requests, then their state words
  // (pinned, mapped: 2 kSrvMaxBatch words)
  uint32_t* h_done = nullptr;
  uint32_t* d_done = nullptr;  // the same words as the device sees them
  uint32_t seq = 0;            // the running batch's sequence number
  std::vector<PendingReq> reqs;
  std::vector<uint8_t> rec;       // the record that the request writes
  std::vector<uint8_t> reported;  // the request's completion has been returned
  std::vector<uint8_t> released;  // the request's state word has been seen
  uint32_t n_reported = 0;
  uint32_t n_released = 0;
  uint32_t polls = 0;  // polls of the running batch
  uint64_t admit_ns = 0;
  uint64_t bytes = 0;
};

}  // namespace

struct hist_server {
  hist_server_config cfg;
  SrvStream* d_streams = nullptr;
  std::vector<HostStream> streams;
  uint64_t scan = 0;  // number of the last admission scan
  std::list<PendingReq> queue;  // FIFO; admission erases from the middle
  std::vector<std::list<PendingReq>::iterator> pick;  // the admission scan's requests
  BatchSlot slot[kSrvMaxSlots];
  uint64_t inflight_bytes = 0;
  uint32_t* h_done = nullptr;  // pinned: 2 kSrvMaxBatch words per batch slot
  uint32_t seq = 0;            // sequence number of the last batch launched
  int sms = 0;
  int max_grid = 0;                          // resident CTAs of the batch kernel
  SrvArgs<kSrvMaxBatch>* args = nullptr;     // parameter block of the next launch
  hist_server_stats stats;
};

namespace {

bool server_config_ok(const hist_server_config* c) {
  return c && c->streams >= 1 && c->streams <= HIST_SERVER_MAX_STREAMS && c->max_batch >= 1 &&
         c->max_batch <= kSrvMaxBatch && c->max_inflight >= 1 && c->max_inflight <= kSrvMaxSlots &&
         c->hbm_budget > 0 && c->theta_milli <= 1000 && c->pattern_budget >= HIST_BUDGET_MIN &&
         c->pattern_budget <= HIST_BUDGET_MAX && c->mode <= HIST_MODE_ADAPTIVE;
}

// Return the completions of finished requests -- those whose completion word
// holds their batch's sequence number -- writing at most `cap` of them to
// `out` (out null: discard them), which gives their streams back to admission,
// and release the slots of the batches whose words are all there; returns how
// many completions were written or discarded.
uint32_t retire(hist_server* s, hist_completion* out, uint32_t cap, int* err) {
  uint32_t n = 0;
  for (uint32_t k = 0; k < s->cfg.max_inflight; ++k) {
    BatchSlot& f = s->slot[k];
    if (!f.busy) continue;
    const uint32_t count = (uint32_t)f.reqs.size();
    // the words are plain reads of host memory; the driver is asked every
    // 32nd poll, so that a failed batch is still seen
    bool all = false;
    if ((++f.polls & 31u) == 0) {
      const cudaError_t q = cudaStreamQuery(f.cs);
      if (q != cudaSuccess && q != cudaErrorNotReady) {
        *err = cuda_fail(q);
        return n;
      }
      all = q == cudaSuccess;
    }
    for (uint32_t i = 0; i < count; ++i) {
      const PendingReq& r = f.reqs[i];
      HostStream& h = s->streams[r.stream];
      // (the acquires pair with the epilogue's releases: what it writes
      // before a word is written when the word is seen)
      if (!f.reported[i] && !(out && n >= cap) && (all || __atomic_load_n(f.h_done + i, __ATOMIC_ACQUIRE) == f.seq)) {
        if (out) {
          hist_completion& c = out[n];
          c.tag = r.tag;
          c.stream = r.stream;
          c.status = 0;
          c.bytes = r.n;
          c.submit_ns = r.submit_ns;
          c.admit_ns = f.admit_ns;
          c.done_ns = now_ns();
        }
        ++n;
        h.busy = false;
        f.reported[i] = 1;
        f.n_reported += 1;
        s->stats.completed += 1;
        s->stats.bytes += r.n;
      }
      if (!f.released[i] && (all || __atomic_load_n(f.h_done + kSrvMaxBatch + i, __ATOMIC_ACQUIRE) == f.seq)) {
        h.owed[f.rec[i]] = false;
        f.released[i] = 1;
        f.n_released += 1;
      }
    }
    if (f.n_reported < count || f.n_released < count) continue;
    // the whole batch is done (the next one in this slot follows it on the
    // slot's CUDA stream): its bytes go back to admission
    s->inflight_bytes -= f.bytes;
    f.reqs.clear();
    f.busy = false;
  }
  return n;
}

// Launch one batch if a slot is free and the queue holds admissible requests.
// FIFO order; only each stream's first queued request is a candidate, and
// only if the completion of the stream's last request has been returned and
// its record is free; the scan stops at the first
// candidate that does not fit the byte budget, so no request waits forever
// behind smaller later ones; it ends once every stream has been met.  A
// batch is launched whatever its size: one formed while the batches on the
// GPU hold every SM starts on the SMs their last CTAs leave (waiting for a
// quarter of a full batch instead measured no faster on a burst of 4000
// requests, and raised p99 at 50k requests/s from 44 to 55 us).
int admit(hist_server* s) {
  BatchSlot* f = nullptr;
  for (uint32_t k = 0; k < s->cfg.max_inflight; ++k)
    if (!s->slot[k].busy) {
      f = &s->slot[k];
      break;
    }
  if (!f || s->queue.empty()) return HIST_OK;
  s->pick.clear();
  uint64_t bytes = 0;
  uint32_t met = 0;  // streams met by the scan
  const uint64_t mark = ++s->scan;
  for (auto it = s->queue.begin();
       it != s->queue.end() && s->pick.size() < s->cfg.max_batch && met < s->cfg.streams; ++it) {
    const PendingReq& r = *it;
    HostStream& h = s->streams[r.stream];
    if (h.scan == mark) continue;  // not the stream's first: keep its order
    h.scan = mark;
    ++met;
    if (h.busy || h.owed[h.admitted & 1u]) continue;
    if (s->inflight_bytes + bytes + r.n > s->cfg.hbm_budget) {
      s->stats.deferred += 1;
      break;
    }
    bytes += r.n;
    s->pick.push_back(it);
  }
  if (s->pick.empty()) return HIST_OK;
  f->reqs.clear();
  f->bytes = bytes;
  for (const auto& it : s->pick) {
    f->reqs.push_back(*it);
    s->queue.erase(it);
  }
  const uint32_t count = (uint32_t)f->reqs.size();
  // the launch's parameters: common fields, then the request table
  if (++s->seq == 0) s->seq = 1;  // completion words start at 0: never a batch's number
  f->seq = s->seq;
  f->reported.assign(count, 0);
  f->released.assign(count, 0);
  f->rec.resize(count);
  f->n_reported = 0;
  f->n_released = 0;
  f->polls = 0;
  SrvArgs<kSrvMaxBatch>* a = s->args;
  a->c.streams = s->d_streams;
  a->c.slot = f->d_slot;
  a->c.done = f->d_done;
  a->c.seq = f->seq;
  a->c.count = count;
  a->c.budget = s->cfg.pattern_budget;
  a->c.theta = s->cfg.theta_milli;
  for (uint32_t i = 0; i < count; ++i) {
    const PendingReq& r = f->reqs[i];
    HostStream& h = s->streams[r.stream];
    f->rec[i] = (uint8_t)(h.admitted++ & 1u);
    h.busy = h.owed[f->rec[i]] = true;
    a->req[i].in = r.in;
    a->req[i].out = r.out;
    a->req[i].n = (uint32_t)r.n;
    a->req[i].stream = 2 * r.stream + f->rec[i];
  }
  PlanCosts<kSrvMaxBatch> pc;
  auto size = [&](uint32_t i) { return (unsigned long long)a->req[i].n; };
  plan_costs(&pc, count, size, [&](uint32_t i) { return srv_cost(a->req[i].n); });
  unsigned long long grid = (pc.pos[count] + kCtaCost - 1) / kCtaCost;
  if (grid > (unsigned long long)s->max_grid) grid = (unsigned long long)s->max_grid;
  if (grid < 1) grid = 1;
  plan_ranges(&a->plan, pc, count, (uint32_t)grid, kSmallReq, size);
  // the smaller variants' parameters are a prefix of the large one's
  static_assert(offsetof(SrvArgs<kSmallCap>, req) == offsetof(SrvArgs<kSrvMaxBatch>, req) &&
                    offsetof(SrvArgs<kMidCap>, req) == offsetof(SrvArgs<kSrvMaxBatch>, req),
                "parameter layout");
  static_assert(sizeof(SrvArgs<kSrvMaxBatch>) <= 32764, "kernel parameters are limited to 32764 bytes");
  void* params[] = {a};
  const void* fn = count <= kSmallCap ? (const void*)server_batch_kernel<kSmallCap>
                   : count <= kMidCap ? (const void*)server_batch_kernel<kMidCap>
                                      : (const void*)server_batch_kernel<kSrvMaxBatch>;
  cudaError_t e = cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(kThreads), params,
                                   a->plan.group_max ? kSrvGroupSmem : kSrvSmem, f->cs);
  if (e != cudaSuccess) {
    // nothing was enqueued: the requests go back to the head of the queue
    for (uint32_t i = 0; i < count; ++i) {
      HostStream& h = s->streams[f->reqs[i].stream];
      h.admitted -= 1;
      h.busy = h.owed[f->rec[i]] = false;
    }
    s->queue.insert(s->queue.begin(), f->reqs.begin(), f->reqs.end());
    f->reqs.clear();
    return cuda_fail(e);
  }
  f->busy = true;
  f->admit_ns = now_ns();
  s->inflight_bytes += f->bytes;
  s->stats.batches += 1;
  return HIST_OK;
}

bool server_idle(const hist_server* s) {
  if (!s->queue.empty()) return false;
  for (uint32_t k = 0; k < s->cfg.max_inflight; ++k)
    if (s->slot[k].busy) return false;
  return true;
}

}  // namespace

extern "C" {

void hist_server_config_init(hist_server_config* c) {
  if (!c) return;
  memset(c, 0, sizeof(*c));
  c->streams = 256;
  c->max_batch = 256;
  c->max_inflight = 4;
  c->theta_milli = HIST_THETA_MILLI_DEFAULT;
  c->pattern_budget = HIST_BUDGET_MAX;
  c->mode = HIST_MODE_AUTO;
  c->hbm_budget = 32ull << 30;
}

int hist_server_create(const hist_server_config* cfg, hist_server** out) {
  if (!out || !server_config_ok(cfg)) return HIST_EINVAL;
  *out = nullptr;
  hist_server* s = new (std::nothrow) hist_server();
  if (!s) return HIST_ENOMEM;
  s->cfg = *cfg;
  s->streams.resize(cfg->streams);
  s->sms = sm_count();
  memset(&s->stats, 0, sizeof(s->stats));
  static int attr_small[kMaxDevices], attr_mid[kMaxDevices], attr_large[kMaxDevices];
  int rc = s->sms > 0 ? HIST_OK : HIST_ECUDA;
  if (rc == HIST_OK) rc = ensure_smem_attr_bytes((const void*)server_batch_kernel<kSmallCap>, attr_small, kSrvGroupSmem);
  if (rc == HIST_OK) rc = ensure_smem_attr_bytes((const void*)server_batch_kernel<kMidCap>, attr_mid, kSrvGroupSmem);
  if (rc == HIST_OK) rc = ensure_smem_attr_bytes((const void*)server_batch_kernel<kSrvMaxBatch>, attr_large, kSrvGroupSmem);
  if (rc == HIST_OK) {
    int per_sm = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, (const void*)server_batch_kernel<kSrvMaxBatch>, kThreads, kSrvGroupSmem);
    if (e != cudaSuccess) rc = cuda_fail(e);
    s->max_grid = s->sms * (per_sm > 0 ? per_sm : 1);
    if (s->max_grid > (int)kPlanCtas) s->max_grid = (int)kPlanCtas;
  }
  s->args = new (std::nothrow) SrvArgs<kSrvMaxBatch>();
  if (!s->args && rc == HIST_OK) rc = HIST_ENOMEM;
  if (rc == HIST_OK) {
    cudaError_t e = cudaMalloc((void**)&s->d_streams, sizeof(SrvStream) * cfg->streams);
    if (e == cudaSuccess) e = cudaMemset(s->d_streams, 0, sizeof(SrvStream) * cfg->streams);
    const size_t done_bytes = sizeof(uint32_t) * 2 * kSrvMaxBatch * kSrvMaxSlots;
    if (e == cudaSuccess) e = cudaHostAlloc((void**)&s->h_done, done_bytes, cudaHostAllocMapped);
    if (e == cudaSuccess) memset(s->h_done, 0, done_bytes);
    for (uint32_t k = 0; e == cudaSuccess && k < cfg->max_inflight; ++k) {
      BatchSlot& f = s->slot[k];
      f.h_done = s->h_done + (size_t)k * 2 * kSrvMaxBatch;
      e = cudaHostGetDevicePointer((void**)&f.d_done, f.h_done, 0);
      if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&f.cs, cudaStreamNonBlocking);
      if (e == cudaSuccess) e = cudaMalloc((void**)&f.d_slot, sizeof(SrvSlot));
      if (e == cudaSuccess) e = cudaMemset(f.d_slot, 0, sizeof(SrvSlot));
    }
    if (e == cudaSuccess) {
      server_init_kernel<<<1, HIST_BINS>>>(s->d_streams, cfg->streams, cfg->pattern_budget);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) rc = e == cudaErrorMemoryAllocation ? HIST_ENOMEM : cuda_fail(e);
  }
  if (rc) {
    hist_server_destroy(s);
    return rc;
  }
  *out = s;
  return HIST_OK;
}

int hist_server_destroy(hist_server* s) {
  if (!s) return HIST_EINVAL;
  cudaError_t e = cudaSuccess;
  for (uint32_t k = 0; k < kSrvMaxSlots; ++k) {
    BatchSlot& f = s->slot[k];
    if (f.cs) {
      const cudaError_t w = cudaStreamSynchronize(f.cs);
      if (e == cudaSuccess) e = w;
    }
  }
  for (uint32_t k = 0; k < kSrvMaxSlots; ++k) {
    BatchSlot& f = s->slot[k];
    if (f.d_slot) cudaFree(f.d_slot);
    if (f.cs) cudaStreamDestroy(f.cs);
  }
  if (s->d_streams) cudaFree(s->d_streams);
  if (s->h_done) cudaFreeHost(s->h_done);
  delete s->args;
  delete s;
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

int hist_server_submit(hist_server* s, uint32_t stream, const uint8_t* d_in, size_t n, uint32_t* d_out,
                       uint64_t tag) {
  if (!s || stream >= s->cfg.streams || (!d_in && n) || n >= ((size_t)1 << 32)) return HIST_EINVAL;
  if (n > s->cfg.hbm_budget) return HIST_EBUDGET;
  s->queue.push_back(PendingReq{stream, d_in, n, d_out, tag, now_ns()});
  s->stats.submitted += 1;
  return HIST_OK;
}

int hist_server_poll(hist_server* s, hist_completion* out, uint32_t cap, uint32_t* n_out) {
  if (n_out) *n_out = 0;
  if (!s || (cap && !out)) return HIST_EINVAL;
  int err = HIST_OK;
  const uint32_t n = retire(s, cap ? out : nullptr, cap, &err);
  if (n_out && cap) *n_out = n;
  if (err) return err;
  return admit(s);
}

int hist_server_drain(hist_server* s, uint32_t timeout_ms) {
  if (!s) return HIST_EINVAL;
  const uint64_t t0 = now_ns();
  while (!server_idle(s)) {
    int err = HIST_OK;
    retire(s, nullptr, 0, &err);
    if (err) return err;
    const int rc = admit(s);
    if (rc) return rc;
    if (timeout_ms && now_ns() - t0 > (uint64_t)timeout_ms * 1000000ull) return HIST_ETIMEDOUT;
  }
  return HIST_OK;
}

int hist_server_stream_state(hist_server* s, uint32_t stream, hist_stream_state* h) {
  if (!s || !h || stream >= s->cfg.streams) return HIST_EINVAL;
  const int rc = hist_server_drain(s, 0);
  if (rc) return rc;
  SrvStream tmp;
  const cudaError_t e = cudaMemcpy(&tmp, s->d_streams + stream, sizeof(SrvStream), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e);
  memset(h, 0, sizeof(*h));
  memcpy(h->totals, tmp.totals, sizeof(h->totals));
  const uint64_t c = s->streams[stream].admitted;
  const SrvRec& last = tmp.rec[(c & 1u) ^ 1u];
  const SrvRec& before = tmp.rec[c & 1u];
  memcpy(h->last_hist, last.hist, sizeof(h->last_hist));
  h->pattern = last.pat;
  h->last_pattern = before.pat;
  h->chunks = c;
  h->flag = last.flag;
  // the last request ran the kernel chosen from the one before
  h->last_kernel = c == 0 || s->cfg.mode == HIST_MODE_PLAIN ? HIST_FLAG_PLAIN
                   : s->cfg.mode == HIST_MODE_AUTO          ? before.flag
                                                            : HIST_FLAG_ADAPTIVE;
  return HIST_OK;
}

int hist_server_get_stats(hist_server* s, hist_server_stats* out) {
  if (!s || !out) return HIST_EINVAL;
  *out = s->stats;
  out->queued = s->queue.size();
  out->inflight_bytes = s->inflight_bytes;
  return HIST_OK;
}

int hist_server_replay(hist_server* s, const hist_request* reqs, uint32_t count, hist_completion* out,
                       uint32_t timeout_ms) {
  if (!s || (count && (!reqs || !out))) return HIST_EINVAL;
  for (uint32_t i = 0; i < count; ++i) {
    const hist_request& r = reqs[i];
    if (r.stream >= s->cfg.streams || (!r.d_in && r.n) || r.n >= (1ull << 32) ||
        (i && r.arrival_ns < reqs[i - 1].arrival_ns))
      return HIST_EINVAL;
    if (r.n > s->cfg.hbm_budget) return HIST_EBUDGET;
  }
  if (!server_idle(s)) return HIST_ESTATE;
  std::vector<hist_completion> buf((size_t)s->cfg.max_batch * s->cfg.max_inflight);
  uint32_t done = 0, next = 0;
  const uint64_t t0 = now_ns();
  while (done < count) {
    const uint64_t now = now_ns() - t0;
    if (timeout_ms && now > (uint64_t)timeout_ms * 1000000ull) return HIST_ETIMEDOUT;
    while (next < count && reqs[next].arrival_ns <= now) {
      const hist_request& r = reqs[next];
      s->queue.push_back(PendingReq{r.stream, r.d_in, (size_t)r.n, r.d_out, next, t0 + r.arrival_ns});
      s->stats.submitted += 1;
      ++next;
    }
    uint32_t n = 0;
    const int rc = hist_server_poll(s, buf.data(), (uint32_t)buf.size(), &n);
    if (rc) return rc;
    for (uint32_t i = 0; i < n; ++i) {
      hist_completion c = buf[i];
      const uint64_t idx = c.tag;
      c.tag = reqs[idx].tag;
      c.submit_ns -= t0;
      c.admit_ns -= t0;
      c.done_ns -= t0;
      out[idx] = c;
    }
    done += n;
  }
  // every request has completed; the last batches retire with their state words
  while (!server_idle(s)) {
    if (timeout_ms && now_ns() - t0 > (uint64_t)timeout_ms * 1000000ull) return HIST_ETIMEDOUT;
    int err = HIST_OK;
    retire(s, nullptr, 0, &err);
    if (err) return err;
  }
  return HIST_OK;
}

}  // extern "C"
