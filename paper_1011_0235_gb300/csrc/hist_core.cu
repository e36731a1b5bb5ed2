// hist_core.cu -- one-shot kernels (hist_plain, hist_adaptive), the device-side
// binning pattern and degeneracy, error handling.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <atomic>

#include "hist.h"
#include "hist_device.cuh"
#include "hist_internal.h"

using namespace histdev;

namespace {

thread_local int g_last_cuda_error = 0;

// ------------------------------------------------------ one-shot kernels --
//
// hist_plain and hist_adaptive count in the lane-private table
// (hist_device.cuh), which refines every pattern: one code path, bound by the
// HBM read on a long input and by launch and latency on a short one.

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The word at shared address `a` of CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_ld(uint32_t a, uint32_t rank) {
  uint32_t r, v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(r) : "memory");
  return v;
}

// A short input: one cluster of 1, 2, 4, 8 or 16 CTAs (as far as the device
// places them: widest_cluster) counts it, each CTA an equal part, and the CTAs sum each other's tables through distributed
// shared memory: no cleared output, no global atomics, one launch.  Bound by
// latency (launch, one round of loads, two barriers of the cluster): 1 MiB of
// uniform pixels 10.3 -> 4.8 us a call in a row (a clearing memset and 16
// CTAs of per-warp tables before), 3.9 us of it on the GPU; 4 KiB 8.0 -> 1.5
// us on the GPU.  Chained: the tables are cleared while the work before ends.
__global__ void __launch_bounds__(kThreads, 1)
    oneshot_cluster_kernel(const uint8_t* __restrict__ in, uint32_t n, uint32_t* __restrict__ out, const Parts parts) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ uint32_t res[HIST_BINS];
  const int t = threadIdx.x;
  const uint32_t C = cluster_size(), rank = cluster_rank();
  const Split sp = split_bytes(in, n);
  const uint4* body = reinterpret_cast<const uint4*>(in + sp.head);
  const uint32_t nvec = (uint32_t)sp.nvec;
  const uint32_t begin = part_begin(parts, nvec, rank), end = part_begin(parts, nvec, rank + 1);
  uint4 v[kLaneLoads];
  const LaneRange r = lane_range(body, begin, end, t);
  zero_table(smem);
  pdl_wait();
  pdl_launch_dependents();
  lane_load<kLaneLoads, kThreads>(v, r);
  __syncthreads();
  lane_count<kLaneLoads, kThreads>(v, r, smem_addr(smem) + ((t & 31) << 2));
  __syncthreads();
  lane_reduce<kThreads, false>(smem, res, t);
  __syncthreads();
  if (rank == 0) count_edges_into(in, sp, res);
  if (C == 1) {
    __syncthreads();
    if (t < HIST_BINS) out[t] = res[t];
    return;
  }
  cluster_sync();
  // CTA r sums bins r 256 / C ..., C neighbouring lanes to a bin, one per CTA
  if (t < HIST_BINS) {
    const uint32_t bin = rank * (HIST_BINS / C) + t / C;
    uint32_t sum = cluster_ld(smem_addr(res + bin), t & (C - 1));
    for (uint32_t o = 1; o < C; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((t & (C - 1)) == 0) out[bin] = sum;
  }
  cluster_sync();  // no CTA leaves while another reads its sums
}

// A longer input: out is cleared by a launch of its own, which lets the
// counting launch start once the work before the call has completed (the
// pixels are there then); that one waits for the clear only before it adds.
__global__ void __launch_bounds__(HIST_BINS) oneshot_clear_kernel(uint32_t* __restrict__ out) {
  pdl_wait();
  pdl_launch_dependents();
  out[threadIdx.x] = 0;
}

// One CTA of 1024 threads per SM with four loads in flight per thread: as
// many bytes in flight as two CTAs with two loads each, without two CTAs on
// one SM finishing their ranges apart.  Bound by the HBM read.  On the GPU,
// clearing launch included: 64 MiB of uniform pixels 30.7 -> 13.1 us, 256 MiB
// 98.4 -> 40.1 us (6.7 TB/s; per-warp tables before).
__global__ void __launch_bounds__(kThreads, 1)
    oneshot_kernel(const uint8_t* __restrict__ in, uint32_t n, uint32_t* __restrict__ out, const Parts parts) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ uint32_t res[HIST_BINS];
  const int t = threadIdx.x;
  pdl_launch_dependents();
  const Split sp = split_bytes(in, n);
  const uint4* body = reinterpret_cast<const uint4*>(in + sp.head);
  const uint32_t nvec = (uint32_t)sp.nvec;
  const uint32_t begin = part_begin(parts, nvec, blockIdx.x), end = part_begin(parts, nvec, blockIdx.x + 1);
  uint4 v[kLaneLoads];
  const LaneRange r = lane_range(body, begin, end, t);
  lane_load<kLaneLoads, kThreads>(v, r);
  zero_table(smem);
  __syncthreads();
  lane_count<kLaneLoads, kThreads>(v, r, smem_addr(smem) + ((t & 31) << 2));
  __syncthreads();
  lane_reduce<kThreads, false>(smem, res, t);
  __syncthreads();
  if (blockIdx.x == 0) {
    count_edges_into(in, sp, res);
    __syncthreads();
  }
  pdl_wait();
  if (t < HIST_BINS && res[t]) atomicAdd(out + t, res[t]);
}

// Change detection between two uint64 histograms (256 threads); chained.
__global__ void __launch_bounds__(HIST_BINS) change_kernel(const unsigned long long* __restrict__ acc,
                                                          const unsigned long long* __restrict__ win,
                                                          uint32_t tau_milli, hist_change_result* __restrict__ res) {
  __shared__ ChangeShared sh;
  const int t = threadIdx.x;
  pdl_launch_dependents();
  pdl_wait();
  const hist_change_result r = change_eval(__ldcg(acc + t), __ldcg(win + t), tau_milli, sh);
  if (t == 0) *res = r;
}

// Sum over the 256 threads of a block of `v` (all threads get it; two
// barriers).
__device__ __forceinline__ unsigned long long block_sum256(unsigned long long v, unsigned long long* sh) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned long long s = 0;
#pragma unroll
  for (int i = 0; i < HIST_BINS / 32; ++i) s += sh[i];
  __syncthreads();
  return s;
}

// The binning pattern of h (or the default pattern if h is null), a bin per
// thread: 256 threads, warp reductions in hardware.  Bound by latency; one
// warp with eight bins a lane spent its time on dependent 64-bit shuffles
// (replayed in a row from a graph: 5.4 -> 2.0 us a call; degeneracy 4.0 ->
// 1.1 us).  Chained: the launch may start while the count that writes h ends.
__global__ void __launch_bounds__(HIST_BINS) pattern_kernel(const uint32_t* __restrict__ h, uint32_t budget,
                                                            hist_pattern* __restrict__ out) {
  __shared__ hist_pattern P;
  __shared__ uint32_t hs[HIST_BINS];
  __shared__ unsigned long long sh[HIST_BINS / 32];
  __shared__ EpiShared es;
  const int t = threadIdx.x;
  pdl_launch_dependents();
  pdl_wait();
  const uint32_t c = h ? __ldcg(h + t) : 0u;
  hs[t] = c;
  const unsigned long long total = block_sum256(c, sh);
  block_epilogue(hs, total, budget, HIST_THETA_MILLI_DEFAULT, P, es);
  __syncthreads();
  const uint32_t* src = reinterpret_cast<const uint32_t*>(&P);
  uint32_t* dst = reinterpret_cast<uint32_t*>(out);
  if (t < (int)(sizeof(hist_pattern) / 4)) dst[t] = src[t];
}

// The degeneracy of h, a bin per thread; chained like pattern_kernel.
template <class T>
__global__ void __launch_bounds__(HIST_BINS) degeneracy_kernel(const T* __restrict__ h, uint32_t theta,
                                                               hist_degeneracy_result* __restrict__ res) {
  __shared__ unsigned long long sh[HIST_BINS / 32], smax[HIST_BINS / 32];
  __shared__ uint32_t sarg[HIST_BINS / 32];
  const int t = threadIdx.x;
  pdl_launch_dependents();
  pdl_wait();
  const unsigned long long c = (unsigned long long)__ldcg(h + t);
  const unsigned long long wm = warp_max(c);
  const uint32_t wa = __reduce_min_sync(0xffffffffu, c == wm ? (uint32_t)t : 0xffffffffu);
  if ((t & 31) == 0) {
    smax[t >> 5] = wm;
    sarg[t >> 5] = wa;
  }
  const unsigned long long total = block_sum256(c, sh);
  if (t == 0) {
    hist_degeneracy_result r;
    r.max = smax[0];
    r.maxbin = sarg[0];
    for (int i = 1; i < HIST_BINS / 32; ++i)  // bins rise with the warp: the first maximum is the lowest bin
      if (smax[i] > r.max) {
        r.max = smax[i];
        r.maxbin = sarg[i];
      }
    if (r.max == 0) r.maxbin = 0;
    r.total = total;
    r.flag = reaches_theta(r.max, total, theta) ? HIST_FLAG_ADAPTIVE : HIST_FLAG_PLAIN;
    *res = r;
  }
}

// Launch a one-block kernel of 256 threads that may start while the work
// before it on `s` ends (it waits before it reads).
template <class... P, class... A>
cudaError_t launch_small(void (*fn)(P...), cudaStream_t s, A... args) {
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute at[1];
  lc.gridDim = dim3(1);
  lc.blockDim = dim3(HIST_BINS);
  lc.stream = s;
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, fn, P(args)...);
}

}  // namespace

namespace histlib {

int cuda_fail(cudaError_t e) {
  g_last_cuda_error = (int)e;
  return HIST_ECUDA;
}

int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) return 148;
  return sms;
}

int ensure_smem_attr_bytes(const void* fn, int* done, size_t bytes) {
  // Kernels using more than 48 KiB of dynamic shared memory need the opt-in,
  // once per (kernel, device); `done` is the caller's per-kernel array of
  // kMaxDevices.
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e);
  if (dev >= 0 && dev < kMaxDevices && done[dev]) return HIST_OK;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return cuda_fail(e);
  if (dev >= 0 && dev < kMaxDevices) done[dev] = 1;
  return HIST_OK;
}

// Bytes of one load per thread of a CTA: a cluster has a CTA for each, up to
// 16.
constexpr size_t kClusterStep = (size_t)kThreads * 16;
// Longest input of the cluster path: one round of four loads per thread of 16
// CTAs.  Calls in a row on 1 MiB (the second launch costs the host 2.5 us):
// 7.7 us against 10.5 with the clearing and the counting launch at 1.5 MiB;
// replayed from a graph both take 3.8 - 3.9 us, and at 2 MiB the cluster 2 us
// more, where 16 SMs are too few.
constexpr size_t kClusterMax = 16 * 4 * kClusterStep;
constexpr size_t kOneshotSmem = (size_t)kTableWords * 4;

// A one-shot launch that may start while the work before it on `s` ends, of
// `grid` CTAs, or of one cluster of that many (`at`: room for its attributes).
static cudaLaunchConfig_t oneshot_launch(unsigned grid, bool cluster, cudaLaunchAttribute (&at)[2], cudaStream_t s) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(grid);
  lc.blockDim = dim3(kThreads);
  lc.dynamicSmemBytes = kOneshotSmem;
  lc.stream = s;
  lc.attrs = at;
  lc.numAttrs = cluster ? 2 : 1;
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = grid;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  return lc;
}

// The widest cluster of oneshot_cluster_kernel (a power of two up to 16) that
// the current device places, asked once per device: a CTA fills an SM, and
// a part of a GPU may have no 16 SMs in one place.
static uint32_t widest_cluster() {
  static std::atomic<uint32_t> known[kMaxDevices];
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) cudaGetLastError();
  const bool keep = dev >= 0 && dev < kMaxDevices;
  if (keep)
    if (const uint32_t w = known[dev].load(std::memory_order_relaxed)) return w;
  bool asked = true;
  uint32_t c = 16;
  for (; c > 1; c >>= 1) {
    cudaLaunchAttribute at[2];
    const cudaLaunchConfig_t lc = oneshot_launch(c, true, at, nullptr);
    int placed = 0;
    cudaError_t e = cudaSuccess;
    if (c > 8)  // (more than the portable size)
      e = cudaFuncSetAttribute((const void*)oneshot_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&placed, oneshot_cluster_kernel, &lc);
    if (e == cudaSuccess && placed > 0) break;
    if (e != cudaSuccess) {
      cudaGetLastError();
      asked = asked && e == cudaErrorInvalidClusterSize;
    }
  }
  if (keep && asked) known[dev].store(c, std::memory_order_relaxed);
  return c;
}

int oneshot(const uint8_t* d_in, size_t n, uint32_t* d_out, cudaStream_t s, uint32_t widest) {
  if (!d_out || (!d_in && n) || n >= ((size_t)1 << 32)) return HIST_EINVAL;
  cudaError_t e;
  if (n == 0) {
    e = cudaMemsetAsync(d_out, 0, HIST_BINS * sizeof(uint32_t), s);
    return e == cudaSuccess ? HIST_OK : cuda_fail(e);
  }
  const uint32_t nvec = (uint32_t)split_bytes(d_in, n).nvec;
  cudaLaunchAttribute at[2];
  if (n <= kClusterMax) {
    unsigned c = 1;
    while (c < 16 && c * kClusterStep < n) c <<= 1;
    // a cluster that cannot be placed leaves the input to the grid below
    if (c == 1 || c <= (widest ? widest : widest_cluster())) {
      const cudaLaunchConfig_t lc = oneshot_launch(c, c > 1, at, s);
      e = cudaLaunchKernelEx(&lc, oneshot_cluster_kernel, d_in, (uint32_t)n, d_out, make_parts(nvec, c));
      if (e == cudaSuccess) return HIST_OK;
      // (the answer is the device's; a context may hold fewer of its SMs)
      const bool placed = e != cudaErrorInvalidClusterSize && e != cudaErrorLaunchOutOfResources &&
                          e != cudaErrorInvalidConfiguration;
      if (c == 1 || placed) return cuda_fail(e);
      cudaGetLastError();
    }
  }
  const uint32_t grid = (uint32_t)sm_count();
  cudaLaunchConfig_t lc = oneshot_launch(1, false, at, s);
  lc.blockDim = dim3(HIST_BINS);
  lc.dynamicSmemBytes = 0;
  e = cudaLaunchKernelEx(&lc, oneshot_clear_kernel, d_out);
  if (e != cudaSuccess) return cuda_fail(e);
  lc = oneshot_launch(grid, false, at, s);
  e = cudaLaunchKernelEx(&lc, oneshot_kernel, d_in, (uint32_t)n, d_out, make_parts(nvec, grid));
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

}  // namespace histlib

using namespace histlib;

extern "C" {

const char* hist_strerror(int code) {
  switch (code) {
    case HIST_OK: return "ok";
    case HIST_EINVAL: return "invalid argument";
    case HIST_ENOMEM: return "out of memory";
    case HIST_EBUDGET: return "request exceeds the admission budget";
    case HIST_ETIMEDOUT: return "bounded wait timed out";
    case HIST_ECUDA: return "CUDA error";
    case HIST_EBUSY: return "no free slot";
    case HIST_ESTATE: return "object in the wrong state";
    default: return "unknown error";
  }
}

int hist_last_cuda_error(void) { return g_last_cuda_error; }

int hist_device_sms(void) { return sm_count(); }

int hist_pattern_check(const hist_pattern* p) {
  if (!p) return HIST_EINVAL;
  if (p->budget < HIST_BUDGET_MIN || p->budget > HIST_BUDGET_MAX) return HIST_EINVAL;
  uint8_t seen[HIST_BUDGET_MAX];
  memset(seen, 0, sizeof(seen));
  uint32_t used = 0;
  for (int b = 0; b < HIST_BINS; ++b) {
    if (p->log2k[b] > 5) return HIST_EINVAL;
    const uint32_t k = 1u << p->log2k[b];
    const uint32_t o = p->off[b];
    if (o % k != 0 || o + k > p->budget) return HIST_EINVAL;
    for (uint32_t j = 0; j < k; ++j) {
      if (seen[o + j]) return HIST_EINVAL;
      seen[o + j] = 1;
    }
    used += k;
  }
  return used == p->used ? HIST_OK : HIST_EINVAL;
}

int hist_plain(const uint8_t* d_in, size_t n, uint32_t* d_out, hist_cuda_stream s) {
  return oneshot(d_in, n, d_out, (cudaStream_t)s, 0);
}

int hist_plain_test_cluster(const uint8_t* d_in, size_t n, uint32_t widest, uint32_t* d_out, hist_cuda_stream s) {
  if (widest < 1 || widest > 16) return HIST_EINVAL;
  return oneshot(d_in, n, d_out, (cudaStream_t)s, widest);
}

int hist_adaptive(const uint8_t* d_in, size_t n, const hist_pattern* d_pat, uint32_t* d_out,
                  hist_cuda_stream s) {
  if (!d_pat) return HIST_EINVAL;
  return oneshot(d_in, n, d_out, (cudaStream_t)s, 0);
}

int binning_pattern(const uint32_t* d_prev_hist, uint32_t budget, hist_pattern* d_pat, hist_cuda_stream s) {
  if (!d_prev_hist || !d_pat || budget < HIST_BUDGET_MIN || budget > HIST_BUDGET_MAX) return HIST_EINVAL;
  const cudaError_t e = launch_small(pattern_kernel, (cudaStream_t)s, d_prev_hist, budget, d_pat);
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

int default_pattern(uint32_t budget, hist_pattern* d_pat, hist_cuda_stream s) {
  if (!d_pat || budget < HIST_BUDGET_MIN || budget > HIST_BUDGET_MAX) return HIST_EINVAL;
  const cudaError_t e = launch_small(pattern_kernel, (cudaStream_t)s, nullptr, budget, d_pat);
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

int degeneracy(const uint32_t* d_hist, uint32_t theta_milli, hist_degeneracy_result* d_res,
               hist_cuda_stream s) {
  if (!d_hist || !d_res || theta_milli > 1000) return HIST_EINVAL;
  const cudaError_t e = launch_small(degeneracy_kernel<uint32_t>, (cudaStream_t)s, d_hist, theta_milli, d_res);
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

int hist_change(const uint64_t* d_acc, const uint64_t* d_win, uint32_t tau_milli, hist_change_result* d_res,
                hist_cuda_stream s) {
  if (!d_acc || !d_win || !d_res || tau_milli > 1000) return HIST_EINVAL;
  const cudaError_t e =
      launch_small(change_kernel, (cudaStream_t)s, reinterpret_cast<const unsigned long long*>(d_acc),
                   reinterpret_cast<const unsigned long long*>(d_win), tau_milli, d_res);
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

int degeneracy_u64(const uint64_t* d_hist, uint32_t theta_milli, hist_degeneracy_result* d_res,
                   hist_cuda_stream s) {
  if (!d_hist || !d_res || theta_milli > 1000) return HIST_EINVAL;
  const cudaError_t e = launch_small(degeneracy_kernel<unsigned long long>, (cudaStream_t)s,
                                     reinterpret_cast<const unsigned long long*>(d_hist), theta_milli, d_res);
  return e == cudaSuccess ? HIST_OK : cuda_fail(e);
}

}  // extern "C"
