// hist_internal.h -- host helpers shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "hist.h"

namespace histlib {

constexpr int kMaxDevices = 64;

// Record a CUDA error for hist_last_cuda_error() and return HIST_ECUDA.
int cuda_fail(cudaError_t e);
// SMs of the current device.
int sm_count();
// Opt a kernel into `bytes` of dynamic shared memory on this device.
int ensure_smem_attr_bytes(const void* fn, int* done, size_t bytes);
// Allow a kernel clusters of more than 8 CTAs on this device (once per kernel
// and device; `done` as above).
int ensure_wide_cluster(const void* fn, int* done);
// The one-shot histogram (hist_plain / hist_adaptive).
int oneshot(const uint8_t* d_in, size_t n, uint32_t* d_out, cudaStream_t s);

}  // namespace histlib
