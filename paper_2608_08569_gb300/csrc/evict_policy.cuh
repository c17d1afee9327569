// Launcher of the eviction under a policy (evict.cu), called by the C ABI (api.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "voxzip.h"

namespace voxzip {

// SMs of the current device (anchor_fuse.cu; looked up once per device).
int sm_count();

// Runs f (which sets kernel attributes: they are per function and device) unless it has succeeded on
// the current device before; `done` is a bit per device. Threads that race both run it.
template <typename F>
cudaError_t once_per_device(std::atomic<uint64_t> &done, F &&f) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = (uint64_t)1 << (dev & 63);
    if (dev < 64 && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    e = f();
    if (e == cudaSuccess && dev < 64) done.fetch_or(bit, std::memory_order_release);
    return e;
}

cudaError_t launch_evict_policy(const voxzip_cache_desc &d, int32_t layer_begin, int32_t layer_count,
                                void *k_cache, void *v_cache, float *score, int32_t *pos, int32_t *len,
                                const int32_t *budget, const voxzip_evict_policy &policy, int32_t *status,
                                cudaStream_t stream);

}  // namespace voxzip
