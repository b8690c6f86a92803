// launch.h -- grid sizing of the persistent fragment kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace rt {

// Number of blocks of a persistent kernel: enough to cover `chunks` 32-fragment
// chunks with `warps` warps per block, at most (SMs x resident blocks per SM).
// The occupancy query is cached per kernel and device.  The kernel is a template
// argument so that each has a cache of its own: kernels of one signature share a
// pointer type, and sized by the first one launched (a flat lookup of 100
// registers, say), the 1080p FP16 forward ran 5 of its 8 blocks per SM: 20 poses
// in 0.675 ms instead of 0.586.  At most `most` blocks per SM where that is given.
template <auto Kernel>
inline unsigned persistent_grid(int threads, int64_t chunks, int most = 0) {
    static std::atomic<int> cached[64];  // SMs << 8 | resident blocks per SM
    int dev = 0;
    cudaGetDevice(&dev);
    const bool known = dev >= 0 && dev < 64;
    int resident = known ? cached[dev].load(std::memory_order_relaxed) : 0;
    if (resident == 0) {
        int sms = 0, per_sm = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, Kernel, threads, 0);
        resident = (sms > 0 ? sms : 1) << 8 | (per_sm > 0 ? per_sm : 1);
        if (known) cached[dev].store(resident, std::memory_order_relaxed);
    }
    const int per_sm = resident & 255;
    const int total = (resident >> 8) * (most > 0 && most < per_sm ? most : per_sm);
    const int warps = threads / 32;
    int64_t want = (chunks + warps - 1) / warps;
    if (want < 1) want = 1;
    return (unsigned)(want < total ? want : total);
}

}  // namespace rt
