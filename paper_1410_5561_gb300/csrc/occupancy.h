// CTAs of a kernel that the current device holds at once.
#pragma once
#include <cuda_runtime_api.h>
#include <stddef.h>

#include <mutex>

namespace stg {

// Resident CTAs of KERNEL per SM times the SM count, by device and warps (the shared memory follows
// from the threads in every caller); 0 where CUDA cannot say. The kernel itself is the template argument: one
// table for each, also among kernels of the same signature.
template <auto KERNEL>
int resident_ctas(int threads, size_t smem = 0) {
    static std::mutex mu;
    static int cached[64][33] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lock(mu);
    int& c = cached[dev][threads / 32];
    if (c == 0) {
        int sms = 0, per = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, reinterpret_cast<const void*>(KERNEL), threads, smem) !=
            cudaSuccess)
            return 0;
        c = sms * (per > 0 ? per : 1);
    }
    return c;
}

}  // namespace stg
