// What the host side keeps of a kernel between launches: its raised shared-memory limit and its
// resident blocks per SM.  Both belong to a device, so they are kept for each; several threads may
// launch at once.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

namespace lat {

class PerDevice {
    static constexpr int kDevices = 64;
    std::atomic<int> value_[kDevices] = {};  // 0: not formed yet

public:
    // The current device's value; make(int*) forms it where there is none (kept as 1 if smaller).
    template <class F>
    cudaError_t get(int* out, F&& make) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const bool kept = dev >= 0 && dev < kDevices;
        int v = kept ? value_[dev].load(std::memory_order_acquire) : 0;
        if (v == 0) {
            e = make(&v);
            if (e != cudaSuccess) return e;
            v = std::max(v, 1);
            if (kept) value_[dev].store(v, std::memory_order_release);
        }
        *out = v;
        return cudaSuccess;
    }
};

template <class... A>
cudaError_t raise_smem(PerDevice& p, void (*kernel)(A...), size_t bytes) {
    int done = 0;
    return p.get(&done, [&](int*) {
        return cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)bytes);
    });
}

// Resident blocks per SM (at least 1), with the shared-memory limit raised to `bytes`.
template <class... A>
cudaError_t resident_blocks(PerDevice& p, void (*kernel)(A...), int threads, size_t bytes, int* out) {
    return p.get(out, [&](int* n) {
        cudaError_t e = cudaFuncSetAttribute((const void*)kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, (const void*)kernel, threads, bytes);
    });
}

}  // namespace lat
