// Launch helpers shared by the superstep launchers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace wsfft {

// Launch with programmatic stream serialization (see pdl_enter): the kernel
// may begin launching while the previous kernel in the stream drains.  Used
// for passes over at most 2 GiB: measured 0.7% faster per transform at 512^3
// and 5% at 256^3, but 14% slower at 1024^3 (8 GiB), so larger passes
// launch plainly.
inline bool pdl_bytes(int64_t bytes) { return bytes <= ((int64_t)2 << 30); }
template <class... KArgs, class... Args>
cudaError_t launch_pdl(bool pdl, void (*kernel)(KArgs...), unsigned grid, unsigned block, int smem,
                       cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Streaming multiprocessors of the current device (0 on failure).  Asked
// once per device; threads that race store the same value.
inline int device_sms() {
    constexpr int kMaxDev = 64;
    static std::atomic<int> sms[kMaxDev];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return 0;
    int n = sms[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        sms[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

}  // namespace wsfft
