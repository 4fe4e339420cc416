// launch.cuh -- launch shapes of the persistent kernels: the device's SM count and a kernel's resident
// blocks per SM.  Both are constants of a device; each is asked of the driver once (the occupancy query
// costs a microsecond or two, several of them in a call whose kernels take 20) and kept in an atomic word
// per device and block size, so that any number of threads may ask.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#define SG_LAUNCH_DEVICES 64

inline int sg_device() {
    int dev = 0;
    cudaGetDevice(&dev);
    return dev;
}

inline int sg_sm_count() {
    static std::atomic<int> known[SG_LAUNCH_DEVICES];
    const int dev = sg_device();
    const bool keep = dev >= 0 && dev < SG_LAUNCH_DEVICES;
    int n = keep ? known[dev].load(std::memory_order_relaxed) : 0;
    if (n <= 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        if (keep) known[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

// resident blocks of `block` threads per SM, at least 1
template <auto KERNEL>
int sg_blocks_per_sm(int block) {
    static std::atomic<int> known[SG_LAUNCH_DEVICES][9];   // [device][block / 32]
    const int dev = sg_device();
    const bool keep = dev >= 0 && dev < SG_LAUNCH_DEVICES && block % 32 == 0 && block >= 0 && block <= 256;
    int n = keep ? known[dev][block / 32].load(std::memory_order_relaxed) : 0;
    if (n <= 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, KERNEL, block, 0) != cudaSuccess) return 1;
        n = std::max(n, 1);
        if (keep) known[dev][block / 32].store(n, std::memory_order_relaxed);
    }
    return n;
}
