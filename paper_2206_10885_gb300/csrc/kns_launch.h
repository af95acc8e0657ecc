// kns_launch.h -- host set-up of kernel launches that belongs to a device, not to the process: a kernel's
// shared-memory limit and carve-out are those of the device that was current when they were set.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace kns {

constexpr int kCachedDevices = 32;  // devices whose answers are kept; others are asked on every launch

// One positive number per device (0: not known yet); a static of this type starts out empty.
struct PerDevice {
    std::atomic<int> n[kCachedDevices];
    int get(int dev) const { return dev < kCachedDevices ? n[dev].load() : 0; }
    void set(int dev, int v) {
        if (dev < kCachedDevices) n[dev].store(v);
    }
};

// Resident blocks per SM of a kernel with `smem` bytes of dynamic shared memory (registers and shared
// memory both count) on the current device, after allowing it the largest shared-memory carve-out there;
// asked once per kernel and device.
template <class K>
cudaError_t resident_blocks(K kernel, int threads, int smem, PerDevice &cache, int &out) {
    const void *f = reinterpret_cast<const void *>(kernel);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    out = cache.get(dev);
    if (out > 0) return cudaSuccess;
    if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 100)) != cudaSuccess ||
        (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&out, f, threads, smem)) != cudaSuccess)
        return e;
    if (out < 1) out = 1;
    cache.set(dev, out);
    return cudaSuccess;
}

}  // namespace kns
