// What a launcher finds out or sets once on each device: function attributes and occupancies belong to the device that was current,
// and a process may use several.
#pragma once

#include <cuda_runtime_api.h>
#include <stdint.h>

#include <atomic>

namespace moe {

class PerDevice {
    static constexpr int MAX_DEVICES = 64;
    std::atomic<int32_t> values[MAX_DEVICES] = {};

  public:
    // The current device's value: find() until it has returned a positive one there, 0 on an error. Threads that come first together
    // may both call find(), which has to give both the same.
    template <typename Find> int32_t get(Find find) {
        int device = -1;
        if (cudaGetDevice(&device) != cudaSuccess || device < 0) return 0;
        if (device >= MAX_DEVICES) return find();
        int32_t v = values[device].load(std::memory_order_acquire);
        if (v <= 0) {
            v = find();
            if (v > 0) values[device].store(v, std::memory_order_release);
        }
        return v;
    }
};

// Raises a kernel's limit of dynamic shared memory, on its first launch on the current device
template <typename Kernel> bool allow_shared(PerDevice &done, Kernel kernel, int bytes) {
    return done.get([&]() { return cudaFuncSetAttribute(reinterpret_cast<const void *>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess ? 1 : 0; }) > 0;
}

}  // namespace moe
