// per_device.h -- what a launcher sets up or finds out once per device.
//
// Kernel attributes (dynamic shared memory, non-portable clusters) belong to the device that is
// current when they are set, and occupancy to the device that is asked, while a launcher's
// static outlives them all: kept once per process, a second device's launches failed for want
// of the attributes and took the first one's launch shape.
#pragma once

#include <atomic>

#include <cuda_runtime.h>

namespace gals {

class PerDevice {
public:
    // The current device's value, a non-negative int: from make(&value) at the device's first
    // call (what fails is tried again at the next one).  Several threads may come first at
    // once; each of them makes the value then, so make only sets attributes and asks.
    template <class Make> cudaError_t get(int *value, Make make)
    {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const bool kept = dev >= 0 && dev < kDevices;
        if (kept) {
            const int v = slot_[dev].load(std::memory_order_acquire);
            if (v > 0) {
                *value = v - 1;
                return cudaSuccess;
            }
        }
        if ((e = make(value)) == cudaSuccess && kept) slot_[dev].store(*value + 1, std::memory_order_release);
        return e;
    }

    // The same for a set-up without a value.
    template <class Make> cudaError_t once(Make make)
    {
        int v = 0;
        return get(&v, [&](int *out) {
            *out = 0;
            return make();
        });
    }

private:
    static constexpr int kDevices = 64;  // devices past these are set up at every call
    std::atomic<int> slot_[kDevices] = {};  // value + 1; 0: not yet
};

// The attribute every launcher of more than the default dynamic shared memory sets.
template <class K> cudaError_t allow_dynamic_smem(K *kern, int bytes)
{
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

}  // namespace gals
