// device.h -- what is set or looked up once for each GPU of the process: a kernel's attributes
// (shared-memory limit, cluster sizes) belong to one GPU's context, so a process that uses a second
// GPU needs them there too.
#pragma once
#include <cuda_runtime.h>

#include <atomic>

namespace mhe {

constexpr int kDeviceSlots = 64;

// the calling thread's current GPU, or -1 (nothing is remembered then)
inline int device_slot()
{
    int d = -1;
    if (cudaGetDevice(&d) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    return d < kDeviceSlots ? d : -1;
}

class OncePerDevice {
    std::atomic<bool> done_[kDeviceSlots] = {};

public:
    template <class F>
    void operator()(F&& f)
    {
        const int d = device_slot();
        if (d >= 0 && done_[d].load(std::memory_order_acquire)) return;
        f();
        if (d >= 0) done_[d].store(true, std::memory_order_release);
    }
};

// a number >= 0 looked up once per GPU (kept plus one: 0 is not looked up yet)
class PerDevice {
    std::atomic<int> v_[kDeviceSlots] = {};

public:
    template <class F>
    int operator()(F&& f)
    {
        const int d = device_slot();
        if (d >= 0) {
            const int v = v_[d].load(std::memory_order_relaxed);
            if (v > 0) return v - 1;
        }
        const int v = f();
        if (d >= 0) v_[d].store(v + 1, std::memory_order_relaxed);
        return v;
    }
};

}  // namespace mhe
