// What the host sets up or asks once per device and process: attributes of a
// kernel (cudaFuncSetAttribute applies to the current device only) and what fits
// on it.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <mutex>

namespace gcvo {

// The device of this thread's call: every entry point that launches names it
// with use_device, so that a launch need not ask the runtime for it.
inline int &call_device() {
    static thread_local int device = 0;
    return device;
}
inline cudaError_t use_device(int device) {
    call_device() = device;
    return cudaSetDevice(device);
}

template <class T>
class PerDevice {
    static constexpr int MOST = 64;
    std::mutex m_;
    std::atomic<bool> known_[MOST] = {};
    T value_[MOST];

public:
    // The value of the call's device, made by make() on its first use there.
    template <class Make>
    T get(Make make) {
        const int d = call_device();
        if (d < 0 || d >= MOST) return make();
        if (!known_[d].load(std::memory_order_acquire)) {
            std::lock_guard<std::mutex> lk(m_);
            if (!known_[d].load(std::memory_order_relaxed)) {
                value_[d] = make();
                known_[d].store(true, std::memory_order_release);
            }
        }
        return value_[d];
    }
};

}  // namespace gcvo
