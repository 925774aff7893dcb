// What the host sets up or asks once per device and process: attributes of a
// kernel (cudaFuncSetAttribute applies to the current device only) and what fits
// on it.
#pragma once

#include <cuda_runtime.h>

#include <mutex>
#include <utility>
#include <vector>

namespace gcvo {

template <class T>
class PerDevice {
    std::mutex m_;
    std::vector<std::pair<int, T>> known_;   // few devices

public:
    // The value of the current device, made by make() on its first use there.
    template <class Make>
    T get(Make make) {
        int d = 0;
        cudaGetDevice(&d);
        std::lock_guard<std::mutex> lk(m_);
        for (const auto &kv : known_)
            if (kv.first == d) return kv.second;
        known_.emplace_back(d, make());
        return known_.back().second;
    }
};

}  // namespace gcvo
