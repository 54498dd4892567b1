// per_device.h -- values made once per device, at the first use on it.  Plain C++,
// so that it can be run on the host.
#pragma once

#include <mutex>

namespace hnet {

// One value per device.  get() makes it at the first call for a device, one thread at
// a time; where init fails nothing is kept, and the next call tries again.
template <typename T> class PerDevice {
    static constexpr int kDevices = 64;
    std::mutex m_;
    T v_[kDevices] = {};
    bool made_[kDevices] = {};

public:
    // init(T &) -> whether it could be made; null where it could not, or dev is none
    template <typename Init> T *get(int dev, Init init) {
        if (dev < 0 || dev >= kDevices) return nullptr;
        std::lock_guard<std::mutex> lock(m_);
        if (!made_[dev]) {
            T v{};
            if (!init(v)) return nullptr;
            v_[dev] = v;
            made_[dev] = true;
        }
        return &v_[dev];
    }
};

}  // namespace hnet
