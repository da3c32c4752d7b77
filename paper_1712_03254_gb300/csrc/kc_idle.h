// What the handles' idle blocks (kc_ctx.h) may come to.  Host code without CUDA.
#pragma once

#include <atomic>
#include <cstddef>

namespace kcapi {

constexpr int kMaxDevices = 64;

// Idle bytes of all handles, device by device.
class IdleTotals {
public:
    // Counts `bytes` more on the device, unless they would pass `limit` there.
    bool reserve(int device, size_t bytes, size_t limit) {
        std::atomic<size_t>& held = of(device);
        if (held.fetch_add(bytes) + bytes <= limit) return true;
        held.fetch_sub(bytes);
        return false;
    }
    void release(int device, size_t bytes) { of(device).fetch_sub(bytes); }
    size_t held(int device) { return of(device).load(); }

private:
    std::atomic<size_t>& of(int device) { return held_[device >= 0 && device < kMaxDevices ? device : 0]; }
    std::atomic<size_t> held_[kMaxDevices] = {};
};

}  // namespace kcapi
