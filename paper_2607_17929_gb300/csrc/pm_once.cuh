// One-time set-up per device, apart from CUDA so that it also compiles for the host.
#pragma once

#include <stdint.h>

#include <atomic>

namespace pm {

// Whoever returns from it finds the device's set-up done: the bit is published after the set-up, so a thread that comes
// while another is at it does it too (it has to be repeatable, as setting a kernel's attributes is) instead of going on
// to a launch that needs it.  Devices from 64 on are set up each time.
struct DeviceOnce {
    std::atomic<uint64_t> done{0};
    template <class F> void operator()(int device, F &&set)
    {
        const uint64_t bit = device >= 0 && device < 64 ? 1ull << device : 0;
        if (done.load(std::memory_order_acquire) & bit) return;
        set();
        done.fetch_or(bit, std::memory_order_release);
    }
};

}  // namespace pm
