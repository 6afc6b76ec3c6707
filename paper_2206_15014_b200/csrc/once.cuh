// Marks for things done once per kernel and device: a hash table of fixed size, so that nothing allocates or throws behind the C interface.
#pragma once
#include <cstdint>
#include <mutex>

namespace nm {

class OncePerDevice {
    static constexpr int kSlots = 1024;  // about 300 kernels
    std::mutex mu;
    const void* key[kSlots] = {};
    uint64_t done[kSlots] = {};  // a bit per device

public:
    // Runs f() unless it has returned 0 for this key and device before; devices from 64 on, and keys beyond the table, run it every time.
    template <typename F>
    int run(const void* k, int dev, F f) {
        if (dev < 0 || dev >= 64) return f();
        std::lock_guard<std::mutex> lock(mu);
        uint32_t at = (uint32_t)(((uint64_t)(uintptr_t)k * 0x9E3779B97F4A7C15ull) >> 54), probes = 0;
        while (key[at] && key[at] != k && ++probes < (uint32_t)kSlots) at = (at + 1) % kSlots;
        if (key[at] && key[at] != k) return f();
        if (done[at] >> dev & 1u) return 0;
        const int rc = f();
        if (rc == 0) {
            key[at] = k;
            done[at] |= 1ull << dev;
        }
        return rc;
    }
};

}  // namespace nm
