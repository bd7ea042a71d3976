// One kernel's dynamic shared memory settings, per device, apart from the CUDA
// calls.
#pragma once

#include <atomic>
#include <cstddef>
#include <mutex>

// The opt-in above 48 KB is set per function and device and the last call wins, so
// it is raised under a lock and never lowered: operators of different classes on
// several threads launch the same kernel with different sizes.
struct SmemOptIn {
    static constexpr int DEVICES = 64;
    static constexpr size_t FREE = 48 * 1024;   // no opt-in needed up to here
    std::mutex lock;
    std::atomic<size_t> size[DEVICES] = {};
    std::atomic<bool> carved[DEVICES] = {};

    // set_size(bytes) and set_carveout() make the runtime's calls for the device
    template <class Size, class Carveout>
    void require(int dev, size_t smem, bool carve, Size set_size, Carveout set_carveout) {
        const bool known = dev >= 0 && dev < DEVICES;
        if (known && (smem <= FREE || size[dev].load(std::memory_order_acquire) >= smem) &&
            (!carve || carved[dev].load(std::memory_order_acquire)))
            return;
        std::lock_guard<std::mutex> hold(lock);
        if (smem > FREE && (!known || size[dev].load() < smem)) {
            set_size(smem);
            if (known) size[dev].store(smem, std::memory_order_release);
        }
        if (carve && (!known || !carved[dev].load())) {
            set_carveout();
            if (known) carved[dev].store(true, std::memory_order_release);
        }
    }
};
