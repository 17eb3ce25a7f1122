// Per-device one-time set-up bookkeeping (plain C++, no CUDA types, so that it can be compiled and tested on its own).
//
// Function attributes (the opt-in to more than 48 KB of dynamic shared memory), occupancy figures and the SM count
// belong to a device, not to the process: a process that drives several GPUs must repeat the set-up on each.  A
// launcher keeps one `static DeviceOnce` (and, where it caches a number, one `static DeviceValue`) and asks it with
// the ordinal of the current device.  Which kernels an entry point launches depends on the sizes, so any later call may be
// the first that needs one of them: the flags are atomic.  Two threads that need the same set-up at once both run it (it is
// idempotent); a thread that finds it marked, or a value known, also sees what was done before.
#pragma once

#include <atomic>

namespace uoe {

constexpr int kMaxDevices = 64;

struct DeviceOnce {
    std::atomic<bool> done[kMaxDevices] = {};
    // true when `dev` is a usable ordinal whose set-up has not run yet
    bool needs(int dev) const { return valid(dev) && !done[dev].load(std::memory_order_acquire); }
    void mark(int dev) { if (valid(dev)) done[dev].store(true, std::memory_order_release); }
    bool valid(int dev) const { return dev >= 0 && dev < kMaxDevices; }
};

struct DeviceValue {
    std::atomic<int> value[kMaxDevices] = {};
    std::atomic<bool> known[kMaxDevices] = {};
    bool has(int dev) const { return dev >= 0 && dev < kMaxDevices && known[dev].load(std::memory_order_acquire); }
    int get(int dev) const { return has(dev) ? value[dev].load(std::memory_order_relaxed) : 0; }
    void set(int dev, int v) {
        if (dev < 0 || dev >= kMaxDevices) return;
        value[dev].store(v, std::memory_order_relaxed);
        known[dev].store(true, std::memory_order_release);
    }
};

}  // namespace uoe
