// rid_once.cuh -- set-up that every thread of the process shares, done once per
// device (host only; no CUDA headers).
#pragma once

#include <atomic>
#include <mutex>

struct RidOnce {
    std::atomic<unsigned long long> done{0};   // one bit per device ordinal
    std::mutex mu;
};

// Runs set() (0: success) for the device `dev` unless a call before it has
// succeeded; returns its error code.  A caller that finds the device done finds
// the set-up complete: the bit is published after set() returned, and callers
// that arrive meanwhile wait for it.  A set-up that failed is tried again.
template <typename F>
int rid_once(RidOnce& once, int dev, F set) {
    const unsigned long long bit = 1ull << (dev & 63);
    if (once.done.load(std::memory_order_acquire) & bit) return 0;
    std::lock_guard<std::mutex> lk(once.mu);
    if (once.done.load(std::memory_order_relaxed) & bit) return 0;
    const int e = set();
    if (e == 0) once.done.fetch_or(bit, std::memory_order_release);
    return e;
}
