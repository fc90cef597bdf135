// Host-side decisions about Gram launches whose CTAs wait on one another (no CUDA in here).
//
// Such a launch ends only if all of its CTAs get to run.  Two of them in different streams could each hold
// half of the SMs and wait for the other half for ever; a cooperative launch, placed whole or not
// at all, rules that out, but the driver then neither places its CTAs while the kernel before
// it drains nor lets them set up meanwhile (measured: 4 to 8 us per call of a chain).  So per
// device ONE stream may launch without the attribute -- in stream order, its launches never
// overlap one another -- and every other stream keeps it, until the first one has been seen idle.
// Captured launches keep it too (where a graph will be replayed is unknown), and so does
// everything under MPS (other processes are not known here).
#pragma once

#include <mutex>

namespace ada {

class SoleStream {
public:
    // May a launch on stream `id` go without the attribute?  Asked right before it; end() right after it.
    bool begin(unsigned long long id) {
        std::lock_guard<std::mutex> hold(lock_);
        if (held_ && id_ != id) return false;
        held_ = true;
        id_ = id;
        ++launches_;
        ++pending_;
        return true;
    }
    void end() {
        std::lock_guard<std::mutex> hold(lock_);
        --pending_;
    }
    // mark() before and idle() after a synchronisation (of one stream, or of everything) tell that the launches
    // so far are done; one that another thread is about to hand to the driver is not among them.
    unsigned long long mark() {
        std::lock_guard<std::mutex> hold(lock_);
        return pending_ == 0 ? launches_ : ~0ull;
    }
    void idle(bool all, unsigned long long id, unsigned long long mark) {
        std::lock_guard<std::mutex> hold(lock_);
        if (held_ && launches_ == mark && (all || id_ == id)) held_ = false;
    }
    bool holds(unsigned long long id) {
        std::lock_guard<std::mutex> hold(lock_);
        return held_ && id_ == id;
    }

private:
    std::mutex lock_;
    bool held_ = false;
    unsigned long long id_ = 0;          // (stream ids are never reused within a process)
    unsigned long long launches_ = 0;    // launches without the attribute so far
    int pending_ = 0;                    // of them, those not handed to the driver yet
};

// Limit of a launch's in-kernel waits, in units of 2^20 ns.  2 s; 20 s for a launch that goes without the attribute on the sole
// stream: its CTAs may have to wait for SMs that another stream's kernel still holds, where a
// cooperative launch is not placed before they are free.
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int wait_limit_units(bool alone) { return alone ? 19073 : 1907; }

}  // namespace ada
