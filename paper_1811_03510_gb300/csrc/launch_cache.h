// What the host keeps about one kernel between launches, per device: the dynamic shared memory limit set on it and the
// resident blocks per SM of the last launch shape.  Plain host C++ so that it can be tested on its own.
//
// Launches of one kernel come from several threads, with leaf depths (shared memory sizes) and devices of their own:
// the limit is an attribute of the kernel on the current device, so it only ever rises, and the lookup, the two runtime
// calls and the store happen under one lock (uncontended about 20 ns, a launch takes 2 us).
#pragma once
#include <stddef.h>
#include <stdint.h>

#include <mutex>

namespace ccs {

class LaunchCache {
public:
    // Resident blocks per SM of `threads` threads with `smem` bytes of dynamic shared memory on `device`, the current
    // one.  set(smem) raises the kernel's limit there and query(threads, smem, active) asks the runtime; both return an
    // error code, zero for none.
    template <class Err, class Set, class Query>
    Err blocks_per_sm(int device, uint32_t threads, size_t smem, Set set, Query query, int *active)
    {
        std::lock_guard<std::mutex> lock(mu_);
        Device none;
        Device &d = device >= 0 && device < kDevices ? dev_[device] : none;   // (beyond the table: asked every time)
        if (smem > d.limit) {
            const Err e = set(smem);
            if (e != Err{}) return e;
            d.limit = smem;
        }
        if (d.threads != threads || d.smem != smem) {
            int a = 0;
            const Err e = query(threads, smem, &a);
            if (e != Err{}) return e;
            d.threads = threads;
            d.smem = smem;
            d.active = a;
        }
        *active = d.active;
        return Err{};
    }

private:
    static constexpr int kDevices = 64;
    struct Device {
        size_t limit = 0;       // largest dynamic shared memory size set
        uint32_t threads = 0;   // the shape last asked for (0: none) and its blocks
        size_t smem = 0;
        int active = 0;
    };
    std::mutex mu_;
    Device dev_[kDevices];
};

}  // namespace ccs
