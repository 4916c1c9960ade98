// nr_once.h -- set-up that a function needs once on every device.
#pragma once

#include <atomic>
#include <cstdint>

namespace nrimpl {

// A kernel's attributes (its dynamic shared memory beyond 48 KB) belong to the
// function on one device.  run(device, set) calls `set` until it has returned
// 0 (cudaSuccess) for that device and returns its result; safe from several
// threads, which may then set the same attribute twice.  Devices from 64 on
// set it on every call.
class OncePerDevice {
public:
    template <class Set>
    auto run(int device, Set &&set) -> decltype(set())
    {
        const uint64_t bit = device >= 0 && device < 64 ? uint64_t{1} << device : 0;
        if (done_.load(std::memory_order_acquire) & bit) return decltype(set()){};
        const auto e = set();
        if (e == decltype(set()){}) done_.fetch_or(bit, std::memory_order_release);
        return e;
    }

private:
    std::atomic<uint64_t> done_{0};
};

} // namespace nrimpl
