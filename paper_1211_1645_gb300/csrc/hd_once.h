// hd_once.h -- settings that belong to one device, made once on each.
#pragma once

#include <atomic>
#include <cstdint>

namespace hd {

// once(device, set): calls set() unless it has succeeded on that device before
// (device numbers of 64 and above: every time), and returns its error, zero
// for success.  Any thread; two at a time may both call set(), which makes the
// same setting twice, but none returns before it is made.
class OncePerDevice {
    std::atomic<uint64_t> made_{0};

public:
    template <class F>
    auto operator()(int device, F&& set) -> decltype(set()) {
        const uint64_t bit = device >= 0 && device < 64 ? uint64_t(1) << device : 0;
        if (made_.load(std::memory_order_acquire) & bit) return decltype(set())(0);
        const auto error = set();
        if (error == decltype(set())(0)) made_.fetch_or(bit, std::memory_order_release);
        return error;
    }
};

}  // namespace hd
