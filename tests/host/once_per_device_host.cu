// Host check of hd_once.h: a device-bound setting is made on every device that
// the process uses, once on each, from any thread, again after a failure.
#include <cstdio>
#include <thread>
#include <vector>

#include "hd_once.h"

int main() {
    hd::OncePerDevice once;
    std::atomic<int> made[80] = {};
    auto set = [&](int dev) { return once(dev, [&] { made[dev] += 1; return 0; }); };
    // two devices in turn
    for (int k = 0; k < 3; ++k)
        for (int dev : {0, 1})
            if (set(dev) != 0) return 1;
    if (made[0] != 1 || made[1] != 1) return 2;
    // a failure is returned and tried again
    int fail = 7;
    if (once(2, [&] { return fail; }) != 7) return 3;
    fail = 0;
    if (once(2, [&] { made[2] += 1; return fail; }) != 0 || once(2, [&] { return 9; }) != 0 || made[2] != 1) return 4;
    // device numbers beyond the set are made on every call
    if (set(63) || set(63) || made[63] != 1 || set(64) || set(64) || made[64] < 1) return 5;
    // several threads: made before any of them goes on
    hd::OncePerDevice shared;
    std::atomic<int> ready{0}, early{0};
    std::vector<std::thread> threads;
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([&, t] {
            const int dev = t & 1;
            if (shared(dev, [&] { ready |= 1 << dev; return 0; }) != 0 || !(ready & (1 << dev))) early += 1;
        });
    for (auto& t : threads) t.join();
    if (early != 0) return 6;
    std::puts("ok");
    return 0;
}
