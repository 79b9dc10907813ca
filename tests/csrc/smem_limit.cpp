// Test harness (host only): threads that raise one kernel's shared-memory limit (pv_smem.h) as launches of
// different sizes do, with a setter that takes a while. Returns the launches whose limit was below their need.
#include <atomic>
#include <thread>
#include <vector>

#include "pv_smem.h"

extern "C" int refused_launches(int threads, int rounds) {
    std::atomic<int> refused{0};
    for (int r = 0; r < rounds; ++r) {
        pv::SmemLimit limit;
        pv::DevicePair pair;
        std::atomic<int> set{0}, ready{0};
        std::vector<std::thread> ts;
        for (int t = 0; t < threads; ++t)
            ts.emplace_back([&, t] {
                const int need = 1000 * (1 + (t * 7 + r) % threads);
                ++ready;
                while (ready < threads) std::this_thread::yield();
                int a = 0, b = 0;
                pair.get(3, a, b, [](int& x, int& y) {
                    x = 152;
                    y = 232448;
                    return 0;
                });
                if (a != 152 || b != 232448) ++refused;
                const int e = limit.raise(3, need, [&](int bytes) {
                    for (int i = 0; i < (t * 13 + r) % 7; ++i) std::this_thread::yield();
                    set = bytes;
                    return 0;
                });
                std::this_thread::yield();
                if (e || set < need) ++refused;
            });
        for (std::thread& t : ts) t.join();
    }
    return refused;
}

// A setter that fails leaves the limit as it was.
extern "C" int failed_raise() {
    pv::SmemLimit limit;
    int calls = 0;
    const int e = limit.raise(0, 100, [&](int) { ++calls; return 7; });
    limit.raise(0, 100, [&](int) { ++calls; return 0; });
    limit.raise(0, 99, [&](int) { ++calls; return 0; });
    limit.raise(1, 99, [&](int) { ++calls; return 0; });
    return 10 * e + calls;
}
