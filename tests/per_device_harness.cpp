// One-time setup per device (svk::PerDevice), from several threads, for ctypes.
#include <atomic>
#include <thread>
#include <vector>

#include "../paper_2604_03816_gb300/csrc/per_device.h"

// calls[d]: how often device d's setup ran when `threads` threads each ask for every device of
// 0 .. devices - 1; returns how many answers were another device's.
extern "C" int per_device_calls(int devices, int threads, int *calls) {
    svk::PerDevice<int> setup;
    std::vector<std::atomic<int>> n(devices);
    for (auto &c : n) c = 0;
    std::atomic<int> wrong{0};
    std::vector<std::thread> th;
    for (int t = 0; t < threads; ++t)
        th.emplace_back([&] {
            for (int r = 0; r < 3; ++r)
                for (int d = 0; d < devices; ++d)
                    wrong += setup.get(d, [&] { ++n[d]; return 100 + d; }) != 100 + d;
        });
    for (auto &t : th) t.join();
    for (int d = 0; d < devices; ++d) calls[d] = n[d];
    return wrong;
}
