// svk::in_groups with a step that stops or throws, for ctypes.
#include <new>

#include "../paper_2604_03816_gb300/csrc/group_threads.h"

// Groups of `workers` parts; the step of group `at` returns false (how = 1) or throws (how = 2), or none does.
// steps[q]: parts of group q that were prepared when its step ran (-1: it did not run).  Returns 1 if the
// step's exception arrived, 2 if any part was prepared twice or threads were still at work, else 0.
extern "C" int run_groups(unsigned workers, int groups, int at, int how, int *steps) {
    std::vector<std::atomic<int>> part(workers * groups);
    for (auto &p : part) p = 0;
    for (int q = 0; q < groups; ++q) steps[q] = -1;
    std::atomic<int> busy{0};
    int r = 0;
    auto share = [&](uint32_t w, size_t q) {
        ++busy;
        std::this_thread::sleep_for(std::chrono::milliseconds(w));
        ++part[q * workers + w];
        --busy;
    };
    try {
        svk::in_groups(workers, (size_t)groups, share, [&](size_t q) {
            steps[q] = 0;
            for (unsigned w = 0; w < workers; ++w) steps[q] += part[q * workers + w];
            if ((int)q == at && how == 2) throw std::bad_alloc();
            return !((int)q == at && how == 1);
        });
    } catch (const std::bad_alloc &) {
        r = 1;
    }
    if (busy) r = 2;
    for (auto &p : part)
        if (p > 1) r = 2;
    return r;
}

// group_cuts into cut[0 .. 4); returns the number of groups.
extern "C" int group_cuts(unsigned long gates, unsigned long table_bytes, int one_chunk, long *cut) {
    const std::vector<size_t> c = svk::group_cuts(gates, table_bytes, one_chunk != 0);
    for (size_t i = 0; i < c.size(); ++i) cut[i] = (long)c[i];
    return (int)c.size() - 1;
}
