// Host threads that prepare groups of work which the calling thread passes on one after the other
// (batch.cu).  Host only.
#pragma once

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <memory>
#include <thread>
#include <vector>

namespace svk {

// Where a batch's gates are cut into groups (ends with the gate count): the first gates' matrices are
// converted, uploaded and their passes launched while host threads convert the rest (18 qubits x
// 96 circuits: 0.9 ms of conversion and upload before the first pass, 0.2 in three groups).  Only
// when the batch is one chunk (several need every gate first), and when the table of all matrices is
// large enough: a group costs one more copy and one more graph launch, and below 512 KiB one group
// was faster on every batch tried (10 qubits x 2 states, 27 gates of two qubits: 121 us in three
// groups, 94 in one; above, three: 16 qubits x 8, 18 gates of five qubits: 204 and 242).
inline std::vector<size_t> group_cuts(size_t ngates, size_t table_bytes, bool one_chunk) {
    if (!one_chunk || ngates < 8 || table_bytes < (size_t(512) << 10)) return {0, ngates};
    return {0, ngates / 8, ngates / 3, ngates};
}

// share(w, q): worker w's part of group q, workers 0 .. nt - 1 (0 is the calling thread; where a thread
// cannot be had it does that worker's part too).  step(q), once group q is prepared, in the
// calling thread and in order; returns false to stop.  The threads have ended when this returns or
// throws (what step throws): they prepare their parts of the remaining groups first.
template <typename Share, typename Step>
void in_groups(uint32_t nt, size_t ngroups, Share share, Step step) {
    const std::unique_ptr<std::atomic<uint32_t>[]> ready(new std::atomic<uint32_t>[ngroups]);
    for (size_t q = 0; q < ngroups; ++q) ready[q].store(0);
    struct Threads {
        std::vector<std::thread> th;
        ~Threads() {
            for (std::thread &t : th) t.join();
        }
    } threads;
    std::vector<std::thread> &th = threads.th;
    th.reserve(nt);
    std::atomic<uint32_t> *done = ready.get();
    try {
        for (uint32_t w = 1; w < nt; ++w)
            th.emplace_back([&share, done, ngroups, w] {
                for (size_t q = 0; q < ngroups; ++q) {
                    share(w, q);
                    done[q].fetch_add(1, std::memory_order_release);
                }
            });
    } catch (...) {
        // no more threads: the calling thread takes the other parts
    }
    for (size_t q = 0; q < ngroups; ++q) {
        share(0u, q);
        for (uint32_t w = (uint32_t)th.size() + 1; w < nt; ++w) share(w, q);
        while (done[q].load(std::memory_order_acquire) < th.size()) std::this_thread::yield();
        if (!step(q)) break;
    }
}

}  // namespace svk
