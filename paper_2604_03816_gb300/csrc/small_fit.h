// Which states the small-state kernel (apply_small.cu) takes: plain integer rules, host only.
#pragma once

#include <algorithm>
#include <cstdint>

namespace svm {

constexpr uint32_t MAX_N = 12;            // qubits
constexpr uint32_t THREADS = 256;         // one amplitude each: 2^12 = 16 CTAs x 256
constexpr uint32_t MAX_C = 4;             // log2 of the largest cluster

// log2 of the cluster that holds n qubits where clusters of 2^max_c CTAs can be scheduled: at
// least 32 amplitudes per CTA.
constexpr uint32_t cluster_log2(uint32_t n, uint32_t max_c) { return n > 5 ? std::min(max_c, n - 5u) : 0u; }

// Every thread owns at most one amplitude, so a CTA's share has to fit its threads: 12 qubits need
// the cluster of 16, and where the device schedules only 8 they go pass by pass.
constexpr bool state_fits(uint32_t n, uint32_t max_c) {
    return n <= MAX_N && ((1u << n) >> cluster_log2(n, max_c)) <= THREADS;
}

}  // namespace svm
