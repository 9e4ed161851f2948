// Which Z strings of a Pauli sum share tiled reads of the state and which go to the kernels that form a
// weight per string and amplitude (expect.cu, batch.cu).  Plain C++, host only.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <utility>
#include <vector>

namespace svx {

constexpr uint32_t Z_CLASSES = 3;         // classes per tiled read
constexpr uint32_t Z_GENERAL = 32;        // strings per read of the general kernels

// Microseconds of a read of N 2^20 amplitudes: tiled, of c classes, tiled_fixed + tiled_class c + N
// (tiled_base + per_class c); general, of m strings, general_fixed + general_string m + N max(general_floor,
// general_base + per_string m).
struct ZCost {
    double tiled_fixed, tiled_class, tiled_base, per_class;
    double general_fixed, general_string, general_floor, general_base, per_string;

    double tiled(uint32_t c, double N) const { return tiled_fixed + tiled_class * c + N * (tiled_base + per_class * c); }
    double tiled_passes(size_t classes, double N) const {
        const size_t full = classes / Z_CLASSES, rest = classes % Z_CLASSES;
        return full * tiled(Z_CLASSES, N) + (rest || !full ? tiled((uint32_t)rest, N) : 0.0);
    }
    double general(size_t strings, double N) const {
        double t = 0.0;
        for (size_t s = 0; s < strings; s += Z_GENERAL) {
            const double m = (double)std::min<size_t>(Z_GENERAL, strings - s);
            t += general_fixed + general_string * m + N * std::max(general_floor, general_base + per_string * m);
        }
        return t;
    }
};

// Fitted to calls with either kernel alone (GB300, less the empty call's time): complex64 and complex128,
// single states of 10 to 27 qubits, batches of 32 to 100 states of 10 to 20, 1 to 96 strings and chains.
// A tiled read is paid per class of strings (one z_hi, see expect.cu) however many strings are in it,
// the general kernels per string: in FP64 on single states, per run of eight amplitudes on
// batches.  Measured, tiled against general, of strings without a common z_hi: 26 qubits, complex128, 3
// strings 1.06 ms and 1.32, 8 strings 2.99 and 2.62, 32 strings 11.2 and 8.8; 20 qubits, complex64,
// 16 strings 144 us and 110; 18 qubits x 96 states, complex64, 8 strings 263 us and 122, complex128 1.83
// ms and 0.40; a chain (one class): 26 qubits, complex128, 0.97 ms and 6.95.
constexpr ZCost Z_COST_SINGLE[2] = {{11.0, 4.0, 1.1, 0.2, 8.0, 0.25, 0.0, 4.0, 4.05},
                                    {11.0, 1.5, 10.3, 2.0, 8.0, 0.25, 0.0, 8.2, 4.1}};
constexpr ZCost Z_COST_BATCH[2] = {{15.0, 2.0, 1.0, 0.35, 10.0, 0.2, 1.8, 1.0, 0.2},
                                   {14.0, 1.0, 10.5, 2.6, 13.0, 0.3, 0.0, 12.2, 0.27}};

// to_general[i]: string z[i] goes to the general kernels.  T: index bits of a tile; amplitudes: of the
// state, or of the whole batch.  The cheapest of: every string tiled; the strings that are alone in
// their class general; those beyond the slots that the other classes' reads leave free; all
// general.
inline std::vector<char> split_z(const uint64_t *z, size_t n, uint32_t T, double amplitudes, const ZCost &cost) {
    std::vector<char> to_general(n, 0);
    const double N = amplitudes / (double)(1u << 20);
    const uint64_t lo = (1ull << T) - 1;
    std::vector<std::pair<uint64_t, size_t>> mixed;      // (z_hi, string); the others lie inside the tile or above it
    for (size_t i = 0; i < n; ++i)
        if ((z[i] >> T) && (z[i] & lo)) mixed.emplace_back(z[i] >> T, i);
    const size_t unclassed = n - mixed.size();
    std::sort(mixed.begin(), mixed.end());
    std::vector<size_t> alone;                           // the only string of their class
    size_t classes = 0;
    for (size_t i = 0, e; i < mixed.size(); i = e, ++classes) {
        for (e = i + 1; e < mixed.size() && mixed[e].first == mixed[i].first; ++e) {}
        if (e == i + 1) alone.push_back(mixed[i].second);
    }
    const size_t shared = classes - alone.size();
    const bool read = unclassed || shared;               // a tiled read is needed without them
    const size_t slots = read ? (shared && shared % Z_CLASSES == 0 ? 0 : Z_CLASSES - shared % Z_CLASSES) : 0;
    const size_t fill = std::min(alone.size(), slots);
    const double t[4] = {
        cost.tiled_passes(classes, N),
        (read ? cost.tiled_passes(shared, N) : 0.0) + cost.general(alone.size(), N),
        (read ? cost.tiled_passes(shared + fill, N) : 0.0) + cost.general(alone.size() - fill, N),
        cost.general(n, N),
    };
    const int best = (int)(std::min_element(t, t + 4) - t);
    if (best == 3) std::fill(to_general.begin(), to_general.end(), 1);
    for (size_t k = best == 2 ? fill : 0; (best == 1 || best == 2) && k < alone.size(); ++k) to_general[alone[k]] = 1;
    return to_general;
}

}  // namespace svx
