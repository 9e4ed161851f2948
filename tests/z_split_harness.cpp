// The choice between tiled and general reads of Z strings, for ctypes.
#include "../paper_2604_03816_gb300/csrc/z_split.h"

extern "C" void split_z(const uint64_t *z, size_t n, unsigned T, double amplitudes, int batch, int dtype, char *out) {
    const std::vector<char> g = svx::split_z(z, n, T, amplitudes, (batch ? svx::Z_COST_BATCH : svx::Z_COST_SINGLE)[dtype]);
    std::copy(g.begin(), g.end(), out);
}
