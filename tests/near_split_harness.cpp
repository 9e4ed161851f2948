// The short cut of the digit split (fxp::offset_fixed_near) beside the general form, for ctypes.
#include "../paper_2604_03816_gb300/csrc/fixed_point.h"

extern "C" long near_split_mismatches(const double *x, const unsigned *spread, long n) {
    long bad = 0;
    for (long i = 0; i < n; ++i) {
        const uint64_t b = fxp::bits_of(x[i]);
        const uint32_t emax = fxp::exp_field(b) + spread[i];
        uint32_t h0, l0, h1, l1;
        fxp::offset_fixed((uint32_t)(b >> 32), (uint32_t)b, emax, h0, l0);
        fxp::offset_fixed_near((uint32_t)(b >> 32), (uint32_t)b, emax << 20 | 0xFFFFFu, h1, l1);
        bad += h0 != h1 || l0 != l1;
    }
    return bad;
}
