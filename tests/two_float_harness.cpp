// The expectation kernels' running sums (svx::SumF, run by run as the launches cut them), for ctypes.
#include "../paper_2604_03816_gb300/csrc/two_float.h"

extern "C" double two_float_sum(const float *x, long n) {
    double acc = 0.0;
    for (long i = 0; i < n;) {
        svx::SumF s;
        s.clear();
        const long end = n - i < (long)svx::RUN_TILES ? n : i + (long)svx::RUN_TILES;
        for (; i < end; ++i) s.add(x[i]);
        acc += s.value();
    }
    return acc;
}
