// Running sums of the Pauli expectations (expect.cu); plain C++, also compiled by the host tests.
#pragma once

#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define TWF_HD __host__ __device__ __forceinline__
#else
#define TWF_HD inline
#endif

namespace svx {

// Two-float sum s + e: an error-free addition, its errors added up in FP32.  e is itself rounded, so
// a long run loses bits (worst of 256 runs: 2^-43 of a sum of 2200 positive terms, 2^-38 of
// 14000), and a launch gives no thread more than RUN_TILES terms: its sums end in FP64, and the launches'
// are added there.  The root-mean-square error of a run then stays below 2^-49, and a
// block adds 4096 independent runs: below FP64's rounding of the total.
constexpr uint32_t RUN_TILES = 128;

struct SumF {
    float s, e;
    TWF_HD void clear() { s = e = 0.f; }
    TWF_HD void add(float x) {
#ifdef __CUDA_ARCH__
        const float t = __fadd_rn(s, x), b = __fsub_rn(t, s);
        e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b)));
#else
        const float t = s + x, b = t - s;
        e = e + ((s - (t - b)) + (x - b));
#endif
        s = t;
    }
    // (an infinite sum has no error term)
    TWF_HD double value() const { return std::isfinite(s) ? (double)s + (double)e : (double)s; }
};

// FP64 (complex128).
struct SumD {
    double s;
    TWF_HD void clear() { s = 0.0; }
    TWF_HD void add(double x) { s += x; }
    TWF_HD double value() const { return s; }
};

}  // namespace svx
