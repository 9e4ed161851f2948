// Pauli expectations sum_t c_t <psi| P_t |psi> (the backend's measurement operation, Section
// 4.1): the terms are grouped by their X-part x, and one read of the state serves many terms.
//
// x = 0 (Z strings), z_sum.  With a tile of 2^T consecutive amplitudes (T = 12; complex128 11)
// and z = (z_lo, z_hi) split at bit T, sum_t c_t sum_k s_t(k) p_k splits into
//   * terms with z_hi = 0: sum over the T low bits of w0[k_lo] (sum of p over all tiles), with
//     the table w0[k_lo] = sum_t c_t s_t(k_lo) formed once by z_table;
//   * terms with z_lo = 0: sum over the tiles of w_hi(tile) (sum of p over the tile);
//   * the others, by their distinct z_hi (a "class"; a nearest-neighbour chain has one): as
//     the first kind, with the tiles' signs: w_c[k_lo] (sum over tiles of s(tile) p).
// So an amplitude costs a few additions however many terms there are, where the general kernel forms
// one weight per term and amplitude in FP64 (25 chain terms on 26 qubits: 6.6 ms).  Terms of many
// classes go there all the same where that is cheaper (z_split.h).
//
// x != 0, x_sum.  A tile of 2^T amplitudes (the low index bits and up to five high ones) is
// staged in shared memory by swizzled tensor-map copies; each thread takes 16 of them, four
// tile bits R in registers, and serves every x inside R; up to three choices of R per tile.
// One read of the state thus serves up to twelve single-qubit flips (26 qubits: 4 reads).
//
// Precision: p_k, re_k and im_k are formed as before (FP32 operations for complex64, runs of
// eight FP32 pairs for x != 0); complex64 then adds up to 128 tiles per thread in two-float
// arithmetic (two_float.h) and everything beyond, weights included, in FP64 -- larger states take
// several launches; complex128 is FP64 throughout.  complex64 groups of more than four terms with one x != 0 had FP64
// products and keep the general kernel.
//
// Measured, a transverse-field Ising chain on 26 qubits, complex64 (25 ZZ and 26 X terms):
// 10.48 ms with one FP64 weight per amplitude and one pass per X-part -> 0.56 ms: z_sum 0.10 ms
// (5.3 TB/s; 25 FP32 operations per amplitude), four x_sum passes of about 0.11 ms (4.8
// TB/s; the latency of 24 warps per SM).
// complex128 is bound by the FP64 pipe.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <type_traits>
#include <vector>

#include "ptx.cuh"
#include "reduce.cuh"
#include "sv_internal.h"
#include "two_float.h"
#include "z_split.h"

namespace svx {

using svk::block_sum;
using svk::prob_of;

template <typename R> struct Sum;
template <> struct Sum<float> { using T = SumF; };
template <> struct Sum<double> { using T = SumD; };

template <typename R> struct Geo;
template <> struct Geo<float> { static constexpr uint32_t T = 12, E = 16; using C = float2; };
template <> struct Geo<double> { static constexpr uint32_t T = 11, E = 8; using C = double2; };

// ---------------------------------------------------------------- Z strings

constexpr uint32_t Z_TERMS = 512;    // terms per pass
constexpr uint32_t THREADS = 256;

struct ZTableArgs {
    uint32_t nterms, t, ntab;                  // tile bits, tables
    double *w;                                 // [ntab][2^t]
    unsigned long long zc[1 + Z_CLASSES];      // z_hi of each table's terms
    unsigned long long z[Z_TERMS];
    double c[Z_TERMS];
};

// w[j][k] = sum of c_t (-1)^{|k & z_t|} over the terms with z_hi = zc[j] (and z_lo != 0, or
// z = 0); one entry per thread.
__global__ void z_table(const __grid_constant__ ZTableArgs a) {
    svk::pass_trigger();
    svk::pass_wait();
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (1u << a.t)) return;
    const unsigned long long zc = a.zc[blockIdx.y];
    double w = 0.0;
    for (uint32_t i = 0; i < a.nterms; ++i) {
        const unsigned long long z = a.z[i], lo = z & ((1ull << a.t) - 1ull);
        if ((z >> a.t) != zc || (lo == 0 && z != 0)) continue;
        w += (__popcll(k & lo) & 1) ? -a.c[i] : a.c[i];
    }
    a.w[((size_t)blockIdx.y << a.t) + k] = w;
}

struct ZArgs {
    const void *psi;
    const double *w;                           // z_table's tables
    double *partial;
    uint32_t t, nhi;
    uint32_t low;                              // 1: this pass adds table 0 (z_hi = 0)
    unsigned long long ntiles;                 // of a state
    unsigned long long begin, end;             // tiles of this launch
    unsigned long long zc[Z_CLASSES];          // z_hi of the classes
    unsigned long long zh[Z_TERMS];            // z_hi of the terms with z_lo = 0
    double ch[Z_TERMS];
};

// blockIdx.y: the state of a batch (states back to back, each of ntiles tiles; its partials follow
// each other).  Amplitude indices of a thread within the tile: e * 2 * THREADS + 2 tid + q for complex64
// (16-byte loads of two), e * THREADS + tid for complex128.
template <typename R, int NC>
__global__ void __launch_bounds__(THREADS, NC >= 2 ? 1 : 2) z_sum(const __grid_constant__ ZArgs a) {
    constexpr uint32_t E = Geo<R>::E;
    constexpr bool F = sizeof(R) == 4;
    constexpr uint32_t NV = F ? E / 2 : E;             // 16-byte loads per tile
    using V = typename std::conditional<F, float4, double2>::type;
    using S = typename Sum<R>::T;
    __shared__ double wh_s[2][8];
    __shared__ uint32_t sg_s[2][8];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t tile_vec = (1u << a.t) / (F ? 2u : 1u);    // vectors per tile (>= 1: t >= 1)
    const V *psi = reinterpret_cast<const V *>(a.psi) + (unsigned long long)blockIdx.y * a.ntiles * tile_vec;
    S U[E], X[NC ? NC * E : 1];
#pragma unroll
    for (uint32_t e = 0; e < E; ++e) U[e].clear();
#pragma unroll
    for (uint32_t e = 0; e < (NC ? NC * E : 1u); ++e) X[e].clear();
    svk::pass_trigger();
    svk::pass_wait();
    double hi_acc = 0.0;
    V next[NV];
    auto load = [&](unsigned long long tile) {
#pragma unroll
        for (uint32_t v = 0; v < NV; ++v) {
            const uint32_t i = v * THREADS + tid;
            next[v] = V{};
            if (tile < a.end && i < tile_vec) next[v] = psi[tile * tile_vec + i];
        }
    };
    load(a.begin + blockIdx.x);
    uint32_t j = 0;
    for (unsigned long long tile = a.begin + blockIdx.x; tile < a.end; tile += gridDim.x, ++j) {
        if ((j & 7u) == 0) {
            // weights and signs of the next eight tiles, one tile per warp
            const unsigned long long t = tile + (unsigned long long)warp * gridDim.x;
            double w = 0.0;
            for (uint32_t i = lane; i < a.nhi; i += 32) w += (__popcll(t & a.zh[i]) & 1) ? -a.ch[i] : a.ch[i];
            if (a.nhi) w = svk::warp_sum(w);
            if (lane == 0) {
                wh_s[(j >> 3) & 1u][warp] = w;
                uint32_t sg = 0;
#pragma unroll
                for (int c = 0; c < NC; ++c) sg |= (uint32_t)(__popcll(t & a.zc[c]) & 1) << c;
                sg_s[(j >> 3) & 1u][warp] = sg;
            }
            __syncthreads();
        }
        R p[E];
#pragma unroll
        for (uint32_t v = 0; v < NV; ++v) {
            if constexpr (F) {
                p[2 * v] = prob_of(next[v].x, next[v].y);
                p[2 * v + 1] = prob_of(next[v].z, next[v].w);
            } else {
                p[v] = prob_of(next[v].x, next[v].y);
            }
        }
        load(tile + gridDim.x);
        if (a.low) {
#pragma unroll
            for (uint32_t e = 0; e < E; ++e) U[e].add(p[e]);
        }
        if constexpr (NC > 0) {
            const uint32_t sg = sg_s[(j >> 3) & 1u][j & 7u];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const R s = ((sg >> c) & 1u) ? R(-1) : R(1);
#pragma unroll
                for (uint32_t e = 0; e < E; ++e) X[c * E + e].add(s * p[e]);
            }
        }
        if (a.nhi) {
            S t;
            t.clear();
#pragma unroll
            for (uint32_t e = 0; e < E; ++e) t.add(p[e]);
            hi_acc += wh_s[(j >> 3) & 1u][j & 7u] * t.value();
        }
    }
    double acc = hi_acc;
#pragma unroll
    for (uint32_t e = 0; e < E; ++e) {
        const uint32_t k = F ? (e >> 1) * 2u * THREADS + 2u * tid + (e & 1u) : e * THREADS + tid;
        if (k >= (1u << a.t)) continue;
        if (a.low) acc += a.w[k] * U[e].value();
#pragma unroll
        for (int c = 0; c < NC; ++c) acc += a.w[((size_t)(c + 1) << a.t) + k] * X[c * E + e].value();
    }
    const double r = block_sum(acc);
    if (tid == 0) a.partial[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = r;
}

// ---------------------------------------------------------------- strings with X or Y

constexpr uint32_t X_TERMS = 16;      // terms per pass
constexpr uint32_t X_SETS = 3;        // register sets R per pass

struct XTerm {
    unsigned long long z;      // on index bits outside the tile (tile base)
    double coef;               // 2 ccr, or -2 cci when |x & z| is odd
    uint32_t zt;               // on tile positions held by the thread index
    uint32_t xr;               // x on the register bits (1..15)
    uint32_t signs;            // bit j: (-1)^{|j & z|} of register index j
    uint32_t odd;              // 1: sum the imaginary parts
};

struct XArgs {
    CUtensorMap tmap;
    uint32_t box_rows, boxes, tb;             // tile bits
    uint32_t L, h, hi[SV_MAX_K];
    unsigned long long begin, end;            // tiles of this launch
    double *partial;
    int *err;
    uint32_t nsets, first[X_SETS], last[X_SETS];   // other terms of set i: first[i] .. last[i] - 1
    uint32_t rbit[X_SETS][4];                 // its register bits, as tile positions, ascending
    // single flips of register bit q without signs inside the registers (an X term of a field,
    // most of what is asked): plain[i][q] is the term, or -1; they come before first[i]
    int32_t plain[X_SETS][4];
    uint32_t nplain[X_SETS];
    uint32_t nterms;
    XTerm term[X_TERMS];
};

__device__ __forceinline__ float flip(float x, uint32_t bit31) { return __uint_as_float(__float_as_uint(x) ^ bit31); }
__device__ __forceinline__ double flip(double x, uint32_t bit31) {
    return __hiloint2double(__double2hiint(x) ^ (int)bit31, __double2loint(x));
}

__device__ __forceinline__ void keep(float2 &v) { asm volatile("" : "+f"(v.x), "+f"(v.y)); }
__device__ __forceinline__ void keep(double2 &v) { asm volatile("" : "+d"(v.x), "+d"(v.y)); }

// acc + (a.x b.x, a.y b.y): one packed instruction in FP32.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 acc) {
    float2 r;
    asm("{\n\t.reg .b64 x, y, z;\n\t"
        "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\t"
        "fma.rn.f32x2 z, x, y, z;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(acc.x), "f"(acc.y));
    return r;
}
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 acc) {
    return make_double2(__fma_rn(a.x, b.x, acc.x), __fma_rn(a.y, b.y, acc.y));
}

// Sum over the eight pairs (k, k ^ XR) of the sixteen register amplitudes, bit hb(XR) of k
// clear, of (-1)^{signs[k]} Re or Im of conj(psi[k ^ XR]) psi[k]: two chains of eight FMAs,
// one per product of the real or imaginary part.
template <typename R, int XR, bool ODD, bool SIGNED, typename C>
__device__ __forceinline__ R pair_sum(const C (&v)[16], uint32_t signs) {
    constexpr int HB = XR >= 8 ? 8 : (XR >= 4 ? 4 : (XR >= 2 ? 2 : 1));
    C acc;
    acc.x = acc.y = 0;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        if (k & HB) continue;
        C p = v[k], q = v[k ^ XR];
        if constexpr (ODD) {                       // Im: q.x p.y - q.y p.x
            const R t = p.x;
            p.x = p.y;
            p.y = t;
        }
        if constexpr (SIGNED) {
            const uint32_t f = (signs << (31 - k)) & 0x80000000u;
            q.x = flip(q.x, f);
            q.y = flip(q.y, f);
        }
        acc = fma2(q, p, acc);
    }
    return ODD ? acc.x - acc.y : acc.x + acc.y;
}

// The four variants of each x; SIGNED only where a sign differs within the registers.
template <typename R, int XR, typename C>
__device__ __forceinline__ R pair_any(const C (&v)[16], uint32_t signs, uint32_t odd) {
    if (signs) return odd ? pair_sum<R, XR, true, true>(v, signs) : pair_sum<R, XR, false, true>(v, signs);
    return odd ? pair_sum<R, XR, true, false>(v, signs) : pair_sum<R, XR, false, false>(v, signs);
}

// PLAIN: every term is a plain flip (at most four per set): running sums in registers, the sets
// unrolled.  Without the sums' 32 KiB three blocks fit an SM (complex64), 24 warps to hide latency:
// a 26-qubit field of 26 X terms and its ZZ chain 693 -> 577 us (two blocks: 641), and 560
// with one block barrier per tile instead of two.
template <typename R, bool PLAIN>
constexpr int x_blocks = PLAIN && sizeof(R) == 4 ? 3 : 2;
template <typename R, bool PLAIN>
__global__ void __launch_bounds__(THREADS, x_blocks<R, PLAIN>) x_sum(const __grid_constant__ XArgs a) {
    using C = typename Geo<R>::C;
    using S = typename Sum<R>::T;
    constexpr uint32_t TILE = (1u << Geo<R>::T) * (uint32_t)sizeof(C);
    constexpr uint32_t NT = (1u << Geo<R>::T) / 16u;           // threads that hold amplitudes
    extern __shared__ __align__(1024) unsigned char smem[];    // two tiles, then the sums
    __shared__ __align__(8) unsigned long long full[2];
    S *sums = reinterpret_cast<S *>(smem + 2 * TILE);          // [term][NT] (not PLAIN)
    S racc[PLAIN ? X_SETS * 4 : 1];                            // PLAIN: [set][register bit]
    const uint32_t tid = threadIdx.x, lane = tid & 31u;
    const uint32_t nseg = 1u << a.h, seg_amps = 1u << a.L;
    const uint32_t nact = 1u << (a.tb - 4u);
    const bool act = tid < nact;
    if (tid == 0) {
        svk::mbar_init(svk::smem_u32(&full[0]), 1);
        svk::mbar_init(svk::smem_u32(&full[1]), 1);
        svk::fence_mbar_init();
    }
    const uint32_t nterms = a.nterms;
    if (PLAIN) {
#pragma unroll
        for (uint32_t t = 0; t < (PLAIN ? X_SETS * 4 : 1); ++t) racc[t].clear();
    } else if (act) {
        for (uint32_t t = 0; t < nterms; ++t) sums[t * NT + tid].clear();
    }
    const unsigned long long my_z = lane < nterms ? a.term[lane].z : 0ull;
    svk::SegLanes sl;
    sl.init(a.L, a.h, a.hi, lane);
    svk::pass_trigger();
    svk::pass_wait();
    __syncthreads();
    constexpr uint32_t ROW = 128u / (uint32_t)sizeof(C);       // amplitudes per 128-byte row
    auto load = [&](unsigned long long t, uint32_t s) {        // warp 0
        const uint32_t bar = svk::smem_u32(&full[s]);
        if (lane == 0) svk::mbar_arrive_expect_tx(bar, (uint32_t)sizeof(C) << a.tb);
        __syncwarp();
        if (lane < nseg) {
            const int32_t row0 = (int32_t)((sl.base(t) + sl.my_off) / ROW);
            const uint32_t d0 = svk::smem_u32(smem + s * TILE) + lane * seg_amps * (uint32_t)sizeof(C);
            for (uint32_t bx = 0; bx < a.boxes; ++bx)
                svk::tma_load_2d(d0 + bx * a.box_rows * 128u, &a.tmap, 0, row0 + (int32_t)(bx * a.box_rows), bar);
        }
    };
    if (tid < 32) {
        load(a.begin + blockIdx.x, 0);
        if (a.begin + blockIdx.x + gridDim.x < a.end) load(a.begin + blockIdx.x + gridDim.x, 1);
    }
    uint32_t j = 0;
    for (unsigned long long t = a.begin + blockIdx.x; t < a.end; t += gridDim.x, ++j) {
        const uint32_t s = j & 1u;
        const bool ok = svk::mbar_wait_bounded(svk::smem_u32(&full[s]), (j >> 1) & 1u);
        const C *tile = reinterpret_cast<const C *>(smem + s * TILE);
        // bit i: (-1)^{|base & z_i|}, lane i's term
        const uint32_t tile_signs = __ballot_sync(0xffffffffu, __popcll(sl.base(t) & my_z) & 1);
        // the sixteen amplitudes of a register set
        auto read_set = [&](uint32_t set, C (&v)[16]) {
            uint32_t g = tid;
            uint32_t rb[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                g = svk::insert_zero32(g, a.rbit[set][q]);
                rb[q] = 1u << a.rbit[set][q];
                rb[q] = sizeof(R) == 4 ? svk::swz128(rb[q]) : svk::swz128_16(rb[q]);
            }
            g = sizeof(R) == 4 ? svk::swz128(g) : svk::swz128_16(g);
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                uint32_t o = g;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if ((k >> q) & 1) o ^= rb[q];
                v[k] = tile[o];
            }
        };
        if constexpr (PLAIN) {
            if (act && ok) {
#pragma unroll
                for (uint32_t set = 0; set < X_SETS; ++set) {
                    if (set >= a.nsets) break;
                    C v[16];
                    read_set(set, v);
                    const R x[4] = {pair_sum<R, 1, false, false>(v, 0), pair_sum<R, 2, false, false>(v, 0),
                                    pair_sum<R, 4, false, false>(v, 0), pair_sum<R, 8, false, false>(v, 0)};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int32_t i = a.plain[set][q];
                        if (i >= 0) racc[set * 4 + q].add(flip(x[q], ((tile_signs >> i) & 1u) << 31));
                    }
                }
            }
        } else if (act && ok) {
            for (uint32_t set = 0; set < a.nsets; ++set) {
                C v[16];
                read_set(set, v);
                auto accumulate = [&](R x, uint32_t i) {
                    S acc = sums[i * NT + tid];
                    acc.add(flip(x, ((tile_signs >> i) & 1u) << 31));
                    sums[i * NT + tid] = acc;
                };
                if (a.nplain[set]) {
                    // all four in one straight line: no dispatch, four chains in flight
                    const R x[4] = {pair_sum<R, 1, false, false>(v, 0), pair_sum<R, 2, false, false>(v, 0),
                                    pair_sum<R, 4, false, false>(v, 0), pair_sum<R, 8, false, false>(v, 0)};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (a.plain[set][q] >= 0) accumulate(x[q], (uint32_t)a.plain[set][q]);
                }
                for (uint32_t i = a.first[set]; i < a.last[set]; ++i) {
                    // keeps the products of all fifteen cases from being moved out of this
                    // loop (they would spill)
#pragma unroll
                    for (int k = 0; k < 16; ++k) keep(v[k]);
                    const uint32_t sg = a.term[i].signs;
                    R x;
                    const uint32_t odd = a.term[i].odd;
                    switch (a.term[i].xr) {
#define SVX_CASE(n) case n: x = pair_any<R, n>(v, sg, odd); break;
                        SVX_CASE(1) SVX_CASE(2) SVX_CASE(3) SVX_CASE(4) SVX_CASE(5) SVX_CASE(6) SVX_CASE(7)
                        SVX_CASE(8) SVX_CASE(9) SVX_CASE(10) SVX_CASE(11) SVX_CASE(12) SVX_CASE(13) SVX_CASE(14)
#undef SVX_CASE
                        default: x = pair_any<R, 15>(v, sg, odd); break;
                    }
                    accumulate(x, i);
                }
            }
        }
        svk::fence_proxy_async_smem();        // reads of this tile before its refill
        if (__syncthreads_or(!ok)) {
            // the copy may still be in flight: wait once more (bounded) before the memory goes
            if (tid == 0) atomicOr(a.err, 8);
            (void)svk::mbar_wait_bounded(svk::smem_u32(&full[s]), (j >> 1) & 1u);
            (void)svk::mbar_wait_bounded(svk::smem_u32(&full[s ^ 1u]), ((j + 1u) >> 1) & 1u);
            return;
        }
        const unsigned long long t2 = t + 2ull * gridDim.x;
        if (tid < 32 && t2 < a.end) load(t2, s);
    }
    double acc = 0.0;
    if (act)
        for (uint32_t set = 0; set < a.nsets; ++set) {
            uint32_t g = tid;
#pragma unroll
            for (int q = 0; q < 4; ++q) g = svk::insert_zero32(g, a.rbit[set][q]);
            auto weigh = [&](const S &sum, uint32_t i) {
                const double v = sum.value() * a.term[i].coef;
                acc += (__popc(g & a.term[i].zt) & 1) ? -v : v;
            };
            if constexpr (PLAIN) {
                // register indices stay constants: each set picks its own four
#pragma unroll
                for (uint32_t t = 0; t < X_SETS * 4; ++t)
                    if (t / 4 == set && a.plain[set][t % 4] >= 0) weigh(racc[t], (uint32_t)a.plain[set][t % 4]);
            } else {
                for (uint32_t i = a.first[set] - a.nplain[set]; i < a.last[set]; ++i) weigh(sums[i * NT + tid], i);
            }
        }
    const double r = block_sum(acc);
    if (tid == 0) a.partial[blockIdx.x] = r;
}

}  // namespace svx

namespace svi {

namespace {

struct Term { uint64_t x, z; double c; };

// Tiles of one launch of nb blocks: all of them, in complex64 at most RUN_TILES per thread.
template <typename R>
unsigned long long run_tiles(unsigned long long nb) {
    return sizeof(R) == 4 ? svx::RUN_TILES * nb : 1ull << SV_MAX_QUBITS;
}

// Block partials of several passes, summed in order by one kernel per full buffer; the sums
// are fetched when their slots run out, and at the end.
struct Partials {
    sv_state *s;
    int used = 0, nres = 0;
    double total = 0.0;
    double *part() const { return reinterpret_cast<double *>(s->ws + WS_PARTIAL) + used; }
    // room for n partials (n <= WS_NPARTIAL)
    sv_status reserve(int n) { return used + n > WS_NPARTIAL ? fold() : SV_OK; }
    // a slot for one more sum
    sv_status slot(double **out) {
        const sv_status st = nres >= 60 ? collect() : SV_OK;
        *out = mail_results(s) + nres++;
        return st;
    }
    sv_status fold() {
        if (!used) return SV_OK;
        double *out;
        const sv_status st = slot(&out);
        if (st != SV_OK) return st;
        const int n = used;
        used = 0;
        return enqueue_sum(s, n, out);
    }
    sv_status collect() {
        double h[64];
        if (!nres) return SV_OK;
        const sv_status st = read_results(s, h, sizeof(double) * nres);
        if (st != SV_OK) return st;
        for (int r = 0; r < nres; ++r) total += h[r];
        nres = 0;
        return SV_OK;
    }
};

// The Z strings t[0 .. n) on `states` states of nq qubits at psi, tables in `tables`: every pass
// asks `reserve` where its partials go (blocks per state, state by state) and says with `ran`
// that it has been enqueued.
template <typename R, typename Reserve, typename Ran>
sv_status z_passes(const void *psi, uint32_t nq, uint32_t states, int num_sms, cudaStream_t stream, double *tables,
                   const Term *t, size_t n, Reserve reserve, Ran ran) {
    using namespace svx;
    const uint32_t T = std::min(nq, Geo<R>::T);
    for (size_t b = 0; b < n; b += Z_TERMS) {
        const uint32_t m = (uint32_t)std::min<size_t>(Z_TERMS, n - b);
        const uint64_t lo = (1ull << T) - 1;
        ZTableArgs ta;
        ZArgs a;
        ta.nterms = m;
        ta.t = T;
        a.nhi = 0;
        std::vector<uint64_t> cls;
        bool low = false;
        for (uint32_t i = 0; i < m; ++i) {
            const uint64_t z = t[b + i].z;
            ta.z[i] = z;
            ta.c[i] = t[b + i].c;
            if ((z >> T) == 0) {
                low = true;
            } else if ((z & lo) == 0) {
                a.zh[a.nhi] = z >> T;
                a.ch[a.nhi++] = t[b + i].c;
            } else if (std::find(cls.begin(), cls.end(), z >> T) == cls.end()) {
                cls.push_back(z >> T);
            }
        }
        a.psi = psi;
        a.t = T;
        a.ntiles = 1ull << (nq - T);
        ta.w = tables;
        a.w = tables;
        size_t done = 0;
        bool first = true;
        while (first || done < cls.size()) {
            const uint32_t nc = (uint32_t)std::min<size_t>(Z_CLASSES, cls.size() - done);
            a.low = first && low;
            if (!first) a.nhi = 0;
            ta.ntab = 1 + nc;
            ta.zc[0] = 0;
            for (uint32_t c = 0; c < nc; ++c) ta.zc[1 + c] = a.zc[c] = cls[done + c];
            // as many blocks as the device holds, shared by the states
            const unsigned long long slots = (unsigned long long)(nc >= 2 ? 1 : 2) * (unsigned long long)num_sms;
            const unsigned long long blocks = std::max<unsigned long long>(1, slots / states);
            if (a.low || nc)
                SV_CUDA(svk::launch_pass(z_table, dim3((unsigned)(((1u << T) + 127) / 128), ta.ntab), 128, 0, stream, ta));
            for (a.begin = 0; a.begin < a.ntiles; a.begin = a.end) {
                a.end = std::min(a.ntiles, a.begin + run_tiles<R>(blocks));
                const int nb = (int)std::min(blocks, a.end - a.begin);
                const dim3 grid(nb, states);
                sv_status st = reserve(nb, &a.partial);
                if (st != SV_OK) return st;
                cudaError_t e = cudaSuccess;
                switch (nc) {
                    case 0: e = svk::launch_pass(z_sum<R, 0>, grid, THREADS, 0, stream, a); break;
                    case 1: e = svk::launch_pass(z_sum<R, 1>, grid, THREADS, 0, stream, a); break;
                    case 2: e = svk::launch_pass(z_sum<R, 2>, grid, THREADS, 0, stream, a); break;
                    default: e = svk::launch_pass(z_sum<R, 3>, grid, THREADS, 0, stream, a); break;
                }
                SV_CUDA(e);
                st = ran(nb);
                if (st != SV_OK) return st;
            }
            done += nc;
            first = false;
        }
    }
    return SV_OK;
}

template <typename R>
sv_status z_group(sv_state *s, Partials &P, const Term *t, size_t n) {
    // the tables lie in the top-k scratch (4 MiB), which no expectation uses
    return z_passes<R>(
        s->buf, s->n, 1, s->num_sms, s->stream, reinterpret_cast<double *>(s->ws + WS_TOPK), t, n,
        [&](int nb, double **out) {
            const sv_status st = P.reserve(nb);
            *out = P.part();
            return st;
        },
        [&](int nb) {
            P.used += nb;
            return SV_OK;
        });
}

// One x_sum pass: the tile's high bits H (ascending, above L), and the terms of `t` that are
// still open (done[i] = 0), lie inside the tile and fit the register sets.
template <typename R>
sv_status x_pass(sv_state *s, Partials &P, const std::vector<Term> &t, std::vector<char> &done,
                 const std::vector<uint32_t> &H, uint32_t L) {
    using namespace svx;
    XArgs a;
    a.tb = L + (uint32_t)H.size();
    a.L = L;
    a.h = (uint32_t)H.size();
    uint64_t tile = (1ull << L) - 1;
    for (uint32_t j = 0; j < SV_MAX_K; ++j) {
        a.hi[j] = j < a.h ? H[j] : 0u;
        if (j < a.h) tile |= 1ull << H[j];
    }
    // a mask on index bits -> on tile positions
    auto to_tile = [&](uint64_t m) {
        uint32_t r = (uint32_t)(m & ((1ull << L) - 1));
        for (uint32_t j = 0; j < a.h; ++j) r |= (uint32_t)((m >> H[j]) & 1ull) << (L + j);
        return r;
    };
    uint32_t sets[X_SETS] = {0, 0, 0};
    std::vector<size_t> in[X_SETS];
    uint32_t ns = 0, total = 0;
    for (size_t i = 0; i < t.size() && total < X_TERMS; ++i) {
        if (done[i] || (t[i].x & ~tile)) continue;
        const uint32_t x = to_tile(t[i].x);
        uint32_t best = X_SETS;
        for (uint32_t q = 0; q < ns && best == X_SETS; ++q)
            if (__builtin_popcount(sets[q] | x) <= 4) best = q;
        if (best == X_SETS) {
            if (ns == X_SETS) continue;
            best = ns++;
        }
        sets[best] |= x;
        in[best].push_back(i);
        done[i] = 1;
        ++total;
    }
    a.nsets = ns;
    a.nterms = total;
    uint32_t m = 0;
    for (uint32_t q = 0; q < ns; ++q) {
        // fill the set up to four bits from the top (bits 0-3 choose the bank)
        for (int p = (int)a.tb - 1; p >= 0 && __builtin_popcount(sets[q]) < 4; --p) sets[q] |= 1u << p;
        uint32_t nb = 0;
        for (uint32_t p = 0; p < a.tb; ++p)
            if ((sets[q] >> p) & 1u) a.rbit[q][nb++] = p;
        auto to_reg = [&](uint32_t tm) {
            uint32_t r = 0;
            for (uint32_t p = 0; p < 4; ++p) r |= ((tm >> a.rbit[q][p]) & 1u) << p;
            return r;
        };
        // plain single flips first, one per register bit
        a.nplain[q] = 0;
        for (int p = 0; p < 4; ++p) a.plain[q][p] = -1;
        std::vector<size_t> order, rest;
        for (size_t i : in[q]) {
            const uint32_t xr = to_reg(to_tile(t[i].x)), zr = to_reg(to_tile(t[i].z & tile));
            const int p = __builtin_ctz(xr);
            if (xr == (1u << p) && !zr && a.plain[q][p] < 0) {
                a.plain[q][p] = (int32_t)(m + order.size());
                ++a.nplain[q];
                order.push_back(i);
            } else {
                rest.push_back(i);
            }
        }
        a.first[q] = m + a.nplain[q];
        order.insert(order.end(), rest.begin(), rest.end());
        for (size_t i : order) {
            XTerm &e = a.term[m++];
            const uint32_t zt = to_tile(t[i].z & tile), zr = to_reg(zt);
            const int y = __builtin_popcountll(t[i].x & t[i].z) & 3;      // i^y
            const double re[4] = {1, 0, -1, 0}, im[4] = {0, 1, 0, -1};
            e.odd = y & 1;
            e.coef = e.odd ? -2.0 * t[i].c * im[y] : 2.0 * t[i].c * re[y];
            e.z = t[i].z & ~tile;
            e.xr = to_reg(to_tile(t[i].x));
            e.zt = zt & ~sets[q];
            e.signs = 0;
            for (uint32_t k = 0; k < 16; ++k) e.signs |= (uint32_t)(__builtin_popcount(k & zr) & 1) << k;
        }
        a.last[q] = m;
    }
    const sv_status st = svk::encode_rows_map(s->buf, (unsigned long long)sizeof(typename Geo<R>::C) << s->n,
                                              (uint32_t)sizeof(typename Geo<R>::C) << L, &a.tmap, &a.box_rows, &a.boxes);
    if (st != SV_OK) return st;
    const unsigned long long ntiles = 1ull << (s->n - a.tb);
    uint32_t flips = 0;
    for (uint32_t q = 0; q < ns; ++q) flips += a.nplain[q];
    const bool plain = flips == total;
    // as many blocks as the device holds
    const unsigned long long blocks = (unsigned long long)(plain ? x_blocks<R, true> : x_blocks<R, false>) *
                                      (unsigned long long)s->num_sms;
    a.err = reinterpret_cast<int *>(s->ws + WS_ERR);
    constexpr size_t tile_bytes = sizeof(typename Geo<R>::C) << Geo<R>::T;
    constexpr size_t smem = 2 * tile_bytes + X_TERMS * ((1u << Geo<R>::T) / 16) * sizeof(typename Sum<R>::T);
    static svk::PerDevice<cudaError_t> setup;
    SV_CUDA(setup.get(svk::current_device(), [] {
        cudaError_t e = cudaFuncSetAttribute(x_sum<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(x_sum<R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(2 * tile_bytes));
        return e;
    }));
    for (a.begin = 0; a.begin < ntiles; a.begin = a.end) {
        a.end = std::min(ntiles, a.begin + run_tiles<R>(blocks));
        const int nb = (int)std::min(blocks, a.end - a.begin);       // every block has a tile
        const sv_status rs = P.reserve(nb);
        if (rs != SV_OK) return rs;
        a.partial = P.part();
        SV_CUDA(plain ? svk::launch_pass(x_sum<R, true>, dim3(nb), THREADS, 2 * tile_bytes, s->stream, a)
                      : svk::launch_pass(x_sum<R, false>, dim3(nb), THREADS, smem, s->stream, a));
        P.used += nb;
    }
    return SV_OK;
}

// Every term with 1 to 4 X or Y factors, in as few reads of the state as the greedy choice of
// tiles gives: first the terms inside the lowest bits, then tiles of the lowest bits and five
// high ones.
template <typename R>
sv_status x_group(sv_state *s, Partials &P, const std::vector<Term> &t) {
    using namespace svx;
    const uint32_t TB = std::min(s->n, Geo<R>::T);
    std::vector<char> done(t.size(), 0);
    const uint32_t L = TB >= 5 ? TB - 5 : 0;       // low bits of a tile with five high ones
    while (true) {
        size_t f = 0;
        bool inside = false;
        for (size_t i = 0; i < t.size() && !inside; ++i) inside = !done[i] && !(t[i].x >> TB);
        std::vector<uint32_t> H;
        uint32_t low = TB;
        if (!inside) {
            while (f < t.size() && done[f]) ++f;
            if (f == t.size()) return SV_OK;
            // high bits of the open terms, as long as five hold them
            low = L;
            uint64_t hm = 0;
            for (size_t i = f; i < t.size(); ++i) {
                if (done[i]) continue;
                const uint64_t m = hm | (t[i].x >> L << L);
                if (__builtin_popcountll(m) <= 5) hm = m;
            }
            for (uint32_t b = L; b < s->n && __builtin_popcountll(hm) < 5; ++b) hm |= 1ull << b;
            for (uint32_t b = L; b < s->n; ++b)
                if ((hm >> b) & 1ull) H.push_back(b);
        }
        const sv_status st = x_pass<R>(s, P, t, done, H, low);
        if (st != SV_OK) return st;
    }
}

}  // namespace

std::vector<char> batch_z_split(uint32_t n, sv_dtype dtype, uint32_t states, const uint64_t *z, size_t nterms) {
    const uint32_t T = std::min(n, dtype == SV_C64 ? svx::Geo<float>::T : svx::Geo<double>::T);
    return svx::split_z(z, nterms, T, std::ldexp((double)states, (int)n), svx::Z_COST_BATCH[dtype]);
}

// Z strings on a batch: the tables (4 x 2^12 doubles) and `partial` (room for `room` doubles) are the
// caller's; after each pass `fold` is called with the number of partials per state that lie there.
sv_status batch_z_terms(const void *psi, uint32_t n, sv_dtype dtype, uint32_t states, int num_sms, cudaStream_t stream,
                        double *tables, double *partial, size_t room, const uint64_t *z, const double *c, size_t nterms,
                        const std::function<sv_status(int)> &fold) {
    std::vector<Term> t(nterms);
    for (size_t i = 0; i < nterms; ++i) t[i] = Term{0, z[i], c[i]};
    auto reserve = [&](int nb, double **out) {
        *out = partial;
        return (size_t)nb * states <= room ? SV_OK : set_error(SV_ERR_ARG, "expectation: too few partials");
    };
    return dtype == SV_C64
               ? z_passes<float>(psi, n, states, num_sms, stream, tables, t.data(), nterms, reserve, fold)
               : z_passes<double>(psi, n, states, num_sms, stream, tables, t.data(), nterms, reserve, fold);
}

// general: every term by the general kernel.
static sv_status expect_terms(sv_state *s, const uint64_t *x, const uint64_t *z, const double *c, size_t nterms,
                              bool general, double *host_out) {
    std::vector<Term> t(nterms);
    for (size_t i = 0; i < nterms; ++i) t[i] = Term{x[i], z[i], c[i]};
    std::stable_sort(t.begin(), t.end(), [](const Term &a, const Term &b) { return a.x < b.x; });
    Partials P{s};
    std::vector<Term> xt;
    for (size_t i = 0; i < nterms;) {
        size_t e = i;
        while (e < nterms && t[e].x == t[i].x) ++e;
        sv_status st = SV_OK;
        size_t g = i;                       // t[g] .. t[e - 1] take the general kernel
        if (t[i].x == 0 && !general) {
            std::vector<uint64_t> zs;
            for (size_t q = i; q < e; ++q) zs.push_back(t[q].z);
            const uint32_t T = std::min(s->n, s->dtype == SV_C64 ? svx::Geo<float>::T : svx::Geo<double>::T);
            const std::vector<char> to_general =
                svx::split_z(zs.data(), zs.size(), T, std::ldexp(1.0, (int)s->n), svx::Z_COST_SINGLE[s->dtype]);
            std::vector<Term> tiled, rest;
            for (size_t q = i; q < e; ++q) (to_general[q - i] ? rest : tiled).push_back(t[q]);
            std::copy(rest.begin(), rest.end(), std::copy(tiled.begin(), tiled.end(), t.begin() + i));
            g = i + tiled.size();
            if (g > i)
                st = s->dtype == SV_C64 ? z_group<float>(s, P, &t[i], g - i) : z_group<double>(s, P, &t[i], g - i);
        } else if (!general && s->n >= 4 && __builtin_popcountll(t[i].x) <= 4 && (s->dtype == SV_C128 || e - i <= 4)) {
            xt.insert(xt.end(), t.begin() + i, t.begin() + e);
            g = e;
        }
        for (size_t b = g; b < e && st == SV_OK; b += 32) {      // up to 32 terms per launch
            uint64_t zz[32];
            double cc[32];
            const int m = (int)std::min<size_t>(32, e - b);
            for (int q = 0; q < m; ++q) {
                zz[q] = t[b + q].z;
                cc[q] = t[b + q].c;
            }
            double *out;
            st = P.fold();
            if (st == SV_OK) st = P.slot(&out);
            if (st == SV_OK) st = enqueue_expect_group(s, t[b].x, zz, cc, m, out);
        }
        if (st != SV_OK) return st;
        i = e;
    }
    if (!xt.empty()) {
        const sv_status st = s->dtype == SV_C64 ? x_group<float>(s, P, xt) : x_group<double>(s, P, xt);
        if (st != SV_OK) return st;
    }
    sv_status st = P.fold();
    if (st == SV_OK) st = P.collect();
    *host_out = P.total;
    return st;
}

// Two-float sums end at 3.4e38 where the general kernel's FP64 sums go on (amplitudes around 1e18):
// a complex64 result that is not finite is formed again there.
sv_status launch_expect(sv_state *s, const uint64_t *x, const uint64_t *z, const double *c,
                        size_t nterms, double *host_out) {
    const sv_status st = expect_terms(s, x, z, c, nterms, false, host_out);
    if (st != SV_OK || s->dtype != SV_C64 || std::isfinite(*host_out)) return st;
    return expect_terms(s, x, z, c, nterms, true, host_out);
}

}  // namespace svi
