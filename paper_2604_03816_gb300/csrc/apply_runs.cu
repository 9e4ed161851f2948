// Runs of consecutive gates that share one read and one write of the state.
//
// Diagonal runs.  A QFT's schedule is mostly diagonal gates, up to 22 of them in a row; one
// pass each is one read and write each for one complex product.  Diagonal gates commute, so a
// run is one factor per amplitude, f(i) = prod_g d_g(i).  It is formed from few products:
//   1. diag_tables (tiny): gates with the same low qubits (below the tile's T bits) are multiplied
//      into tables of at most 8 qubits, in FP64;
//   2. apply_diag_run: the T low bits are split into two bins so that every table's low qubits
//      lie in one bin (connected sets of low qubits, packed).  For each tile of 2^T consecutive
//      amplitudes the tile's high bits fix the rest of every index, so the tables collapse to
//      two small ones, H0 over bin 0 and H1 over bin 1 (up to 128 entries, shared memory), and
//      f = H0[a] H1[b]: two products per amplitude however long the run is.  Tiles whose two
//      tables are all 1 are not touched; amplitudes whose factor is exactly 1 keep their bits.
// Where all the run's qubits lie below T, f is one table of 2^T entries, the same for every tile:
// diag_tables forms it whole, and apply_low_run keeps each thread's entries in registers.
// Measured, 28 qubits, complex64: one pass of 0.37 ms per gate -> 0.64 ms per run (the copy
// speed), the QFT's 72 diagonal gates 26.9 -> 4.9 ms; 23 qubits, complex128: 36 us per gate ->
// 157 us per run (the FP64 pipe: 8 operations per amplitude, and its tables; 82 inside the low
// bits), 69 gates 2.5 -> 0.9 ms.
//
// Swap runs.  Consecutive gates that only permute index bits, whose product swaps pairs of
// bits (the bit reversal that ends a QFT: 13 passes of half the state each on 28 qubits, 5.07 ms),
// are one pass (0.84 ms): the tile is the a low bits and their partners (and pairs of other bits up to 12),
// so it is closed under the permutation, and tiles r and pi(r) trade places through shared
// memory, read and written in rows of 2^a amplitudes.
//
// When: a run moves the whole state once, so it pays when its gates, one pass each, touch more
// than that; the thresholds and what they were measured at stand at ONE_PRODUCT and least_gates.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "ptx.cuh"
#include "sv_internal.h"

namespace svr {

template <typename R> struct Cx;
template <> struct Cx<float> { using T = float2; };
template <> struct Cx<double> { using T = double2; };
__device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mk(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ float fmar(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmar(double a, double b, double c) { return __fma_rn(a, b, c); }
template <typename C>
__device__ __forceinline__ C cmul(C a, C b) {
    return mk(fmar(a.x, b.x, -(a.y * b.y)), fmar(a.x, b.y, a.y * b.x));
}

// Is the factor exactly 1 (+-0 i)?  In FP64 by its bits: a compare costs as much as a product on
// this GPU's FP64 pipe.
__device__ __forceinline__ bool is_one(float2 f) { return f.x == 1.f && f.y == 0.f; }
__device__ __forceinline__ bool is_one(double2 f) {
    return __double_as_longlong(f.x) == 0x3FF0000000000000ll && (__double_as_longlong(f.y) << 1) == 0ll;
}

constexpr uint32_t MAX_GATES = 40;      // gates of a run
constexpr uint32_t TAB_Q = 8;           // qubits of a merged table
constexpr uint32_t MAX_TABS = 12;
constexpr uint32_t BIN_Q = 7;           // low bits of a bin
constexpr uint32_t THREADS = 256;

// Tile bits: 2^T amplitudes are 64 KiB in both precisions.
template <typename R> constexpr uint32_t tile_bits() { return sizeof(R) == 4 ? 13u : 12u; }

// ---------------------------------------------------------------- diagonal runs

struct TablesArgs {
    uint32_t ngates, ntabs;
    uint8_t nq[MAX_TABS];                   // qubits of each table
    uint8_t tab[MAX_GATES];                 // the table a gate goes into
    uint8_t k[MAX_GATES];
    uint8_t pos[MAX_GATES][SV_MAX_K];       // its qubits as positions in the table's qubits
    uint32_t first[MAX_GATES];              // its entries
    uint32_t lg;                            // entries per table: 2^lg
    void *out;                              // [ntabs][2^lg], in the state's precision
    double2 d[MAX_GATES << SV_MAX_K];
};
static_assert(sizeof(TablesArgs) <= 32764, "kernel parameters");

// Entry e of table t, one per thread: the product of its gates' entries.
template <typename R>
__global__ void diag_tables(const __grid_constant__ TablesArgs a) {
    svk::pass_trigger();
    const uint32_t t = blockIdx.x, e = blockIdx.y * blockDim.x + threadIdx.x;
    double2 p = make_double2(1.0, 0.0);
    if (e < (1u << a.nq[t]))
        for (uint32_t g = 0; g < a.ngates; ++g) {
            if (a.tab[g] != t) continue;
            uint32_t l = 0;
            for (uint32_t j = 0; j < a.k[g]; ++j) l |= ((e >> a.pos[g][j]) & 1u) << j;
            const double2 d = a.d[a.first[g] + l];
            if (!is_one(d)) p = is_one(p) ? d : cmul(d, p);
        }
    svk::pass_wait();                       // the previous run's pass may still read the tables
    typename Cx<R>::T *out = reinterpret_cast<typename Cx<R>::T *>(a.out);
    out[(t << a.lg) + e] = mk((R)p.x, (R)p.y);
}

struct DiagRunArgs {
    void *psi;
    const void *tabs;
    unsigned long long ntiles;
    uint32_t ntabs, nbin[2];                // bits of each bin
    uint8_t bin[MAX_TABS];                  // the bin a table multiplies into
    uint8_t nq[MAX_TABS];
    uint8_t qubit[MAX_TABS][TAB_Q];
    uint8_t bit_of[2][BIN_Q];               // the index bits of each bin
};

template <typename R>
__global__ void __launch_bounds__(THREADS, 3) apply_diag_run(const __grid_constant__ DiagRunArgs a) {
    using C = typename Cx<R>::T;
    constexpr uint32_t T = tile_bits<R>();
    constexpr bool F = sizeof(R) == 4;
    constexpr uint32_t NV = 16;                           // 16-byte words per thread and tile
    extern __shared__ __align__(16) unsigned char smem[];
    C *tab = reinterpret_cast<C *>(smem);                                    // [ntabs][2^TAB_Q]
    C *H = tab + (a.ntabs << TAB_Q);                                         // two tables of 2^BIN_Q
    uint16_t *low = reinterpret_cast<uint16_t *>(H + (2u << BIN_Q));         // [ntabs][2^BIN_Q]
    __shared__ uint32_t hi_s[MAX_TABS];
    const uint32_t tid = threadIdx.x;
    svk::pass_trigger();
    // entry x of table t's bin: the low part of its table index (the same for every tile)
    for (uint32_t i = tid; i < (a.ntabs << BIN_Q); i += THREADS) {
        const uint32_t t = i >> BIN_Q, x = i & ((1u << BIN_Q) - 1u), b = a.bin[t];
        uint32_t l = 0;
        for (uint32_t j = 0; j < a.nq[t]; ++j)
            for (uint32_t q = 0; q < a.nbin[b]; ++q)
                if (a.qubit[t][j] == a.bit_of[b][q]) l |= ((x >> q) & 1u) << j;
        low[i] = (uint16_t)l;
    }
    // Byte offsets into H of both bins' entries, packed (bin 0 in the low half): the part of this
    // thread's words (word number e THREADS + tid), of e, and of the amplitude within a word.
    uint32_t at = (uint32_t)(sizeof(C) << BIN_Q) << 16, aq = 0;
    __shared__ uint32_t ae[NV];
    {
        uint32_t mine = 0;                                // thread e < NV: the part of e
        for (uint32_t b = 0; b < 2; ++b)
            for (uint32_t q = 0; q < a.nbin[b]; ++q) {
                const uint32_t p = a.bit_of[b][q], w = F ? p - 1u : p;   // bit of the word number
                const uint32_t o = (uint32_t)(sizeof(C) << q) << (16 * b);
                if (F && p == 0) aq = o;
                else if (w < 8) at += (tid >> w) & 1u ? o : 0u;
                else mine += (tid >> (w - 8u)) & 1u ? o : 0u;
            }
        if (tid < NV) ae[tid] = mine;
    }
    svk::pass_wait();
    const C *gt = reinterpret_cast<const C *>(a.tabs);
    for (uint32_t i = tid; i < (a.ntabs << TAB_Q); i += THREADS) tab[i] = gt[i];
    using V = typename std::conditional<F, float4, double2>::type;
    V *psi = reinterpret_cast<V *>(a.psi);
    for (unsigned long long tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
        __syncthreads();                                  // H and hi_s are free
        if (tid < a.ntabs) {                              // the high part of each table's index
            const unsigned long long base = tile << T;
            uint32_t h = 0;
            for (uint32_t j = 0; j < a.nq[tid]; ++j)
                if (a.qubit[tid][j] >= T) h |= (uint32_t)((base >> a.qubit[tid][j]) & 1ull) << j;
            hi_s[tid] = h;
        }
        __syncthreads();
        bool other = false;
        {
            const uint32_t b = tid >> BIN_Q, x = tid & ((1u << BIN_Q) - 1u);
            C p = mk(R(1), R(0));
            if (x < (1u << a.nbin[b]))
                for (uint32_t t = 0; t < a.ntabs; ++t) {
                    if (a.bin[t] != b) continue;
                    const C d = tab[(t << TAB_Q) + (hi_s[t] | low[(t << BIN_Q) + x])];
                    if (!is_one(d)) {
                        p = is_one(p) ? d : cmul(d, p);
                        other = true;
                    }
                }
            H[tid] = p;
        }
        // which bins have a factor other than 1 (the halves of the block hold one bin each)
        const uint32_t any0 = __syncthreads_or(other && tid < (1u << BIN_Q));
        const uint32_t any1 = __syncthreads_or(other && tid >= (1u << BIN_Q));
        if (!any0 && !any1) continue;
        V *p = psi + tile * (NV * THREADS) + tid;
        const unsigned char *h = reinterpret_cast<const unsigned char *>(H);
        auto run_tile = [&](auto both) {
            constexpr int B = decltype(both)::value;      // 0, 1: that bin alone; 2: both
            auto factor = [&](uint32_t x) {
                const C f0 = *reinterpret_cast<const C *>(h + (B == 1 ? x >> 16 : x & 0xFFFFu));
                if constexpr (B < 2) return f0;
                return cmul(f0, *reinterpret_cast<const C *>(h + (x >> 16)));
            };
#pragma unroll
            for (uint32_t e0 = 0; e0 < NV; e0 += 8) {
                V v[8];
#pragma unroll
                for (uint32_t e = 0; e < 8; ++e) v[e] = p[(e0 + e) * THREADS];
#pragma unroll
                for (uint32_t e = 0; e < 8; ++e) {
                    const uint32_t x = at + ae[e0 + e];
                    const C f = factor(x);
                    V w = v[e];
                    if (!is_one(f)) {
                        const C y = cmul(f, mk(v[e].x, v[e].y));
                        w.x = y.x;
                        w.y = y.y;
                    }
                    if constexpr (F) {
                        const C f1 = factor(x + aq);
                        if (!is_one(f1)) {
                            const C y = cmul(f1, mk(v[e].z, v[e].w));
                            w.z = y.x;
                            w.w = y.y;
                        }
                    }
                    p[(e0 + e) * THREADS] = w;
                }
            }
        };
        if (!any1) run_tile(std::integral_constant<int, 0>());
        else if (!any0) run_tile(std::integral_constant<int, 1>());
        else run_tile(std::integral_constant<int, 2>());
    }
}

// The run's factors of the T low bits, f[0 .. 2^T), on every tile.
template <typename R>
__global__ void __launch_bounds__(THREADS, 2) apply_low_run(void *psi_, const void *f_, unsigned long long ntiles) {
    using C = typename Cx<R>::T;
    constexpr bool F = sizeof(R) == 4;
    constexpr uint32_t NV = 16;
    using V = typename std::conditional<F, float4, double2>::type;
    const uint32_t tid = threadIdx.x;
    svk::pass_trigger();
    svk::pass_wait();
    const V *ft = reinterpret_cast<const V *>(f_);
    V f[NV];
#pragma unroll
    for (uint32_t e = 0; e < NV; ++e) f[e] = ft[e * THREADS + tid];
    for (unsigned long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        V *p = reinterpret_cast<V *>(psi_) + tile * (NV * THREADS) + tid;
#pragma unroll
        for (uint32_t e0 = 0; e0 < NV; e0 += 8) {
            V v[8];
#pragma unroll
            for (uint32_t e = 0; e < 8; ++e) v[e] = p[(e0 + e) * THREADS];
#pragma unroll
            for (uint32_t e = 0; e < 8; ++e) {
                const V g = f[e0 + e];
                V w = v[e];
                if (!is_one(mk(g.x, g.y))) {
                    const C y = cmul(mk(g.x, g.y), mk(v[e].x, v[e].y));
                    w.x = y.x;
                    w.y = y.y;
                }
                if constexpr (F) {
                    if (!is_one(mk(g.z, g.w))) {
                        const C y = cmul(mk(g.z, g.w), mk(v[e].z, v[e].w));
                        w.z = y.x;
                        w.w = y.y;
                    }
                }
                p[(e0 + e) * THREADS] = w;
            }
        }
    }
}

// ---------------------------------------------------------------- swap runs

constexpr uint32_t SWAP_TILE = 12;          // bits of a tile at most (complex128: 11)

struct SwapArgs {
    void *psi;
    unsigned long long ntiles;
    uint32_t n, a, h;                        // row bits, rows = 2^h
    uint8_t hi[SWAP_TILE];                   // index bits of the row number, ascending
    uint8_t rest[SV_MAX_QUBITS];             // index bits outside the tile, ascending
    uint8_t pi[SV_MAX_QUBITS];               // the partner of every index bit
};

// Column j of row r of a tile lies at r (2^a + 1) + j: reads down a column then spread over the
// banks.
template <typename R>
__global__ void __launch_bounds__(THREADS, 3) apply_swap_run(const __grid_constant__ SwapArgs a) {
    using C = typename Cx<R>::T;
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t tid = threadIdx.x, cols = 1u << a.a, pitch = cols + 1u, rows = 1u << a.h;
    const uint32_t size = rows << a.a;
    C *buf[2] = {reinterpret_cast<C *>(smem), reinterpret_cast<C *>(smem) + rows * pitch};
    svk::pass_trigger();
    // where element k of a tile comes from in the other tile: column bits and row bits trade
    // places as pi says; k = e THREADS + tid, linear over XOR
    auto tile_pos = [&](uint32_t bit) -> uint32_t {      // index bit -> tile position
        if (bit < a.a) return bit;
        for (uint32_t j = 0; j < a.h; ++j)
            if (a.hi[j] == bit) return a.a + j;
        return 0;
    };
    __shared__ uint32_t src_bit[SWAP_TILE];              // image of tile position p
    __shared__ unsigned long long out_bit[SWAP_TILE];    // its index bit
    if (tid < a.a + a.h) {
        const uint32_t bit = tid < a.a ? tid : a.hi[tid - a.a];
        src_bit[tid] = 1u << tile_pos(a.pi[bit]);
        out_bit[tid] = 1ull << bit;
    }
    __syncthreads();
    // element k = e THREADS + tid of a tile: its offset in the state and the place (in the
    // partner's buffer) it comes from are sums of a part of tid and a part of e
    constexpr uint32_t E = (1u << (sizeof(R) == 4 ? SWAP_TILE : SWAP_TILE - 1)) / THREADS;
    auto place = [&](uint32_t k, uint32_t &from, uint32_t &to, unsigned long long &off) {
        uint32_t s = 0;
        off = 0;
        for (uint32_t p = 0; p < a.a + a.h; ++p)
            if ((k >> p) & 1u) {
                s |= src_bit[p];
                off |= out_bit[p];
            }
        from = (s >> a.a) * pitch + (s & (cols - 1u));
        to = (k >> a.a) * pitch + (k & (cols - 1u));
    };
    __shared__ uint32_t from_e[E], to_e[E];
    __shared__ unsigned long long off_e[E];
    uint32_t from_t, to_t;
    unsigned long long off_t;
    place(tid < size ? tid : 0u, from_t, to_t, off_t);
    if (tid < E) {
        uint32_t f, t;
        unsigned long long o;
        place(tid * THREADS < size ? tid * THREADS : 0u, f, t, o);
        from_e[tid] = f;
        to_e[tid] = t;
        off_e[tid] = o;
    }
    __syncthreads();
    svk::pass_wait();
    C *psi = reinterpret_cast<C *>(a.psi);
    const uint32_t nrest = a.n - a.a - a.h, lane = tid & 31u;        // at most 29
    const unsigned long long my_base = lane < nrest ? 1ull << a.rest[lane] : 0ull;
    const unsigned long long my_other = lane < nrest ? 1ull << a.pi[a.rest[lane]] : 0ull;
    for (unsigned long long t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        // lane j places bit j of the tile number
        const bool on = lane < nrest && ((t >> lane) & 1ull);
        const unsigned long long b0 = on ? my_base : 0ull, o0 = on ? my_other : 0ull;
        const unsigned long long base = (unsigned long long)__reduce_or_sync(0xffffffffu, (uint32_t)(b0 >> 32)) << 32 |
                                        __reduce_or_sync(0xffffffffu, (uint32_t)b0);
        const unsigned long long other = (unsigned long long)__reduce_or_sync(0xffffffffu, (uint32_t)(o0 >> 32)) << 32 |
                                         __reduce_or_sync(0xffffffffu, (uint32_t)o0);
        if (other < base) continue;                      // the partner's turn does both
        const bool two = other != base;
        __syncthreads();                                 // the buffers are free
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            if (half == 1 && !two) break;
            const C *src = psi + (half ? other : base) + off_t;
            C v[E];
#pragma unroll
            for (uint32_t e = 0; e < E; ++e)
                if (e * THREADS + tid < size) v[e] = src[off_e[e]];
#pragma unroll
            for (uint32_t e = 0; e < E; ++e)
                if (e * THREADS + tid < size) buf[half][to_t + to_e[e]] = v[e];
        }
        __syncthreads();
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            if (half == 1 && !two) break;
            C *dst = psi + (half ? other : base) + off_t;
            const C *in = buf[two ? 1 - half : 0] + from_t;
#pragma unroll
            for (uint32_t e = 0; e < E; ++e)
                if (e * THREADS + tid < size) dst[off_e[e]] = in[from_e[e]];
        }
    }
}

}  // namespace svr

namespace svi {

namespace {

// A run moves the state once: 0.64 ms on 28 qubits in complex64, against 0.33-0.37 ms for a
// gate that touches half of it, so it pays from a touched share of 1.25 on.  complex128 with two
// tables per tile takes two products per amplitude on the FP64 pipe, against one per touched
// amplitude: from 2.25 on.
constexpr double ONE_PRODUCT = 1.25;
double two_products(const sv_state *s) { return s->dtype == SV_C128 ? 2.25 : 1.25; }

// A diagonal run is two launches, so below 20 qubits, where launches are what counts, two gates stay
// two passes (two rotations on 15 qubits: 15.0 us, 18.4 as a run; complex128, inside the low bits, 19.4
// and 22.7; on 20 qubits 19.0 and 18.4, 31 and 28).  Three gates: 17 us and 19 alone, the same in a
// longer circuit; complex128 with two tables per tile 24 and 28, four gates 28 either way.
size_t least_gates(const sv_state *s, bool two) {
    return s->n >= 20 ? 2 : two && s->dtype == SV_C128 ? 4 : 3;
}

// Is the gate a permutation of its index bits?  Then out bit j of its targets comes from target
// perm[j]: U |c> = |r> with bit perm[j] of r equal to bit j of c.
bool bit_permutation(const Gate &g, uint32_t (&perm)[SV_MAX_K]) {
    const uint32_t D = 1u << g.k;
    for (uint32_t c = 0; c < D; ++c) {
        uint32_t hits = 0, row = 0;
        for (uint32_t r = 0; r < D; ++r) {
            const cplx u = g.u[(size_t)r * D + c];
            if (u == cplx(0.0, 0.0)) continue;
            if (u != cplx(1.0, 0.0)) return false;
            row = r;
            ++hits;
        }
        if (hits != 1) return false;
        if (c == 0 && row != 0) return false;
        if ((c & (c - 1)) == 0 && c) {                  // a single bit must go to a single bit
            if (row & (row - 1)) return false;
            perm[__builtin_ctz(c)] = (uint32_t)__builtin_ctz(row);
        } else if (c) {                                 // the others follow from those
            uint32_t want = 0;
            for (uint32_t j = 0; j < g.k; ++j)
                if ((c >> j) & 1u) want |= 1u << perm[j];
            if (row != want) return false;
        }
    }
    return true;
}

struct Table {
    uint64_t qubits = 0;
    std::vector<uint32_t> gates;        // positions in the run
};

// The merged tables of a run and the bins of their low qubits; false if they do not fit.
struct DiagPlan {
    uint32_t T;
    std::vector<Table> tabs;
    uint64_t bin[2] = {0, 0};

    bool pack() {
        const uint64_t low = (1ull << T) - 1;
        std::vector<uint64_t> comp;                     // connected sets of low qubits
        for (const Table &t : tabs) {
            uint64_t m = t.qubits & low;
            if (!m) continue;
            for (size_t i = 0; i < comp.size();) {
                if (comp[i] & m) {
                    m |= comp[i];
                    comp.erase(comp.begin() + i);
                } else {
                    ++i;
                }
            }
            comp.push_back(m);
        }
        std::sort(comp.begin(), comp.end(), [](uint64_t a, uint64_t b) {
            return __builtin_popcountll(a) != __builtin_popcountll(b)
                       ? __builtin_popcountll(a) > __builtin_popcountll(b) : a < b;
        });
        bin[0] = bin[1] = 0;
        for (uint64_t m : comp) {
            const int c = __builtin_popcountll(bin[0]) <= __builtin_popcountll(bin[1]) ? 0 : 1;
            const int b = __builtin_popcountll(bin[c] | m) <= (int)svr::BIN_Q ? c : 1 - c;
            if (__builtin_popcountll(bin[b] | m) > (int)svr::BIN_Q) return false;
            bin[b] |= m;
        }
        return true;
    }
    // Add gate number i with these qubits; false (and unchanged) if the run is full.
    bool add(uint32_t i, uint64_t q) {
        const uint64_t low = (1ull << T) - 1;
        Table *best = nullptr;
        for (Table &t : tabs) {
            if ((t.qubits & low) != (q & low) || __builtin_popcountll(t.qubits | q) > (int)svr::TAB_Q) continue;
            if (!best || __builtin_popcountll(t.qubits | q) - __builtin_popcountll(t.qubits) <
                             __builtin_popcountll(best->qubits | q) - __builtin_popcountll(best->qubits))
                best = &t;
        }
        if (!best) {
            if (tabs.size() == svr::MAX_TABS) return false;
            tabs.push_back(Table());
            best = &tabs.back();
        }
        const uint64_t before = best->qubits;
        if (before && (before | q) == before) {              // nothing new to pack
            best->gates.push_back(i);
            return true;
        }
        best->qubits |= q;
        best->gates.push_back(i);
        if (pack()) return true;
        best->gates.pop_back();
        best->qubits = before;
        if (!before) tabs.pop_back();
        pack();
        return false;
    }
};

// The factors of a run are multiplied before they meet an amplitude, so the product of any of them
// has to stay inside FP32: a run ends before a gate with which the largest or the smallest nonzero
// product could pass 2^+-64 (gate by gate, 0 times 1e20 twice is 0; times their product, NaN).
// Unitary gates never come near.
struct Range {
    double hi = 1.0, lo = 1.0;
    bool add(const Gate &g) {
        const uint32_t D = 1u << g.k;
        double h = 1.0, l = 1.0;
        for (uint32_t r = 0; r < D; ++r) {
            const cplx z = g.u[(size_t)r * D + r];
            const double m = std::max(std::fabs(z.real()), std::fabs(z.imag()));
            if (!(m <= 0x1p64) || !(std::fabs(z.real()) <= m) || !(std::fabs(z.imag()) <= m)) return false;   // NaN too
            h = std::max(h, m);
            if (m > 0.0) l = std::min(l, m);
        }
        if (!(hi * h <= 0x1p64) || !(lo * l >= 0x1p-64)) return false;
        hi *= h;
        lo *= l;
        return true;
    }
};

uint64_t qubit_mask(const Gate &g) {
    uint64_t m = 0;
    for (uint32_t j = 0; j < g.k; ++j) m |= 1ull << g.t[j];
    return m;
}

// The gates' entries into the arguments; the caller places them in tables.
void fill_entries(svr::TablesArgs &ta, const std::vector<Gate> &gates, size_t begin, size_t end) {
    ta.ngates = (uint32_t)(end - begin);
    uint32_t used = 0;
    for (uint32_t g = 0; g < ta.ngates; ++g) {
        const Gate &gg = gates[begin + g];
        const uint32_t D = 1u << gg.k;
        ta.k[g] = (uint8_t)gg.k;
        ta.first[g] = used;
        for (uint32_t r = 0; r < D; ++r) {
            const cplx z = gg.u[(size_t)r * D + r];
            ta.d[used++] = make_double2(z.real(), z.imag());
        }
    }
}

// All qubits of gates [begin, end) lie below the tile bits T.
template <typename R>
sv_status launch_low_run(sv_state *s, const std::vector<Gate> &gates, size_t begin, size_t end) {
    using namespace svr;
    constexpr uint32_t T = tile_bits<R>();
    TablesArgs ta;
    fill_entries(ta, gates, begin, end);
    ta.ntabs = 1;
    ta.nq[0] = T;
    ta.lg = T;
    for (uint32_t g = 0; g < ta.ngates; ++g) {
        ta.tab[g] = 0;
        for (uint32_t j = 0; j < ta.k[g]; ++j) ta.pos[g][j] = (uint8_t)gates[begin + g].t[j];
    }
    ta.out = s->ws + WS_TOPK;
    SV_CUDA(svk::launch_pass(diag_tables<R>, dim3(1, (1u << T) / 64), 64, 0, s->stream, ta));
    const unsigned long long ntiles = 1ull << (s->n - T);
    const unsigned grid = (unsigned)std::min<unsigned long long>(ntiles, 2ull * s->num_sms);
    SV_CUDA(svk::launch_pass(apply_low_run<R>, dim3(grid), THREADS, 0, s->stream, s->buf, (const void *)ta.out, ntiles));
    return SV_OK;
}

template <typename R>
sv_status launch_diag_run(sv_state *s, const std::vector<Gate> &gates, size_t begin, size_t end,
                          const DiagPlan &plan) {
    using namespace svr;
    using C = typename Cx<R>::T;
    TablesArgs ta;
    DiagRunArgs a;
    fill_entries(ta, gates, begin, end);
    ta.ntabs = a.ntabs = (uint32_t)plan.tabs.size();
    ta.lg = TAB_Q;
    for (uint32_t b = 0; b < 2; ++b) {
        a.nbin[b] = 0;
        for (uint32_t q = 0; q < plan.T; ++q)
            if ((plan.bin[b] >> q) & 1ull) a.bit_of[b][a.nbin[b]++] = (uint8_t)q;
    }
    const uint64_t low = (1ull << plan.T) - 1;
    for (uint32_t t = 0; t < a.ntabs; ++t) {
        const Table &tb = plan.tabs[t];
        uint32_t nq = 0;
        for (uint32_t q = 0; q < s->n; ++q)
            if ((tb.qubits >> q) & 1ull) a.qubit[t][nq++] = (uint8_t)q;
        a.nq[t] = ta.nq[t] = (uint8_t)nq;
        const uint64_t m = tb.qubits & low;
        // tables without low qubits go to the bin with fewer entries
        a.bin[t] = (uint8_t)(m ? !(plan.bin[0] & m) : a.nbin[1] < a.nbin[0]);
        for (uint32_t g : tb.gates) {
            ta.tab[g] = (uint8_t)t;
            for (uint32_t j = 0; j < ta.k[g]; ++j)
                for (uint32_t p = 0; p < nq; ++p)
                    if (a.qubit[t][p] == gates[begin + g].t[j]) ta.pos[g][j] = (uint8_t)p;
        }
    }
    ta.out = s->ws + WS_TOPK;
    a.tabs = ta.out;
    a.psi = s->buf;
    a.ntiles = 1ull << (s->n - plan.T);
    SV_CUDA(svk::launch_pass(diag_tables<R>, dim3(ta.ntabs), 1u << TAB_Q, 0, s->stream, ta));
    const size_t smem = ((size_t)a.ntabs << TAB_Q) * sizeof(C) + (2u << BIN_Q) * sizeof(C) + ((size_t)a.ntabs << BIN_Q) * 2;
    static svk::PerDevice<cudaError_t> setup;
    SV_CUDA(setup.get(svk::current_device(), [] {
        return cudaFuncSetAttribute(apply_diag_run<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(((size_t)MAX_TABS << TAB_Q) * sizeof(C) + (2u << BIN_Q) * sizeof(C) +
                                          ((size_t)MAX_TABS << BIN_Q) * 2));
    }));
    const unsigned grid = (unsigned)std::min<unsigned long long>(a.ntiles, 3ull * s->num_sms);
    SV_CUDA(svk::launch_pass(apply_diag_run<R>, dim3(grid), THREADS, smem, s->stream, a));
    return SV_OK;
}

template <typename R>
sv_status launch_swap_run(sv_state *s, const uint8_t (&pi)[SV_MAX_QUBITS]) {
    using namespace svr;
    using C = typename Cx<R>::T;
    const uint32_t most = sizeof(R) == 4 ? SWAP_TILE : SWAP_TILE - 1;
    SwapArgs a;
    a.psi = s->buf;
    a.n = s->n;
    a.a = sizeof(R) == 4 ? 6 : 5;           // rows of 512 bytes
    uint64_t tile = (1ull << a.a) - 1;
    for (uint32_t q = 0; q < a.a; ++q) tile |= 1ull << pi[q];
    // more bits, closed under the permutation
    for (uint32_t q = 0; q < s->n; ++q) {
        const uint64_t m = tile | 1ull << q | 1ull << pi[q];
        if (__builtin_popcountll(m) <= (int)most) tile = m;
    }
    a.h = 0;
    uint32_t nr = 0;
    for (uint32_t q = 0; q < SV_MAX_QUBITS; ++q) a.pi[q] = pi[q];
    for (uint32_t q = a.a; q < s->n; ++q) {
        if ((tile >> q) & 1ull) a.hi[a.h++] = (uint8_t)q;
        else a.rest[nr++] = (uint8_t)q;
    }
    a.ntiles = 1ull << nr;
    const size_t smem = 2 * sizeof(C) * (size_t)((1u << a.h) * ((1u << a.a) + 1u));
    static svk::PerDevice<cudaError_t> setup;
    SV_CUDA(setup.get(svk::current_device(), [] {
        return cudaFuncSetAttribute(apply_swap_run<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, 72 * 1024);
    }));
    // an odd stride: which of a pair of tiles does the work depends on the tile number's low
    // bits first, and an even stride gave half of the blocks three quarters of it (1.45 -> 0.94 ms,
    // and 0.84 with a tile's place formed by the lanes together)
    const unsigned grid = (unsigned)std::min<unsigned long long>(a.ntiles, (3ull * s->num_sms - 1) | 1ull);
    SV_CUDA(svk::launch_pass(apply_swap_run<R>, dim3(grid), THREADS, smem, s->stream, a));
    return SV_OK;
}

}  // namespace

size_t launch_run(sv_state *s, const std::vector<Gate> &gates, const Structure *st, const double *touched,
                  size_t begin, size_t end, size_t *tried, sv_status *status) {
    auto share = [&](size_t upto) { return touched[upto - begin] - touched[0]; };       // of gates begin .. upto - 1
    *status = SV_OK;
    *tried = 0;
    const uint32_t T = s->dtype == SV_C64 ? svr::tile_bits<float>() : svr::tile_bits<double>();
    if (s->n < T) return 0;
    const uint32_t kind = st[0].kind;
    if (kind == SV_STRUCT_DIAGONAL) {
        end = std::min(end, begin + svr::MAX_GATES);
        if (end - begin < least_gates(s, false) || share(end) < ONE_PRODUCT) return 0;     // not even all of them
        // the longer of a run inside the low bits and one with tables per tile
        size_t low_end = begin, i = begin;
        Range low_range, range;
        while (low_end < end && !(qubit_mask(gates[low_end]) >> T) && low_range.add(gates[low_end])) ++low_end;
        const bool low = low_end - begin >= least_gates(s, false) && share(low_end) >= ONE_PRODUCT;
        if (!low && share(end) < two_products(s)) return 0;
        DiagPlan plan;
        plan.T = T;
        while (i < end && range.add(gates[i]) && plan.add((uint32_t)(i - begin), qubit_mask(gates[i]))) ++i;
        *tried = std::max(i, low_end) - begin;
        if (low && low_end >= i) {
            *status = s->dtype == SV_C64 ? launch_low_run<float>(s, gates, begin, low_end)
                                         : launch_low_run<double>(s, gates, begin, low_end);
            return low_end - begin;
        }
        if (i - begin < least_gates(s, true) || share(i) < two_products(s)) return 0;
        *status = s->dtype == SV_C64 ? launch_diag_run<float>(s, gates, begin, i, plan)
                                     : launch_diag_run<double>(s, gates, begin, i, plan);
        return i - begin;
    }
    if (kind == SV_STRUCT_MONOMIAL) {
        // the product of the run's bit permutations, as long as it only swaps pairs
        uint8_t pi[SV_MAX_QUBITS], good[SV_MAX_QUBITS];
        for (uint32_t q = 0; q < SV_MAX_QUBITS; ++q) pi[q] = (uint8_t)q;
        std::memcpy(good, pi, sizeof(pi));
        size_t i = begin, upto = begin;
        uint32_t perm[SV_MAX_K];
        for (; i < end && bit_permutation(gates[i], perm); ++i) {
            const Gate &g = gates[i];
            uint8_t to[SV_MAX_QUBITS];
            for (uint32_t q = 0; q < SV_MAX_QUBITS; ++q) to[q] = (uint8_t)q;
            for (uint32_t j = 0; j < g.k; ++j) to[g.t[j]] = (uint8_t)g.t[perm[j]];
            for (uint32_t q = 0; q < SV_MAX_QUBITS; ++q) pi[q] = to[pi[q]];   // this gate after the others
            bool pairs = true;
            for (uint32_t q = 0; q < SV_MAX_QUBITS; ++q) pairs = pairs && pi[pi[q]] == q;
            if (pairs) {
                upto = i + 1;
                std::memcpy(good, pi, sizeof(pi));
            }
        }
        *tried = i - begin;
        // one launch, like a pass: from the same share on at every size
        if (upto - begin < 2 || share(upto) < ONE_PRODUCT) return 0;
        *status = s->dtype == SV_C64 ? launch_swap_run<float>(s, good) : launch_swap_run<double>(s, good);
        return upto - begin;
    }
    return 0;
}

}  // namespace svi
