// Fused k = 4, 5 gates in complex64 on the 5th-generation tensor cores (tcgen05).
//
// Per group of 2^k amplitudes the update v' = U v (Eq. 3 with k targets) is a real
// dense contraction: with amplitudes interleaved (re, im), v' = R v where R is the
// 2^{k+1} x 2^{k+1} real embedding of U
//     R[2j][2l] = Re U[j][l],  R[2j][2l+1] = -Im U[j][l],
//     R[2j+1][2l] = Im U[j][l], R[2j+1][2l+1] = Re U[j][l].
// A tile of 128 groups is the GEMM D[128 x N] = A[128 x K] B[N x K]^T with A = the
// groups' amplitudes, B = R and N = K = 2^{k+1} (64 for k = 5, 32 for k = 4).
//
// Precision: the tensor cores' FP32 accumulation truncates, so a plain split of the
// FP32 operands into TF32 parts gives errors biased toward zero (a measurable loss of
// norm per pass).  Instead each operand is cut into three 9-bit integer slices on a
// fixed-point grid -- per row of A (scale 2^{8-e}, e = exponent of the row's largest
// component) and for all of B -- so that x = (a1 + a2 2^-9 + a3 2^-18) / s.  The
// slices at their scale (a2 2^-9, a3 2^-18) are exact in FP16 and every product of slices is
// an integer below 2^16 times a power of two, so
//     D0  = A1 B1                                      (below 2^22: exact in FP32)
//     D12 = A1 B2 + A2 B1 + A1 B3 + A2 B2 + A3 B1
// are accumulated by the tensor cores (kind::f16, FP32 accumulators in TMEM).  D0, which
// carries the leading 2^22 of the result, is exact; D12 sits 2^-9 below it, so the
// truncation of its accumulation costs about 2^-31 of the output per step -- the error
// stays unbiased to well below FP32 rounding.  The epilogue forms
// out = (D0 + D12) / (s s_B) with round-to-nearest (the dropped slice products are
// below 2^-27 of the row's largest amplitude).  With every slice at its own scale no scaled
// copies are needed (three slices of each operand, 20 MMA instructions per 128 groups instead of
// 24), and the slices are cut by magic-number rounding in packed FP32x2 instructions (tc.cuh)
// instead of six conversions per amplitude on the conversion pipe, which bound the transform:
// a 20-qubit pass 8.7 -> 7.8 us, 24 qubits 53 -> 47, 28 qubits 675 -> 670 (92 -> 94% of the copy
// rate), a batched pass of 18 qubits x 96 states 86 -> 75.
//
// One persistent CTA per SM, warp-specialised, every hand-off an mbarrier:
//   warp 8               TMA producer: lane i issues the load of segment i of each tile
//                        into a ring of NS raw stages (a 1-D bulk copy, or 2-D tensor-map
//                        boxes of 128-byte rows with the 128-byte swizzle, SW);
//   warps 0-7            transform: two warps per TMEM lane quadrant, one group (row of A)
//                        and half of its members per thread -- gather from the raw stage,
//                        cut into three 9-bit slices and write them into tensor memory
//                        with tcgen05.st (the thread's own TMEM lane);
//   warp 9 (one thread)  MMA issuer: 5 x K/16 tcgen05.mma.kind::f16, A from TMEM and B
//                        from shared memory, into two TMEM accumulators
//                        (double-buffered), committed to mbarriers;
//   warps 10-17          epilogue: two warps per quadrant, tcgen05.ld of half the columns,
//                        combine, scatter into an output staging tile;
//   warp 18              issues the staging tiles' TMA bulk stores.
// The epilogue warps never meet: they hand accumulators and staging tiles on by counted mbarrier
// arrivals (an epilogue barrier and stores by one of its warps cost a batched pass of 18 qubits x
// 96 states 4%, 75 -> 71 us).  The transform warps meet three times per tile; letting them meet
// in pairs instead measured the same within 1% (faster on 24-qubit states, slower on 28).
// Targets among tile bits 0..3 (where 8-byte accesses pick their bank) would make the
// lanes of a warp hit one bank.  Width-5 launches on states of 13 qubits or more, and
// batched launches, avoid that with the swizzled staging (SW); the others take each group's
// members in a lane-dependent XOR order (XP), undone in registers.  The others are width 4 on 11
// qubits (K = 4) and widths 4 and 5 on 12; circuits on such states run in apply_small.cu, so only
// single gates, the server's requests and passes that a policy flag asks for come here.
// So loads, slicing, MMAs and stores of consecutive tiles overlap.  With A in tensor
// memory, shared memory holds only B, the raw stages and the output staging: four tiles (k = 5) or
// eight (k = 4), of which two loads are in flight except where launch_tc_t says more.  Every wait is bounded and any
// role that gives up makes the others leave too (abort flag).
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "plan.h"
#include "ptx.cuh"
#include "sv_internal.h"
#include "tc.cuh"

namespace svk {

// One tile is one MMA (128 groups).  BT: a batched launch over many states with their own matrices (see apply_tc): two B
// sets (the current state's and the next one's).
template <int K, bool BT = false>
struct TcShape {
    static constexpr uint32_t D = 1u << K;            // amplitudes per group
    static constexpr uint32_t KD = 2u * D;            // real K = N
    static constexpr uint32_t ROWS = 128;             // groups per tile (MMA M)
    static constexpr uint32_t TB = K + 7;             // tile bits
    static constexpr uint32_t TILE_BYTES = ROWS * D * 8u;
    static constexpr uint32_t B_BYTES = KD * KD * 2u;     // one FP16 slice of B
    static constexpr uint32_t NB = 3;                     // B1, B2 2^-9, B3 2^-18
    static constexpr uint32_t SBO = (KD / 8u) * 128u;     // 8-row group stride of B
    static constexpr uint32_t NS = BT ? 3u : (K == 5 ? 4u : 8u);   // raw stages
    static constexpr uint32_t NOUT = 2u;              // output staging tiles
    static constexpr uint32_t ACC = 2u * KD;              // TMEM columns of one D set (D0, D12)
    static constexpr uint32_t A_COLS = KD / 2u;           // TMEM columns of one A slice
    static constexpr uint32_t NA = 3;                     // A1, A2 2^-9, A3 2^-18
    static constexpr uint32_t A_SET = NA * A_COLS;        // one A buffer
    static constexpr uint32_t A_COL0 = 2u * ACC;          // first column of the A buffers
    static constexpr uint32_t TMEM_COLS = K == 5 ? 512u : 256u;
    static_assert(A_COL0 + 2u * A_SET <= TMEM_COLS, "TMEM layout");
    static constexpr uint32_t NBSET = BT ? 2u : 1u;       // B sets
    static constexpr uint32_t B_SET = NB * B_BYTES;
    static constexpr uint32_t OFF_RAW = NBSET * B_SET;
    static constexpr uint32_t OFF_OUT = OFF_RAW + NS * TILE_BYTES;
    static constexpr uint32_t SMEM = OFF_OUT + NOUT * TILE_BYTES;
    static constexpr uint32_t THREADS = 608;              // 19 warps
    // warps 0-7 transform, 8 TMA producer, 9 MMA issuer, 10-17 epilogue, 18 TMA stores
    static constexpr uint32_t W_PROD = 8, W_MMA = 9, W_EPI = 10, W_STORE = 18;
    static constexpr uint32_t HALF = D / 2;               // group members per worker thread
};

template <int K>
struct TcArgs {
    // swizzled launches (SW): the state as a 2-D tensor of 128-byte rows (32 floats), boxes
    // of box_rows rows, `boxes` boxes per segment, 128-byte swizzle in shared memory
    CUtensorMap tmap;                      // 128-byte aligned by its type
    // U on a fixed-point grid: entry (r, c) = (bx[..].x + i bx[..].y) 2^-18 b_inv_scale, row-major;
    // |bx| <= 2^26.  The prologue cuts each into three 9-bit slices (cut_b).
    alignas(16) int2 bx[(1u << K) * (1u << K)];
    uint32_t box_rows, boxes;
    uint32_t depth;                        // tile loads in flight, 1 .. NS
    float b_inv_scale;
    void *psi;
    int *err;
    unsigned long long ntiles;
    uint32_t L, h;
    uint32_t hi[SV_MAX_K];
    uint32_t lp[K];
    // bank-conflict avoidance: the xt lowest targets sit at tile bits below 4; lane l
    // takes group members in the order c ^ x(l), x(l) = (l >> xs) & (2^xt - 1)
    uint32_t xs, xt;
    // batched launches: ntiles = states x 2^tps tiles, state i at amplitude offset
    // i 2^n; state i's operand (the B set as it lies in shared memory) is images + i B_SET, its
    // scale bscale[i] (pack_images)
    const unsigned char *images;
    const float *bscale;
    uint32_t tps;                  // log2 of tiles_per_state
    uint32_t n;
};

// v[c] <- v[c ^ x] for the low xt bits of x: one conditional-swap stage per bit.
template <int N>
__device__ __forceinline__ void xor_unpermute(float2 (&v)[N], uint32_t x, uint32_t xt) {
    constexpr int NBITS = N >= 16 ? 4 : (N >= 8 ? 3 : (N >= 4 ? 2 : 1));
#pragma unroll
    for (int j = 0; j < NBITS; ++j) {
        if (xt > (uint32_t)j) {                       // uniform over the launch
            const bool f = (x >> j) & 1u;
#pragma unroll
            for (int c = 0; c < N; ++c) {
                if (c & (1 << j)) continue;
                const float2 lo = v[c], hi = v[c | (1 << j)];
                v[c] = make_float2(f ? hi.x : lo.x, f ? hi.y : lo.y);
                v[c | (1 << j)] = make_float2(f ? lo.x : hi.x, f ? lo.y : hi.y);
            }
        }
    }
}

// Three 9-bit slices of a fixed-point entry, x = b1 2^18 + b2 2^9 + b3, |b1|, |b2|, |b3| <= 256.
__device__ __forceinline__ void cut_b(int x, float &b1, float &b2, float &b3) {
    const int i1 = (x + (1 << 17)) >> 18;
    x -= i1 << 18;
    const int i2 = (x + (1 << 8)) >> 9;
    b1 = (float)i1;
    b2 = (float)i2;
    b3 = (float)(x - (i2 << 9));
}

// B = the FP16 slices (B1, B2 2^-9, B3 2^-18) of R, from the fixed-point entries in the
// kernel's parameters: complex entry (r, c) fills R's rows 2r (re, -im) and 2r + 1 (im, re) at
// columns 2c, 2c + 1, one FP16 pair each.  Entries i0, i0 + stride, ... two at a time.
// Why here and in this form: the operand used to travel as three int16 copies of all of R
// (24 KiB of parameters) read entry by entry, i.e. as constant-bank loads that serialise over
// a warp's 16 different words and miss line by line.  That was most of a launch on a small
// state: a 20-qubit pass took 25.0 us (12 qubits: 21.0) and takes 11.1 (7.8) with 8 KiB of
// parameters, 16-byte generic loads and the first tiles already in flight meanwhile; a
// 28-qubit pass 693 -> 678 us.
template <int K>
__device__ __forceinline__ void expand_b(unsigned char *sB, const int2 *bx, uint32_t b_bytes, uint32_t sbo,
                                         uint32_t i0, uint32_t stride) {
    for (uint32_t e = 2u * i0; e < (1u << (2 * K)); e += 2u * stride) {
        const int4 v = ld_param16(bx + e);
        const uint32_t r = e >> K, c = e & ((1u << K) - 1u);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            float re[3], im[3];
            cut_b(q ? v.z : v.x, re[0], re[1], re[2]);
            cut_b(q ? v.w : v.y, im[0], im[1], im[2]);
            const uint32_t o0 = kmajor_off16(2u * r, 2u * (c + q), sbo);
            const uint32_t o1 = kmajor_off16(2u * r + 1u, 2u * (c + q), sbo);
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                const float f = s == 0 ? 1.f : s == 1 ? 1.f / 512.f : 1.f / 262144.f;   // exact: 9-bit integers
                *reinterpret_cast<uint32_t *>(sB + s * b_bytes + o0) = pack_h2(re[s] * f, -im[s] * f);
                *reinterpret_cast<uint32_t *>(sB + s * b_bytes + o1) = pack_h2(im[s] * f, re[s] * f);
            }
        }
    }
}

// sb = 2^(8 - eb) and 1 / sb for a matrix whose largest |entry| is m < 2^eb.
__device__ __forceinline__ void b_grid(float m, float &sb, float &inv) {
    int eb = 0;
    frexpf(m, &eb);
    eb = max(eb, -100);
    sb = ldexpf(1.f, 8 - eb);
    inv = ldexpf(1.f, eb - 8);
}

// Operands of batched launches.  Every (gate, state) of a batch has its own matrix; pack_images
// cuts them into B sets in global memory, laid out as in shared memory, before the passes, and a
// pass then loads a state's set with one bulk copy.  (Built inside the pass by its producer
// warp, a set cost about 20 us of stalled loads whenever a CTA met a new state: 18 qubits x 96
// states 115 us per pass -> 86.)
struct PackGate {
    unsigned long long tab;          // offset of the gate's FP32 matrices in the table (bytes)
    unsigned long long image;        // and of its images in units of B sets
    uint32_t kin;
    uint32_t idm;                    // identity bits of the width-5 gate it is widened to
    uint8_t pos[SV_MAX_K];           // its local bits' places there
};
constexpr uint32_t PACK_GATES = 64;
struct PackArgs {
    const unsigned char *utab;       // matrices of the first state
    unsigned char *images;
    float *bscale;
    PackGate g[PACK_GATES];
};

// One block per (state, gate).  R is the real embedding of the widened U times sb, so |R sb| <
// 256 and the three 9-bit slices of the FP32 values are exact.  A thread writes 16-byte chunks of
// the slices B1, B2 2^-9, B3 2^-18: eight columns of one row.
__global__ void __launch_bounds__(256) pack_images(const __grid_constant__ PackArgs a) {
    using S = TcShape<5, true>;
    __shared__ float red[8];
    const uint32_t tid = threadIdx.x;
    const PackGate &g = a.g[blockIdx.y];
    const uint32_t kin = g.kin, size = 2u << (2u * kin);
    pass_trigger();
    pass_wait();
    const float *U = reinterpret_cast<const float *>(a.utab + g.tab) + (size_t)blockIdx.x * size;
    float m = 0.f;
    for (uint32_t i = tid; i < size; i += 256) m = fmaxf(m, fabsf(U[i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31u) == 0) red[tid >> 5] = m;
    __syncthreads();
    m = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) m = fmaxf(m, red[w]);
    float sb, inv;
    b_grid(m, sb, inv);
    const unsigned long long at = g.image + blockIdx.x;
    if (tid == 0) a.bscale[at] = inv;
    unsigned char *img = a.images + at * S::B_SET;
    auto local = [&](uint32_t x) {                       // the gate's own local index of x
        uint32_t l = 0;
        for (uint32_t j = 0; j < kin; ++j) l |= ((x >> g.pos[j]) & 1u) << j;
        return l;
    };
    for (uint32_t q = tid; q < S::B_BYTES / 16u; q += 256) {
        // the chunk's place (kmajor_off16): row n, columns kk .. kk + 7
        const uint32_t n = (q / (S::SBO / 16u)) * 8u + (q & 7u), kk = ((q >> 3) & 7u) * 8u;
        const uint32_t r = n >> 1, lr = local(r);
        uint32_t w[3][4];
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i) {
            const uint32_t c = (kk >> 1) + i;
            float2 u = make_float2(0.f, 0.f);
            if (!((r ^ c) & g.idm)) u = reinterpret_cast<const float2 *>(U)[(lr << kin) + local(c)];
            const float x[2] = {(n & 1u ? u.y : u.x) * sb, (n & 1u ? u.x : -u.y) * sb};
            slices(make_float2(x[0], x[1]), make_float2(1.f, 1.f), w[0][i], w[1][i], w[2][i]);
        }
#pragma unroll
        for (uint32_t s = 0; s < 3; ++s)
            *reinterpret_cast<uint4 *>(img + s * S::B_BYTES + q * 16u) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
    }
}

// XP: the launch has targets among tile bits 0..3 and takes members in the lane's XOR
// order; otherwise every lane takes them in member order (no permutation code at all).
// The pipelines count this CTA's tiles (j).
// BT: one launch over a batch of states, each with its own matrix: a CTA takes a
// contiguous range of tiles (so it meets few states), B is double-buffered and the producer
// loads the next state's set a few tiles into the current one (b_full: arrived; b_empty: the
// MMAs of the state that last used the set have completed).
// SW: tiles move by 2-D tensor-map copies that store them in shared memory with the
// 128-byte swizzle (16-byte chunk index XOR the 128-byte row within each 1 KiB), and the
// roles address the tile through the same swizzle.  A warp's lanes (consecutive groups)
// then reach different banks whatever the targets, so no lane-dependent member order is
// needed (XP = false).  The swizzle is linear
// over XOR, so it is applied to the group base and to the target bits once, and member
// offsets combine them by XOR.
// P0 (with SW): the targets include index bits 0-3, so members c and c + 1 are neighbours, also
// under the swizzle, and take 16-byte accesses: a group is then one or two whole 128-byte rows and the
// swizzle spreads a warp's lanes over few chunks (8-way conflicts in 8-byte accesses).  Targets
// 0-4: 28 qubits 848 -> 626 us per pass, 24 qubits 62.9 -> 46.1.  With only bit 0 or bits 0 and 1
// among the targets 8-byte accesses are as fast.
template <int K, bool XP, bool BT = false, bool SW = false, bool P0 = false>
__global__ void __launch_bounds__(608, 1) apply_tc(const __grid_constant__ TcArgs<K> a) {
    using S = TcShape<K, BT>;
    constexpr uint32_t KD = S::KD, NS = S::NS, NOUT = S::NOUT, HALF = S::HALF;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long full[NS], empty[NS];
    __shared__ __align__(8) unsigned long long a_full[2], a_empty[2], d_full[2], d_empty[2];
    __shared__ __align__(8) unsigned long long scale_full[4];   // row scales, tile j -> j & 3
    __shared__ float row_scale[4][128];
    __shared__ __align__(8) unsigned long long out_full[NOUT], out_free[NOUT];   // staging tiles
    __shared__ float max_part[2][128];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ __align__(8) unsigned long long b_full[2], b_empty[2];   // batched launches
    // B slices, the raw stages and the output staging tiles; B operand reads stay inside
    // the CTA's shared memory whatever the descriptor strides.
    unsigned char *sB = smem;
    float2 *psi = reinterpret_cast<float2 *>(a.psi);
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    const uint32_t seg_amps = 1u << a.L;
    const uint32_t seg_bytes = seg_amps * 8u;
    const uint32_t nseg = 1u << a.h;

    if (tid == 0) pass_trigger();
    if (warp == S::W_MMA) {
        tmem_alloc(smem_u32(&tmem_slot), S::TMEM_COLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (uint32_t s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&a_full[b]), 1);
            mbar_init(smem_u32(&a_empty[b]), 1);
            mbar_init(smem_u32(&d_full[b]), 1);
            mbar_init(smem_u32(&d_empty[b]), 8);      // the epilogue warps
        }
        for (int q = 0; q < 4; ++q) mbar_init(smem_u32(&scale_full[q]), 1);
        for (uint32_t o = 0; o < NOUT; ++o) {
            mbar_init(smem_u32(&out_full[o]), 8);
            mbar_init(smem_u32(&out_free[o]), 1);
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(smem_u32(&b_full[q]), 1);
            mbar_init(smem_u32(&b_empty[q]), 1);
        }
        abort_flag = 0;
        fence_mbar_init();
    }
    // tiles of this CTA: strided over the grid, or (batched) a contiguous range
    unsigned long long first = blockIdx.x, step = gridDim.x, tend = a.ntiles;
    if constexpr (BT) {
        const unsigned long long per = (a.ntiles + gridDim.x - 1) / gridDim.x;
        first = min(a.ntiles, (unsigned long long)blockIdx.x * per);
        tend = min(a.ntiles, first + per);
        step = 1;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (!BT && warp != S::W_PROD) {
        // every warp but the producer, which is already loading the first tiles
        const uint32_t i = tid < S::W_PROD * 32u ? tid : tid - 32u;
        expand_b<K>(sB, a.bx, S::B_BYTES, S::SBO, i, S::THREADS - 32u);
        fence_proxy_async_smem();
        named_bar(3, S::THREADS - 32u);
    }
    const uint32_t tmem = tmem_slot;
    volatile int *abort = &abort_flag;
    // amplitude offset of tile t (batched: the state's offset plus the tile's base)
    auto tile_base = [&](const SegLanes &sl, unsigned long long t) -> unsigned long long {
        if constexpr (BT) {
            const unsigned long long st = t >> a.tps;
            return (st << a.n) + sl.base(t - (st << a.tps));
        } else {
            return sl.base(t);
        }
    };

    auto group_base = [&](uint32_t row) {
        uint32_t g = row;
#pragma unroll
        for (int j = 0; j < K; ++j) g = insert_zero32(g, a.lp[j]);
        return SW ? swz128(g) : g;
    };
    // offset of group member c (bit j of c at tile bit lp[j]); for the unrolled constant
    // c this is an XOR of the (swizzled) bits 1 << lp[j] held in K registers, and a
    // member's index is group base XOR offset
    uint32_t tbit[K];
#pragma unroll
    for (int j = 0; j < K; ++j) tbit[j] = SW ? swz128(1u << a.lp[j]) : 1u << a.lp[j];
    auto member_off = [&](uint32_t c) {
        uint32_t o = 0;
#pragma unroll
        for (int j = 0; j < K; ++j)
            if ((c >> j) & 1u) o ^= tbit[j];
        return o;
    };

    if (warp == S::W_PROD) {
        // ------------------------------------------------------------ TMA producer
        // lane i issues the bulk copy of segment i of every tile
        SegLanes sl;
        sl.init(a.L, a.h, a.hi, lane);
        pass_wait();
        uint32_t j = 0;
        // batched: B sets are requested state by state, from the range's first one
        const unsigned long long st0 = BT ? first >> a.tps : 0;
        unsigned long long asked = st0;
        auto ask = [&]() -> bool {
            const uint32_t i = (uint32_t)(asked - st0), set = i & 1u, use = i >> 1;
            bool okb = true;
            if (lane == 0) {
                if (use >= 1) okb = mbar_wait_or_abort(smem_u32(&b_empty[set]), (use - 1u) & 1u, abort);
                if (okb) {
                    const uint32_t bar = smem_u32(&b_full[set]);
                    mbar_arrive_expect_tx(bar, S::B_SET);
                    bulk_g2s(smem_u32(sB + set * S::B_SET), a.images + asked * S::B_SET, S::B_SET, bar);
                }
            }
            ++asked;
            return __shfl_sync(0xffffffffu, (int)okb, 0) != 0;
        };
        for (unsigned long long t = first; t < tend; t += step, ++j) {
            if constexpr (BT) {
                const unsigned long long st = t >> a.tps, in = t - (st << a.tps);
                if (asked <= st && !ask()) break;
                // the next state's set, once the previous state's last MMAs must be done (its
                // tiles left the raw stages), or at the last tile of this one
                if (asked == st + 1 && (in >= 3 || in + 1 == 1ull << a.tps) && (asked << a.tps) < tend &&
                    !ask())
                    break;
            }
            const uint32_t s = j % NS, u = j / NS;
            bool ok = true;
            if (lane == 0) {
                ok = mbar_wait_or_abort(smem_u32(&empty[s]), (u & 1u) ^ 1u, abort);
                // at most `depth` tiles on their way (launch_tc_t)
                const uint32_t i = j - a.depth;
                if (ok && a.depth < NS && j >= a.depth) ok = mbar_wait_or_abort(smem_u32(&full[i % NS]), (i / NS) & 1u, abort);
            }
            if (!__shfl_sync(0xffffffffu, (int)ok, 0)) break;
            const uint32_t bar = smem_u32(&full[s]);
            if (lane == 0) mbar_arrive_expect_tx(bar, S::TILE_BYTES);
            __syncwarp();
            if (lane < nseg) {
                float2 *dst = reinterpret_cast<float2 *>(smem + S::OFF_RAW + s * S::TILE_BYTES);
                if constexpr (SW) {
                    // segment = `boxes` boxes of box_rows 128-byte rows (16 amplitudes each)
                    const int32_t row0 = (int32_t)((tile_base(sl, t) + sl.my_off) >> 4);
                    const uint32_t d0 = smem_u32(dst + (size_t)lane * seg_amps);
                    for (uint32_t bx = 0; bx < a.boxes; ++bx)
                        tma_load_2d(d0 + bx * a.box_rows * 128u, &a.tmap, 0, row0 + (int32_t)(bx * a.box_rows), bar);
                } else {
                    bulk_g2s(smem_u32(dst + (size_t)lane * seg_amps), psi + tile_base(sl, t) + sl.my_off,
                             seg_bytes, bar);
                }
            }
        }
    } else if (warp == S::W_MMA) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            const uint32_t idesc = idesc_f16(S::ROWS, KD), idesc2 = idesc_f16(S::ROWS, 2u * KD);
            uint32_t B0 = smem_u32(sB);
            const unsigned long long ntile = tend > first ? (tend - first + step - 1) / step : 0;
            unsigned long long cur = ~0ull;
            uint32_t nsw = 0;
            for (unsigned long long j = 0; j < ntile; ++j) {
                if constexpr (BT) {
                    const unsigned long long st = (first + j * step) >> a.tps;
                    if (st != cur) {
                        if (cur != ~0ull) {
                            mma_commit(smem_u32(&b_empty[nsw & 1u]));   // the old state's MMAs
                            ++nsw;
                        }
                        cur = st;
                        const uint32_t set = nsw & 1u, use = nsw >> 1;
                        if (!mbar_wait_or_abort(smem_u32(&b_full[set]), use & 1u, abort)) break;
                        tc_fence_after();
                        B0 = smem_u32(sB) + set * S::B_SET;
                    }
                }
                const uint32_t b = (uint32_t)j & 1u, u = (uint32_t)(j >> 1);
                if (!mbar_wait_or_abort(smem_u32(&a_full[b]), u & 1u, abort)) break;
                if (!mbar_wait_or_abort(smem_u32(&d_empty[b]), (u & 1u) ^ 1u, abort)) break;
                tc_fence_after();
                const uint32_t A0 = tmem + S::A_COL0 + b * S::A_SET;
                const uint32_t dset = tmem + b * S::ACC;
                // A1 [B1 B2] -> [D0 D12] (the accumulators and the slices are adjacent: N =
                // 2 KD), then A2 B1, A2 B2, A1 B3, A3 B1 -> D12
                const uint32_t prod[5][2] = {{0, 0}, {1, 0}, {1, 1}, {0, 2}, {2, 0}};
#pragma unroll
                for (int p = 0; p < 5; ++p) {
                    const uint32_t Aa = A0 + prod[p][0] * S::A_COLS;
                    const uint32_t Bb = B0 + prod[p][1] * S::B_BYTES;
#pragma unroll
                    for (uint32_t ks = 0; ks < KD / 16; ++ks)
                        mma_f16_tmem_a(p == 0 ? dset : dset + KD, Aa + ks * 8u,
                                       smem_desc(Bb + ks * 256u, 128u, S::SBO), p == 0 ? idesc2 : idesc,
                                       (p == 0 && ks == 0) ? 0u : 1u);
                }
                mma_commit(smem_u32(&a_empty[b]));
                mma_commit(smem_u32(&d_full[b]));
            }
        }
    } else if (warp < S::W_PROD) {
        // ------------------------------------------------------------ transform
        // Two warps per TMEM lane quadrant: warp w takes rows 32 (w & 3) .. + 31 of each
        // tile and group members HALF (w >> 2) .. + HALF - 1.
        const uint32_t row = (warp & 3u) * 32u + lane;
        const uint32_t part = warp >> 2;
        const uint32_t gbase = group_base(row);
        const uint32_t xl = (lane >> a.xs) & ((1u << a.xt) - 1u);
        uint32_t cx = 0;
#pragma unroll
        for (int q = 0; q < K; ++q)
            if ((xl >> q) & 1u) cx |= tbit[q];
        uint32_t j = 0;
        unsigned long long cur = ~0ull;
        float bsc = a.b_inv_scale;
        for (unsigned long long t = first; t < tend; t += step, ++j) {
            const uint32_t s = j % NS;
            const bool okf = mbar_wait_or_abort(smem_u32(&full[s]), (j / NS) & 1u, abort);
            if constexpr (BT) {
                const unsigned long long st = t >> a.tps;
                if (st != cur) bsc = __ldcg(a.bscale + st);       // after the first tile's arrival
                cur = st;
            }
            const float2 *rs = reinterpret_cast<const float2 *>(smem + S::OFF_RAW + s * S::TILE_BYTES);
            // this half of the row (members in the lane's order c ^ x), its largest component
            float2 v[HALF];
            float m = 0.f;
#pragma unroll
            for (uint32_t c = 0; c < HALF; c += P0 ? 2 : 1) {
                const uint32_t mo = member_off(part * HALF + c);
                if constexpr (P0) {
                    const float4 f = *reinterpret_cast<const float4 *>(rs + (gbase ^ mo));
                    v[c] = make_float2(f.x, f.y);
                    v[c + 1] = make_float2(f.z, f.w);
                    m = max_abs2(m, f.z, f.w);
                } else {
                    v[c] = rs[gbase ^ (XP ? (mo ^ cx) : mo)];
                }
                m = max_abs2(m, v[c].x, v[c].y);
            }
            max_part[part][row] = m;
            fence_proxy_async_smem();         // reads of the raw stage before its refill
            if (!named_bar_and(1, 256, okf)) break;
            if (tid == 0) mbar_arrive(smem_u32(&empty[s]));
            m = fmaxf(max_part[0][row], max_part[1][row]);
            int ex = 0;
            frexpf(m, &ex);                   // m < 2^ex (m = 0: ex = 0)
            ex = max(ex, -100);               // keep 2^(8-ex) finite
            const float sc = ldexpf(1.f, 8 - ex);      // |x * sc| < 256
            const float2 scale = make_float2(sc, sc);
            const uint32_t ab = j & 1u;
            const bool oka = mbar_wait_or_abort(smem_u32(&a_empty[ab]), ((j >> 1) & 1u) ^ 1u, abort);
            if (!named_bar_and(1, 256, oka)) break;
            tc_fence_after();
            // slot j & 3 was last read by the epilogue of tile j - 4, which finished
            // before the MMAs of tile j - 2 were issued, whose completion released
            // a_empty[ab]
            if (part == 0) row_scale[j & 3u][row] = ldexpf(bsc, ex - 8);
            if constexpr (XP) xor_unpermute(v, xl, a.xt);   // back in member order (x < HALF)
            // three 9-bit slices, one FP16 pair (re, im) per 32-bit TMEM column, stored
            // eight members at a time
            const uint32_t arow = tmem + S::A_COL0 + ab * S::A_SET + (((warp & 3u) * 32u) << 16) +
                                  part * HALF;
#pragma unroll
            for (uint32_t c0 = 0; c0 < HALF; c0 += 8) {
                uint32_t w1[8], w2[8], w3[8];
#pragma unroll
                for (uint32_t c = 0; c < 8; ++c) slices(v[c0 + c], scale, w1[c], w2[c], w3[c]);
                tmem_st8_async(arow + c0, w1);
                tmem_st8_async(arow + S::A_COLS + c0, w2);
                tmem_st8_async(arow + 2 * S::A_COLS + c0, w3);
            }
            tmem_wait_st();
            tc_fence_before();
            named_bar(1, 256);                // also: max_part is free for the next tile
            if (tid == 0) {
                mbar_arrive(smem_u32(&a_full[ab]));
                mbar_arrive(smem_u32(&scale_full[j & 3u]));
            }
        }
    } else if (warp < S::W_STORE) {
        // ------------------------------------------------------------ epilogue
        // Two warps per lane quadrant, each over half of the accumulator columns.
        const uint32_t quad = warp & 3u;          // TMEM lanes 32*quad .. 32*quad+31
        const uint32_t row = quad * 32u + lane;
        const uint32_t part = (warp - S::W_EPI) >> 2;
        const uint32_t gbase = group_base(row);
        const uint32_t xl = (lane >> a.xs) & ((1u << a.xt) - 1u);
        uint32_t cx = 0;
#pragma unroll
        for (int q = 0; q < K; ++q)
            if ((xl >> q) & 1u) cx |= tbit[q];
        uint32_t j = 0;
        bool ok = true;
        for (unsigned long long t = first; t < tend && ok; t += step, ++j) {
            const uint32_t ob = j % NOUT;
            float2 *out = reinterpret_cast<float2 *>(smem + S::OFF_OUT + ob * S::TILE_BYTES);
            const uint32_t b = j & 1u;
            ok = ok && mbar_wait_or_abort(smem_u32(&d_full[b]), (j >> 1) & 1u, abort);
            ok = ok && mbar_wait_or_abort(smem_u32(&scale_full[j & 3u]), (j >> 2) & 1u, abort);
            ok = ok && mbar_wait_or_abort(smem_u32(&out_free[ob]), ((j / NOUT) & 1u) ^ 1u, abort);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const float osc1 = row_scale[j & 3u][row];
            const float2 osc = make_float2(osc1, osc1);
            const uint32_t lane_addr = tmem + b * S::ACC + ((quad * 32u) << 16) + part * HALF * 2u;
            float2 o[XP ? HALF : 1];
#pragma unroll
            for (uint32_t c0 = 0; c0 < 2u * HALF; c0 += 16) {
                float d0[16], d12[16];
                tmem_ld16x2(lane_addr + c0, lane_addr + KD + c0, d0, d12);
#pragma unroll
                for (uint32_t i = 0; i < 16; i += P0 ? 4 : 2) {
                    const float2 x = __fmul2_rn(__fadd2_rn(make_float2(d0[i], d0[i + 1]),
                                                           make_float2(d12[i], d12[i + 1])), osc);
                    if constexpr (P0) {
                        const float2 y = __fmul2_rn(__fadd2_rn(make_float2(d0[i + 2], d0[i + 3]),
                                                               make_float2(d12[i + 2], d12[i + 3])), osc);
                        *reinterpret_cast<float4 *>(out + (gbase ^ member_off(part * HALF + (c0 + i) / 2))) =
                            make_float4(x.x, x.y, y.x, y.y);
                        continue;
                    }
                    // in member order each chunk of eight members is written as soon as it
                    // is formed (fewer live registers than holding the half row)
                    if constexpr (XP) o[(c0 + i) / 2] = x;
                    else out[gbase ^ member_off(part * HALF + (c0 + i) / 2)] = x;
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&d_empty[b]));
            if constexpr (XP) {
                xor_unpermute(o, xl, a.xt);   // o[c] = member c ^ x (x < HALF)
#pragma unroll
                for (uint32_t c = 0; c < HALF; ++c) out[gbase ^ member_off(part * HALF + c) ^ cx] = o[c];
            }
            fence_proxy_async_smem();             // the bulk store reads them
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&out_full[ob]));
        }
    } else {
        // ------------------------------------------------------------ TMA stores
        // lane i stores segment i of every tile
        SegLanes sl;
        sl.init(a.L, a.h, a.hi, lane);
        uint32_t j = 0;
        for (unsigned long long t = first; t < tend; t += step, ++j) {
            const uint32_t ob = j % NOUT;
            const float2 *out = reinterpret_cast<const float2 *>(smem + S::OFF_OUT + ob * S::TILE_BYTES);
            const bool ok = mbar_wait_or_abort(smem_u32(&out_full[ob]), (j / NOUT) & 1u, abort);
            if (!__all_sync(0xffffffffu, ok)) break;
            if (lane < nseg) {
                if constexpr (SW) {
                    const int32_t row0 = (int32_t)((tile_base(sl, t) + sl.my_off) >> 4);
                    const uint32_t s0 = smem_u32(out + (size_t)lane * seg_amps);
                    for (uint32_t bx = 0; bx < a.boxes; ++bx)
                        tma_store_2d(&a.tmap, 0, row0 + (int32_t)(bx * a.box_rows), s0 + bx * a.box_rows * 128u);
                } else {
                    bulk_s2g(psi + tile_base(sl, t) + sl.my_off, smem_u32(out + (size_t)lane * seg_amps),
                             seg_bytes);
                }
            }
            bulk_commit();
            bulk_wait_read_all();                 // the staging tile is free again
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&out_free[ob]));
        }
        bulk_wait_all();
    }
    if (tid == 0 && abort_flag) atomicOr(a.err, 2);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == S::W_MMA) tmem_dealloc(tmem, S::TMEM_COLS);
}

// The driver's tensor-map encoder, looked up once through the runtime.
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// `bytes` bytes at buf as a 2-D tensor of 128-byte rows (32 floats), boxes of box_rows
// rows, 128-byte swizzle in shared memory; a segment of seg_bytes (a multiple of 128) is
// `boxes` boxes.
sv_status encode_rows_map(void *buf, unsigned long long bytes, uint32_t seg_bytes, CUtensorMap *map,
                          uint32_t *box_rows, uint32_t *boxes) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return svi::set_error(SV_ERR_CUDA, "tensor-core kernel setup: cuTensorMapEncodeTiled unavailable");
    const uint32_t seg_rows = seg_bytes / 128u;
    *box_rows = std::min(seg_rows, 256u);
    *boxes = seg_rows / *box_rows;
    const cuuint64_t dims[2] = {32, bytes / 128u};
    const cuuint64_t strides[1] = {128};
    const cuuint32_t box[2] = {32, *box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, buf, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        return svi::set_error(SV_ERR_CUDA, "tensor-core kernel setup: cuTensorMapEncodeTiled failed (" +
                                               std::to_string((int)r) + ")");
    return SV_OK;
}

template <int K>
sv_status launch_tc_t(sv_state *s, const svi::Gate &g) {
    using S = TcShape<K>;
    constexpr uint32_t D = S::D;
    static PerDevice<cudaError_t> setup;
    const cudaError_t init_err = setup.get(current_device(), [] {
        cudaError_t e = cudaSuccess;
        auto allow = [&e](auto kernel) {
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
        };
        allow(apply_tc<K, false>);
        allow(apply_tc<K, true>);
        if constexpr (K == 5) {
            allow(apply_tc<K, false, false, true>);
            allow(apply_tc<K, false, false, true, true>);
        }
        return e;
    });
    if (init_err != cudaSuccess)
        return svi::set_error(SV_ERR_CUDA, std::string("tensor-core kernel setup: ") +
                                               cudaGetErrorString(init_err));
    Plan p = make_plan(s->n, K, g.t, S::TB);
    // 8-byte accesses: bank pair = tile bits 0..3; targets there get lane-dependent order
    uint32_t tl = 0;
    while (tl < (uint32_t)K && p.lp[tl] < 4u) ++tl;
    // width 5 on states of at least 13 qubits: the swizzled tensor-map staging, whatever the
    // targets (no XOR member order); otherwise XOR order for bank-bit targets
    const bool swz = K == 5 && s->n >= K + 8u;
    if (swz) tl = 0;
    TcArgs<K> a;
    a.box_rows = a.boxes = 0;
    if (swz) {
        const sv_status st = encode_rows_map(s->buf, 8ull << s->n, 8u << p.L, &a.tmap, &a.box_rows, &a.boxes);
        if (st != SV_OK) return st;
    }
    // U on its fixed-point grid, in FP64 on the host
    const double *u = reinterpret_cast<const double *>(g.u.data());
    double m4[4] = {0.0, 0.0, 0.0, 0.0};
    for (uint32_t i = 0; i < 2 * D * D; i += 4)
        for (uint32_t q = 0; q < 4; ++q) m4[q] = std::fabs(u[i + q]) > m4[q] ? std::fabs(u[i + q]) : m4[q];
    const double rmax = std::max(std::max(m4[0], m4[1]), std::max(m4[2], m4[3]));
    int eb = 0;
    std::frexp(rmax, &eb);                                   // rmax < 2^eb
    // nearest integers (ties to even) by adding 1.5 2^52: |u sx| <= 2^26, the integer is the low
    // word of the sum (lrint was a library call per entry, a third of a launch's host time)
    const double sx = std::ldexp(1.0, 26 - eb);
    int32_t *bx = reinterpret_cast<int32_t *>(a.bx);
    for (uint32_t i = 0; i < 2 * D * D; ++i) {
        const double t = u[i] * sx + 6755399441055744.0;
        int64_t w;
        std::memcpy(&w, &t, 8);
        bx[i] = (int32_t)w;
    }
    a.b_inv_scale = (float)std::ldexp(1.0, eb - 8);
    a.psi = s->buf;
    a.err = reinterpret_cast<int *>(s->ws + svi::WS_ERR);
    a.ntiles = p.ntiles;
    // Two tiles in flight per SM (64 KiB at K = 5, 10 MB in all) keep HBM busy; more of them queue up
    // in front of the stores: 28 qubits, targets 6-10, 694 us per pass with four tiles in flight, 641
    // with two; targets 7 and 24-27 699 and 640.  Tiles in 1 KiB pieces (five high targets)
    // have longer latencies and want all stages: targets 23-27 636 us with four, 671 with two.
    // (Two 32 KiB tiles per stage and transfer, the form for more than 22 qubits before: 657-669 us,
    // 24 qubits 47-48.5 against 45-46 us.)
    a.depth = K == 5 && p.h < K ? 2u : S::NS;
    a.L = p.L;
    a.h = p.h;
    for (int j = 0; j < SV_MAX_K; ++j) a.hi[j] = p.hi[j];
    for (int j = 0; j < K; ++j) a.lp[j] = p.lp[j];
    a.xs = 4u - tl;
    a.xt = std::min(tl, (uint32_t)K - 1u);   // permute within a worker's half of the members
    const unsigned grid = (unsigned)std::min<unsigned long long>(p.ntiles, (unsigned long long)s->num_sms);
    // with eight worker warps per role the permutation costs less than even 2-way conflicts
    auto kernel = a.xt >= 1 ? apply_tc<K, true> : apply_tc<K, false>;
    if constexpr (K == 5)
        if (swz) kernel = p.lp[3] == 3 ? apply_tc<K, false, false, true, true> : apply_tc<K, false, false, true>;
    SV_CUDA(launch_pass(kernel, dim3(grid), S::THREADS, S::SMEM, s->stream, a));
    return SV_OK;
}

// Batched launches (sv_batch_apply): complex64 gates of widths 4 and 5 on states of at least 12
// qubits, the former widened by an identity qubit (chosen as in widen_gate), with the swizzled
// tensor-map staging (SW) like single states.
static cudaError_t tc_batch_setup() {
    static PerDevice<cudaError_t> setup;
    return setup.get(current_device(), [] {
        constexpr int smem = (int)TcShape<5, true>::SMEM;
        cudaError_t e = cudaFuncSetAttribute(apply_tc<5, false, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(apply_tc<5, false, true, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        return e;
    });
}

// Also looks up the tensor-map encoder, so that a launch inside a stream capture finds it.
cudaError_t tc_batch_prepare() {
    const cudaError_t e = tc_batch_setup();
    if (e == cudaSuccess && !tensor_map_encoder()) return cudaErrorNotSupported;
    return e;
}

// The width-5 targets of a gate, and where its own local bits lie among them.
static void widen_targets(uint32_t n, uint32_t k, const uint32_t *t, uint32_t (&t5)[5], uint8_t *pos, uint32_t *idm) {
    uint64_t used = 0;
    for (uint32_t j = 0; j < k; ++j) used |= 1ull << t[j];
    uint32_t m = k;
    for (uint32_t q = 5; q < n && m < 5; ++q)
        if (!((used >> q) & 1ull)) { used |= 1ull << q; ++m; }
    for (uint32_t q = 0; q < n && m < 5; ++q)
        if (!((used >> q) & 1ull)) { used |= 1ull << q; ++m; }
    uint32_t i = 0, own = 0;
    *idm = 0;
    for (uint32_t q = 0; q < n && i < 5; ++q)
        if ((used >> q) & 1ull) {
            t5[i] = q;
            if (own < k && t[own] == q) pos[own++] = (uint8_t)i;
            else *idm |= 1u << i;
            ++i;
        }
}

size_t tc_batch_image_bytes() { return TcShape<5, true>::B_SET; }

sv_status launch_tc_pack(const sv_batch_launch *L, const size_t *tab_off, uint32_t ngates, const void *utab,
                         void *images, float *bscale) {
    for (uint32_t g0 = 0; g0 < ngates; g0 += PACK_GATES) {
        const uint32_t m = std::min(PACK_GATES, ngates - g0);
        PackArgs a;
        a.utab = static_cast<const unsigned char *>(utab);
        a.images = static_cast<unsigned char *>(images);
        a.bscale = bscale;
        for (uint32_t i = 0; i < m; ++i) {
            const sv_batch_launch &l = L[g0 + i];
            uint32_t t5[5];
            a.g[i].tab = tab_off[g0 + i];
            a.g[i].image = (unsigned long long)(g0 + i) * l.states;
            a.g[i].kin = l.k;
            widen_targets(l.n, l.k, l.t, t5, a.g[i].pos, &a.g[i].idm);
        }
        SV_CUDA(launch_pass(pack_images, dim3(L[g0].states, m), 256, 0, L[g0].stream, a));
    }
    return SV_OK;
}

sv_status launch_tc_batch(const sv_batch_launch &L) {
    using S = TcShape<5, true>;
    const cudaError_t e0 = tc_batch_prepare();
    if (e0 != cudaSuccess)
        return svi::set_error(SV_ERR_CUDA, std::string("batched tensor-core kernel setup: ") + cudaGetErrorString(e0));
    uint32_t t5[5], idm;
    uint8_t pos[SV_MAX_K];
    widen_targets(L.n, L.k, L.t, t5, pos, &idm);
    const Plan p = make_plan(L.n, 5, t5, S::TB);
    TcArgs<5> a;
    // the whole batch (states back to back) as one tensor; the swizzle spreads the banks
    const sv_status st = encode_rows_map(L.psi, (8ull * L.states) << L.n, 8u << p.L, &a.tmap, &a.box_rows,
                                         &a.boxes);
    if (st != SV_OK) return st;
    std::memset(a.bx, 0, sizeof(a.bx));
    a.b_inv_scale = 1.f;
    a.psi = L.psi;
    a.err = L.err;
    a.ntiles = p.ntiles * L.states;
    a.L = p.L;
    a.h = p.h;
    for (int j = 0; j < SV_MAX_K; ++j) a.hi[j] = p.hi[j];
    for (int j = 0; j < 5; ++j) a.lp[j] = p.lp[j];
    a.xs = 0;
    a.xt = 0;
    a.depth = S::NS;
    a.images = static_cast<const unsigned char *>(L.images);
    a.bscale = L.bscale;
    a.tps = (uint32_t)__builtin_ctzll(p.ntiles);
    a.n = L.n;
    const unsigned grid = (unsigned)std::min<unsigned long long>(a.ntiles, (unsigned long long)L.num_sms);
    SV_CUDA(launch_pass(p.lp[3] == 3 ? apply_tc<5, false, true, true, true> : apply_tc<5, false, true, true>,
                        dim3(grid), S::THREADS, S::SMEM, L.stream, a));
    return SV_OK;
}

}  // namespace svk

namespace svi {

// Width 4 and 5, and on states of at least 13 qubits every dense width (narrower gates run
// as width-5 ones, U (x) I, on the swizzled kernel: at 30 qubits its passes
// take 2.59-2.74 ms against 2.74 for the width-2/3 CUDA-core kernel).
bool tc_eligible(const sv_state *s, const Gate &g) {
    if (s->dtype != SV_C64 || (s->policy & SV_POLICY_NO_TENSOR_CORES)) return false;
    if (g.k == 4 || g.k == 5) return s->n >= g.k + 7;
    return g.k >= 1 && s->n >= svk::TcShape<5>::TB + 1;
}

// Width-4 gates run as width-5 ones (U (x) I) where the state allows: the k = 5 kernel
// moves a tile with half the per-tile overhead of the k = 4 one for the same bytes.
sv_status launch_apply_tc(sv_state *s, const Gate &g) {
    if (g.k == 5) return svk::launch_tc_t<5>(s, g);
    if (s->n >= svk::TcShape<5>::TB) return svk::launch_tc_t<5>(s, widen_gate(g, s->n, 5));
    return svk::launch_tc_t<4>(s, g);
}

}  // namespace svi
