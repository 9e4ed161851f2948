// Gates in complex128 on the 5th-generation tensor cores (tcgen05), to FP64 accuracy.
//
// As in the complex64 kernel, a tile of 128 groups of 2^4 amplitudes is the real GEMM
// D[128 x 32] = A[128 x 32] R^T (R = real embedding of the 16 x 16 gate, Eq. 3), but every
// operand is cut into six exact FP16 digits (fixed_point.h): per row of A on the grid of
// the row's largest exponent, for R on the grid of its largest entry,
//     A = sum_i A_i 2^(-9 i),  R = sum_j B_j 2^(-9 j),  i, j = 0..5, |A_i|, |B_j| <= 256.
// Level s collects the digit pairs with i + j = s; with 32 products of at most 2^16 per
// pair, the levels s = 0..4 (1 to 5 pairs) stay below 2^24 and are accumulated EXACTLY by the FP32
// tensor-core accumulators; level 5 is added at its scale to level 4's accumulator (B_j 2^-9, also
// exact FP16).  Levels 6..10 are dropped (below 2^-46 of the row's largest term).  The epilogue
// converts the accumulators to integers, forms Z = L0 2^40 + L1 2^31 + L2 2^22 + L3 2^13 +
// rint(16 D45) in 64 bits and builds the nearest double of Z 2^p (an identity gate returns its
// input bit for bit).
// The split and the products never touch the FP64 pipe (this GPU runs it at about 1/64 of the
// FP32 rate), only the final int64 -> double conversion of each output does, which balances the
// integer and FP64 pipes.
//
// The five accumulators and the slices of R lie side by side, so the products of digit A_i with
// B_0 .. B_{4-i} are one MMA per K step into D_i .. D_4 (N = 160, 128, .. 32): 22 instructions
// per 128 groups instead of 42 of N = 32, which took about 140 cycles each.
//
// What bounds it: issue and the integer pipe (about 160 instructions per amplitude, 4250 cycles
// per 2048 amplitudes where HBM needs 3030).  So the workers do not meet: two transform groups of
// four warps take alternate tiles, whole rows per warp (eight warps on one tile exchanged
// row maxima and met twice: 2430 cycles more), the epilogue's hand over by counted arrivals, and
// the short forms of the split and of the scaling (rows whose exponents allow them, a vote per warp)
// save a quarter of the integer instructions.  More workers do not help (16 epilogue warps: the
// same time; 16 transform warps: 5% slower).  28-qubit grid circuit: 238.5 -> 196 ms, with a store warp and
// one swizzled tile per stage 169.8 ms.
//
// Gates on fewer than four qubits are widened to four (U (x) I on extra qubits chosen
// above bit 4, so a warp's rows stay contiguous in shared memory).
//
// Roles: warps 0-7 digit transform into TMEM (tcgen05.st), warp 8 TMA producer (lane i copies
// segment i), warp 9 lane 0 the MMA issuer, warps 10-17 the epilogue, warp 18 the bulk stores; A
// and D double-buffered in TMEM (2 x 96 + 2 x 160 = 512 columns); every wait bounded with a shared
// abort flag.
#include <cuda_fp16.h>
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "fixed_point.h"
#include "plan.h"
#include "ptx.cuh"
#include "sv_internal.h"
#include "tc.cuh"

namespace svk {

// One tile is one MMA (128 groups): 32 KiB.
struct Tc64 {
    static constexpr uint32_t K = 4;
    static constexpr uint32_t D = 16;                     // amplitudes per group
    static constexpr uint32_t KD = 32;                    // real K = N
    static constexpr uint32_t ROWS = 128;                 // groups per tile (MMA M)
    static constexpr uint32_t TB = 11;                    // tile bits
    static constexpr uint32_t TILE_BYTES = ROWS * D * 16u;
    static constexpr uint32_t B_BYTES = KD * KD * 2u;     // one FP16 digit slice of R
    static constexpr uint32_t NB = 12;                    // B_j and B_j 2^-9, j = 0..5
    static constexpr uint32_t SBO = (KD / 8u) * 128u;
    static constexpr uint32_t NS = 4;                     // raw stages
    static constexpr uint32_t NOUT = 2;                   // output staging tiles
    static constexpr uint32_t NACC = 5;                   // D0, D1, D2, D3, D45
    static constexpr uint32_t ACC = NACC * KD;            // TMEM columns of one D set
    static constexpr uint32_t A_COLS = KD / 2u;           // TMEM columns of one A digit slice
    static constexpr uint32_t A_SET = 6u * A_COLS;        // one A buffer (six slices)
    static constexpr uint32_t A_COL0 = 2u * ACC;
    static constexpr uint32_t TMEM_COLS = 512;
    static_assert(A_COL0 + 2u * A_SET <= TMEM_COLS, "TMEM layout");
    static constexpr uint32_t OFF_RAW = NB * B_BYTES;
    static constexpr uint32_t OFF_OUT = OFF_RAW + NS * TILE_BYTES;
    static constexpr uint32_t SMEM = OFF_OUT + NOUT * TILE_BYTES;
    static constexpr uint32_t THREADS = 608;              // 19 warps
    // warps 0-7 transform, 8 producer, 9 MMA issuer, 10-17 epilogue, 18 TMA stores
    static constexpr uint32_t W_PROD = 8, W_MMA = 9, W_EPI = 10, W_STORE = 18;
};

struct Tc64Args {
    // the state as a 2-D tensor of 128-byte rows (8 amplitudes), `boxes` boxes of box_rows rows per
    // segment, 128-byte swizzle in shared memory
    CUtensorMap tmap;
    // U on the fixed-point grid of its largest entry: (re, im) of entry (r, c), row-major; the
    // prologue cuts each into six digits (expand_b64)
    alignas(16) longlong2 bx[16 * 16];
    uint32_t box_rows, boxes;
    int b_exp;               // max |U| < 2^b_exp
    int *err;
    unsigned long long ntiles;
    uint32_t L, h;
    uint32_t hi[SV_MAX_K];
    uint32_t lp[4];
};

// Digit-pair word -> FP16 pair of digits: the patterns read 2048 + 2u, and
// (2048 + 2u) 0.5 - 1280 = u - 256 is exact in one half2 multiply-add.
__device__ __forceinline__ uint32_t digit_pair(uint32_t word) {
    const __half2 h = __hfma2(*reinterpret_cast<const __half2 *>(&word), __float2half2_rn(0.5f),
                              __float2half2_rn(-1280.f));
    return *reinterpret_cast<const uint32_t *>(&h);
}

// The twelve FP16 slices of R (B_j, then B_j 2^-9) from the fixed-point entries in the
// kernel's parameters: complex entry (r, c) fills R's rows 2r (re, -im) and 2r + 1 (im, re)
// at columns 2c, 2c + 1, one FP16 pair each.  Entries i0, i0 + stride, ...  4 KiB of
// parameters in 16-byte generic loads instead of 12 KiB of int16 digits in constant-bank
// loads (see expand_b in apply_tc.cu): a 12-qubit pass 17.2 -> 9.4 us, a 23-qubit one 97 -> 90.
__device__ __forceinline__ void expand_b64(unsigned char *sB, const longlong2 *bx, uint32_t i0, uint32_t stride) {
    using S = Tc64;
    for (uint32_t e = i0; e < 256u; e += stride) {
        const int4 v = ld_param16(bx + e);
        const uint64_t re = ((uint64_t)(uint32_t)v.y << 32 | (uint32_t)v.x) + fxp::OFFSET;
        const uint64_t im = ((uint64_t)(uint32_t)v.w << 32 | (uint32_t)v.z) + fxp::OFFSET;
        const uint32_t r = e >> 4, c = e & 15u;
        const uint32_t o0 = kmajor_off16(2u * r, 2u * c, S::SBO), o1 = kmajor_off16(2u * r + 1u, 2u * c, S::SBO);
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const float dr = (float)((int)fxp::field(re, j) - 256), di = (float)((int)fxp::field(im, j) - 256);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float f = h ? 1.f / 512.f : 1.f;      // exact: an integer of at most 9 bits
                *reinterpret_cast<__half2 *>(sB + (6 * h + j) * S::B_BYTES + o0) = __floats2half2_rn(dr * f, -di * f);
                *reinterpret_cast<__half2 *>(sB + (6 * h + j) * S::B_BYTES + o1) = __floats2half2_rn(di * f, dr * f);
            }
        }
    }
}

// Levels as integers (L0, L1 below 2^22 by the bit-pattern trick, the others by
// conversion; 16 D45 below 2^28), Z = L0 2^40 + L1 2^31 + L2 2^22 + L3 2^13 + rint(16 D45)
// in 64 bits, and the nearest double of Z 2^p.  The int64 -> double conversion runs on the
// FP64 pipe, which the rest of the kernel leaves idle: it rounds to nearest even exactly
// like fxp::assemble_words (the integer-pipe form, about 30 instructions; converting every
// second output in integers measured the same), and the scaling by 2^p is an add to the exponent
// field while the result stays normal: always, for nonzero |Z| < 2^63, with P_SAFE (-1022 <= p
// <= 960).
template <bool P_SAFE>
__device__ __forceinline__ double combine_levels(float f0, float f1, float f2, float f3, float f45, int p) {
    constexpr uint32_t MAGIC = 0x4B400000u;                 // pattern of 1.5 2^23
    const uint32_t b0 = __float_as_uint(f0 + 12582912.f), b1 = __float_as_uint(f1 + 12582912.f);
    const unsigned long long c0 = 0ull - ((unsigned long long)MAGIC << 31) - ((unsigned long long)MAGIC << 40);
    unsigned long long u = (unsigned long long)((long long)__float2int_rn(f45 * 16.f)) + c0;
    u += (unsigned long long)((long long)__float2int_rn(f3) * (1 << 13));
    u += (unsigned long long)((long long)__float2int_rn(f2) * (1 << 22));
    u += (unsigned long long)b1 * 0x80000000u;
    u += (unsigned long long)(b0 << 8) << 32;               // the bits above 2^64 cancel with c0's
    const long long z = (long long)u;
    const double x = __ll2double_rn(z);
    if (P_SAFE) {
        const int hi = __double2hiint(x);
        return __hiloint2double(hi ? hi + (p << 20) : 0, __double2loint(x));
    }
    if (z == 0) return 0.0;
    const long long b = __double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FF) + p;
    if (e < 1 || e > 2046) return fxp::assemble_slow(z, p);
    return __longlong_as_double(b + ((long long)p << 52));
}

// The digit words of group members c0 .. c0 + 3 of one row.  NEAR: every component's exponent
// field is nonzero and at most 31 below the row's largest.
template <bool NEAR>
__device__ __forceinline__ void cut_members(const uint4 (&v)[4], uint32_t emax, uint32_t (&w)[6][4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint32_t rh, rl, ih, il, t[6];
        if (NEAR) {
            const uint32_t ew = emax << 20 | 0xFFFFFu;
            fxp::offset_fixed_near(v[c].y, v[c].x, ew, rh, rl);
            fxp::offset_fixed_near(v[c].w, v[c].z, ew, ih, il);
        } else {
            fxp::offset_fixed(v[c].y, v[c].x, emax, rh, rl);
            fxp::offset_fixed(v[c].w, v[c].z, emax, ih, il);
        }
        fxp::digit_pair_words(rh, rl, ih, il, t);
#pragma unroll
        for (int i = 0; i < 6; ++i) w[i][c] = digit_pair(t[i]);
    }
}

// The pipelines count this CTA's tiles (j).
// Tiles move by 2-D tensor-map copies with the 128-byte swizzle and the roles address
// them through it, so a warp's lanes reach different banks whatever the targets.  The swizzle is
// applied to the group base and the target bits, which then combine by XOR.  (1-D bulk copies where
// at most one target is among bits 0-2: the same time, 8% more with one.)
__global__ void __launch_bounds__(608, 1) apply_tc64(const __grid_constant__ Tc64Args a) {
    using S = Tc64;
    constexpr uint32_t KD = S::KD, NS = S::NS;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long full[NS], empty[NS];
    __shared__ __align__(8) unsigned long long a_full[2], a_empty[2], d_full[2], d_empty[2];
    __shared__ __align__(8) unsigned long long scale_full[4];   // row exponents, tile j -> j & 3
    __shared__ __align__(8) unsigned long long out_full[2], out_free[2];   // staged tiles
    __shared__ int row_exp[4][128];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    unsigned char *sB = smem;
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    const uint32_t seg_amps = 1u << a.L;
    const uint32_t nseg = 1u << a.h;

    if (tid == 0) pass_trigger();
    if (warp == S::W_MMA) {
        tmem_alloc(smem_u32(&tmem_slot), S::TMEM_COLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (uint32_t s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 4);            // one transform group
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&a_full[b]), 4);       // one transform group
            mbar_init(smem_u32(&a_empty[b]), 1);
            mbar_init(smem_u32(&d_full[b]), 1);
            mbar_init(smem_u32(&d_empty[b]), 8);      // the epilogue warps
            mbar_init(smem_u32(&out_full[b]), 8);
            mbar_init(smem_u32(&out_free[b]), 1);
        }
        for (int q = 0; q < 4; ++q) mbar_init(smem_u32(&scale_full[q]), 4);
        abort_flag = 0;
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp != S::W_PROD) {
        // every warp but the producer, which is already loading the first tiles
        expand_b64(sB, a.bx, tid < S::W_PROD * 32u ? tid : tid - 32u, S::THREADS - 32u);
        fence_proxy_async_smem();
        named_bar(3, S::THREADS - 32u);
    }
    const uint32_t tmem = tmem_slot;
    volatile int *abort = &abort_flag;
    const unsigned long long first = blockIdx.x, step = gridDim.x;
    const uint32_t ntile = a.ntiles > first ? (uint32_t)((a.ntiles - first + step - 1) / step) : 0u;

    auto group_base = [&](uint32_t row) {
        uint32_t g = row;
#pragma unroll
        for (int j = 0; j < 4; ++j) g = insert_zero32(g, a.lp[j]);
        return swz128_16(g);
    };
    // tile offset of target j (swizzled; four registers), and of group member c:
    // the XOR of the offsets of its set bits; a member's index is group base XOR offset
    uint32_t tb[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) tb[j] = swz128_16(1u << a.lp[j]);
    auto member_off = [&](uint32_t c) {
        uint32_t o = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if ((c >> j) & 1u) o ^= tb[j];
        return o;
    };

    if (warp == S::W_PROD) {
        // ------------------------------------------------------------ TMA producer
        SegLanes sl;
        sl.init(a.L, a.h, a.hi, lane);
        pass_wait();
        uint32_t j = 0;
        for (unsigned long long t = first; t < a.ntiles; t += step, ++j) {
            const uint32_t s = j % NS, u = j / NS;
            bool ok = true;
            if (lane == 0) ok = mbar_wait_or_abort(smem_u32(&empty[s]), (u & 1u) ^ 1u, abort);
            if (!__shfl_sync(0xffffffffu, (int)ok, 0)) break;
            const uint32_t bar = smem_u32(&full[s]);
            if (lane == 0) mbar_arrive_expect_tx(bar, S::TILE_BYTES);
            __syncwarp();
            if (lane < nseg) {
                double2 *dst = reinterpret_cast<double2 *>(smem + S::OFF_RAW + s * S::TILE_BYTES);
                // segment = `boxes` boxes of box_rows 128-byte rows (8 amplitudes each)
                const int32_t row0 = (int32_t)((sl.base(t) + sl.my_off) >> 3);
                const uint32_t d0 = smem_u32(dst + (size_t)lane * seg_amps);
                for (uint32_t bx = 0; bx < a.boxes; ++bx)
                    tma_load_2d(d0 + bx * a.box_rows * 128u, &a.tmap, 0, row0 + (int32_t)(bx * a.box_rows), bar);
            }
        }
    } else if (warp == S::W_MMA) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            const uint32_t B0 = smem_u32(sB);
            for (uint32_t j = 0; j < ntile; ++j) {
                const uint32_t b = j & 1u, u = j >> 1;
                if (!mbar_wait_or_abort(smem_u32(&a_full[b]), u & 1u, abort)) break;
                if (!mbar_wait_or_abort(smem_u32(&d_empty[b]), (u & 1u) ^ 1u, abort)) break;
                tc_fence_after();
                const uint32_t A0 = tmem + S::A_COL0 + b * S::A_SET;
                const uint32_t dset = tmem + b * S::ACC;
                // A_i [B_0 .. B_{4-i}] -> [D_i .. D_4]: N rows from the first slice of B on
#pragma unroll
                for (uint32_t i = 0; i < 5; ++i)
#pragma unroll
                    for (uint32_t ks = 0; ks < KD / 16; ++ks)
                        mma_f16_tmem_a(dset + i * KD, A0 + i * S::A_COLS + ks * 8u,
                                       smem_desc(B0 + ks * 256u, 128u, S::SBO), idesc_f16(S::ROWS, (5u - i) * KD),
                                       (i == 0 && ks == 0) ? 0u : 1u);
                // level 5 at its scale, after the exact sums of level 4: A_i (B_{5-i} 2^-9) -> D_4
#pragma unroll
                for (uint32_t i = 0; i < 6; ++i)
#pragma unroll
                    for (uint32_t ks = 0; ks < KD / 16; ++ks)
                        mma_f16_tmem_a(dset + 4u * KD, A0 + i * S::A_COLS + ks * 8u,
                                       smem_desc(B0 + (11u - i) * S::B_BYTES + ks * 256u, 128u, S::SBO),
                                       idesc_f16(S::ROWS, KD), 1u);
                mma_commit(smem_u32(&a_empty[b]));
                mma_commit(smem_u32(&d_full[b]));
            }
        }
    } else if (warp < S::W_PROD) {
        // ------------------------------------------------------------ digit transform
        // Two groups of four warps take alternate tiles, one warp per TMEM lane quadrant and
        // whole rows each, so that no warp waits for another.  Rolled loops over four members at
        // a time keep the code small (the roles run different code on every SM sub-partition).
        const uint32_t quad = warp & 3u, grp = warp >> 2;
        const uint32_t row = quad * 32u + lane;
        const uint32_t lo_off[4] = {0u, tb[0], tb[1], tb[0] ^ tb[1]};
        const uint32_t gbase = group_base(row);
        const uint32_t arow = tmem + S::A_COL0 + grp * S::A_SET + ((quad * 32u) << 16);
        for (uint32_t j = grp; j < ntile; j += 2) {
            const uint32_t s = j % NS;
            const bool okf = mbar_wait_or_abort(smem_u32(&full[s]), (j / NS) & 1u, abort);
            if (!__all_sync(0xffffffffu, okf)) break;
            const double2 *rs = reinterpret_cast<const double2 *>(smem + S::OFF_RAW + s * S::TILE_BYTES);
            uint32_t em = 0, mn = 0x7FFFFFFFu;    // largest and smallest |high word| of the row
#pragma unroll 1
            for (uint32_t c0 = 0; c0 < 16u; c0 += 4) {
                const uint32_t hoff = gbase ^ (((c0 >> 2) & 1u) ? tb[2] : 0u) ^ (((c0 >> 3) & 1u) ? tb[3] : 0u);
#pragma unroll
                for (uint32_t c = 0; c < 4; ++c) {
                    const uint4 v = *reinterpret_cast<const uint4 *>(rs + (hoff ^ lo_off[c]));
                    const uint32_t r = v.y & 0x7FFFFFFFu, i = v.w & 0x7FFFFFFFu;
                    em = max(em, max(r, i));
                    mn = min(mn, min(r, i));
                }
            }
            const uint32_t emax = max(em >> 20, 1u);
            const uint32_t emin = mn >> 20;
            const bool near = __all_sync(0xffffffffu, emin != 0u && emax - emin < 32u);
            bool oka = true;
#pragma unroll 1
            for (uint32_t c0 = 0; c0 < 16u; c0 += 4) {
                const uint32_t hoff = gbase ^ (((c0 >> 2) & 1u) ? tb[2] : 0u) ^ (((c0 >> 3) & 1u) ? tb[3] : 0u);
                uint32_t w[6][4];
                uint4 va[4];
#pragma unroll
                for (uint32_t c = 0; c < 4; ++c) va[c] = *reinterpret_cast<const uint4 *>(rs + (hoff ^ lo_off[c]));
                if (near) cut_members<true>(va, emax, w);
                else cut_members<false>(va, emax, w);
                if (c0 == 0) {
                    // the A buffer is free once the MMAs of tile j - 2 have completed
                    oka = __all_sync(0xffffffffu,
                                     mbar_wait_or_abort(smem_u32(&a_empty[grp]), ((j >> 1) & 1u) ^ 1u, abort));
                    if (!oka) break;
                    tc_fence_after();
                    // slot j & 3 was last read by the epilogue of tile j - 4, which finished
                    // before the MMAs of tile j - 2
                    row_exp[j & 3u][row] = (int)emax;
                }
#pragma unroll
                for (int i = 0; i < 6; ++i) tmem_st4_async(arow + i * S::A_COLS + c0, w[i]);
            }
            if (!oka) break;
            fence_proxy_async_smem();             // reads of the raw stage before its refill
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(smem_u32(&empty[s]));
                mbar_arrive(smem_u32(&a_full[grp]));
                mbar_arrive(smem_u32(&scale_full[j & 3u]));
            }
        }
    } else if (warp < S::W_STORE) {
        // ------------------------------------------------------------ epilogue
        // Two warps per lane quadrant, each over 16 of the 32 accumulator columns.
        const uint32_t quad = warp & 3u;
        const uint32_t row = quad * 32u + lane;
        const uint32_t part = (warp - S::W_EPI) >> 2;
        const uint32_t gbase = group_base(row);
        for (uint32_t j = 0; j < ntile; ++j) {
            const uint32_t b = j & 1u;
            double2 *out = reinterpret_cast<double2 *>(smem + S::OFF_OUT + b * S::TILE_BYTES);
            bool ok = mbar_wait_or_abort(smem_u32(&d_full[b]), (j >> 1) & 1u, abort);
            ok = ok && mbar_wait_or_abort(smem_u32(&scale_full[j & 3u]), (j >> 2) & 1u, abort);
            ok = ok && mbar_wait_or_abort(smem_u32(&out_free[b]), ((j >> 1) & 1u) ^ 1u, abort);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const int p = row_exp[j & 3u][row] + a.b_exp - 1078;   // out = Z 2^p
            const uint32_t lane_addr = tmem + b * S::ACC + ((quad * 32u) << 16);
            const bool p_safe = __all_sync(0xffffffffu, p >= -1022 && p <= 960);
            // eight columns (four members) of the five accumulators per step, both steps
            // unrolled so that their recombinations overlap
            auto finish = [&](auto safe, uint32_t c0) {
                float d[5][8];
                tmem_ld8x5(lane_addr + part * 16u + c0, KD, d);
                const uint32_t hoff = gbase ^ (c0 ? tb[2] : 0u) ^ (part ? tb[3] : 0u);
#pragma unroll
                for (uint32_t c = 0; c < 4; ++c) {
                    const double re = combine_levels<decltype(safe)::value>(
                        d[0][2 * c], d[1][2 * c], d[2][2 * c], d[3][2 * c], d[4][2 * c], p);
                    const double im = combine_levels<decltype(safe)::value>(
                        d[0][2 * c + 1], d[1][2 * c + 1], d[2][2 * c + 1], d[3][2 * c + 1], d[4][2 * c + 1], p);
                    out[hoff ^ member_off(c)] = make_double2(re, im);
                }
            };
            if (p_safe) {
                finish(std::true_type{}, 0u);
                finish(std::true_type{}, 8u);
            } else {
#pragma unroll 1
                for (uint32_t c0 = 0; c0 < 16u; c0 += 8) finish(std::false_type{}, c0);
            }
            tc_fence_before();
            fence_proxy_async_smem();                 // the bulk store reads what this thread wrote
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(smem_u32(&d_empty[b]));
                mbar_arrive(smem_u32(&out_full[b]));
            }
        }
    } else {
        // ------------------------------------------------------------ TMA stores
        SegLanes sl;
        sl.init(a.L, a.h, a.hi, lane);
        for (uint32_t j = 0; j < ntile; ++j) {
            const uint32_t ob = j & 1u;
            const unsigned long long t = first + (unsigned long long)j * step;
            const double2 *out = reinterpret_cast<const double2 *>(smem + S::OFF_OUT + ob * S::TILE_BYTES);
            const bool ok = mbar_wait_or_abort(smem_u32(&out_full[ob]), (j >> 1) & 1u, abort);
            if (!__all_sync(0xffffffffu, ok)) break;
            if (lane < nseg) {
                const int32_t row0 = (int32_t)((sl.base(t) + sl.my_off) >> 3);
                const uint32_t s0 = smem_u32(out + (size_t)lane * seg_amps);
                for (uint32_t bx = 0; bx < a.boxes; ++bx)
                    tma_store_2d(&a.tmap, 0, row0 + (int32_t)(bx * a.box_rows), s0 + bx * a.box_rows * 128u);
            }
            bulk_commit();
            bulk_wait_read_all();                 // the staging is free again
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

sv_status launch_tc64(sv_state *s, const svi::Gate &g0) {
    using S = Tc64;
    static PerDevice<cudaError_t> setup;
    const cudaError_t init_err = setup.get(current_device(), [] {
        return cudaFuncSetAttribute(apply_tc64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
    });
    if (init_err != cudaSuccess)
        return svi::set_error(SV_ERR_CUDA, std::string("tensor-core kernel setup: ") +
                                               cudaGetErrorString(init_err));
    svi::Gate gw;
    const svi::Gate *g = &g0;
    if (g0.k < 4) {
        gw = svi::widen_gate(g0, s->n, 4);
        g = &gw;
    }
    const Plan p = make_plan(s->n, 4, g->t, S::TB);
    // (Tiles of two MMAs for high targets, 64 KiB per stage, took 68 us per pass on 23 qubits against
    // 63, and 0.8% more on 28.)
    Tc64Args a;
    const sv_status st = encode_rows_map(s->buf, 16ull << s->n, 16u << p.L, &a.tmap, &a.box_rows, &a.boxes);
    if (st != SV_OK) return st;
    // U on its fixed-point grid, exactly, on the host (the kernel cuts the digits)
    double rmax = 0.0;
    for (uint32_t i = 0; i < 256; ++i)
        rmax = std::max(rmax, std::max(std::fabs(g->u[i].real()), std::fabs(g->u[i].imag())));
    int eb = 0;
    std::frexp(rmax, &eb);                                   // rmax < 2^eb
    const uint32_t ebias = (uint32_t)std::max(eb + 1022, 1);    // as a biased exponent field
    for (uint32_t i = 0; i < 256; ++i)
        a.bx[i] = make_longlong2(fxp::to_fixed(fxp::bits_of(g->u[i].real()), ebias),
                                 fxp::to_fixed(fxp::bits_of(g->u[i].imag()), ebias));
    a.b_exp = (int)ebias - 1022;
    a.err = reinterpret_cast<int *>(s->ws + svi::WS_ERR);
    a.ntiles = p.ntiles;
    a.L = p.L;
    a.h = p.h;
    for (int j = 0; j < SV_MAX_K; ++j) a.hi[j] = p.hi[j];
    for (int j = 0; j < 4; ++j) a.lp[j] = p.lp[j];
    const unsigned grid = (unsigned)std::min<unsigned long long>(p.ntiles, (unsigned long long)s->num_sms);
    SV_CUDA(launch_pass(apply_tc64, dim3(grid), S::THREADS, S::SMEM, s->stream, a));
    return SV_OK;
}

}  // namespace svk

namespace svi {

bool tc64_eligible(const sv_state *s, const Gate &g) {
    return s->dtype == SV_C128 && g.k <= 4 && s->n >= svk::Tc64::TB &&
           !(s->policy & SV_POLICY_NO_TENSOR_CORES);
}

sv_status launch_apply_tc64(sv_state *s, const Gate &g) { return svk::launch_tc64(s, g); }

}  // namespace svi
