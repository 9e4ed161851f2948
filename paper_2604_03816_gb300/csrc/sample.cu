// Measurement sampling, the backend's third operation next to initialisation and gate
// application (Section 4.1).  The paper prints no procedure; this one draws from an exact
// integer cumulative distribution, so the sampled indices are reproducible bit for bit
// and every prefix sum may be formed in parallel:
//
// 1. p_k = |alpha_k|^2 in the state's precision (FP32 for complex64, FP64 for
//    complex128), no contraction.
// 2. P_k = floor(p_k 2^58), from the bits of p_k (exponent and mantissa, integer shifts).
// 3. Blocks of B = min(64, 2^n) outcomes: S_b = sum of the block's P_k (uint64, one warp
//    per block); chunks of C = min(4096, #blocks) blocks: L_b = exclusive prefix of the
//    S_b within the chunk (a shared-memory scan), chunk totals, O_c = their exclusive
//    prefix and T = the total; the block prefix is P_b = O_{chunk(b)} + L_b.
// 4. Shot i: z = SplitMix64(seed + (i + 1) * 0x9E3779B97F4A7C15) (Steele, Lea and Flood's
//    generator as an output function of a counter), target = floor((z >> 11) T / 2^53),
//    one 64 x 64 -> 128-bit high product.
// 5. b = the largest block with P_b <= target (then target < P_b + S_b: S_b > 0); the
//    outcome is the block's first k whose running sum of P exceeds target - P_b.
//
// Step 3 reads the state once (coalesced, integer work only for complex64; complex128
// computes p_k on the FP64 pipe); each shot reads one block of the state.  The scratch
// arrays stay allocated in the state between calls (2^n / 4 bytes plus the shots).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <string>
#include <type_traits>

#include "ptx.cuh"
#include "sv_internal.h"

namespace svk {

constexpr unsigned long long SM_GAMMA = 0x9E3779B97F4A7C15ull;
constexpr int SCALE_BITS = 58;
constexpr uint32_t SCAN_THREADS = 512, SCAN_ITEMS = 8;   // chunk = 4096 blocks

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// floor(p 2^58) from the IEEE bits of p >= 0.  p = m 2^(e - 150) with m < 2^24; below p = 2
// (e <= 127) the floor is (m 2^35) >> (127 - e), one 64-bit shift.
__device__ __forceinline__ unsigned long long fixed_of(float p) {
    const uint32_t b = __float_as_uint(p);
    const int e = (int)(b >> 23);
    const uint32_t m = e ? (b & 0x7FFFFFu) | 0x800000u : 0u;  // below 2^-126: floor is 0
    if (e > 127) return (unsigned long long)m << (e - 150 + SCALE_BITS);
    return ((unsigned long long)m << 35) >> min(127 - e, 63);
}
__device__ __forceinline__ unsigned long long fixed_of(double p) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(p);
    const int e = (int)(b >> 52);
    if (e == 0) return 0ull;
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);   // p = m 2^(e - 1075)
    const int sh = e - 1075 + SCALE_BITS;
    if (sh >= 0) return m << sh;
    return sh <= -64 ? 0ull : m >> (-sh);
}

// P_k of amplitude k: |alpha|^2 in the state's precision, no contraction.
__device__ __forceinline__ unsigned long long pfix(const float2 *psi, unsigned long long k) {
    const float2 v = psi[k];
    return fixed_of(__fadd_rn(__fmul_rn(v.x, v.x), __fmul_rn(v.y, v.y)));
}
__device__ __forceinline__ unsigned long long pfix(const double2 *psi, unsigned long long k) {
    const double2 v = psi[k];
    return fixed_of(__dadd_rn(__dmul_rn(v.x, v.x), __dmul_rn(v.y, v.y)));
}

// P of the two adjacent amplitudes 2j, 2j + 1 (one 16-byte load for complex64).
__device__ __forceinline__ unsigned long long pfix2(const float2 *psi, unsigned long long j) {
    const float4 v = reinterpret_cast<const float4 *>(psi)[j];
    return fixed_of(__fadd_rn(__fmul_rn(v.x, v.x), __fmul_rn(v.y, v.y))) +
           fixed_of(__fadd_rn(__fmul_rn(v.z, v.z), __fmul_rn(v.w, v.w)));
}
__device__ __forceinline__ unsigned long long pfix2(const double2 *psi, unsigned long long j) {
    return pfix(psi, 2 * j) + pfix(psi, 2 * j + 1);
}

// P of eight adjacent amplitudes in 16-byte loads.
__device__ __forceinline__ void pfix8(const float2 *psi, unsigned long long k, unsigned long long (&p)[8]) {
    const float4 *v = reinterpret_cast<const float4 *>(psi + k);
    float4 w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = v[q];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        p[2 * q] = fixed_of(__fadd_rn(__fmul_rn(w[q].x, w[q].x), __fmul_rn(w[q].y, w[q].y)));
        p[2 * q + 1] = fixed_of(__fadd_rn(__fmul_rn(w[q].z, w[q].z), __fmul_rn(w[q].w, w[q].w)));
    }
}
__device__ __forceinline__ void pfix8(const double2 *psi, unsigned long long k, unsigned long long (&p)[8]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) p[q] = pfix(psi, k + q);
}

// Eight consecutive blocks of B = 64 outcomes per warp and step (two adjacent outcomes of
// each per lane, 4 KiB of complex64 in flight per warp).  The eight sums over 32 lanes are formed
// together: each exchange halves the sums a lane carries, 9 shuffles of 64 bits instead of 40
// (28 qubits, complex64: 484 -> 355 us, 6.1 TB/s).  B < 64 (n < 6): one block, lane l takes outcomes
// l and l + 32.
template <typename C>
__global__ void block_sums(const C *__restrict__ psi, unsigned long long nb, uint32_t B,
                           unsigned long long *__restrict__ S) {
    pass_trigger();
    pass_wait();
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned long long wid = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const unsigned long long nw = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    if (B < 64) {
        if (wid == 0) {
            unsigned long long s = 0;
            if (lane < B) s = pfix(psi, lane);
            if (lane + 32 < B) s += pfix(psi, lane + 32);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) S[0] = s;
        }
        return;
    }
    for (unsigned long long b0 = 8 * wid; b0 < nb; b0 += 8 * nw) {
        unsigned long long s[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) s[u] = b0 + u < nb ? pfix2(psi, (b0 + u) * 32 + lane) : 0ull;
        // lane bits 4, 3, 2 choose the block kept: halves of 4, 2, 1 sums change hands
#pragma unroll
        for (int h = 4, o = 16; h > 0; h >>= 1, o >>= 1) {
            const bool up = (lane & (uint32_t)o) != 0;
#pragma unroll
            for (int u = 0; u < h; ++u) {
                const unsigned long long give = up ? s[u] : s[u + h];
                s[u] = (up ? s[u + h] : s[u]) + __shfl_xor_sync(0xffffffffu, give, o);
            }
        }
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
        const unsigned long long b = b0 + (((lane >> 4) & 1u) * 4u + ((lane >> 3) & 1u) * 2u + ((lane >> 2) & 1u));
        if ((lane & 3u) == 0 && b < nb) S[b] = s[0];
    }
}

// Chunk c of C = SCAN_THREADS x SCAN_ITEMS blocks (or all nb < C): exclusive prefix L of
// its S and its total tot[c], by a shared-memory scan (the sums are exact integers, so
// the order does not matter).
__global__ void __launch_bounds__(SCAN_THREADS) chunk_scan(const unsigned long long *__restrict__ S,
                                                           unsigned long long nb, uint32_t C,
                                                           unsigned long long *__restrict__ L,
                                                           unsigned long long *__restrict__ tot,
                                                           unsigned long long *__restrict__ O) {
    __shared__ unsigned long long part[SCAN_THREADS];
    pass_trigger();
    pass_wait();
    const unsigned long long c = blockIdx.x;
    const unsigned long long base = c * C;
    const uint32_t t = threadIdx.x;
    unsigned long long v[SCAN_ITEMS];
    unsigned long long s = 0;
#pragma unroll
    for (uint32_t i = 0; i < SCAN_ITEMS; ++i) {
        const unsigned long long j = base + (unsigned long long)t * SCAN_ITEMS + i;
        v[i] = (t * SCAN_ITEMS + i < C && j < nb) ? S[j] : 0ull;
        s += v[i];
    }
    part[t] = s;
    __syncthreads();
    for (uint32_t o = 1; o < SCAN_THREADS; o <<= 1) {          // inclusive Hillis-Steele
        const unsigned long long add = t >= o ? part[t - o] : 0ull;
        __syncthreads();
        part[t] += add;
        __syncthreads();
    }
    unsigned long long run = t ? part[t - 1] : 0ull;            // exclusive
#pragma unroll
    for (uint32_t i = 0; i < SCAN_ITEMS; ++i) {
        const unsigned long long j = base + (unsigned long long)t * SCAN_ITEMS + i;
        if (t * SCAN_ITEMS + i < C && j < nb) L[j] = run;
        run += v[i];
    }
    if (t == SCAN_THREADS - 1) {
        tot[c] = part[t];
        if (gridDim.x == 1) {                                   // one chunk: no second scan
            O[0] = 0;
            O[1] = part[t];
        }
    }
}

// One block: O_c = exclusive prefix of the chunk totals, and T at O[nc].
__global__ void __launch_bounds__(1024) chunk_offsets(const unsigned long long *__restrict__ tot,
                                                      unsigned long long nc,
                                                      unsigned long long *__restrict__ O) {
    __shared__ unsigned long long part[1024];
    __shared__ unsigned long long carry;
    pass_trigger();
    pass_wait();
    const uint32_t t = threadIdx.x;
    if (t == 0) carry = 0;
    __syncthreads();
    for (unsigned long long c0 = 0; c0 < nc; c0 += 1024) {
        const unsigned long long j = c0 + t;
        const unsigned long long x = j < nc ? tot[j] : 0ull;
        part[t] = x;
        __syncthreads();
        for (uint32_t o = 1; o < 1024; o <<= 1) {
            const unsigned long long add = t >= o ? part[t - o] : 0ull;
            __syncthreads();
            part[t] += add;
            __syncthreads();
        }
        if (j < nc) O[j] = carry + part[t] - x;
        __syncthreads();
        if (t == 0) carry += part[1023];
        __syncthreads();
    }
    if (t == 0) O[nc] = carry;
}

// One lane per shot finds its block (a binary search over the chunks, then inside one); then
// eight lanes per shot scan the block's 64 outcomes, eight outcomes each, so that the 512 bytes
// of a block arrive in few requests (28 qubits, 2^20 shots: one thread per shot through both
// steps 464 us; 203 with 8-byte loads, bound by L1; 155 with 16-byte ones).
template <typename C>
__global__ void __launch_bounds__(256) draw_shots(const C *__restrict__ psi, const unsigned long long *__restrict__ L,
                           const unsigned long long *__restrict__ O, unsigned long long nb, uint32_t B,
                           uint32_t Cb, unsigned long long nc, unsigned long long seed,
                           unsigned long long nshots, unsigned long long *__restrict__ out, const int *err,
                           unsigned char *mail) {
    pass_trigger();
    pass_wait();
    const unsigned long long T = O[nc];
    if (blockIdx.x == 0 && threadIdx.x == 0) {                   // the call's result: T, the error word
        *reinterpret_cast<unsigned long long *>(mail + svi::WS_RESULT) = T;
        *reinterpret_cast<int *>(mail + svi::WS_ERR) = *err;
    }
    if (T == 0) return;                                          // reported by the host
    const uint32_t lane = threadIdx.x & 31u;
    for (unsigned long long i0 = blockIdx.x * (unsigned long long)blockDim.x + (threadIdx.x & ~31u);
         i0 < nshots; i0 += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long i = i0 + lane;
        const unsigned long long z = splitmix64(seed + (i + 1) * SM_GAMMA);
        const unsigned long long target = __umul64hi((z >> 11) << 11, T);   // floor(u53 T / 2^53)
        // the largest b with P_b = O[b / Cb] + L[b] <= target (P_0 = 0 <= target): first the
        // largest chunk with O_c <= target, then the block in it (L is 0 at its start)
        unsigned long long lo = 0, hi = nc - 1;
        while (lo < hi) {
            const unsigned long long mid = lo + (hi - lo + 1) / 2;
            if (O[mid] <= target) lo = mid;
            else hi = mid - 1;
        }
        unsigned long long r = target - O[lo];
        lo *= Cb;
        hi = min(nb, lo + Cb) - 1;
        while (lo < hi) {
            const unsigned long long mid = lo + (hi - lo + 1) / 2;
            if (L[mid] <= r) lo = mid;
            else hi = mid - 1;
        }
        r -= L[lo];                                              // < S_b
        if (B < 64) {
            unsigned long long c = 0;
            uint32_t k = B - 1;
            for (uint32_t j = 0; j < B; ++j) {
                c += pfix(psi, j);
                if (c > r) {
                    k = j;
                    break;
                }
            }
            if (i < nshots) out[i] = k;
            continue;
        }
        const uint32_t sub = lane & 7u;
#pragma unroll 4
        for (uint32_t it = 0; it < 8; ++it) {
            const int src = (int)(4u * it + (lane >> 3));        // this group's shot
            const unsigned long long b = __shfl_sync(0xffffffffu, lo, src), rs = __shfl_sync(0xffffffffu, r, src);
            unsigned long long p[8], sum = 0;
            pfix8(psi, b * 64 + sub * 8, p);
#pragma unroll
            for (uint32_t j = 0; j < 8; ++j) sum += p[j];
            unsigned long long end = sum;                        // inclusive prefix over the group
#pragma unroll
            for (uint32_t o = 1; o < 8; o <<= 1) {
                const unsigned long long up = __shfl_up_sync(0xffffffffu, end, o, 8);
                if (sub >= o) end += up;
            }
            unsigned long long c = end - sum;
            if (c <= rs && rs < end && i0 + (unsigned)src < nshots) {
                uint32_t k = 0;
#pragma unroll
                for (uint32_t j = 0; j < 8; ++j) {
                    c += p[j];
                    k += c <= rs;
                }
                out[i0 + (unsigned)src] = b * 64 + sub * 8 + k;
            }
        }
    }
}

}  // namespace svk

using namespace svi;

extern "C" sv_status sv_sample(sv_state *s, uint64_t seed, size_t nshots, uint64_t *out,
                               int out_on_device) {
    clear_error();
    if (!s || !out) return set_error(SV_ERR_ARG, "sv_sample: null argument");
    if (check_live(s, "sv_sample") != SV_OK) return SV_ERR_STATE;
    if (nshots == 0) return SV_OK;
    const unsigned long long N = 1ull << s->n;
    const uint32_t B = (uint32_t)std::min<unsigned long long>(64, N);
    const unsigned long long nb = N / B;
    const uint32_t Cb = (uint32_t)std::min<unsigned long long>(svk::SCAN_THREADS * svk::SCAN_ITEMS, nb);
    const unsigned long long nc = (nb + Cb - 1) / Cb;
    cudaStream_t st = s->stream;
    sv_status rc = SV_OK;
    auto fail = [&](cudaError_t e, const char *what) {
        if (rc == SV_OK && e != cudaSuccess)
            rc = set_error(e == cudaErrorMemoryAllocation ? SV_ERR_OOM : SV_ERR_CUDA,
                           std::string("sv_sample: ") + what + ": " + cudaGetErrorString(e));
    };
    // scratch S, L, tot, O (and the shots for host output), kept in the state across calls
    const size_t words = 2 * nb + 2 * nc + 1 + (out_on_device ? 0 : nshots);
    if (s->samp_cap < words * sizeof(unsigned long long)) {
        SV_CUDA(cudaStreamSynchronize(st));
        if (s->samp) cudaFree(s->samp);
        s->samp = nullptr;
        s->samp_cap = 0;
        SV_CUDA(cudaMalloc(&s->samp, words * sizeof(unsigned long long)));
        s->samp_cap = words * sizeof(unsigned long long);
    }
    unsigned long long *S = static_cast<unsigned long long *>(s->samp);
    unsigned long long *L = S + nb, *tot = L + nb, *O = tot + nc;
    unsigned long long *dout = out_on_device ? nullptr : O + nc + 1;
    if (rc == SV_OK) {
        const unsigned grid = (unsigned)std::min<unsigned long long>((nb * 4 + 255) / 256,
                                                                     (unsigned long long)s->num_sms * 16);
        unsigned long long *dst = out_on_device ? reinterpret_cast<unsigned long long *>(out) : dout;
        const unsigned dgrid = (unsigned)std::min<unsigned long long>((nshots + 255) / 256,
                                                                      (unsigned long long)s->num_sms * 32);
        auto enqueue = [&](auto *psi) {
            using C = std::remove_pointer_t<decltype(psi)>;
            fail(svk::launch_pass(svk::block_sums<C>, dim3(grid), 256, 0, st, psi, nb, B, S), "block sums");
            fail(svk::launch_pass(svk::chunk_scan, dim3((unsigned)nc), svk::SCAN_THREADS, 0, st, S, nb, Cb, L, tot, O),
                 "chunk scan");
            if (nc > 1) fail(svk::launch_pass(svk::chunk_offsets, dim3(1), 1024, 0, st, tot, nc, O), "chunk offsets");
            fail(svk::launch_pass(svk::draw_shots<C>, dim3(dgrid), 256, 0, st, psi, L, O, nb, B, Cb, nc,
                                  (unsigned long long)seed, (unsigned long long)nshots, dst, device_error(s),
                                  s->mail_dev),
                 "shots");
        };
        if (s->dtype == SV_C64) enqueue(reinterpret_cast<float2 *>(s->buf));
        else enqueue(reinterpret_cast<double2 *>(s->buf));
    }
    if (rc != SV_OK) return rc;
    unsigned long long T = 0;
    rc = read_results(s, &T, sizeof(T));
    if (rc != SV_OK) return rc;
    if (T == 0) return set_error(SV_ERR_STATE, "sv_sample: the state has no probability mass to sample");
    if (!out_on_device) {
        SV_CUDA(cudaMemcpyAsync(out, dout, nshots * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
        SV_CUDA(cudaStreamSynchronize(st));
    }
    return SV_OK;
}
