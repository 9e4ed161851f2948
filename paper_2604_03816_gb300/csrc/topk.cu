// The 64 most probable outcomes, p descending, ties to the lower index (Eq. 1; the backend's
// measurement operation of Section 4.1 reduced to its head).
//
// Selection by maxima: if the amplitudes are cut into chunks, the 64 best outcomes lie in the
// 64 chunks with the best (maximum, then lowest chunk) -- any other chunk's outcomes come after
// the 64 maxima of those.  So
//   1. chunk_max reads the state once and keeps the largest p of every chunk (and, from 23
//      qubits, of every 64 chunks);
//   2. topk_select, one block, narrows 64 groups -> 64 chunks -> 64 sub-chunks of 16 -> 64
//      outcomes.  Each step picks 64 of at most 4096 keys held in registers: the 64th largest
//      key by building its bits from the top (one block-wide count per two bits, until a count
//      is exactly 64), ties by position.
// States of up to 16 qubits take step 2 alone.  Step 1 is one HBM read with a max per amplitude;
// the per-warp insertion lists it replaces spent most of their time inserting (28 qubits,
// complex64: 938 + 447 us -> 295 + 30; 13 qubits: 144 + 146 -> 16).
//
// Keys are the bits of p, plus one so that 0 means "no outcome": they order like the values.
// p is formed in the state's precision without contraction (prob_of), so a host that does the
// same IEEE operations takes the same decisions.  complex64 outcomes whose p is NaN are not
// listed; complex128 ones come first.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "ptx.cuh"
#include "reduce.cuh"
#include "sv_internal.h"

namespace svt {

constexpr uint32_t K = 64;
constexpr uint32_t SEL_THREADS = 1024;

template <typename R> struct Ty;
template <> struct Ty<float> {
    using C = float2;
    using Key = uint32_t;
    __device__ static Key key(float2 v) {
        const float p = svk::prob_of(v.x, v.y);
        return p >= 0.f ? __float_as_uint(p) + 1u : 0u;      // NaN: no outcome
    }
    __device__ static double value(Key k) { return (double)__uint_as_float(k - 1u); }
};
template <> struct Ty<double> {
    using C = double2;
    using Key = unsigned long long;
    __device__ static Key key(double2 v) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(svk::prob_of(v.x, v.y));
        return (b >> 63) ? 0ull : b + 1ull;
    }
    __device__ static double value(Key k) { return __longlong_as_double((long long)(k - 1ull)); }
};

// Largest key of this lane's 16 bytes: amplitudes 2 i, 2 i + 1 (complex64) or i (complex128).
__device__ __forceinline__ uint32_t lane_key(const float4 &v) {
    return max(Ty<float>::key(make_float2(v.x, v.y)), Ty<float>::key(make_float2(v.z, v.w)));
}
__device__ __forceinline__ unsigned long long lane_key(const double2 &v) { return Ty<double>::key(v); }
template <typename R> struct Vec;
template <> struct Vec<float> { using T = float4; };
template <> struct Vec<double> { using T = double2; };

// fine[c] = the largest key of chunk c (2^lf amplitudes, lf >= 10), one warp per chunk;
// coarse[c / 64] (zeroed before) = the largest of 64 chunks, if coarse is given.
template <typename R>
__global__ void __launch_bounds__(256) chunk_max(const typename Vec<R>::T *__restrict__ v, uint32_t lf,
                                                 unsigned long long nchunks, typename Ty<R>::Key *fine,
                                                 typename Ty<R>::Key *coarse) {
    using Key = typename Ty<R>::Key;
    svk::pass_trigger();
    svk::pass_wait();
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned long long nw = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    const unsigned long long per = (sizeof(R) == 4 ? 1ull : 2ull) << (lf - 1);     // 16-byte words of a chunk
    for (unsigned long long c = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
         c < nchunks; c += nw) {
        const typename Vec<R>::T *p = v + c * per;
        Key m = 0;
        for (unsigned long long i = lane; i < per; i += 256) {
            typename Vec<R>::T w[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) w[q] = p[i + 32ull * q];
#pragma unroll
            for (int q = 0; q < 8; ++q) m = max(m, lane_key(w[q]));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) {
            fine[c] = m;
            if (coarse) atomicMax(coarse + (c >> 6), m);
        }
    }
}

struct Shared {
    uint32_t count[2][32];       // the warps' counts of a bit-search step
    uint32_t warp_sum[32];
    uint32_t total;
    uint32_t sel[K];             // selected positions, ascending
    unsigned long long list[2][K];   // chunks (then sub-chunks) in play, ascending
};

// Positions (4 tid + j) of the 64 largest nonzero keys, ties to the lower position, ascending
// into sh.sel; returns how many there are (at most 64).
template <typename Key>
__device__ uint32_t select64(const Key (&k)[4], Shared &sh) {
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    constexpr int STEPS = 4 * (int)sizeof(Key);      // two bits per step
    Key T = 0;
    for (int b = STEPS - 1; b >= 0; --b) {
        // counts of keys at or above the three larger candidates, 10 bits each over a warp; the
        // warps' counts pass through shared memory (two copies: one barrier per step)
        uint32_t c = 0;
#pragma unroll
        for (uint32_t d = 1; d < 4; ++d) {
            const Key cand = T | (Key(d) << (2 * b));
#pragma unroll
            for (int j = 0; j < 4; ++j) c += (k[j] >= cand ? 1u : 0u) << (10 * (d - 1));
        }
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) sh.count[b & 1][warp] = c;
        __syncthreads();
        c = sh.count[b & 1][lane];
        const uint32_t n12 = __reduce_add_sync(0xffffffffu, (c & 1023u) | ((c >> 10) & 1023u) << 16);
        const uint32_t n[4] = {0, n12 & 0xFFFFu, n12 >> 16, __reduce_add_sync(0xffffffffu, c >> 20)};
        uint32_t d = 0, got = 0;
#pragma unroll
        for (uint32_t q = 1; q < 4; ++q) {
            if (n[q] >= K) {
                d = q;
                got = n[q];
            }
        }
        T |= Key(d) << (2 * b);
        if (got == K) break;
    }
    if (T == 0) T = 1;                               // fewer than 64 keys: all of them
    // counts of keys above and at T, scanned over the block in position order
    uint32_t mine = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) mine += k[j] > T ? 1u : (k[j] == T ? 0x10000u : 0u);
    uint32_t inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= (uint32_t)o) inc += up;
    }
    if (lane == 31) sh.warp_sum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = sh.warp_sum[lane], s = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t up = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= (uint32_t)o) s += up;
        }
        sh.warp_sum[lane] = s - w;
        if (lane == 31) sh.total = s;
    }
    __syncthreads();
    const uint32_t total = sh.total, gt = total & 0xFFFFu, limit = K - min(gt, K);   // ties taken
    uint32_t before = sh.warp_sum[warp] + inc - mine;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t g = before & 0xFFFFu, e = before >> 16;
        const bool above = k[j] > T, at = k[j] == T;
        if (above || (at && e < limit)) sh.sel[g + min(e, limit)] = 4u * tid + (uint32_t)j;
        before += above ? 1u : (at ? 0x10000u : 0u);
    }
    __syncthreads();
    return min(K, gt + min(total >> 16, limit));
}

struct SelectArgs {
    const void *psi;
    const void *fine, *coarse;           // chunk_max's maxima, or null
    unsigned long long nchunks;          // chunks in all (without maxima: at most 64, or one)
    uint32_t lf, ncoarse;
    double *out_p;
    unsigned long long *out_i;
    const int *err;                      // error word and where it goes (or null)
    int *mail;
};

template <typename R>
__global__ void __launch_bounds__(SEL_THREADS) topk_select(const __grid_constant__ SelectArgs a) {
    using C = typename Ty<R>::C;
    using Key = typename Ty<R>::Key;
    using V = typename Vec<R>::T;
    __shared__ Shared sh;
    __shared__ Key sub[4096];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const Key *fine = reinterpret_cast<const Key *>(a.fine), *coarse = reinterpret_cast<const Key *>(a.coarse);
    svk::pass_trigger();
    svk::pass_wait();
    if (tid == 0 && a.mail) *a.mail = *a.err;
    uint32_t cur = 0, nl;                // list in use, its length
    Key k[4];
    if (coarse) {
#pragma unroll
        for (int j = 0; j < 4; ++j) k[j] = 4u * tid + j < a.ncoarse ? coarse[4u * tid + j] : Key(0);
        nl = select64(k, sh);
        if (tid < nl) sh.list[0][tid] = sh.sel[tid];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t q = 4u * tid + j;
            k[j] = (q >> 6) < nl ? fine[sh.list[0][q >> 6] * 64ull + (q & 63u)] : Key(0);
        }
        nl = select64(k, sh);
        if (tid < nl) sh.list[1][tid] = sh.list[0][sh.sel[tid] >> 6] * 64ull + (sh.sel[tid] & 63u);
        cur = 1;
    } else if (fine) {
#pragma unroll
        for (int j = 0; j < 4; ++j) k[j] = 4u * tid + j < a.nchunks ? fine[4u * tid + j] : Key(0);
        nl = select64(k, sh);
        if (tid < nl) sh.list[0][tid] = sh.sel[tid];
    } else {
        nl = (uint32_t)a.nchunks;
        if (tid < nl) sh.list[0][tid] = tid;
    }
    // chunks of 2^lf amplitudes -> sub-chunks of 2^ls, until 64 chunks are at most 4096 outcomes
    uint32_t lf = a.lf;
    while (nl > 1 ? lf > 6 : lf > 12) {
        const uint32_t ls = lf > 10 ? lf - 6 : 4, lper = lf - ls;     // 2^lper sub-chunks per chunk
        for (uint32_t q = tid; q < 4096; q += SEL_THREADS) sub[q] = 0;
        __syncthreads();
        // a warp reads 32 16-byte words at a time (2^lu amplitudes); lanes of one group of 16
        // amplitudes, all in one sub-chunk, reduce first
        constexpr uint32_t lu = sizeof(R) == 4 ? 6 : 5, group = sizeof(R) == 4 ? 8 : 16;
        const uint32_t lun = lf - lu;                                  // units per chunk
        const uint32_t units = nl << lun;
        for (uint32_t u0 = warp; u0 < units; u0 += 8 * 32) {
            V w[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint32_t u = u0 + 32u * q;
                if (u < units)
                    w[q] = reinterpret_cast<const V *>(a.psi)[(((sh.list[cur][u >> lun] << lf) +
                                                                ((unsigned long long)(u & ((1u << lun) - 1u)) << lu)) >>
                                                               (lu - 5)) + lane];
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint32_t u = u0 + 32u * q;
                Key m = u < units ? lane_key(w[q]) : Key(0);
#pragma unroll
                for (uint32_t o = group / 2; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
                if (u < units && (lane & (group - 1u)) == 0) {
                    const uint32_t at = ((u & ((1u << lun) - 1u)) << lu) + ((lane / group) << 4);
                    atomicMax(&sub[((u >> lun) << lper) + (at >> ls)], m);
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) k[j] = sub[4u * tid + j];
        const uint32_t ns = select64(k, sh);
        if (tid < ns)
            sh.list[cur ^ 1u][tid] = (sh.list[cur][sh.sel[tid] >> lper] << lper) + (sh.sel[tid] & ((1u << lper) - 1u));
        cur ^= 1u;
        nl = ns;
        lf = ls;
        __syncthreads();
    }
    __syncthreads();
    // outcomes: position q is amplitude q mod 2^lf of chunk q / 2^lf
    const C *psi = reinterpret_cast<const C *>(a.psi);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t q = 4u * tid + j;
        k[j] = (q >> lf) < nl ? Ty<R>::key(psi[(sh.list[cur][q >> lf] << lf) + (q & ((1u << lf) - 1u))]) : Key(0);
    }
    const uint32_t m = select64(k, sh);
    // the selected keys and indices by selection order, then by rank
    unsigned long long *idx = sh.list[cur ^ 1u];
#pragma unroll
    for (int j = 0; j < 4; ++j) sub[4u * tid + j] = k[j];
    __syncthreads();
    Key mine = 0;
    if (tid < m) {
        const uint32_t q = sh.sel[tid];
        mine = sub[q];
        idx[tid] = (sh.list[cur][q >> lf] << lf) + (q & ((1u << lf) - 1u));
    }
    __syncthreads();
    if (tid < K) {
        if (tid < m) sub[tid] = mine;
    }
    __syncthreads();
    if (tid < m) {
        uint32_t rank = 0;
        for (uint32_t i = 0; i < m; ++i) rank += sub[i] > mine || (sub[i] == mine && i < tid);
        a.out_p[rank] = Ty<R>::value(mine);
        a.out_i[rank] = idx[tid];
    } else if (tid < K) {
        a.out_p[tid] = -1.0;
        a.out_i[tid] = ~0ull;
    }
}

}  // namespace svt

namespace svi {

template <typename R>
static sv_status topk_t(sv_state *s, double *out, int *mail) {
    using Key = typename svt::Ty<R>::Key;
    using V = typename svt::Vec<R>::T;
    svt::SelectArgs a;
    a.psi = s->buf;
    a.fine = a.coarse = nullptr;
    a.ncoarse = 0;
    a.out_p = out;
    a.out_i = reinterpret_cast<unsigned long long *>(out) + 64;
    a.err = device_error(s);
    a.mail = mail;
    // up to 12 qubits the outcomes themselves are the keys; up to 16 there are at most 64 chunks
    // of 1024; above, chunks of 1024 (from 29 qubits 2^(n - 18), so that there are at most 2^18)
    a.lf = s->n <= 12 ? s->n : std::max(10u, s->n > 18 ? s->n - 18 : 0u);
    a.nchunks = 1ull << (s->n - a.lf);
    if (s->n > 16) {
        Key *fine = reinterpret_cast<Key *>(s->ws + WS_TOPK);
        Key *coarse = nullptr;
        if (a.nchunks > 4096) {
            coarse = fine + a.nchunks;
            a.ncoarse = (uint32_t)(a.nchunks >> 6);
            SV_CUDA(cudaMemsetAsync(coarse, 0, a.ncoarse * sizeof(Key), s->stream));
        }
        const unsigned blocks = (unsigned)std::min<unsigned long long>((a.nchunks + 7) / 8, 8ull * s->num_sms);
        SV_CUDA(svk::launch_pass(svt::chunk_max<R>, dim3(blocks), 256, 0, s->stream,
                                 reinterpret_cast<const V *>(s->buf), a.lf, a.nchunks, fine, coarse));
        a.fine = fine;
        a.coarse = coarse;
    }
    SV_CUDA(svk::launch_pass(svt::topk_select<R>, dim3(1), svt::SEL_THREADS, 0, s->stream, a));
    return SV_OK;
}

// The top 64 as p[64], index[64] at `out`; empty places hold (-1, ~0).
static sv_status enqueue_topk_to(sv_state *s, double *out, int *mail) {
    return s->dtype == SV_C64 ? topk_t<float>(s, out, mail) : topk_t<double>(s, out, mail);
}

// Enqueue the top-64 search and asynchronous copies of the 64 (p, index) pairs, best
// first, into host_p / host_i (pinned memory for a truly asynchronous copy).
sv_status enqueue_topk(sv_state *s, double *host_p, unsigned long long *host_i) {
    double *r = reinterpret_cast<double *>(s->ws + WS_RESULT);
    const sv_status st = enqueue_topk_to(s, r, nullptr);
    if (st != SV_OK) return st;
    SV_CUDA(cudaMemcpyAsync(host_p, r, 64 * 8, cudaMemcpyDeviceToHost, s->stream));
    SV_CUDA(cudaMemcpyAsync(host_i, r + 64, 64 * 8, cudaMemcpyDeviceToHost, s->stream));
    return SV_OK;
}

sv_status launch_topk(sv_state *s, uint32_t k, uint64_t *idx, double *p) {
    sv_status st = enqueue_topk_to(s, mail_results(s), mail_error(s));
    if (st != SV_OK) return st;
    unsigned char h[128 * 8];
    st = read_results(s, h, sizeof(h));
    if (st != SV_OK) return st;
    const uint32_t m = (uint32_t)std::min<unsigned long long>(k, 1ull << s->n);
    std::memcpy(p, h, m * sizeof(double));
    std::memcpy(idx, h + 64 * 8, m * sizeof(uint64_t));
    return SV_OK;
}

}  // namespace svi
