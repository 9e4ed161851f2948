// Read-only reductions over the state: norm (Eq. 1), Z-basis probabilities and the general Pauli
// expectations (the ones that share reads are in expect.cu, the top-k outcomes in topk.cu), plus the
// small initialisation kernels.
//
// Every reduction reads the state once with 16-byte vector loads from a fixed-size
// grid (so the partial-sum layout, and therefore the FP64 result, is the same on every
// run), folds per-thread values in FP64, reduces each block with warp shuffles and
// finishes with a single-block pass over the block partials in a fixed order.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "ptx.cuh"
#include "reduce.cuh"
#include "sv_internal.h"

namespace svk {

// ---------------------------------------------------------------- norm

// err, mail: a single block's sum is the result; the error word goes with it (else null).
__global__ void norm_c64(const float4 *__restrict__ v, unsigned long long nvec, double *partial, const int *err,
                         int *mail) {
    pass_trigger();
    pass_wait();
    double acc = 0.0;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 3 * stride < nvec; i += 4 * stride) {
        float4 a = v[i], b = v[i + stride], c = v[i + 2 * stride], d = v[i + 3 * stride];
        const float sa = __fadd_rn(prob_of(a.x, a.y), prob_of(a.z, a.w));
        const float sb = __fadd_rn(prob_of(b.x, b.y), prob_of(b.z, b.w));
        const float sc = __fadd_rn(prob_of(c.x, c.y), prob_of(c.z, c.w));
        const float sd = __fadd_rn(prob_of(d.x, d.y), prob_of(d.z, d.w));
        // eight amplitudes summed pairwise in FP32, one FP64 operation per eight (the FP64
        // pipe of this GPU runs at about 1/64 of the FP32 rate)
        acc += (double)__fadd_rn(__fadd_rn(sa, sb), __fadd_rn(sc, sd));
    }
    for (; i < nvec; i += stride) {
        float4 a = v[i];
        acc += (double)__fadd_rn(prob_of(a.x, a.y), prob_of(a.z, a.w));
    }
    const double r = block_sum(acc);
    if (threadIdx.x == 0) {
        partial[blockIdx.x] = r;
        if (mail) *mail = *err;
    }
}

__global__ void norm_c128(const double2 *__restrict__ v, unsigned long long n, double *partial, const int *err,
                          int *mail) {
    pass_trigger();
    pass_wait();
    double acc = 0.0;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n; i += 4 * stride) {
        double2 a = v[i], b = v[i + stride], c = v[i + 2 * stride], d = v[i + 3 * stride];
        acc += prob_of(a.x, a.y) + prob_of(b.x, b.y) + prob_of(c.x, c.y) + prob_of(d.x, d.y);
    }
    for (; i < n; i += stride) acc += prob_of(v[i].x, v[i].y);
    const double r = block_sum(acc);
    if (threadIdx.x == 0) {
        partial[blockIdx.x] = r;
        if (mail) *mail = *err;
    }
}

// out[0] = sum of partial[0..n) in a fixed order (one block); *mail = *err if given.
__global__ void sum_partials(const double *partial, int n, double *out, const int *err, int *mail) {
    pass_trigger();
    pass_wait();
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) acc += partial[i];
    const double r = block_sum(acc);
    if (threadIdx.x == 0) {
        out[0] = r;
        if (mail) *mail = *err;
    }
}

// ---------------------------------------------------------------- probabilities

__global__ void probs_c64(const float4 *__restrict__ v, unsigned long long nvec, float2 *out) {
    pass_trigger();
    pass_wait();
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < nvec;
         i += stride) {
        const float4 a = v[i];
        out[i] = make_float2(prob_of(a.x, a.y), prob_of(a.z, a.w));
    }
}

__global__ void probs_c128(const double2 *__restrict__ v, unsigned long long n, double *out) {
    pass_trigger();
    pass_wait();
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += stride)
        out[i] = prob_of(v[i].x, v[i].y);
}

// Diagonal of a density matrix held as the 2m-qubit vector v[r + 2^m c] = rho[r, c]:
// p(x) = Re rho[x, x] = Re v[x (2^m + 1)], in the state's precision.
template <typename C, typename R>
__global__ void density_diag(const C *__restrict__ v, uint32_t m, R *__restrict__ out) {
    const unsigned long long M = 1ull << m;
    for (unsigned long long x = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; x < M;
         x += (unsigned long long)gridDim.x * blockDim.x)
        out[x] = v[x * (M + 1)].x;
}

// ---------------------------------------------------------------- Pauli expectation

constexpr int EXP_MAX_TERMS = 32;

// Terms sharing one X-part x.  cc = coef * i^{|x & z|} (complex, FP64).
struct ExpectArgs {
    unsigned long long x;
    unsigned long long z[EXP_MAX_TERMS];
    double ccr[EXP_MAX_TERMS], cci[EXP_MAX_TERMS];
    int nterms;
    int hb;                   // highest set bit of x (x != 0)
    unsigned long long npairs;
};

// sum_k Re[ conj(psi[k ^ x]) psi[k] w(k) ],  w(k) = sum_t cc_t (-1)^{|k & z_t|}.
// x = 0: sum_k |psi_k|^2 Re w(k).  x != 0: the pair (k, k ^ x) with bit hb of k clear
// contributes both of its orderings.
template <typename R>
__global__ void expect_kernel(const __grid_constant__ ExpectArgs a, const void *psi_, double *partial) {
    using C = typename std::conditional<sizeof(R) == 4, float2, double2>::type;
    const C *psi = reinterpret_cast<const C *>(psi_);
    double acc = 0.0;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
         i < a.npairs; i += stride) {
        if (a.x == 0) {
            const C v = psi[i];
            double w = 0.0;
            for (int t = 0; t < a.nterms; ++t)
                w += (__popcll(i & a.z[t]) & 1) ? -a.ccr[t] : a.ccr[t];
            acc += w * (double)prob_of(v.x, v.y);
        } else {
            const unsigned long long k = insert_zero64(i, (uint32_t)a.hb), k2 = k ^ a.x;
            const C p = psi[k], q = psi[k2];
            // conj(q) p and conj(p) q = conj(conj(q) p)
            const double re = (double)q.x * p.x + (double)q.y * p.y;
            const double im = (double)q.x * p.y - (double)q.y * p.x;
            double w1r = 0, w1i = 0, w2r = 0, w2i = 0;
            for (int t = 0; t < a.nterms; ++t) {
                const bool s1 = __popcll(k & a.z[t]) & 1, s2 = __popcll(k2 & a.z[t]) & 1;
                w1r += s1 ? -a.ccr[t] : a.ccr[t];
                w1i += s1 ? -a.cci[t] : a.cci[t];
                w2r += s2 ? -a.ccr[t] : a.ccr[t];
                w2i += s2 ? -a.cci[t] : a.cci[t];
            }
            // Re[(re + i im) w1] + Re[(re - i im) w2]
            acc += re * w1r - im * w1i + re * w2r + im * w2i;
        }
    }
    const double r = block_sum(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = r;
}

// complex64, up to NT terms of one X-part x != 0: per term FP32 partial sums over runs of
// eight pairs, one FP64 step per run and term.  With s_t(k) = (-1)^{|k & z_t|} and
// cc_t = ccr_t + i cci_t, the pair (k, k2 = k ^ x) with bit hb of k clear and
// c = conj(psi_k2) psi_k = re + i im contributes ccr_t (s_t(k) + s_t(k2)) re - cci_t (s_t(k) -
// s_t(k2)) im.
template <int NT>
__global__ void expect_c64(const __grid_constant__ ExpectArgs a, const float2 *__restrict__ psi,
                           double *partial) {
    double A[NT], B[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) A[t] = B[t] = 0.0;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long i0 = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
         i0 < a.npairs; i0 += 8 * stride) {
        float sa[NT], sb[NT];
#pragma unroll
        for (int t = 0; t < NT; ++t) sa[t] = sb[t] = 0.f;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const unsigned long long i = i0 + r * stride;
            if (i >= a.npairs) break;
            const unsigned long long k = insert_zero64(i, (uint32_t)a.hb), k2 = k ^ a.x;
            const float2 p = psi[k], q = psi[k2];
            const float re = __fadd_rn(__fmul_rn(q.x, p.x), __fmul_rn(q.y, p.y));
            const float im = __fsub_rn(__fmul_rn(q.x, p.y), __fmul_rn(q.y, p.x));
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const bool s1 = __popcll(k & a.z[t]) & 1, s2 = __popcll(k2 & a.z[t]) & 1;
                if (s1 == s2) sa[t] = __fadd_rn(sa[t], s1 ? -2.f * re : 2.f * re);
                else sb[t] = __fadd_rn(sb[t], s1 ? -2.f * im : 2.f * im);
            }
        }
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            A[t] += (double)sa[t];
            B[t] += (double)sb[t];
        }
    }
    double acc = 0.0;
#pragma unroll
    for (int t = 0; t < NT; ++t) acc += a.ccr[t] * A[t] - a.cci[t] * B[t];
    const double r = block_sum(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = r;
}

// ---------------------------------------------------------------- init helpers

__global__ void set_amp_one(void *psi, unsigned long long x, int is_c128) {
    if (is_c128) reinterpret_cast<double2 *>(psi)[x] = make_double2(1.0, 0.0);
    else reinterpret_cast<float2 *>(psi)[x] = make_float2(1.0f, 0.0f);
}

// |x> of a small state in one launch: 16-byte words, zero but for the amplitude of x.
__global__ void set_basis_small(uint4 *psi, unsigned long long words, unsigned long long x, int is_c128) {
    pass_trigger();
    pass_wait();
    const unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= words) return;
    uint4 w = make_uint4(0, 0, 0, 0);
    if (is_c128) {
        if (i == x) w.y = (uint32_t)__double2hiint(1.0);
    } else if (i == x >> 1) {
        (x & 1 ? w.z : w.x) = __float_as_uint(1.f);
    }
    psi[i] = w;
}

__global__ void widen_kernel(const float2 *__restrict__ src, double2 *__restrict__ dst,
                             unsigned long long n) {
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += stride)
        dst[i] = make_double2((double)src[i].x, (double)src[i].y);
}

}  // namespace svk

namespace svi {

static int red_blocks(const sv_state *s) { return std::min(WS_NPARTIAL, s->num_sms * 8); }

sv_status enqueue_sum(sv_state *s, int n, double *dev_out) {
    SV_CUDA(svk::launch_pass(svk::sum_partials, dim3(1), svk::RED_THREADS, 0, s->stream,
                             reinterpret_cast<double *>(s->ws + WS_PARTIAL), n, dev_out, device_error(s),
                             mail_error(s)));
    return SV_OK;
}

sv_status launch_norm(sv_state *s, double *dev_out) {
    double *partial = reinterpret_cast<double *>(s->ws + WS_PARTIAL);
    const unsigned long long N = 1ull << s->n;
    // fixed by n, so the sum's order is; at least four 16-byte words per thread
    const unsigned long long words = (N * (s->dtype == SV_C64 ? 8 : 16)) / 16;
    const int nb = (int)std::min<unsigned long long>(red_blocks(s), std::max(1ull, words / (4 * svk::RED_THREADS)));
    int *mail = nb == 1 ? mail_error(s) : nullptr;
    if (nb == 1) partial = dev_out;
    if (s->dtype == SV_C64)
        SV_CUDA(svk::launch_pass(svk::norm_c64, dim3(nb), svk::RED_THREADS, 0, s->stream,
                                 reinterpret_cast<const float4 *>(s->buf), N / 2, partial, device_error(s), mail));
    else
        SV_CUDA(svk::launch_pass(svk::norm_c128, dim3(nb), svk::RED_THREADS, 0, s->stream,
                                 reinterpret_cast<const double2 *>(s->buf), N, partial, device_error(s), mail));
    return nb == 1 ? SV_OK : enqueue_sum(s, nb, dev_out);
}

sv_status launch_probs(sv_state *s, void *dev_out) {
    const unsigned long long N = 1ull << s->n;
    const int nb = (int)std::min<unsigned long long>(s->num_sms * 8, (N + 511) / 512);
    if (s->dtype == SV_C64)
        SV_CUDA(svk::launch_pass(svk::probs_c64, dim3(nb), 256, 0, s->stream, reinterpret_cast<const float4 *>(s->buf),
                                 N / 2, reinterpret_cast<float2 *>(dev_out)));
    else
        SV_CUDA(svk::launch_pass(svk::probs_c128, dim3(nb), 256, 0, s->stream,
                                 reinterpret_cast<const double2 *>(s->buf), N, reinterpret_cast<double *>(dev_out)));
    return SV_OK;
}

sv_status launch_density_probs(sv_state *s, void *dev_out) {
    const uint32_t m = s->n / 2;
    const int nb = s->num_sms * 8;
    if (s->dtype == SV_C64)
        svk::density_diag<<<nb, 256, 0, s->stream>>>(reinterpret_cast<const float2 *>(s->buf), m,
                                                     reinterpret_cast<float *>(dev_out));
    else
        svk::density_diag<<<nb, 256, 0, s->stream>>>(reinterpret_cast<const double2 *>(s->buf), m,
                                                     reinterpret_cast<double *>(dev_out));
    SV_CUDA(cudaGetLastError());
    return SV_OK;
}

// One X-part's terms (at most 32) by the general kernels, the sum into *dev_out.
sv_status enqueue_expect_group(sv_state *s, uint64_t x, const uint64_t *z, const double *c, int nterms,
                               double *dev_out) {
    double *partial = reinterpret_cast<double *>(s->ws + WS_PARTIAL);
    const int nb = red_blocks(s);
    svk::ExpectArgs a;
    std::memset(&a, 0, sizeof(a));
    a.x = x;
    a.nterms = nterms;
    for (int t = 0; t < nterms; ++t) {
        const int y = __builtin_popcountll(x & z[t]) & 3;   // i^y
        const double re[4] = {1, 0, -1, 0}, im[4] = {0, 1, 0, -1};
        a.z[t] = z[t];
        a.ccr[t] = c[t] * re[y];
        a.cci[t] = c[t] * im[y];
    }
    a.hb = x ? 63 - __builtin_clzll(x) : 0;
    a.npairs = x ? 1ull << (s->n - 1) : 1ull << s->n;
    if (s->dtype == SV_C64 && x != 0 && nterms <= 4) {
        const float2 *v = reinterpret_cast<const float2 *>(s->buf);
        switch (nterms) {
            case 1: svk::expect_c64<1><<<nb, svk::RED_THREADS, 0, s->stream>>>(a, v, partial); break;
            case 2: svk::expect_c64<2><<<nb, svk::RED_THREADS, 0, s->stream>>>(a, v, partial); break;
            case 3: svk::expect_c64<3><<<nb, svk::RED_THREADS, 0, s->stream>>>(a, v, partial); break;
            default: svk::expect_c64<4><<<nb, svk::RED_THREADS, 0, s->stream>>>(a, v, partial);
        }
    } else if (s->dtype == SV_C64) {
        svk::expect_kernel<float><<<nb, svk::RED_THREADS, 0, s->stream>>>(a, s->buf, partial);
    } else {
        svk::expect_kernel<double><<<nb, svk::RED_THREADS, 0, s->stream>>>(a, s->buf, partial);
    }
    SV_CUDA(cudaGetLastError());
    return enqueue_sum(s, nb, dev_out);
}

// Enqueue sum_t coef[t] <P_t> for a raw device state into *out_dev, with block partials
// in caller-provided scratch (nb_fixed doubles per batch of up to EXP_MAX_TERMS terms
// sharing one X-part).  Uses no heap memory: the term order lives on the stack, so
// nterms is limited to ENQ_MAX_TERMS.  SV_ERR_ARG if the batches need more scratch.
sv_status enqueue_expect_sum(const void *psi, uint32_t n, sv_dtype dtype, const uint64_t *x,
                             const uint64_t *z, const double *c, size_t nterms, double *scratch,
                             size_t scratch_doubles, int nb_fixed, double *out_dev,
                             cudaStream_t stream) {
    constexpr size_t ENQ_MAX_TERMS = 2048;
    if (nterms > ENQ_MAX_TERMS)
        return set_error(SV_ERR_ARG, "expectation: at most 2048 terms per call");
    if (nterms == 0) {
        SV_CUDA(cudaMemsetAsync(out_dev, 0, sizeof(double), stream));
        return SV_OK;
    }
    uint16_t order[ENQ_MAX_TERMS];
    for (size_t i = 0; i < nterms; ++i) {          // stable insertion sort by X-part
        size_t j = i;
        while (j > 0 && x[order[j - 1]] > x[i]) {
            order[j] = order[j - 1];
            --j;
        }
        order[j] = (uint16_t)i;
    }
    size_t nbatches = 0;
    for (size_t i = 0, run = 0; i < nterms; ++i) {
        run = (i > 0 && x[order[i]] == x[order[i - 1]]) ? run + 1 : 0;
        if (run % svk::EXP_MAX_TERMS == 0) ++nbatches;
    }
    if (nbatches * (size_t)nb_fixed > scratch_doubles)
        return set_error(SV_ERR_ARG, "expectation: too many term batches for the scratch array");
    size_t i = 0, b = 0;
    while (i < nterms) {
        svk::ExpectArgs a;
        std::memset(&a, 0, sizeof(a));
        a.x = x[order[i]];
        while (i < nterms && x[order[i]] == a.x && a.nterms < svk::EXP_MAX_TERMS) {
            const size_t t = order[i++];
            const int y = __builtin_popcountll(a.x & z[t]) & 3;
            const double re[4] = {1, 0, -1, 0}, im[4] = {0, 1, 0, -1};
            a.z[a.nterms] = z[t];
            a.ccr[a.nterms] = c[t] * re[y];
            a.cci[a.nterms] = c[t] * im[y];
            ++a.nterms;
        }
        a.hb = a.x ? 63 - __builtin_clzll(a.x) : 0;
        a.npairs = a.x ? (1ull << (n - 1)) : (1ull << n);
        double *part = scratch + (b++) * (size_t)nb_fixed;
        if (dtype == SV_C64)
            svk::expect_kernel<float><<<nb_fixed, svk::RED_THREADS, 0, stream>>>(a, psi, part);
        else
            svk::expect_kernel<double><<<nb_fixed, svk::RED_THREADS, 0, stream>>>(a, psi, part);
        SV_CUDA(cudaGetLastError());
    }
    svk::sum_partials<<<1, svk::RED_THREADS, 0, stream>>>(scratch, (int)(nbatches * nb_fixed),
                                                          out_dev, nullptr, nullptr);
    SV_CUDA(cudaGetLastError());
    return SV_OK;
}

sv_status launch_widen(sv_state *s, const void *src_c64, void *dst_c128) {
    const unsigned long long N = 1ull << s->n;
    svk::widen_kernel<<<s->num_sms * 8, 256, 0, s->stream>>>(
        reinterpret_cast<const float2 *>(src_c64), reinterpret_cast<double2 *>(dst_c128), N);
    SV_CUDA(cudaGetLastError());
    return SV_OK;
}

// The state becomes |x>.  Up to 16 qubits in one launch; larger states by a memset and a
// one-amplitude kernel (the memset runs at copy speed).
sv_status launch_set_basis(sv_state *s, uint64_t x) {
    const int wide = s->dtype == SV_C128;
    const unsigned long long bytes = (wide ? 16ull : 8ull) << s->n;
    if (s->n <= 16) {
        const unsigned long long words = bytes / 16;
        SV_CUDA(svk::launch_pass(svk::set_basis_small, dim3((unsigned)((words + 255) / 256)), 256, 0, s->stream,
                                 reinterpret_cast<uint4 *>(s->buf), words, (unsigned long long)x, wide));
        return SV_OK;
    }
    SV_CUDA(cudaMemsetAsync(s->buf, 0, bytes, s->stream));
    svk::set_amp_one<<<1, 1, 0, s->stream>>>(s->buf, x, wide);
    SV_CUDA(cudaGetLastError());
    return SV_OK;
}

}  // namespace svi
