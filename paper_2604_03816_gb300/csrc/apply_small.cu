// Whole schedules on small states (up to 12 qubits): many gates per launch.
//
// A state of 12 qubits is 32 KiB (complex64) or 64 KiB (complex128): a pass per gate is all
// launch latency, fill and drain (6-8 us for work of well under one).  Measured on the 12-qubit
// brickwork circuit, pass per gate -> this: 350 gates in complex128 2169 -> 251 us, 21 width-5
// gates in complex64 208 -> 66 us.  Here one cluster of up
// to 16 CTAs keeps the state on chip and runs the gates one after the other, as many per
// launch as fit the kernel's parameters (28 KiB: 350 unfused gates, or three dense width-5
// ones).  Thread j of rank r owns amplitude i = r 2^(n-c) + j in registers for the whole launch.
//
// * diagonal gates multiply the owner's amplitude: no exchange, no barrier;
// * monomial and dense gates read other amplitudes: every owner first writes its amplitude to
//   its CTA's shared-memory copy of the state and, for targets among the top c index bits, to
//   the copies of the peers that will read it (stores into distributed shared memory, which
//   nobody waits for), then one barrier -- of the cluster if a target is among those bits, of
//   the CTA otherwise -- and each owner forms its own output row from its own CTA's copy.
//
// Two copies alternate, so one barrier per gate is enough: copy b is written again two
// exchanges later, and the barrier in between (a cluster one, added where the schedule has
// none there) lies after every read of it.
//
// What bounds it: complex128 the FP64 pipe (4 2^k FP64 operations per amplitude and gate at
// about 1.9 per clock and SM: 0.5 us for a one-qubit gate on 12 qubits over 16 SMs); complex64
// the barriers (0.1-0.4 us) and, at width 5, the host, which needs about 12 us to classify and pack
// the three matrices of a launch that runs 7.6 (two threads per amplitude: the same time).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "ptx.cuh"
#include "small_fit.h"
#include "sv_internal.h"

namespace svm {

template <typename R> struct Cx;
template <> struct Cx<float> { using T = float2; };
template <> struct Cx<double> { using T = double2; };
__device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mk(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ float fmar(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmar(double a, double b, double c) { return __fma_rn(a, b, c); }

constexpr uint32_t BLOB = 28 * 1024;      // ops, then their entries
// Parameters of a few gates go in a smaller block: launching costs time by the size of the block (one
// single-qubit gate 14.7 us with 28 KiB, 12.7 with 2).
constexpr uint32_t SMALL_BLOB = 2 * 1024;

enum OpKind : uint32_t { OP_DIAG = 0, OP_MONO = 1, OP_DENSE = 2 };

// One gate: its remainder V on `k` targets (4 bits each in `t`, ascending) where every bit of
// `ctrl` is 1.  Entries at blob + 16 `off`: diagonal d[r]; monomial: phase[r], then 2^k source
// rows as uint32; dense: V transposed (entry (r, c) at c 2^k + r), so that lanes in different
// rows read consecutive words.
struct Op {
    uint32_t kind_k;       // kind | k << 8
    uint32_t ctrl;
    uint32_t t;
    uint32_t off;
};

template <uint32_t B>
struct SmallArgs {
    void *psi;
    uint32_t n, c, nops, blob_bytes;
    alignas(16) unsigned char blob[B];
};

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_peer(uint32_t addr, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t addr, double2 v) {
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(addr), "d"(v.x), "d"(v.y) : "memory");
}

// Is the entry exactly 1 (+-0 i)?  In FP64 by its bits: two compares cost as much as half the product
// on the FP64 pipe.
__device__ __forceinline__ bool is_one(float2 d) { return d.x == 1.f && d.y == 0.f; }
__device__ __forceinline__ bool is_one(double2 d) {
    return __double_as_longlong(d.x) == 0x3FF0000000000000ll && (__double_as_longlong(d.y) << 1) == 0ll;
}

template <typename C>
__device__ __forceinline__ C cmul(C a, C b) {
    return mk(fmar(a.x, b.x, -(a.y * b.y)), fmar(a.x, b.y, a.y * b.x));
}

// Row r of V times the 2^K inputs at base ^ offset.  From K = 3 on two chains of FMAs (even
// and odd columns), which halves the latency and the growth of the rounding error; narrower
// rows are one chain, since adding two up costs a fifth more FP64 operations at K = 1.
template <typename R, int K>
__device__ __forceinline__ typename Cx<R>::T dense_row(const typename Cx<R>::T *in, const typename Cx<R>::T *vt,
                                                       uint32_t base, uint32_t r, uint32_t t) {
    using C = typename Cx<R>::T;
    uint32_t tb[K];
#pragma unroll
    for (int j = 0; j < K; ++j) tb[j] = 1u << ((t >> (4 * j)) & 15u);
    constexpr int M = K >= 3 ? 1 : 0;
    R re[2] = {0, 0}, im[2] = {0, 0};
#pragma unroll
    for (int c = 0; c < (1 << K); ++c) {
        uint32_t o = base;
#pragma unroll
        for (int j = 0; j < K; ++j)
            if ((c >> j) & 1) o |= tb[j];
        const C x = in[o], u = vt[(c << K) + r];
        re[c & M] = c <= M ? u.x * x.x : fmar(u.x, x.x, re[c & M]);
        re[c & M] = fmar(-u.y, x.y, re[c & M]);
        im[c & M] = c <= M ? u.x * x.y : fmar(u.x, x.y, im[c & M]);
        im[c & M] = fmar(u.y, x.x, im[c & M]);
    }
    return M ? mk(re[0] + re[1], im[0] + im[1]) : mk(re[0], im[0]);
}

template <typename R, uint32_t B>
__global__ void __launch_bounds__(THREADS, 1) apply_small(const __grid_constant__ SmallArgs<B> a) {
    using C = typename Cx<R>::T;
    extern __shared__ __align__(16) unsigned char smem[];
    svk::pass_trigger();
    const uint32_t N = 1u << a.n, own = N >> a.c;             // amplitudes in all, per CTA
    const uint32_t rank = blockIdx.x, tid = threadIdx.x;
    C *copy0 = reinterpret_cast<C *>(smem);                   // two copies of the state
    unsigned char *blob = smem + 2u * N * (uint32_t)sizeof(C);
    for (uint32_t o = 16u * tid; o < a.blob_bytes; o += 16u * THREADS)
        *reinterpret_cast<int4 *>(blob + o) = svk::ld_param16(a.blob + o);
    const Op *ops = reinterpret_cast<const Op *>(blob);
    const bool mine = tid < own;
    const uint32_t i = rank * own + tid;
    // the peers' shared memory may be written once their CTAs have started
    if (a.c) cluster_barrier();
    else __syncthreads();
    svk::pass_wait();
    C *psi = reinterpret_cast<C *>(a.psi);
    C v = mk(R(0), R(0));
    if (mine) v = psi[i];
    uint32_t b = 0;                                           // the copy of this exchange
    bool fenced = true;                                       // was the last barrier the cluster's?
    const uint32_t shift = a.n - a.c;
    for (uint32_t g = 0; g < a.nops; ++g) {
        const Op op = ops[g];
        const uint32_t kind = op.kind_k & 255u, k = (op.kind_k >> 8) & 255u;
        const C *ent = reinterpret_cast<const C *>(blob + 16u * op.off);
        const bool act = mine && (i & op.ctrl) == op.ctrl;
        uint32_t r = 0, tmask = 0;
#pragma unroll
        for (uint32_t j = 0; j < SV_MAX_K; ++j) {
            const uint32_t t = (op.t >> (4u * j)) & 15u, on = j < k ? 1u : 0u;
            r |= ((i >> t) & on) << j;
            tmask |= on << t;
        }
        if (kind == OP_DIAG) {
            if (act) {
                const C d = ent[r];
                if (!is_one(d)) v = cmul(d, v);
            }
            continue;
        }
        C *buf = copy0 + b * N;
        const uint32_t far = tmask >> shift;                  // rank bits among the targets
        if (far) {
            if (!fenced) cluster_barrier();
            if (mine)
                for (uint32_t m = far; m; m = (m - 1u) & far)
                    st_peer(peer_addr(svk::smem_u32(buf + i), rank ^ m), v);
        }
        if (mine) buf[i] = v;
        if (far) cluster_barrier();
        else __syncthreads();
        fenced = far != 0;
        if (act) {
            const uint32_t base = i & ~tmask;
            if (kind == OP_MONO) {
                const uint32_t src = reinterpret_cast<const uint32_t *>(ent + (1u << k))[r];
                uint32_t o = base;
                for (uint32_t j = 0; j < k; ++j)
                    if ((src >> j) & 1u) o |= 1u << ((op.t >> (4u * j)) & 15u);
                const C x = buf[o], d = ent[r];
                v = is_one(d) ? x : cmul(d, x);
            } else {
                switch (k) {
                    case 1: v = dense_row<R, 1>(buf, ent, base, r, op.t); break;
                    case 2: v = dense_row<R, 2>(buf, ent, base, r, op.t); break;
                    case 3: v = dense_row<R, 3>(buf, ent, base, r, op.t); break;
                    case 4: v = dense_row<R, 4>(buf, ent, base, r, op.t); break;
                    default: v = dense_row<R, 5>(buf, ent, base, r, op.t); break;
                }
            }
        }
        b ^= 1u;
    }
    if (mine) psi[i] = v;
}

// Collects gates until the parameters are full, then launches.
template <typename R>
struct Builder {
    sv_state *s;
    std::vector<Op> ops;
    uint32_t used = 0;                        // bytes of entries
    alignas(16) unsigned char data[BLOB];

    explicit Builder(sv_state *s_) : s(s_) {}

    void put(const svi::cplx &z) {
        R *p = reinterpret_cast<R *>(data + used);
        p[0] = static_cast<R>(z.real());
        p[1] = static_cast<R>(z.imag());
        used += 2 * (uint32_t)sizeof(R);
    }

    static uint32_t entry_bytes(const svi::Structure &st) {
        const uint32_t D = 1u << st.v.k, e = 2u * (uint32_t)sizeof(R);
        const uint32_t b = st.kind == SV_STRUCT_DENSE ? D * D * e : st.kind == SV_STRUCT_MONOMIAL ? D * (e + 4u) : D * e;
        return (b + 15u) & ~15u;
    }

    sv_status add(const svi::Structure &st) {
        if ((ops.size() + 1) * sizeof(Op) + used + entry_bytes(st) > BLOB) {
            const sv_status rc = flush();
            if (rc != SV_OK) return rc;
        }
        const uint32_t k = st.v.k, D = 1u << k;
        Op op;
        op.off = used / 16;                                   // relative to the entries for now
        op.ctrl = op.t = 0;
        for (uint32_t j = 0; j < st.nctrl; ++j) op.ctrl |= 1u << st.ctrl_q[j];
        for (uint32_t j = 0; j < k; ++j) op.t |= st.v.t[j] << (4 * j);
        uint32_t kind = OP_DENSE;
        if (st.kind == SV_STRUCT_DIAGONAL) {
            kind = OP_DIAG;
            for (uint32_t r = 0; r < D; ++r) put(st.v.u[(size_t)r * D + r]);
        } else if (st.kind == SV_STRUCT_MONOMIAL) {
            kind = OP_MONO;
            std::vector<uint32_t> src(D);
            for (uint32_t r = 0; r < D; ++r) {
                uint32_t c = 0;
                while (st.v.u[(size_t)r * D + c] == svi::cplx(0.0, 0.0)) ++c;   // the row's nonzero
                src[r] = c;
                put(st.v.u[(size_t)r * D + c]);
            }
            std::memcpy(data + used, src.data(), 4 * D);
            used += 4 * D;
        } else {
            for (uint32_t c = 0; c < D; ++c)
                for (uint32_t r = 0; r < D; ++r) put(st.v.u[(size_t)r * D + c]);
        }
        used = (used + 15u) & ~15u;
        op.kind_k = kind | k << 8;
        ops.push_back(op);
        return SV_OK;
    }

    template <uint32_t B>
    sv_status launch(uint32_t max_c);
    sv_status flush();
};

// Cluster size (log2) for this device: 16 CTAs where the device schedules them, else 8.
template <typename R>
static cudaError_t setup(uint32_t *max_c) {
    struct Setup { cudaError_t err; uint32_t max_c; };
    static svk::PerDevice<Setup> setup;
    const Setup done = setup.get(svk::current_device(), [] {
        const int smem = int((2u << MAX_N) * 2u * sizeof(R) + BLOB);
        Setup r = {cudaSuccess, 3};
        r.err = cudaFuncSetAttribute(apply_small<R, BLOB>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (r.err == cudaSuccess)
            r.err = cudaFuncSetAttribute(apply_small<R, SMALL_BLOB>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (r.err != cudaSuccess) return r;
        if (cudaFuncSetAttribute(apply_small<R, BLOB>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaFuncSetAttribute(apply_small<R, SMALL_BLOB>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
                cudaSuccess) {
            cudaLaunchAttribute at;
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = 16;
            at.val.clusterDim.y = at.val.clusterDim.z = 1;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(16);
            cfg.blockDim = dim3(THREADS);
            cfg.dynamicSmemBytes = (size_t)smem;
            cfg.attrs = &at;
            cfg.numAttrs = 1;
            int nc = 0;
            if (cudaOccupancyMaxActiveClusters(&nc, apply_small<R, BLOB>, &cfg) == cudaSuccess && nc > 0) r.max_c = MAX_C;
        }
        (void)cudaGetLastError();
        return r;
    });
    *max_c = done.max_c;
    return done.err;
}

template <typename R>
sv_status Builder<R>::flush() {
    if (ops.empty()) return SV_OK;
    uint32_t max_c = 0;
    const cudaError_t e = setup<R>(&max_c);
    if (e != cudaSuccess)
        return svi::set_error(SV_ERR_CUDA, std::string("small-state kernel setup: ") + cudaGetErrorString(e));
    return ops.size() * sizeof(Op) + used <= SMALL_BLOB ? launch<SMALL_BLOB>(max_c) : launch<BLOB>(max_c);
}

template <typename R>
template <uint32_t B>
sv_status Builder<R>::launch(uint32_t max_c) {
    SmallArgs<B> a;
    const size_t ob = ops.size() * sizeof(Op);
    for (Op &op : ops) op.off += (uint32_t)(ob / 16);
    std::memcpy(a.blob, ops.data(), ob);
    std::memcpy(a.blob + ob, data, used);
    a.psi = s->buf;
    a.n = s->n;
    a.c = cluster_log2(s->n, max_c);
    a.nops = (uint32_t)ops.size();
    a.blob_bytes = (uint32_t)ob + used;
    ops.clear();
    used = 0;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 1u << a.c;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1u << a.c);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = (size_t)(2u << a.n) * 2u * sizeof(R) + ((a.blob_bytes + 15u) & ~15u);
    cfg.stream = s->stream;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    SV_CUDA(cudaLaunchKernelEx(&cfg, apply_small<R, B>, a));
    return SV_OK;
}

}  // namespace svm

namespace svi {

bool small_state(const sv_state *s) {
    if (s->n > svm::MAX_N || (s->policy & (SV_POLICY_NO_TENSOR_CORES | SV_POLICY_DENSE_ONLY | SV_POLICY_TWO_GATE_PASSES)))
        return false;
    uint32_t max_c = 0;
    const cudaError_t e = s->dtype == SV_C64 ? svm::setup<float>(&max_c) : svm::setup<double>(&max_c);
    return e == cudaSuccess && svm::state_fits(s->n, max_c);
}

template <typename R>
static sv_status launch_small_t(sv_state *s, const std::vector<Gate> &gates, size_t begin, size_t end,
                                uint64_t *bytes) {
    svm::Builder<R> build(s);
    for (size_t i = begin; i < end; ++i) {
        const Structure st = classify(gates[i]);
        *bytes += struct_preferred(s, st) ? struct_bytes(s, st) : (uint64_t)(4 * sizeof(R)) << s->n;
        if (st.kind == SV_STRUCT_IDENTITY) continue;
        const sv_status rc = build.add(st);
        if (rc != SV_OK) return rc;
    }
    return build.flush();
}

sv_status launch_small(sv_state *s, const std::vector<Gate> &gates, size_t begin, size_t end, uint64_t *bytes) {
    return s->dtype == SV_C64 ? launch_small_t<float>(s, gates, begin, end, bytes)
                              : launch_small_t<double>(s, gates, begin, end, bytes);
}

}  // namespace svi
