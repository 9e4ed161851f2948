// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include <complex>
#include <cstdint>
#include <functional>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "per_device.h"
#include "sv.h"

namespace svi {

using cplx = std::complex<double>;

// Thread-local last error message; set() returns the status for `return svi::set(...)`.
sv_status set_error(sv_status st, const std::string &msg);
void clear_error();

// A gate on sorted targets with its FP64 matrix (row-major, 2^k x 2^k).
struct Gate {
    uint32_t k = 0;
    uint32_t t[SV_MAX_K] = {0, 0, 0, 0, 0};
    std::vector<cplx> u;
};

// Relabel a gate's local bits so that its targets are ascending (same operator).
Gate sorted_gate(uint32_t k, const uint32_t *targets, const double *u);

// Exact structure of a sorted gate (structure.cpp): its control qubits and the reduced
// gate V on the other targets (U = I except where every control bit is 1, V there).
struct Structure {
    uint32_t kind = SV_STRUCT_DENSE;   // of V: SV_STRUCT_*
    uint32_t ctrl = 0;                 // local control bits of the gate
    uint32_t nctrl = 0;
    uint32_t ctrl_q[SV_MAX_K] = {0, 0, 0, 0, 0};   // their qubits, ascending
    Gate v;                            // reduced gate (k = 0 for a 1 x 1 V)
};
Structure classify(const Gate &g);

// The decisions of one run of Algorithm 2: contractions (u absorbs v) in order and the
// final topological order of the surviving vertices.
struct FusePlan {
    std::vector<std::pair<int, int>> contractions;
    std::vector<int> order;
};

// Algorithm 2 over sorted gates (fuse.cpp); records its decisions in *plan if given;
// commute: the commutation-aware DAG and contractions of commuting vertices.
std::vector<Gate> fuse_gates(const std::vector<Gate> &in, uint32_t n, uint32_t max_k,
                             FusePlan *plan = nullptr, bool commute = false);
// Bit j set when the gate never changes its local bit j (fuse.cpp).
uint32_t diagonal_mask(const Gate &g);
// g as an m-qubit gate U (x) I (m >= g.k, m <= n; fuse.cpp).
Gate widen_gate(const Gate &g, uint32_t n, uint32_t m);
// g as an m-qubit gate U (x) I on the sorted qubits qs (containing g's targets).
Gate widen_gate_on(const Gate &g, const uint32_t *qs, uint32_t m);
// Apply a recorded plan to gates with the same qubit sets (fuse.cpp).
std::vector<Gate> replay_fusion(std::vector<Gate> nodes, const FusePlan &plan);

}  // namespace svi

struct sv_circuit {
    uint32_t n = 0;
    std::vector<svi::Gate> gates;
    // the input gates (targets sorted), kept so that complex128 states can run the same
    // circuit fused at the tensor-core kernel's widest width (4) instead of applying
    // width-5 gates on the FP64 CUDA cores; that schedule is built on first use
    std::vector<svi::Gate> in_gates;
    mutable std::once_flag narrow_once;
    mutable std::vector<svi::Gate> narrow;
    // how it was fused, for sv_fuse_like: input qubit sets and the recorded plan
    uint32_t max_k = 0;
    uint32_t flags = 0;               // SV_FUSE_* it was fused with
    std::vector<uint32_t> in_k;
    std::vector<uint32_t> in_t;       // SV_MAX_K per input gate, sorted
    std::vector<uint32_t> in_diag;    // with SV_FUSE_COMMUTE: diagonal_mask of each input gate
    svi::FusePlan plan;
};

// Device workspace layout (bytes), carved from one allocation.
namespace svi {
constexpr size_t WS_ERR = 0;                   // int error word (+ padding)
// 64 doubles, then the 64 indices of a top-k (server states; others use the mailbox)
constexpr size_t WS_RESULT = 16;
constexpr size_t WS_PARTIAL = 2048;            // double partials[WS_NPARTIAL]
constexpr int WS_NPARTIAL = 8192;
constexpr size_t WS_TOPK = WS_PARTIAL + WS_NPARTIAL * 8;   // chunk maxima of a top-k; tables of an expectation
constexpr size_t WS_TOPK_BYTES = size_t(4) << 20;
constexpr size_t WS_BYTES = WS_TOPK + WS_TOPK_BYTES;
}  // namespace svi

struct sv_state {
    uint32_t n = 0;
    sv_dtype dtype = SV_C64;
    void *buf = nullptr;        // amplitudes
    size_t cap = 0;             // bytes available at buf
    bool owned = false;
    cudaStream_t stream = nullptr;
    int device = 0;
    unsigned char *ws = nullptr;   // device workspace (WS_BYTES)
    // what the state holds, for adaptive replay: a basis state or a snapshot
    bool basis_known = true;
    uint64_t basis_x = 0;
    void *snap = nullptr;       // library-owned snapshot of the initial state (c64)
    size_t snap_cap = 0;
    int num_sms = 0;
    uint32_t policy = 0;        // SV_POLICY_* flags (kernel selection)
    void *samp = nullptr;       // sampling scratch (sample.cu), kept across calls
    size_t samp_cap = 0;
    // results and the error word in page-locked host memory that kernels write (sv_alloc): a
    // call that returns a number then needs no copy.  Layout as WS_ERR / WS_RESULT.
    unsigned char *mail = nullptr, *mail_dev = nullptr;
    void *probs_buf = nullptr;  // SV_POLICY_STAGED_PROBS: device probabilities, kept across calls
    size_t probs_cap = 0;
};

namespace svi {
// Where a reduction's last kernel writes: results, and a copy of the error word.
inline double *mail_results(const sv_state *s) { return reinterpret_cast<double *>(s->mail_dev + WS_RESULT); }
inline int *mail_error(const sv_state *s) { return reinterpret_cast<int *>(s->mail_dev + WS_ERR); }
inline const int *device_error(const sv_state *s) { return reinterpret_cast<const int *>(s->ws + WS_ERR); }

// Which kernel family ran a pass (launch_apply's optional out-parameter).
enum PassKind { PASS_CUDA_CORE = 0, PASS_TENSOR_CORE = 1, PASS_STRUCTURED = 2 };
}  // namespace svi

// One batched launch: gate k/t applied to `states` consecutive states at psi with
// per-state matrices at utab (batch.cu).
struct sv_batch_launch {
    sv_dtype dtype = SV_C64;
    uint32_t k = 0, n = 0;
    uint32_t t[SV_MAX_K] = {0, 0, 0, 0, 0};
    uint32_t states = 0;
    void *psi = nullptr;
    const void *utab = nullptr;
    int *err = nullptr;
    cudaStream_t stream = nullptr;
    int num_sms = 0;
    bool tc = false;            // complex64 on the tensor cores (apply_tc.cu): its operands
    const void *images = nullptr;   // are packed first (launch_tc_pack)
    const float *bscale = nullptr;
    uint32_t tile_bits = 0;     // CUDA-core passes: 2^tile_bits amplitudes per CTA (0: default)
};

namespace svk {
inline int current_device() {
    int dev = 0;
    (void)cudaGetDevice(&dev);
    return dev;
}

// Launch a kernel that calls pass_wait() before its first access to memory that other kernels touch: its
// launch latency and prologue overlap the previous kernel's tail -- or all of it, where that begins
// with pass_trigger().  Short kernels whose blocks fill the SMs leave the trigger to their end: blocks
// that come in early take the places of the current kernel's own (3000 permutations on 20 qubits,
// complex128: 28.1 ms launched in order, 30.1 with the trigger first, 20.9 without it; 13 qubits,
// complex64: 12.4, 7.1 and 6.3).
// Measured on whole circuits, in-order launches -> this: 350 gates on 12 qubits (complex128)
// 3094 -> 2169 us, 50 passes on 20 qubits 573 -> 481 us, 74 on 28 qubits 50.21 -> 49.93 ms.
template <typename... P, typename... A>
cudaError_t launch_pass(void (*kern)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t stream,
                        A &&...args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

cudaError_t tc_batch_prepare();
sv_status launch_tc_batch(const sv_batch_launch &L);
// Operand images of `ngates` gates (L[i]; all with the same states and stream) into images,
// gate by gate, tc_batch_image_bytes() each, and their scales into bscale; gate i's FP32 matrices
// start tab_off[i] bytes into utab.
size_t tc_batch_image_bytes();
sv_status launch_tc_pack(const sv_batch_launch *L, const size_t *tab_off, uint32_t ngates, const void *utab,
                         void *images, float *bscale);
// `bytes` bytes at buf as a 2-D tensor of 128-byte rows for TMA tensor copies with the
// 128-byte shared-memory swizzle; a segment of seg_bytes is *boxes boxes of *box_rows rows
// (apply_tc.cu).  `map` points to a CUtensorMap.
sv_status encode_rows_map(void *buf, unsigned long long bytes, uint32_t seg_bytes, struct CUtensorMap_st *map,
                          uint32_t *box_rows, uint32_t *boxes);
}  // namespace svk

namespace svi {
// ---- kernels (apply_kernels.cu / reduce_kernels.cu); all enqueue on s->stream ----
// One pass of g; *bytes (if given) gets the pass's algorithmic HBM bytes: a full read and
// write of the state, or of the amplitudes a structure-aware pass touches.
// st: the gate's structure where the caller has it.
sv_status launch_apply(sv_state *s, const Gate &g, uint64_t *bytes = nullptr, int *kind = nullptr,
                       const Structure *st = nullptr);
// Gates from `begin` on that share one pass (apply_runs.cu; st[i - begin]: gate i's structure, share[i -
// begin + 1] - share[i - begin]: the share of the state it touches; all of one kind): how many it ran, 0
// if there is no run there that pays -- then *tried is how many gates a plan in vain went over.
constexpr size_t RUN_GATES = 64;      // gates looked at for a run
size_t launch_run(sv_state *s, const std::vector<Gate> &gates, const Structure *st, const double *share, size_t begin,
                  size_t end, size_t *tried, sv_status *status);
// Structure-aware pass (apply_struct.cu): is it preferred over the dense kernels, and run it.
bool struct_preferred(const sv_state *s, const Structure &st);
sv_status launch_apply_struct(sv_state *s, const Structure &st);
uint64_t struct_bytes(const sv_state *s, const Structure &st);   // 2 s per amplitude it touches
// States of up to 12 qubits (small_fit.h) without kernel-selection flags: gates [begin, end) in as few
// launches as their matrices allow (apply_small.cu); *bytes is added to as by launch_apply.
bool small_state(const sv_state *s);
sv_status launch_small(sv_state *s, const std::vector<Gate> &gates, size_t begin, size_t end, uint64_t *bytes);
bool tc_eligible(const sv_state *s, const Gate &g);        // apply_tc.cu
sv_status launch_apply_tc(sv_state *s, const Gate &g);
bool tc64_eligible(const sv_state *s, const Gate &g);      // apply_tc64.cu
sv_status launch_apply_tc64(sv_state *s, const Gate &g);
// Two complex64 gates in one pass (apply_tc2.cu): do they fit one tile, and run them
// (g0 first).
bool tc2_pair_fits(const sv_state *s, const Gate &g0, const Gate &g1);
sv_status launch_apply_tc2(sv_state *s, const Gate &g0, const Gate &g1);
sv_status launch_norm(sv_state *s, double *dev_out);     // writes one double on device
sv_status launch_probs(sv_state *s, void *dev_out);
sv_status launch_density_probs(sv_state *s, void *dev_out);   // Re v[x + 2^(n/2) x]
sv_status launch_expect(sv_state *s, const uint64_t *x, const uint64_t *z, const double *c,
                        size_t nterms, double *host_out);
sv_status enqueue_sum(sv_state *s, int n, double *dev_out);   // of the first n block partials
sv_status enqueue_expect_group(sv_state *s, uint64_t x, const uint64_t *z, const double *c, int nterms,
                               double *dev_out);
sv_status batch_z_terms(const void *psi, uint32_t n, sv_dtype dtype, uint32_t states, int num_sms, cudaStream_t stream,
                        double *tables, double *partial, size_t room, const uint64_t *z, const double *c, size_t nterms,
                        const std::function<sv_status(int)> &fold);
std::vector<char> batch_z_split(uint32_t n, sv_dtype dtype, uint32_t states, const uint64_t *z, size_t nterms);
sv_status launch_topk(sv_state *s, uint32_t k, uint64_t *idx, double *p);
sv_status enqueue_topk(sv_state *s, double *host_p, unsigned long long *host_i);
sv_status launch_widen(sv_state *s, const void *src_c64, void *dst_c128);
sv_status launch_set_basis(sv_state *s, uint64_t x);
sv_status check_device_error(sv_state *s);   // synchronises; reads and clears the error word
// Synchronise and read the first `bytes` (<= 1024) of the results that the stream's last kernel
// left in the state's mailbox, with the error word; one found set is cleared and reported.
sv_status read_results(sv_state *s, void *dst, size_t bytes);
// The circuit's input gates fused again at width <= 4 when its schedule has width-5 gates
// (built once per circuit), else its schedule: what complex128 runs on the tensor cores.
const std::vector<Gate> &narrow_schedule(const sv_circuit *c);
// cudaMalloc that sv_debug_fail_allocs can make fail.
cudaError_t alloc_state_buffer(void **p, size_t bytes);
// SV_ERR_STATE (with a message) when a failed reallocation left the state without a buffer.
sv_status check_live(const sv_state *s, const char *who);
sv_status enqueue_expect_sum(const void *psi, uint32_t n, sv_dtype dtype, const uint64_t *x,
                             const uint64_t *z, const double *c, size_t nterms, double *scratch,
                             size_t scratch_doubles, int nb_fixed, double *out_dev,
                             cudaStream_t stream);
}  // namespace svi

#define SV_CUDA(call)                                                                    \
    do {                                                                                 \
        cudaError_t e_ = (call);                                                         \
        if (e_ != cudaSuccess)                                                           \
            return svi::set_error(e_ == cudaErrorMemoryAllocation ? SV_ERR_OOM : SV_ERR_CUDA, \
                                  std::string(#call) + ": " + cudaGetErrorString(e_));  \
    } while (0)
