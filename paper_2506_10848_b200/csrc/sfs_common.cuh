// Shared host/device helpers of libsfs (error reporting, small device utilities).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stdio.h>
#include <stdarg.h>
#include <tuple>
#include <utility>
#include <vector>

#include "../../include/sfs.h"

static_assert(sizeof(sfs_state) == 128, "sfs_state is 32 int32");

namespace sfs {

// ---- host-side error reporting ---------------------------------------------------------------------
void set_error(const char *fmt, ...);          // stores a message for sfs_last_error() (thread-local)

#define SFS_REQUIRE(cond, code, ...)                                   \
    do {                                                               \
        if (!(cond)) { ::sfs::set_error(__VA_ARGS__); return (code); } \
    } while (0)

#define SFS_CUDA(call)                                                                           \
    do {                                                                                         \
        cudaError_t e__ = (call);                                                                \
        if (e__ != cudaSuccess) {                                                                \
            ::sfs::set_error("%s failed: %s (%s:%d)", #call, cudaGetErrorString(e__), __FILE__, __LINE__); \
            return (e__ == cudaErrorMemoryAllocation) ? SFS_ERR_OOM : SFS_ERR_CUDA;              \
        }                                                                                        \
    } while (0)

#define SFS_LAUNCH_CHECK()  SFS_CUDA(cudaGetLastError())

static inline bool aligned_to(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Per-device bookkeeping (kernel attributes, the sticky status word) is indexed by the ordinal of the current device.
constexpr int kMaxDevices = 64;
static inline int current_device_slot()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
    return dev;
}
// The current device's sticky status word (set by kernels whose bounded waits give up, or that skip an invalid row);
// allocated on first use, null if that allocation fails.  The _if_any form never allocates.
int32_t *device_status_word();
int32_t *device_status_word_if_any();

// ---- programmatic dependent launch -----------------------------------------------------------------------
// A kernel launched with launch_pdl may start (be scheduled, run its prologue) while the kernel before it in the stream is
// still running; it calls pdl_wait() before its first access to global memory, which returns once that kernel has completed
// and its writes are visible.  pdl_trigger() tells the runtime that the kernels after this one may be scheduled.  Kernels call it
// when about one launch latency of their own work is left: after their wait if they are short, before the last epilogue if they
// are GEMMs.  Called first thing, a whole row of kernels becomes resident, and each reaches its wait so long before its input is
// there that the code behind the wait has left the instruction cache by then (small projection after attention, 192 tokens: 4.9
// us from wait to end, 2.8 when released late; tiny step 55 -> 49 us, 8B forward at 104 rows 3990 -> 3946).  Never before the wait: where a
// QKV projection leaves SMs idle, all CTAs of an attention of few queries fit beside it, and if those release the output projection at
// once its CTAs fill the rest, long before their input (us a layer of 128 rows, 16 / 20 / 28 / 32 heads of 128: 67.7 / 76.9 / 102.4 / 118.6,
// released behind the wait 64.1 / 73.7 / 99.7 / 117.9).
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launches whose arguments change from call to call (a caller's pointers, step counts) inside a recorded graph: while a sink is
// installed on the thread, launch_pdl either notes the node it has just recorded, or sets that node's arguments instead of launching.
struct NodeSink {
    cudaGraphExec_t exec = nullptr;          // NULL: recording
    std::vector<cudaGraphNode_t> *nodes = nullptr;
    size_t next = 0;
};
inline thread_local NodeSink *g_node_sink = nullptr;
cudaError_t note_recorded_node(NodeSink *sink, cudaStream_t stream);
template <typename Tuple, size_t... I>
static inline cudaError_t set_node_args(NodeSink *sink, void *kernel, dim3 grid, dim3 block, size_t smem, Tuple &vals, std::index_sequence<I...>)
{
    void *ptrs[] = {(void *)&std::get<I>(vals)...};
    cudaKernelNodeParams p = {};
    p.func = kernel; p.gridDim = grid; p.blockDim = block; p.sharedMemBytes = (unsigned)smem; p.kernelParams = ptrs;
    if (sink->next >= sink->nodes->size()) return cudaErrorInvalidValue;
    return cudaGraphExecKernelNodeSetParams(sink->exec, (*sink->nodes)[sink->next++], &p);
}
template <typename... KArgs, typename... Args>
static inline bool redirect_launch(cudaError_t *e, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, Args... args)
{
    if (g_node_sink == nullptr || g_node_sink->exec == nullptr) return false;
    std::tuple<KArgs...> vals{static_cast<KArgs>(args)...};
    *e = set_node_args(g_node_sink, (void *)kernel, grid, block, smem, vals, std::index_sequence_for<KArgs...>());
    return true;
}

template <typename... KArgs, typename... Args>
static inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args... args)
{
    cudaError_t e;
    if (redirect_launch(&e, kernel, grid, block, smem, args...)) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
    return (e == cudaSuccess && g_node_sink) ? note_recorded_node(g_node_sink, stream) : e;
}
// the same with clusters of `cluster` CTAs
template <typename... KArgs, typename... Args>
static inline cudaError_t launch_pdl_cluster(void (*kernel)(KArgs...), int cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args... args)
{
    cudaError_t e;
    if (redirect_launch(&e, kernel, grid, block, smem, args...)) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
    return (e == cudaSuccess && g_node_sink) ? note_recorded_node(g_node_sink, stream) : e;
}
#endif

// A launch may use 48 KB of shared memory unasked, static arrays included (these kernels have a few KB of them at most): more is asked
// for here.  Comparing the dynamic part alone with 48 KB left a band of sizes just below it that no launch accepted.
#ifdef __CUDACC__
constexpr size_t kUnaskedShared = 40 * 1024;
template <typename... KArgs>
static inline cudaError_t allow_shared(void (*kernel)(KArgs...), size_t dynamic)
{
    return dynamic > kUnaskedShared ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dynamic) : cudaSuccess;
}
#endif

// ---- device helpers ---------------------------------------------------------------------------------
#ifdef __CUDACC__
__device__ __forceinline__ float bf16_bits_to_f32(uint32_t h16) { return __uint_as_float(h16 << 16); }

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ int warp_sum_i32(int v) { return __reduce_add_sync(0xffffffffu, v); }
__device__ __forceinline__ int warp_min_i32(int v) { return __reduce_min_sync(0xffffffffu, v); }
__device__ __forceinline__ int warp_max_i32(int v) { return __reduce_max_sync(0xffffffffu, v); }

// Algorithm 1's initial state of a sequence with L masked positions
__device__ __forceinline__ sfs_state initial_state(int L, int max_steps)
{
    sfs_state s;
    memset(&s, 0, sizeof(s));
    s.phase = SFS_PHASE_SLOW;
    s.k_remaining = max_steps > 0 ? max_steps : L;
    s.n_masked = L;
    s.done = (L == 0) ? 1 : 0;
    return s;
}

// block structure of the LLaDA strategies: which positions the step with index t works on, and the block's countdown
struct BlockStep { int j, lo, hi, k_b, steps_per_block; };
__device__ __forceinline__ BlockStep block_step(const sfs_params &p, int L, int t)
{
    const int N = p.max_steps > 0 ? p.max_steps : L;
    const int bl = (p.block_len > 0 && p.block_len < L) ? p.block_len : max(L, 1);
    const int nb = (L + bl - 1) / bl;
    BlockStep s;
    s.steps_per_block = max(N / max(nb, 1), 1);
    s.j = t / s.steps_per_block;
    s.k_b = s.steps_per_block - (t - s.j * s.steps_per_block);
    s.lo = min(L, s.j * bl);
    s.hi = min(L, s.lo + bl);
    return s;
}

// what one denoising step asks of the row statistics of sequence state `st`: the candidate window [lo, hi) of response
// positions, the confidence threshold whose outcome is read (0 = none) and how many most-confident candidates are ranked
// (k_top; n_cand = number of masked positions in the window, needed by the low-confidence rule only)
struct StepAsk { int lo, hi; float tau; bool rank_needed; };
__device__ __forceinline__ StepAsk step_ask(const sfs_params &p, const sfs_state &st, int L)
{
    StepAsk a;
    a.tau = 0.f; a.rank_needed = false;
    if (p.sampler != SFS_SAMPLER_SLOWFAST) {
        const BlockStep b = block_step(p, L, st.steps_done);
        a.lo = b.lo; a.hi = b.hi;
        a.rank_needed = (p.sampler == SFS_SAMPLER_LOW_CONFIDENCE);
    } else if (st.k_remaining == 1) {
        a.lo = 0; a.hi = L;                                 // last permitted step: everything is unmasked, nothing is compared
    } else if (st.phase == SFS_PHASE_SLOW) {
        a.lo = st.s_cycle; a.hi = L; a.tau = p.tau_min_conf; a.rank_needed = true;
    } else {
        a.lo = st.s_cycle; a.hi = st.hi; a.tau = p.tau_high_conf; a.rank_needed = true;
    }
    return a;
}

// c > tau  <=>  S_q * tau < 2^28, one IEEE double multiply
__device__ __forceinline__ bool conf_exceeds(unsigned long long sq, float tau) {
    return __dmul_rn((double)sq, (double)tau) < (double)(1u << SFS_CONF_QBITS);
}
#endif

// ---- internal launchers (defined in the .cu files) --------------------------------------------------
// The token positions that statistics are scattered to: n = B * S of them, the first P of every S a prompt's.  Rows of prompt positions
// are left out: the selection reads, and clears again, response positions only, and what stayed behind would be taken for the
// statistics of a later call whose prompt is shorter (with a logits row that may lie beyond that call's buffer).
struct TokenGrid {
    int32_t n, S, P;
#ifdef __CUDACC__
    __device__ __forceinline__ bool inside(int p) const { return (unsigned)p < (unsigned)n; }
    __device__ __forceinline__ bool response(int p) const { return p % S >= P; }
#endif
};

// Row statistics (Section 3.1: greedy token and confidence).  Results are written densely by logits row
// (d_argmax/d_sq/d_conf, each optional) and, when d_rows is given, scattered to d_pos_sq/d_pos_arg at the
// flat token index of each row; an index outside the grid is skipped and reported as SFS_ERR_INVALID_ARG
// in *d_err (a device status word, optional), as is a bounded wait that gives up (SFS_ERR_TIMEOUT).
int32_t launch_row_stats(const void *d_logits, int32_t logits_dtype, int32_t vocab, int64_t ld,
                         const int32_t *d_n_rows, int32_t max_rows, const int32_t *d_rows,
                         int32_t *d_argmax, unsigned long long *d_sq, float *d_conf,
                         unsigned long long *d_pos_sq, int32_t *d_pos_arg, TokenGrid grid, int32_t *d_err,
                         cudaStream_t stream);

// Row statistics for the selection step in two passes over long bf16 rows (the filter + exact form):
//   pass 1 streams every row from HBM once and finds the exact maximum and argmax plus an APPROXIMATE denominator (special-
//     function exponentials, fp32 sum) with a proven enclosure [lo, lo + w] of the canonical S_q;
//   pass 2, inside the selection kernel, looks at what the step's rule will ask of a sequence's rows (which threshold, which
//     top-k), recomputes the canonical S_q of those whose enclosure leaves an answer open and takes every other one's lower bound.
// The decisions equal those taken on all-canonical values.
struct BoundsScratch {
    unsigned long long *pos_lo, *pos_hi;                    // [positions] enclosures written by pass 1 (lo == 0: no row supplied)
    int32_t *pos_arg;                                       // [positions] what the selection kernel reads
    float *slice_partials; int32_t *row_tickets;            // scratch of pass 1: [max rows * 8 * 4] floats, [max rows] (zeroed)
    int32_t *pos_row; float *pos_max;                       // [positions] logits row and exact row maximum of each position (pass 1)
    TokenGrid grid;
};
constexpr int kRowStatsSlices = 8;
// true when the two-pass form applies to this logits layout (long bf16 rows, 16-byte aligned)
bool row_stats_two_pass_applies(const void *d_logits, int32_t logits_dtype, int32_t vocab, int64_t ld);
int32_t launch_row_stats_two_pass(const void *d_logits, int32_t vocab, int64_t ld, const int32_t *d_n_rows, int32_t max_rows,
                                  const int32_t *d_rows, const BoundsScratch &rf, int32_t *d_err, cudaStream_t stream);
// Which columns a record of the LM head's statistics covers: blocks of `block` columns, each with two records (epilogue-warp
// parities) that take its 64-column units in turn; record 2 b + p holds the units p, p + 2, ... of block b.
struct StatsLayout {
    int block, per_part;                                    // columns of a block, columns a record covers at most
    __host__ __device__ int column(int rec, int i) const    // i-th column of a record, -1 beyond its block
    {
        const int c = 64 * ((rec & 1) + 2 * (i >> 6)) + (i & 63);
        return c < block ? (rec >> 1) * block + c : -1;
    }
};
// the same with pass 1 already taken by the LM head's epilogue: `stats` holds n_parts records per row (stats_ld apart)
int32_t launch_row_stats_from_partials(const void *stats, int32_t stats_ld, int32_t n_parts, const StatsLayout &lay, const void *d_logits, int64_t ld, int32_t vocab, const int32_t *d_n_rows, int32_t max_rows,
                                       const int32_t *d_rows, const BoundsScratch &rf, int32_t *d_err, cudaStream_t stream);
// pass 1 alone, dense outputs by logits row (for tests): d_lo / d_hi enclose the canonical S_q
int32_t launch_row_stats_bounds(const void *d_logits, int32_t vocab, int64_t ld, const int32_t *d_n_rows, int32_t max_rows,
                                unsigned long long *d_lo, unsigned long long *d_hi, int32_t *d_argmax, int32_t *d_err, cudaStream_t stream);

struct LogitsRows { const uint4 *base; long long ld; int32_t chunks; };          // bf16 logits as 16-byte chunks, ld chunks between rows
constexpr int32_t kMayEnd = 1 << 30;
struct SelectArgs {
    int32_t *tokens; uint8_t *mask; int32_t B, S, P, L;
    sfs_state *state; sfs_params params;
    unsigned long long *pos_sq; int32_t *pos_arg;          // [B*S] scratch written by the row-stats kernel
    // two-pass form (pos_lo != NULL): the enclosures (pos_lo is cleared with pos_sq), and what recomputing a row takes
    unsigned long long *pos_lo; const unsigned long long *pos_hi;           // [B*S]
    const int32_t *pos_row; const float *pos_max;                           // [B*S]
    LogitsRows lrows;
    int32_t *seq_ticket;                                    // [B] scratch counters (zero between launches)
    int32_t groups;                                         // CTAs per sequence (set by the launcher)
    int32_t *sel_count, *sel_pos, *sel_tok;                 // [B], [B,L], [B,L]   (optional)
    int32_t *seq_rows, *seq_row_count;                      // [B,L], [B] scratch: next step's rows per sequence
    int32_t *next_rows, *next_n_rows;                       // optional flat list (sequence-major) + count
    int32_t *n_active;                                      // optional: sequences not done after this step
    int32_t *ticket;                                        // scratch counter (zero between launches)
    int32_t *trace;                                         // optional [B, SFS_TRACE_INTS]
    // host_active: [0] sequences still decoding, [1] steps finished, with kMayEnd when the next one may be the last
    int32_t *host_active, *step_count;                      // optional: the host's mirror, and the device's count of steps
};
int32_t select_fits(int32_t L);                             // SFS_OK, or the error of a response too long (before any statistics are written)
int32_t launch_select(const SelectArgs &a, cudaStream_t stream);
int32_t launch_state_init(sfs_state *d_state, int32_t B, int32_t L, const sfs_params &p, cudaStream_t stream);

}  // namespace sfs
