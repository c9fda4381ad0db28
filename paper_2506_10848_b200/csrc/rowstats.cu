// Row statistics of the sampling epilogue (paper Section 3.1): per logits row the greedy token
// r_hat = argmax_v x_v and the canonical fixed-point softmax denominator S_q (c = 2^28 / S_q).
//
// A thread-block cluster owns one row and HBM is read once.  Pass 1 finds the exact row maximum, the CTAs send their slice
// maxima to each other through distributed shared memory, pass 2 evaluates the fixed-point exponentials with packed f32x2
// arithmetic and sums them as integers; sums and first-maximum candidates go to rank 0 the same way.  Integer sums make the result independent of how the row is split over threads, warps and
// CTAs.  Rows stay in registers between the passes (any element type, length and alignment); many long aligned bf16 rows are
// staged: each of 8 CTAs brings its contiguous slice into shared memory with one bulk asynchronous copy (no registers tied up
// in flight, seven CTAs per SM).
#include "sfs_common.cuh"
#include "canonical.cuh"
#include "tc05.cuh"

#include <math_constants.h>

namespace sfs {
namespace {

// ---- what the CTAs of a row's cluster tell each other -------------------------------------------------------------
// Every CTA its slice maximum to every CTA, then its sum and its candidate for the argmax to rank 0.  Each value is a remote store
// that completes its bytes on a barrier of the receiver, who waits for exactly what it needs.  Nobody leaves while something is on its way
// to it: every CTA waits for all maxima, rank 0 for all sums.  With a cluster barrier for the maxima and remote atomics, a fence and an
// arrival counter for the sums, 64 rows of 126464 bf16 logits spent 1700 and 3800 of 13700 clocks here.
constexpr int kMostCtas = 8;
struct Exchange {
    float max_of[kMostCtas];
    uint4 part_of[kMostCtas];                               // rank 0: sum (two words) and candidate of every CTA
    unsigned long long bar_max, bar_part;
};
__device__ __forceinline__ void exchange_init(Exchange &x, int C)      // one thread; then the cluster's start barrier
{
    const uint32_t bar_max = tc::smem_u32(&x.bar_max), bar_part = tc::smem_u32(&x.bar_part);
    tc::mbar_init(bar_max, 1); tc::mbar_init(bar_part, 1);
    tc::mbar_init_fence();
    tc::mbar_expect_tx(bar_max, 4 * C); tc::mbar_expect_tx(bar_part, 16 * C);
}
__device__ __forceinline__ void send_max(Exchange &x, int rank, int to, float v)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
                 ::"r"(tc::mapa(tc::smem_u32(&x.max_of[rank]), to)), "r"(__float_as_uint(v)), "r"(tc::mapa(tc::smem_u32(&x.bar_max), to)) : "memory");
}
__device__ __forceinline__ void send_part(Exchange &x, int rank, unsigned long long sum, int arg)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(tc::mapa(tc::smem_u32(&x.part_of[rank]), 0)), "r"((uint32_t)sum), "r"((uint32_t)(sum >> 32)), "r"(arg), "r"(0), "r"(tc::mapa(tc::smem_u32(&x.bar_part), 0)) : "memory");
}
// the whole row's maximum: `mine` is this CTA's, the same in threads 0 .. C - 1 (called by all threads, after the start barrier)
__device__ __forceinline__ float exchange_max(Exchange &x, int C, int rank, float mine, int32_t *err)
{
    if ((int)threadIdx.x < C) send_max(x, rank, threadIdx.x, mine);
    tc::mbar_await(tc::smem_u32(&x.bar_max), err);
    float m = x.max_of[0];
    for (int r = 1; r < C; ++r) m = fmaxf(m, x.max_of[r]);
    return m;
}
// one thread of every CTA; true in rank 0, where `sum` and `arg` then are the row's
__device__ __forceinline__ bool exchange_parts(Exchange &x, int C, int rank, unsigned long long &sum, int &arg, int32_t *err)
{
    send_part(x, rank, sum, arg);
    if (rank != 0) return false;
    tc::mbar_await(tc::smem_u32(&x.bar_part), err);
    sum = 0; arg = 0x7FFFFFFF;
    for (int r = 0; r < C; ++r) { const uint4 p = x.part_of[r]; sum += (unsigned long long)p.y << 32 | p.x; arg = min(arg, (int)p.z); }
    return true;
}

__device__ __forceinline__ uint4 ld_stream(const uint4 *p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ __nv_bfloat162 as_bf162(uint32_t w) { return *reinterpret_cast<__nv_bfloat162 *>(&w); }
__device__ __forceinline__ float bf162_max(uint32_t w) {
    return fmaxf(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
}

struct RowOut {
    const int32_t *rows;            // flat token index per logits row, or null
    int32_t *argmax; unsigned long long *sq; float *conf;       // dense by logits row (optional)
    unsigned long long *pos_sq; int32_t *pos_arg;               // scattered by flat token index (optional)
    TokenGrid grid;                                             // positions of the scattered arrays
    int32_t *err;                                               // device status word (optional)
};

__device__ __forceinline__ void write_row(const RowOut &o, int row, int arg, unsigned long long S) {
    if (o.argmax) o.argmax[row] = arg;
    if (o.sq) o.sq[row] = S;
    if (o.conf) o.conf[row] = (float)((double)(1u << SFS_CONF_QBITS) / (double)S);
    if (o.rows && o.pos_sq) {
        const int p = o.rows[row];
        if (o.grid.inside(p)) {
            if (o.grid.response(p)) { o.pos_sq[p] = S; o.pos_arg[p] = arg; }
        } else if (o.err) {
            atomicExch(o.err, SFS_ERR_INVALID_ARG);               // a row index outside the token grid: skipped, reported
        }
    }
}

constexpr int kThreads = 256;
constexpr uint32_t kNegInf2 = 0xFF80FF80u;

// ---- a logits row as 16-byte chunks -----------------------------------------------------------------------------
// A row may start anywhere (its stride need not be a multiple of 16 bytes).  The `whole` chunks between its first and last 16-byte
// boundary come first, one vector load each; the elements before and after them, together, are the last one or two chunks, put
// together from the row's own elements with -inf in the places beyond (adds nothing, never is the maximum's first position).
// So an unaligned row has as many chunks as an aligned one: one more took another chunk of every thread's registers, or a
// second sweep, at every length that fills them (fp32 65536, 2048 rows: 345 us instead of 178 under the same rule).
template <typename T> struct RowChunks {
    static constexpr int PER = 16 / (int)sizeof(T);
    const uint4 *first;
    int head, whole, vocab;                                 // elements before the whole chunks, their number, elements in all
    __device__ __forceinline__ RowChunks(const T *logits, long long ld, int r, int V) {
        const T *row = logits + (long long)r * ld;
        const int off = (int)((unsigned long long)row & 15u) / (int)sizeof(T);
        vocab = V;
        head = off ? min(V, PER - off) : 0;
        first = reinterpret_cast<const uint4 *>(row + head);
        whole = (V - head) / PER;
    }
    __device__ __forceinline__ int chunks() const { return (vocab + PER - 1) / PER; }
    static __device__ __forceinline__ uint4 nothing();      // PER times -inf
    __device__ __forceinline__ uint4 load(int c) const { return c < whole ? ld_stream(first + c) : nothing(); }      // a whole chunk
    __device__ __forceinline__ uint4 load_edge(int c) const { return edge(first, head, whole, vocab, c); }          // whole <= c < chunks()
    // The chunks made of the row's two ends.  By value: with an address taken, the chunks a thread keeps would not stay in registers.
    static __device__ __forceinline__ int edge_index(int head, int whole, int vocab, int c, int e) {      // position of element e, -1: none
        const int k = (c - whole) * PER + e, ends = vocab - whole * PER;
        return k < head ? k : (k < ends ? k + whole * PER : -1);
    }
    static __device__ __noinline__ uint4 edge(const uint4 *first, int head, int whole, int vocab, int c);
    static __device__ __noinline__ int first_edge(int head, int whole, int vocab, int c, uint4 q, float m);      // first position of m in one
};
template <> __device__ __forceinline__ uint4 RowChunks<__nv_bfloat16>::nothing() { return make_uint4(kNegInf2, kNegInf2, kNegInf2, kNegInf2); }
template <> __device__ __forceinline__ uint4 RowChunks<float>::nothing() { return make_uint4(0xFF800000u, 0xFF800000u, 0xFF800000u, 0xFF800000u); }
template <> __device__ __noinline__ uint4 RowChunks<__nv_bfloat16>::edge(const uint4 *first, int head, int whole, int vocab, int c) {
    const unsigned short *row = reinterpret_cast<const unsigned short *>(first) - head;
    uint32_t h[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int i = edge_index(head, whole, vocab, c, e);
        h[e] = i >= 0 ? row[i] : 0xFF80u;
    }
    return make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
}
template <> __device__ __noinline__ uint4 RowChunks<float>::edge(const uint4 *first, int head, int whole, int vocab, int c) {
    const float *row = reinterpret_cast<const float *>(first) - head;
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int i = edge_index(head, whole, vocab, c, e);
        w[e] = i >= 0 ? __float_as_uint(row[i]) : 0xFF800000u;
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
// element e of a chunk, its maximum, and the sum of its terms (8 terms < 8 * 1.42 * 2^28 < 2^32)
template <typename T> __device__ __forceinline__ float chunk_elem(const uint4 &v, int e);
template <> __device__ __forceinline__ float chunk_elem<__nv_bfloat16>(const uint4 &v, int e) {
    const uint32_t w = (e >> 1) == 0 ? v.x : ((e >> 1) == 1 ? v.y : ((e >> 1) == 2 ? v.z : v.w));
    return (e & 1) ? __uint_as_float(w & 0xFFFF0000u) : __uint_as_float(w << 16);
}
template <> __device__ __forceinline__ float chunk_elem<float>(const uint4 &v, int e) {
    return __uint_as_float(e == 0 ? v.x : (e == 1 ? v.y : (e == 2 ? v.z : v.w)));
}
template <typename T> __device__ __noinline__ int RowChunks<T>::first_edge(int head, int whole, int vocab, int c, uint4 q, float m) {
    int best = 0x7FFFFFFF;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
        const int i = edge_index(head, whole, vocab, c, e);
        if (i >= 0 && chunk_elem<T>(q, e) == m) best = min(best, i);
    }
    return best;
}
template <typename T> __device__ __forceinline__ float chunk_max(const uint4 &v);
template <> __device__ __forceinline__ float chunk_max<__nv_bfloat16>(const uint4 &v) {
    __nv_bfloat162 m = __hmax2(__hmax2(as_bf162(v.x), as_bf162(v.y)), __hmax2(as_bf162(v.z), as_bf162(v.w)));
    return bf162_max(*reinterpret_cast<uint32_t *>(&m));
}
template <> __device__ __forceinline__ float chunk_max<float>(const uint4 &v) {
    return fmaxf(fmaxf(__uint_as_float(v.x), __uint_as_float(v.y)), fmaxf(__uint_as_float(v.z), __uint_as_float(v.w)));
}
template <typename T> __device__ __forceinline__ uint32_t chunk_terms(const uint4 &v, const Consts2 &k);
template <> __device__ __forceinline__ uint32_t chunk_terms<__nv_bfloat16>(const uint4 &v, const Consts2 &k) {
    return canon_pair(v.x, k) + canon_pair(v.y, k) + canon_pair(v.z, k) + canon_pair(v.w, k);
}
template <> __device__ __forceinline__ uint32_t chunk_terms<float>(const uint4 &v, const Consts2 &k) {
    return canon2(pack2(__uint_as_float(v.x), __uint_as_float(v.y)), k) + canon2(pack2(__uint_as_float(v.z), __uint_as_float(v.w)), k);
}

// One cluster (1, 2, 4 or 8 CTAs) of NT threads each per logits row, any element type, length and alignment; a thread keeps NV 16-byte
// chunks of the row in registers between the two passes (rows of more than C * NT * NV chunks read the rest a second time, from L2).
template <typename T, int NV, int NT>
__global__ void __launch_bounds__(NT, NT < 256 ? 16 : (NV > 8 ? 2 : 4))
rowstats_cluster(const T *__restrict__ logits, long long ld, int vocab, const int32_t *__restrict__ n_rows_ptr, int max_rows, RowOut out, int32_t *err)
{
    const int C = (int)tc::cluster_nctarank(), rank = (int)tc::cluster_ctarank();
    const int row  = blockIdx.x / C;
    pdl_wait();
    pdl_trigger();
    const int n_rows = n_rows_ptr ? min(*n_rows_ptr, max_rows) : max_rows;
    if (row >= n_rows) return;                              // uniform over the cluster

    __shared__ float s_wmax[NT / 32];
    __shared__ unsigned long long s_wsum[NT / 32];
    __shared__ __align__(16) Exchange s_x;
    __shared__ int s_cta_arg;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const RowChunks<T> rc(logits, ld, row, vocab);
    const int stride = C * NT, c0 = rank * NT + tid, n = rc.chunks();

    // this thread's chunks at the row's ends beyond those it keeps
    auto rest_of_edges = [&](auto &&f) {
        if (rc.whole < n)
            for (int c = max(rc.whole, NV * stride); c < n; ++c) if ((c - c0) % stride == 0) f(c, rc.load_edge(c));
    };

    // ---- the only pass over HBM: this thread's chunks of the row, kept in registers
    uint4 v[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] = rc.load(c0 + j * stride);
    if (rc.whole < n)
#pragma unroll
        for (int j = 0; j < NV; ++j) if (c0 + j * stride >= rc.whole && c0 + j * stride < n) v[j] = rc.load_edge(c0 + j * stride);
    if (tid == 0) { s_cta_arg = 0x7FFFFFFF; if (C > 1) exchange_init(s_x, C); }
    __syncwarp();                                           // (here and not only below: the compiler then has registers for all of v)
    // every CTA of the cluster announces that it runs (its shared memory exists) before anybody writes into a peer
    if (C > 1) tc::cluster_arrive();

    // ---- pass 1: exact maximum
    float lmax = -INFINITY;
#pragma unroll
    for (int j = 0; j < NV; ++j) lmax = fmaxf(lmax, chunk_max<T>(v[j]));
    for (int c = c0 + NV * stride; c < rc.whole; c += 4 * stride) {                  // the rest of a longer row: four loads in flight
        uint4 q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) q[u] = rc.load(c + u * stride);
#pragma unroll
        for (int u = 0; u < 4; ++u) lmax = fmaxf(lmax, chunk_max<T>(q[u]));
    }
    rest_of_edges([&](int, const uint4 &q) { lmax = fmaxf(lmax, chunk_max<T>(q)); });
    float m = warp_max(lmax);
    if (lane == 0) s_wmax[warp] = m;
    __syncthreads();
    m = s_wmax[0];
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) m = fmaxf(m, s_wmax[w]);
    if (C > 1) {
        tc::cluster_wait();                                 // all peers run
        m = exchange_max(s_x, C, rank, m, err);
    }

    // ---- first position of the maximum (only threads that hold it look)
    if (lmax == m) {
        int best = 0x7FFFFFFF;
        auto look = [&](int c, const uint4 &q) {
            int at = -1;
#pragma unroll
            for (int e = RowChunks<T>::PER - 1; e >= 0; --e) if (chunk_elem<T>(q, e) == m) at = e;
            if (at < 0 || c >= n) return;
            if (c < rc.whole) best = min(best, rc.head + c * RowChunks<T>::PER + at);
            else best = min(best, RowChunks<T>::first_edge(rc.head, rc.whole, rc.vocab, c, q, m));
        };
#pragma unroll
        for (int j = 0; j < NV; ++j) look(c0 + j * stride, v[j]);
        for (int c = c0 + NV * stride; c < rc.whole && best == 0x7FFFFFFF; c += stride) look(c, rc.load(c));
        rest_of_edges(look);                                                      // (they may hold the row's beginning)
        if (best != 0x7FFFFFFF) atomicMin(&s_cta_arg, best);
    }

    // ---- pass 2: fixed-point exponentials, integer sum
    const Consts2 k = canon_consts(m);
    unsigned long long acc = 0;
#pragma unroll
    for (int j = 0; j < NV; ++j) acc += chunk_terms<T>(v[j], k);
    for (int c = c0 + NV * stride; c < rc.whole; c += 4 * stride) {
        uint4 q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) q[u] = rc.load(c + u * stride);
#pragma unroll
        for (int u = 0; u < 4; ++u) acc += chunk_terms<T>(q[u], k);
    }
    rest_of_edges([&](int, const uint4 &q) { acc += chunk_terms<T>(q, k); });
    acc = warp_sum_u64(acc);
    if (lane == 0) s_wsum[warp] = acc;
    __syncthreads();
    if (tid == 0) {
        unsigned long long t = 0;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) t += s_wsum[w];
        int arg = s_cta_arg;
        if (C == 1 || exchange_parts(s_x, C, rank, t, arg, err)) write_row(out, row, arg == 0x7FFFFFFF ? 0 : arg, t);
    }
}

// ---- long rows: slices staged in shared memory ------------------------------------------------------------------
// Same arithmetic, other staging: a cluster of 8 CTAs of 128 threads owns a row, and each CTA brings its contiguous slice
// into shared memory with ONE bulk asynchronous copy, so no registers are tied up while the bytes are in flight and seven
// CTAs (seven 32 KB slices) fit an SM instead of four.  The two passes then read shared memory.
constexpr int kStagedThreads = 128;
constexpr int kStagedCluster = 8;

__global__ void __launch_bounds__(kStagedThreads)
rowstats_staged_bf16(const uint4 *__restrict__ logits, long long ld_chunks, int nchunks, int per_cta, int vocab,
                     const int32_t *__restrict__ n_rows_ptr, int max_rows, RowOut out, int32_t *err)
{
    const int C = (int)tc::cluster_nctarank(), rank = (int)tc::cluster_ctarank();
    const int row  = blockIdx.x / C;
    pdl_wait();
    pdl_trigger();
    const int n_rows = n_rows_ptr ? min(*n_rows_ptr, max_rows) : max_rows;
    if (row >= n_rows) return;                              // uniform over the cluster

    extern __shared__ __align__(16) uint4 s_slice[];
    __shared__ __align__(8) unsigned long long s_bar;
    __shared__ float s_wmax[kStagedThreads / 32];
    __shared__ unsigned long long s_wsum[kStagedThreads / 32];
    __shared__ __align__(16) Exchange s_x;
    __shared__ int s_cta_arg;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c0 = rank * per_cta;                          // first 16-byte chunk of this CTA's slice
    const int n = max(0, min(per_cta, nchunks - c0));
    const uint32_t bar = tc::smem_u32(&s_bar);
    if (tid == 0) {
        s_cta_arg = 0x7FFFFFFF;
        exchange_init(s_x, C);
        tc::mbar_init(bar, 1);
        tc::mbar_init_fence();
        if (n > 0) {
            const uint32_t bytes = (uint32_t)n * 16u;
            tc::mbar_expect_tx(bar, bytes);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(tc::smem_u32(s_slice)), "l"(logits + (long long)row * ld_chunks + c0), "r"(bytes), "r"(bar) : "memory");
        } else {
            tc::mbar_arrive(bar);
        }
    }
    __syncthreads();
    // every CTA of the cluster announces that it runs (its shared memory exists) before anybody writes into a peer
    tc::cluster_arrive();
    tc::mbar_await(bar, err);                               // the slice

    // ---- pass 1: exact maximum
    __nv_bfloat162 mx = as_bf162(kNegInf2);
    for (int c = tid; c < n; c += kStagedThreads) {
        const uint4 v = s_slice[c];
        mx = __hmax2(mx, __hmax2(__hmax2(as_bf162(v.x), as_bf162(v.y)), __hmax2(as_bf162(v.z), as_bf162(v.w))));
    }
    const float lmax = bf162_max(*reinterpret_cast<uint32_t *>(&mx));
    float m = warp_max(lmax);
    if (lane == 0) s_wmax[warp] = m;
    __syncthreads();
    tc::cluster_wait();                                     // all peers run
    m = s_wmax[0];
#pragma unroll
    for (int w = 1; w < kStagedThreads / 32; ++w) m = fmaxf(m, s_wmax[w]);
    m = exchange_max(s_x, C, rank, m, err);

    // ---- first position of the maximum (only threads that hold it look), then pass 2
    if (lmax == m) {
        int best = 0x7FFFFFFF;
        for (int c = tid; c < n && best == 0x7FFFFFFF; c += kStagedThreads) {
            const uint4 v = s_slice[c];
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 7; e >= 0; --e) {
                const float x = (e & 1) ? __uint_as_float(w[e >> 1] & 0xFFFF0000u) : __uint_as_float(w[e >> 1] << 16);
                const int idx = (c0 + c) * 8 + e;
                if (x == m && idx < vocab) best = idx;
            }
        }
        if (best != 0x7FFFFFFF) atomicMin(&s_cta_arg, best);
    }
    const Consts2 k = canon_consts(m);
    unsigned long long acc = 0;
#pragma unroll 4
    for (int c = tid; c < n; c += kStagedThreads) {
        const uint4 v = s_slice[c];
        const uint32_t a = canon_pair(v.x, k) + canon_pair(v.y, k) + canon_pair(v.z, k) + canon_pair(v.w, k);
        acc += a;                                           // 8 terms < 8 * 1.42 * 2^28 < 2^32
    }
    acc = warp_sum_u64(acc);
    if (lane == 0) s_wsum[warp] = acc;
    __syncthreads();
    if (tid == 0) {
        unsigned long long t = 0;
#pragma unroll
        for (int w = 0; w < kStagedThreads / 32; ++w) t += s_wsum[w];
        int arg = s_cta_arg;
        if (exchange_parts(s_x, C, rank, t, arg, err)) write_row(out, row, arg == 0x7FFFFFFF ? 0 : arg, t);
    }
}

// ---- pass 1 of the two-pass form: exact maximum / argmax, approximate denominator with a proven enclosure -----------------
// No staging and no cluster here: a row is cut into kSlices slices, one CTA per (row, slice) streams its slice straight from
// HBM into registers (kInFlight 16-byte loads per thread in flight) and evaluates it as it arrives.  Measured on 256 rows of
// 126464 logits, back to back, cold: a bare read of the 64.75 MB takes 12.5 us, this kernel 18.4 us, the staged cluster form
// of the same arithmetic 27 us (its staging and cluster barrier, not its arithmetic, set the pace).  Packed f32x2 arithmetic,
// a deeper or software-pipelined load queue and fewer registers each moved the time by less than 1 us: the special-function
// unit (two ex2 per 32-bit word: 7 us of its time) overlaps the loads only in part, and every CTA ends with the same short
// serial tail (block reduction, ticket).  The canonical kernel needs the row maximum before its first term and keeps the
// staged form.  The exponentials are taken against a reference c = the maximum of the WARP's first batch of chunks (no
// CTA-wide barrier before the stream starts); a warp's sum is moved to the slice maximum when the CTA reduces, and the CTA
// that completes a row (a ticket per row) moves the slice sums to the row maximum and adds them in slice order:
//     S~ = sum over slices, warps of ex2((c - m) log2 e) * sum_v ex2.approx(fma(x_v, log2 e, -c log2 e))       (fp32)
// The canonical S_q = sum_v trunc(2^28 exp~(x_v - m)) lies in
//     [ 2^28 S~ (1 - eps) - V - 1 ,  2^28 S~ (1 + eps) + 1 ]  intersected with [2^28, inf):
// the canonical exponential is within 1e-5 relative of exp (degree-4 fit 3.3e-6, its fp32 steps < 1e-6) and truncation loses
// less than 1 per term (V terms); on this side an exponent (x - c) log2 e of magnitude up to 100 is rounded to 2^-24
// relative (< 6e-6 absolute, i.e. < 4.2e-6 relative in the term), the same again for each of the two moves, ex2.approx is
// within 2^-22 three times, and the fp32 sums (at most 32 sequential adds per thread, then pairwise levels) within 3e-6.
// Worst case 2.8e-5.  Besides, -c log2 e, and the same of a slice's and of the row's maximum, are rounded to 2^-24 of their magnitude,
// which shifts every term of a sum alike: relative 2^-24 |c| each, and a reference lies at most 100 log 2 below the maximum, so
// 3 * 2^-24 (|m| + 70) in all.  The enclosure takes 6e-5, which holds both up to |m| = 100, and their sum beyond (with 6e-5 throughout rows
// with logits of 600 and more lay outside theirs).  A reference more than 100 (in log2 units) below the maximum it is moved to, and a sum
// that is not a finite number >= 1, yield an enclosure that contains everything, which sends the row to the canonical pass.
constexpr double kEps = 6e-5, kEpsTerms = 2.8e-5, kEpsPerUnit = 1.8e-7;
constexpr int kSlices = 8;
constexpr int kBoundsThreads = 128;

__device__ __forceinline__ float ex2_fast(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }

struct BoundsOut {
    const int32_t *rows;                                    // flat token index per logits row, or null (dense outputs only)
    unsigned long long *lo, *hi; int32_t *argmax;           // dense by logits row (optional)
    unsigned long long *pos_lo, *pos_hi; int32_t *pos_arg;  // scattered by flat token index (optional)
    int32_t *pos_row;                                       // with them: the logits row a position's statistics came from
    float *pos_max;                                         //            and the exact row maximum
    TokenGrid grid; int32_t *err;
    float4 *partial;                                        // scratch [max_rows * kSlices]: (slice max, reference, sum, argmax bits)
    int32_t *tickets;                                       // scratch [max_rows], zero between launches
};

// the enclosure of the canonical S_q from the approximate sum `tot` (relative to the row maximum m), and the scattered outputs
__device__ __forceinline__ void write_enclosure(const BoundsOut &out, int row, float tot, int arg, float m, bool open, int vocab, bool certain = false)
{
    if (arg == 0x7FFFFFFF) arg = 0;
    const double Sd = (double)tot * (double)(1u << SFS_CONF_QBITS);
    const double eps = fmax(kEps, kEpsTerms + kEpsPerUnit * (fabs((double)m) + 70.0));
    const double dlo = Sd * (1.0 - eps) - (double)vocab - 1.0, dhi = Sd * (1.0 + eps) + 1.0;
    const unsigned long long floor_q = 1ull << SFS_CONF_QBITS;     // the maximum alone contributes 2^28
    unsigned long long lo = dlo > (double)floor_q ? (unsigned long long)dlo : floor_q;
    unsigned long long hi = (unsigned long long)dhi + 1ull;
    if (open || !(eps <= 0.25) || !(tot >= 0.999f) || !(tot <= 3.0e38f)) { lo = 1ull; hi = ~0ull >> 1; }
    if (certain) lo = hi = floor_q;
    if (out.lo) out.lo[row] = lo;
    if (out.hi) out.hi[row] = hi;
    if (out.argmax) out.argmax[row] = arg;
    if (out.rows && out.pos_lo) {
        const int p = out.rows[row];
        if (out.grid.inside(p)) {
            if (!out.grid.response(p)) return;
            out.pos_lo[p] = lo; out.pos_hi[p] = hi; out.pos_arg[p] = arg; out.pos_row[p] = row; out.pos_max[p] = m;
        } else if (out.err) {
            atomicExch(out.err, SFS_ERR_INVALID_ARG);
        }
    }
}

// Pass 1 when the LM head has already taken the statistics in its epilogue: per row, n_parts records (maximum, reference,
// sum of 2^((x - reference) log2 e), first position of the maximum) are combined exactly like the slices of the streaming
// kernel — one warp per row, the lanes' shares added in a fixed order — into the row's argmax and enclosure.  Of the logits
// only the columns of the record that holds the maximum are read: with the other records' maxima they give the second largest
// logit, and when that is more than 19.5 below the maximum every other term of the canonical S_q is trunc(2^28 exp(< -19.5)) = 0
// (2^28 exp(-19.5) = 0.91), so S_q is 2^28 exactly.  Such rows (confidence above 0.9996, most of a confident model's) all lie in
// each other's enclosures otherwise, and a ranking step recomputed every one of them (256 rows: 50 us).
__global__ void __launch_bounds__(128)
combine_partials_kernel(const float4 *__restrict__ stats, int stats_ld, int n_parts, const int32_t *__restrict__ n_rows_ptr, int max_rows,
                        int vocab, BoundsOut out, const __nv_bfloat16 *__restrict__ logits, long long ld, StatsLayout lay)
{
    pdl_wait();
    pdl_trigger();
    const int row = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int n_rows = n_rows_ptr ? min(*n_rows_ptr, max_rows) : max_rows;
    if (row >= n_rows) return;
    const float4 *ps = stats + (long long)row * stats_ld;
    float m = -INFINITY;
    for (int q = lane; q < n_parts; q += 32) m = fmaxf(m, __ldg(&ps[q]).x);
    m = warp_max(m);
    const float nm = __fmul_rn(-m, kLog2e);
    int arg = 0x7FFFFFFF;
    float tot = 0.f;
    int open = 0;
    for (int q = lane; q < n_parts; q += 32) {
        const float4 r = __ldg(&ps[q]);
        if (r.x == m) arg = min(arg, __float_as_int(r.w));
        if (r.z != 0.f) {
            const float shift = __fmaf_rn(r.y, kLog2e, nm);
            if (!(shift >= -100.f) || !(shift <= 100.f)) open = 1;
            tot += r.z * ex2_fast(shift);
        }
    }
    tot = warp_sum(tot);
    arg = warp_min_i32(arg);
    open = warp_max_i32(open);
    // the second largest logit: the other records' maxima, and the other columns of the record that holds position arg
    float m2 = -INFINITY;
    int own = -1;
    for (int q = lane; q < n_parts; q += 32) {
        const float4 r = __ldg(&ps[q]);
        if (r.x == m && __float_as_int(r.w) == arg) own = q;
        else m2 = fmaxf(m2, r.x);
    }
    own = warp_max_i32(own);
    if (own >= 0) {
        const __nv_bfloat16 *rp = logits + (long long)row * ld;
        for (int i = lane; i < lay.per_part; i += 32) {
            const int c = lay.column(own, i);
            if (c >= 0 && c < vocab && c != arg) m2 = fmaxf(m2, __bfloat162float(rp[c]));
        }
    }
    m2 = warp_max(m2);
    const bool certain = own >= 0 && fabsf(m) <= 3.0e38f && m2 - m < -19.5f;
    if (lane == 0) write_enclosure(out, row, tot, arg, m, open != 0, vocab, certain);
}

__device__ __forceinline__ uint32_t chunk_max2(const uint4 &v) {
    __nv_bfloat162 m = __hmax2(__hmax2(as_bf162(v.x), as_bf162(v.y)), __hmax2(as_bf162(v.z), as_bf162(v.w)));
    return *reinterpret_cast<uint32_t *>(&m);
}

template <int kInFlight>
__global__ void __launch_bounds__(kBoundsThreads)
rowstats_bounds_bf16(const uint4 *__restrict__ logits, long long ld_chunks, int nchunks, int vocab,
                     const int32_t *__restrict__ n_rows_ptr, int max_rows, int slices, BoundsOut out)
{
    const int row = blockIdx.x / slices, sl = blockIdx.x - row * slices;
    pdl_wait();
    pdl_trigger();
    const int n_rows = n_rows_ptr ? min(*n_rows_ptr, max_rows) : max_rows;
    if (row >= n_rows) return;
    const int per = (nchunks + slices - 1) / slices;
    const int c0 = sl * per, c1 = min(nchunks, c0 + per);
    const uint4 *rp = logits + (long long)row * ld_chunks;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NW = kBoundsThreads / 32;
    __shared__ float s_wmax[NW], s_wsum[NW], s_wref[NW];
    __shared__ int s_arg;
    const uint4 neg = make_uint4(kNegInf2, kNegInf2, kNegInf2, kNegInf2);

    // ---- first batch: also gives the reference, per warp (no CTA-wide barrier before the stream starts)
    uint4 v[kInFlight], nx[kInFlight];
#pragma unroll
    for (int u = 0; u < kInFlight; ++u) { const int c = c0 + tid + u * kBoundsThreads; v[u] = c < c1 ? ld_stream(rp + c) : neg; }
    int c = c0 + tid + kInFlight * kBoundsThreads;
#pragma unroll
    for (int u = 0; u < kInFlight; ++u) { const int cc = c + u * kBoundsThreads; nx[u] = cc < c1 ? ld_stream(rp + cc) : neg; }
    if (tid == 0) s_arg = 0x7FFFFFFF;
    float fm = -INFINITY;
#pragma unroll
    for (int u = 0; u < kInFlight; ++u) fm = fmaxf(fm, bf162_max(chunk_max2(v[u])));
    float cref = warp_max(fm);
    if (!(fabsf(cref) <= 3.0e38f)) cref = 0.f;
    const float nc = __fmul_rn(-cref, kLog2e);

    float mx = -INFINITY, a0 = 0.f, a1 = 0.f;
    int best_c = -1;
    auto eat = [&](const uint4 &q, int cq) {
        const float cm = bf162_max(chunk_max2(q));
        if (cm > mx) { mx = cm; best_c = cq; }              // strict: the first chunk of this thread that holds its maximum
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
        float e[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            e[2 * k] = ex2_fast(__fmaf_rn(__uint_as_float(w[k] << 16), kLog2e, nc));
            e[2 * k + 1] = ex2_fast(__fmaf_rn(__uint_as_float(w[k] & 0xFFFF0000u), kLog2e, nc));
        }
        a0 += (e[0] + e[1]) + (e[2] + e[3]); a1 += (e[4] + e[5]) + (e[6] + e[7]);
    };
    int cur = c0 + tid;
#pragma unroll
    for (int u = 0; u < kInFlight; ++u) if (cur + u * kBoundsThreads < c1) eat(v[u], cur + u * kBoundsThreads);
    cur += kInFlight * kBoundsThreads;
#pragma unroll
    for (int u = 0; u < kInFlight; ++u) if (cur + u * kBoundsThreads < c1) eat(nx[u], cur + u * kBoundsThreads);
    cur += kInFlight * kBoundsThreads;
    for (; cur < c1; cur += kInFlight * kBoundsThreads) {
#pragma unroll
        for (int u = 0; u < kInFlight; ++u) { const int cc = cur + u * kBoundsThreads; v[u] = cc < c1 ? ld_stream(rp + cc) : neg; }
#pragma unroll
        for (int u = 0; u < kInFlight; ++u) if (cur + u * kBoundsThreads < c1) eat(v[u], cur + u * kBoundsThreads);
    }

    // ---- slice maximum, its first position, slice sum
    const float wm = warp_max(mx), ws = warp_sum(a0 + a1);
    if (lane == 0) { s_wmax[warp] = wm; s_wsum[warp] = ws; s_wref[warp] = cref; }
    __syncthreads();
    const float m_slice = fmaxf(fmaxf(s_wmax[0], s_wmax[1]), fmaxf(s_wmax[2], s_wmax[3]));
    if (mx == m_slice && best_c >= 0) {
        const uint4 q = rp[best_c];                         // this thread's first chunk that holds the slice maximum
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
        int best = 0x7FFFFFFF;
#pragma unroll
        for (int e = 7; e >= 0; --e) {
            const float x = (e & 1) ? __uint_as_float(w[e >> 1] & 0xFFFF0000u) : __uint_as_float(w[e >> 1] << 16);
            const int idx = best_c * 8 + e;
            if (x == m_slice && idx < vocab) best = idx;
        }
        if (best != 0x7FFFFFFF) atomicMin(&s_arg, best);
    }
    __syncthreads();
    if (tid != 0) return;
    // the warps' sums, moved from each warp's reference to the slice maximum (the table holds sums relative to it)
    float sum = 0.f;
    bool far = false;
    const float nms = __fmul_rn(-m_slice, kLog2e);
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        if (s_wsum[w] == 0.f) continue;                     // nothing finite in this warp's share
        const float shift = __fmaf_rn(s_wref[w], kLog2e, nms);
        if (!(shift >= -100.f)) far = true;
        sum += s_wsum[w] * ex2_fast(shift);
    }
    if (far) sum = CUDART_INF_F;                            // leaves the row to the canonical pass
    out.partial[(long long)row * kSlices + sl] = make_float4(m_slice, m_slice, c1 > c0 ? sum : 0.f, __int_as_float(s_arg));
    __threadfence();
    if (atomicAdd(&out.tickets[row], 1) != slices - 1) return;

    // ---- the CTA that completes the row combines its slices, in slice order
    __threadfence();
    out.tickets[row] = 0;
    float4 ps[kSlices];
#pragma unroll
    for (int q = 0; q < kSlices; ++q)
        ps[q] = q < slices ? __ldcg(&out.partial[(long long)row * kSlices + q]) : make_float4(-INFINITY, 0.f, 0.f, __int_as_float(0x7FFFFFFF));
    float m = ps[0].x;
#pragma unroll
    for (int q = 1; q < kSlices; ++q) m = fmaxf(m, ps[q].x);
    int arg = 0x7FFFFFFF;
    float tot = 0.f;
    bool open = false;
    const float nm = __fmul_rn(-m, kLog2e);
#pragma unroll
    for (int q = 0; q < kSlices; ++q) {
        if (ps[q].x == m && arg == 0x7FFFFFFF) arg = __float_as_int(ps[q].w);     // slices are in position order
        if (ps[q].z != 0.f) {
            const float shift = __fmaf_rn(ps[q].y, kLog2e, nm);                      // (c - m) log2 e <= 0
            if (!(shift >= -100.f)) open = true;                                     // the reference was too far below the maximum
            tot += ps[q].z * ex2_fast(shift);
        }
    }
    write_enclosure(out, row, tot, arg, m, open, vocab);
}

int num_sms_rowstats()
{
    static int n[kMaxDevices] = {};
    int &v = n[current_device_slot()];
    if (v == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 148;
    }
    return v;
}

int32_t launch_staged(const uint4 *logits, long long ld_chunks, int nchunks, int vocab, const int32_t *d_n_rows,
                      int max_rows, const RowOut &out, cudaStream_t stream)
{
    const int per_cta = (nchunks + kStagedCluster - 1) / kStagedCluster;
    SFS_CUDA(launch_pdl_cluster(rowstats_staged_bf16, kStagedCluster, dim3((unsigned)(max_rows * kStagedCluster)), dim3(kStagedThreads),
                                (size_t)per_cta * 16, stream, logits, ld_chunks, nchunks, per_cta, vocab, d_n_rows, max_rows, out, out.err));
    return SFS_OK;
}

int32_t launch_bounds(const uint4 *logits, long long ld_chunks, int nchunks, int vocab, const int32_t *d_n_rows, int max_rows,
                      const BoundsOut &out, cudaStream_t stream)
{
    // slices per row (at most kSlices): the count whose CTAs fill whole waves best at 9 resident CTAs per SM, longer slices
    // winning ties (fewer reductions); a last wave that is nearly empty costs as much as a full one
    const int per_wave = 9 * num_sms_rowstats();
    int slices = kSlices;
    double best = -1.0;
    for (int sl = kSlices; sl >= 3; --sl) {
        const long long ctas = (long long)max_rows * sl, waves = (ctas + per_wave - 1) / per_wave;
        const double fill = (double)ctas / (double)(waves * per_wave);
        if (fill > best + 0.02) { best = fill; slices = sl; }
    }
    SFS_CUDA(launch_pdl(rowstats_bounds_bf16<4>, dim3((unsigned)(max_rows * slices)), dim3(kBoundsThreads), 0, stream, logits, ld_chunks,
                        nchunks, vocab, d_n_rows, max_rows, slices, out));
    return SFS_OK;
}

template <typename T, int NV, int NT = kThreads>
int32_t launch_cluster(const void *logits, long long ld, int vocab, const int32_t *d_n_rows, int max_rows, int C, const RowOut &out, cudaStream_t stream)
{
    SFS_CUDA(launch_pdl_cluster(rowstats_cluster<T, NV, NT>, C, dim3((unsigned)(max_rows * C)), dim3(NT), 0, stream,
                                reinterpret_cast<const T *>(logits), ld, vocab, d_n_rows, max_rows, out, out.err));
    return SFS_OK;
}

template <typename T>
int32_t launch_rows(const void *logits, long long ld, int vocab, const int32_t *d_n_rows, int max_rows, const RowOut &out, cudaStream_t stream)
{
    // Cluster size and chunks kept per thread.  A cluster costs a barrier and each of its CTAs ~2 us besides its chunks, so the fewest
    // CTAs are best that leave a thread no more chunks than the other rows' CTAs hide: the more rows, the more of a row may be read a
    // second time (from L2).  Below one CTA per SM more of them, down to 4 chunks a thread.  16 chunks are kept while two CTAs per SM
    // hold all rows, or where that saves the second reading without a cluster.  us at 64 / 256 / 512 / 2048 rows, in brackets with the rule
    // before (65 % of every row in registers):
    //   bf16 16384 3.9 / 5.0 / 7.8 / 25 [3.9 / 6.8 / 8.5 / 27], 32000 4.9 / 7.6 / 14.3 / 45 [4.9 / 9.8 / 17.2 / 58], 50257 7.3 / 17.2 / 27.8 / 83 [7.3 / 17.4 / 31 / 103];
    //   fp32 16384 4.2 / 5.8 / 11.2 / 33 [4.2 / 7.6 / 13.6 / 44], 65536 7.1 / 24 / 43 / 133 [7.5 / 25 / 47 / 172], 100000 11.6 / 36 / 62 / 210 [12.3 / 42 / 80 / 307];
    //   at odd addresses bf16 126464 8.9 / 33 / 58 / 184 [10.3 / 35 / 66 / 250], fp32 65536 7.1 / 26 / 46 / 139 [12.5 / 46 / 90 / 346].
    // Rows of up to 2 KB take CTAs of 64 threads: 2048 rows of 64 bf16 values 5.8 [8.0].
    const int nchunks = (int)((vocab * (long long)sizeof(T) + 15) / 16);
    if (nchunks <= 128) return launch_cluster<T, 2, 64>(logits, ld, vocab, d_n_rows, max_rows, 1, out, stream);
    const int most = max_rows >= 1024 ? 33 : (max_rows >= 384 ? 25 : 19);      // chunks per thread
    int C = 1;
    while (C < 8 && nchunks > C * kThreads * most) C *= 2;
    while (C < 8 && (long long)max_rows * C < 128 && nchunks > C * 4 * kThreads) C *= 2;
    const int per_thread = (nchunks + C * kThreads - 1) / (C * kThreads);
    if (per_thread <= 1) return launch_cluster<T, 1>(logits, ld, vocab, d_n_rows, max_rows, C, out, stream);
    if (per_thread <= 2) return launch_cluster<T, 2>(logits, ld, vocab, d_n_rows, max_rows, C, out, stream);
    if (per_thread <= 4) return launch_cluster<T, 4>(logits, ld, vocab, d_n_rows, max_rows, C, out, stream);
    if (per_thread <= 8 || !((long long)max_rows * C <= 400 || (C == 1 && per_thread <= 16)))
        return launch_cluster<T, 8>(logits, ld, vocab, d_n_rows, max_rows, C, out, stream);
    return launch_cluster<T, 16>(logits, ld, vocab, d_n_rows, max_rows, C, out, stream);
}

}  // namespace

static bool staged_shape(int32_t logits_dtype, int32_t vocab, int64_t ld, const void *d_logits)
{
    const bool fast = logits_dtype == SFS_LOGITS_BF16 && (vocab % 8) == 0 && (ld % 8) == 0 && aligned_to(d_logits, 16);
    const int nchunks = vocab / 8;
    return fast && nchunks >= 8192 && (nchunks + kStagedCluster - 1) / kStagedCluster <= 2560;
}

int32_t launch_row_stats(const void *d_logits, int32_t logits_dtype, int32_t vocab, int64_t ld,
                         const int32_t *d_n_rows, int32_t max_rows, const int32_t *d_rows,
                         int32_t *d_argmax, unsigned long long *d_sq, float *d_conf,
                         unsigned long long *d_pos_sq, int32_t *d_pos_arg, TokenGrid grid, int32_t *d_err,
                         cudaStream_t stream)
{
    if (max_rows <= 0) return SFS_OK;
    RowOut out{d_rows, d_argmax, d_sq, d_conf, d_pos_sq, d_pos_arg, grid, d_err};
    if (staged_shape(logits_dtype, vocab, ld, d_logits)) {
        const int nchunks = vocab / 8;
        // Long rows (128 KB and more, slices of at most 40 KB): staged through shared memory, seven CTAs to an SM, unless the rows
        // are so few that the register form's CTAs are resident at once.  us, staged against registers: 126464 bf16 logits 64 rows 10.0 /
        // 8.6, 128 rows 17.0 / 17.1, 512 rows 46 / 54; 151936, more than eight chunks a thread of eight CTAs, 4 rows 7.0 / 6.3, 16 rows 6.9 / 8.2,
        // 64 rows 10.8 / 11.7.
        const long long resident = nchunks > 8 * 8 * kThreads ? 32 : 4 * num_sms_rowstats();
        if ((long long)max_rows * kStagedCluster > resident)
            return launch_staged(reinterpret_cast<const uint4 *>(d_logits), ld / 8, nchunks, vocab, d_n_rows, max_rows, out, stream);
    }
    return logits_dtype == SFS_LOGITS_BF16 ? launch_rows<__nv_bfloat16>(d_logits, ld, vocab, d_n_rows, max_rows, out, stream)
                                           : launch_rows<float>(d_logits, ld, vocab, d_n_rows, max_rows, out, stream);
}

bool row_stats_two_pass_applies(const void *d_logits, int32_t logits_dtype, int32_t vocab, int64_t ld)
{
    return staged_shape(logits_dtype, vocab, ld, d_logits);
}

int32_t launch_row_stats_bounds(const void *d_logits, int32_t vocab, int64_t ld, const int32_t *d_n_rows, int32_t max_rows,
                                unsigned long long *d_lo, unsigned long long *d_hi, int32_t *d_argmax, int32_t *d_err, cudaStream_t stream)
{
    if (max_rows <= 0) return SFS_OK;
    SFS_REQUIRE(staged_shape(SFS_LOGITS_BF16, vocab, ld, d_logits), SFS_ERR_UNSUPPORTED,
                "row-statistics enclosures: bf16 rows of 65536 to 163840 entries, 16-byte aligned, only");
    // scratch of this entry point: one table per device, grown on demand and kept (the selection path brings its session's)
    static float4 *s_partial[kMaxDevices] = {};
    static int32_t *s_tickets[kMaxDevices] = {};
    static int s_rows[kMaxDevices] = {};
    const int dev = current_device_slot();
    if (s_rows[dev] < max_rows) {
        SFS_CUDA(cudaDeviceSynchronize());
        if (s_partial[dev]) { cudaFree(s_partial[dev]); cudaFree(s_tickets[dev]); s_partial[dev] = nullptr; s_tickets[dev] = nullptr; s_rows[dev] = 0; }
        SFS_CUDA(cudaMalloc(&s_partial[dev], (size_t)max_rows * kSlices * sizeof(float4)));
        SFS_CUDA(cudaMalloc(&s_tickets[dev], (size_t)max_rows * sizeof(int32_t)));
        SFS_CUDA(cudaMemset(s_tickets[dev], 0, (size_t)max_rows * sizeof(int32_t)));
        s_rows[dev] = max_rows;
    }
    BoundsOut out{nullptr, d_lo, d_hi, d_argmax, nullptr, nullptr, nullptr, nullptr, nullptr, TokenGrid{0, 1, 0}, d_err, s_partial[dev], s_tickets[dev]};
    return launch_bounds(reinterpret_cast<const uint4 *>(d_logits), ld / 8, vocab / 8, vocab, d_n_rows, max_rows, out, stream);
}

int32_t launch_row_stats_two_pass(const void *d_logits, int32_t vocab, int64_t ld, const int32_t *d_n_rows, int32_t max_rows,
                                  const int32_t *d_rows, const BoundsScratch &rf, int32_t *d_err, cudaStream_t stream)
{
    if (max_rows <= 0) return SFS_OK;
    const uint4 *lp = reinterpret_cast<const uint4 *>(d_logits);
    BoundsOut bo{d_rows, nullptr, nullptr, nullptr, rf.pos_lo, rf.pos_hi, rf.pos_arg, rf.pos_row, rf.pos_max, rf.grid, d_err,
                 reinterpret_cast<float4 *>(rf.slice_partials), rf.row_tickets};
    int32_t rc = launch_bounds(lp, ld / 8, vocab / 8, vocab, d_n_rows, max_rows, bo, stream);
    if (rc != SFS_OK) return rc;
    return SFS_OK;
}

int32_t launch_row_stats_from_partials(const void *stats, int32_t stats_ld, int32_t n_parts, const StatsLayout &lay, const void *d_logits, int64_t ld, int32_t vocab, const int32_t *d_n_rows, int32_t max_rows, const int32_t *d_rows, const BoundsScratch &rf, int32_t *d_err,
                                       cudaStream_t stream)
{
    if (max_rows <= 0) return SFS_OK;
    BoundsOut bo{d_rows, nullptr, nullptr, nullptr, rf.pos_lo, rf.pos_hi, rf.pos_arg, rf.pos_row, rf.pos_max, rf.grid, d_err,
                 nullptr, nullptr};
    SFS_CUDA(launch_pdl(combine_partials_kernel, dim3((unsigned)((max_rows + 3) / 4)), dim3((unsigned)(128)), (size_t)(0), stream, reinterpret_cast<const float4 *>(stats), stats_ld, n_parts, d_n_rows, max_rows, vocab, bo,
                        reinterpret_cast<const __nv_bfloat16 *>(d_logits), (long long)ld, lay));
    return SFS_OK;
}

}  // namespace sfs
