// Feature cache of the mask predictor (the adaptive caching the paper's sampler integrates, Section 2.2 and the
// (K_p, K_r) settings of Table 4): value-similarity sums, the least-similar row choice, and the gathers / scatters
// that move the recomputed rows between the compact buffers the GEMMs work on and the per-layer caches.
#include "sfs_common.cuh"
#include "cache.cuh"

namespace sfs {
namespace {

// Fresh (a) and cached (b) values are bf16, features x tokens; a's columns begin with token t_first.  An unchanged row's fresh values
// equal its cached ones bit for bit (one sum over all of K gives both), so its three sums are one number.
// grid (ceil(tokens / 64), kSimSlices), 256 threads: lane = two neighbouring tokens, warp = every 8th feature of the slice
__global__ void __launch_bounds__(256)
sim_partial_kernel(const __nv_bfloat16 *__restrict__ a, long long lda, const __nv_bfloat16 *__restrict__ b, long long ldb, int d, int t_first, int t_end, int T,
                   float *__restrict__ partial)
{
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t0 = t_first + blockIdx.x * 64 + 2 * lane;             // t_first is even: 4-byte loads of two tokens stay aligned
    const int per = (d + kSimSlices - 1) / kSimSlices;
    const int f0 = blockIdx.y * per, f1 = min(d, f0 + per);
    float acc[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (t0 < t_end) {
        const __nv_bfloat16 *ap = a + (t0 - t_first);
        auto term = [&](uint32_t wa, uint32_t wb) {
            const float a0 = bf16_bits_to_f32(wa & 0xFFFFu), a1 = bf16_bits_to_f32(wa >> 16);
            const float b0 = bf16_bits_to_f32(wb & 0xFFFFu), b1 = bf16_bits_to_f32(wb >> 16);
            acc[0] = fmaf(a0, b0, acc[0]); acc[1] = fmaf(a0, a0, acc[1]); acc[2] = fmaf(b0, b0, acc[2]);
            acc[3] = fmaf(a1, b1, acc[3]); acc[4] = fmaf(a1, a1, acc[4]); acc[5] = fmaf(b1, b1, acc[5]);
        };
        constexpr int U = 8;
        for (int f = f0 + warp; f < f1; f += 8 * U) {                // eight features per round, all their loads in flight
            uint32_t wa[U], wb[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int fu = f + 8 * u;
                if (fu < f1) {
                    wa[u] = *reinterpret_cast<const uint32_t *>(ap + (long long)fu * lda);
                    wb[u] = *reinterpret_cast<const uint32_t *>(b + (long long)fu * ldb + t0);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) if (f + 8 * u < f1) term(wa[u], wb[u]);
        }
    }
    __shared__ float s[8][32][6];
#pragma unroll
    for (int i = 0; i < 6; ++i) s[warp][lane][i] = acc[i];
    __syncthreads();
    if (warp == 0 && t0 < t_end) {
        float r[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) { r[i] = s[0][lane][i]; for (int w = 1; w < 8; ++w) r[i] += s[w][lane][i]; }   // fixed order
        float *o = partial + ((long long)blockIdx.y * T + t0) * 3;
        o[0] = r[0]; o[1] = r[1]; o[2] = r[2];
        if (t0 + 1 < t_end) { o[3] = r[3]; o[4] = r[4]; o[5] = r[5]; }
    }
}

__device__ __forceinline__ float ld_nc(const float *p) {              // (volatile: issued where it stands, not where it is used)
    float v;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t float_order_key(float f) {       // monotone map float -> uint32
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// One CTA per sequence; dynamic shared memory: u32 keys[L].  The similarities of a position are summed by two lanes; the k-th
// smallest key is found bit by bit (one block-wide count per bit), the chosen positions are those below it and the first of those
// equal to it, and their slots are running counts.  It is one link of every layer's chain: 512 positions took 18 us when each
// candidate's rank was counted over all keys (262 thousand 64-bit comparisons on one SM).
constexpr int kChoiceThreads = 1024;
__global__ void __launch_bounds__(kChoiceThreads) cache_select_kernel(CacheSelectArgs a)
{
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) uint32_t s_key[];
    __shared__ int s_cnt[kChoiceThreads / 32], s_last;
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, L = a.L, P = a.P, S = a.S;
    int32_t *out = a.sel_rows + (long long)b * a.n_sel;
    int base = 0;
    if (a.refresh_p) {
        for (int i = tid; i < P; i += kChoiceThreads) out[i] = b * S + i;
        base = P;
    }
    if (a.refresh_r) {
        for (int i = tid; i < L; i += kChoiceThreads) out[base + i] = b * S + P + i;
    } else if (a.n_adapt > 0) {
        // (the four fields in one round trip, beside that of the similarities)
        int4 span = make_int4(SFS_PHASE_SLOW, 0, 0, L);              // phase, done, first, end
        if (a.state != nullptr) span = make_int4(a.state[b].phase, a.state[b].done, a.state[b].s_cycle, a.state[b].hi);
        constexpr int HS = kSimSlices / 2;
        for (int it = tid; it < 2 * L; it += kChoiceThreads) {        // (2 L is even: both lanes of a position are there)
            const int i = it >> 1, half = it & 1;
            const float *__restrict__ p = a.partial + ((long long)(half * HS) * a.T + (long long)b * S + P + i) * 3;
            float pd[HS], pa[HS], pb[HS];
#pragma unroll
            for (int sl = 0; sl < HS; ++sl) {                        // all loads first: one latency, not HS of them
                const float *q = p + (long long)sl * a.T * 3;
                pd[sl] = ld_nc(q); pa[sl] = ld_nc(q + 1); pb[sl] = ld_nc(q + 2);
            }
            // added in slice order, the odd lane going on where the even one stopped: equal vectors' last bits decide among unchanged rows
            float dot = 0.f, na = 0.f, nb = 0.f;
            const unsigned both = 3u << (lane & 30);
#pragma unroll
            for (int turn = 0; turn < 2; ++turn) {
                if (half == turn)
#pragma unroll
                    for (int sl = 0; sl < HS; ++sl) { dot += pd[sl]; na += pa[sl]; nb += pb[sl]; }
                if (turn == 0) {
                    const float d0 = __shfl_sync(both, dot, lane & 30), a0 = __shfl_sync(both, na, lane & 30), b0 = __shfl_sync(both, nb, lane & 30);
                    if (half == 1) { dot = d0; na = a0; nb = b0; }
                }
            }
            const float den = __fmul_rn(__fsqrt_rn(na), __fsqrt_rn(nb));
            const float sim = den > 0.f ? __fdiv_rn(dot, den) : 0.f;
            if (half == 1) {
                if (a.sims_dump) a.sims_dump[(long long)b * L + i] = sim;
                s_key[i] = float_order_key(sim);
            }
        }
        const bool fast = span.x == SFS_PHASE_FAST && !span.y;
        const int lo = fast ? max(0, min(span.z, L)) : 0, hi = fast ? max(lo, min(span.w, L)) : L;
        if (tid == 0) s_last = -1;
        __syncthreads();
        const int n_cand = hi - lo, k = min(a.n_adapt, n_cand);
        // candidates whose key is below v
        auto count_below = [&](uint32_t v) {
            if (L <= kChoiceThreads) return __syncthreads_count(tid >= lo && tid < hi && s_key[tid] < v);
            int c = 0;
            for (int i = lo + tid; i < hi; i += kChoiceThreads) c += s_key[i] < v ? 1 : 0;
            c = warp_sum_i32(c);
            __syncthreads();
            if (lane == 0) s_cnt[warp] = c;
            __syncthreads();
            return warp_sum_i32(s_cnt[lane]);
        };
        uint32_t kth = 0xFFFFFFFFu;                                  // the k-th smallest key, when not all are chosen
        int need = n_cand;                                           // how many of those equal to it are chosen
        if (k > 0 && k < n_cand) {
            kth = 0;
            for (int bit = 31; bit >= 0; --bit) {
                const uint32_t v = kth | (1u << bit);
                if (count_below(v) < k) kth = v;
            }
            need = k - count_below(kth);
        }
        int run_less = 0, run_eq = 0;
        for (int i0 = 0; i0 < L && k > 0; i0 += kChoiceThreads) {
            const int i = i0 + tid;
            const bool cand = i >= lo && i < hi, all = k == n_cand;
            const uint32_t key = cand ? s_key[i] : 0u;
            const bool less = cand && !all && key < kth, eq = cand && (all || key == kth);
            const unsigned bl = __ballot_sync(0xffffffffu, less), be = __ballot_sync(0xffffffffu, eq);
            __syncthreads();
            if (lane == 0) s_cnt[warp] = __popc(bl) | (__popc(be) << 16);
            __syncthreads();
            const int c = s_cnt[lane];
            const int before = warp_sum_i32(lane < warp ? c : 0), total = warp_sum_i32(c);
            const unsigned lt = (1u << lane) - 1u;
            const int n_less = run_less + (before & 0xFFFF) + __popc(bl & lt), n_eq = run_eq + (before >> 16) + __popc(be & lt);
            if (less || (eq && n_eq < need)) {
                const int slot = n_less + min(n_eq, need);
                out[base + slot] = b * S + P + i;
                if (slot == k - 1) s_last = b * S + P + i;
            }
            run_less += total & 0xFFFF; run_eq += total >> 16;
        }
        __syncthreads();
        const int pad = (k > 0) ? s_last : b * S + P;                  // nothing to choose from: recompute the first response row
        for (int j = k + tid; j < a.n_adapt; j += kChoiceThreads) out[base + j] = pad;
    }
    if (a.sets_dump) {
        __syncthreads();
        for (int j = tid; j < a.n_sel; j += blockDim.x) a.sets_dump[(long long)b * a.n_sel + j] = out[j];
    }
}

__global__ void gather_rows_bf16_kernel(const uint4 *__restrict__ src, const int32_t *__restrict__ rows, int chunks, uint4 *__restrict__ dst)
{
    pdl_wait();
    pdl_trigger();
    const int j = blockIdx.x;
    const uint4 *s = src + (long long)rows[j] * chunks;
    uint4 *o = dst + (long long)j * chunks;
    for (int c = threadIdx.x; c < chunks; c += blockDim.x) o[c] = s[c];
}

// the split-K partial products of one 16-byte chunk, added in slab order; up to six slabs are one round trip
constexpr int kSlabRegs = 6;
__device__ __forceinline__ float4 sum_slabs(const float4 *s, int n_slabs, long long slab_chunks)
{
    float4 p[kSlabRegs];
#pragma unroll
    for (int k = 0; k < kSlabRegs; ++k) if (k < n_slabs) p[k] = s[(long long)k * slab_chunks];
    float4 v = p[0];
#pragma unroll
    for (int k = 1; k < kSlabRegs; ++k) if (k < n_slabs) { v.x += p[k].x; v.y += p[k].y; v.z += p[k].z; v.w += p[k].w; }
    for (int k = kSlabRegs; k < n_slabs; ++k) { const float4 q = s[(long long)k * slab_chunks]; v.x += q.x; v.y += q.y; v.z += q.z; v.w += q.w; }
    return v;
}

__global__ void scatter_rows_f32_kernel(const float4 *__restrict__ src, int n_slabs, long long slab_chunks, const int32_t *__restrict__ rows,
                                        int chunks, float4 *__restrict__ dst)
{
    pdl_wait();
    pdl_trigger();
    const int j = blockIdx.x;
    const float4 *s = src + (long long)j * chunks;
    float4 *o = dst + (long long)rows[j] * chunks;
    for (int c = blockIdx.y * blockDim.x + threadIdx.x; c < chunks; c += gridDim.y * blockDim.x) {
        o[c] = sum_slabs(s + c, n_slabs, slab_chunks);
    }
}

// One launch for what follows the QKV projection of the recomputed rows: the rotary embedding of q and k (in place, on the
// compact rows; the arithmetic of rope_kernel), the rotated k also written to the token's row of the K cache, and the new
// value columns scattered into V^T.  Blocks [0, rope_blocks) rotate, the rest scatter values (8 features per block).
__global__ void __launch_bounds__(256)
rope_scatter_kv_kernel(__nv_bfloat16 *__restrict__ qk, long long ld, int n_rows, int S, int n_heads, int dh, const float2 *__restrict__ table,
                       const int32_t *__restrict__ rows, __nv_bfloat16 *__restrict__ k_dst, const __nv_bfloat16 *__restrict__ vt_src,
                       long long ld_vt_src, __nv_bfloat16 *__restrict__ vt_dst, long long ld_vt_dst, int rope_blocks)
{
    pdl_wait();
    pdl_trigger();
    const int d = n_heads * dh;
    if ((int)blockIdx.x >= rope_blocks) {
        const int f0 = ((int)blockIdx.x - rope_blocks) * 8;
        for (int idx = threadIdx.x; idx < 8 * n_rows; idx += blockDim.x) {
            const int f = f0 + idx / n_rows, j = idx - (idx / n_rows) * n_rows;
            if (f < d) vt_dst[(long long)f * ld_vt_dst + rows[j]] = vt_src[(long long)f * ld_vt_src + j];
        }
        return;
    }
    const int half = dh / 2, groups = half / 8;
    const unsigned idx = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned total = (unsigned)n_rows * 2u * (unsigned)n_heads * (unsigned)groups;
    if (idx >= total) return;
    const unsigned per_token = (unsigned)groups * 2u * (unsigned)n_heads;
    const int t = (int)(idx / per_token);
    const unsigned rem = idx - (unsigned)t * per_token;
    const int hh = (int)(rem / (unsigned)groups);              // q heads then k heads: contiguous columns
    const int g = (int)(rem - (unsigned)hh * (unsigned)groups);
    const int tok = rows[t], pos = tok % S;
    __nv_bfloat16 *base = qk + (long long)t * ld + (long long)hh * dh + g * 8;
    uint4 lo = *reinterpret_cast<uint4 *>(base), hi = *reinterpret_cast<uint4 *>(base + half);
    const float2 *tb = table + (long long)pos * half + g * 8;
    uint32_t *lw = reinterpret_cast<uint32_t *>(&lo), *hw = reinterpret_cast<uint32_t *>(&hi);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        float x1[2] = {bf16_bits_to_f32(lw[w] & 0xFFFFu), bf16_bits_to_f32(lw[w] >> 16)};
        float x2[2] = {bf16_bits_to_f32(hw[w] & 0xFFFFu), bf16_bits_to_f32(hw[w] >> 16)};
        float o1[2], o2[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float2 cs = tb[2 * w + e];
            o1[e] = x1[e] * cs.x - x2[e] * cs.y;
            o2[e] = x2[e] * cs.x + x1[e] * cs.y;
        }
        __nv_bfloat162 a = __floats2bfloat162_rn(o1[0], o1[1]), b2 = __floats2bfloat162_rn(o2[0], o2[1]);
        lw[w] = *reinterpret_cast<uint32_t *>(&a);
        hw[w] = *reinterpret_cast<uint32_t *>(&b2);
    }
    *reinterpret_cast<uint4 *>(base) = lo;
    *reinterpret_cast<uint4 *>(base + half) = hi;
    if (hh >= n_heads) {                                       // a key head: also the token's row of the K cache
        __nv_bfloat16 *kd = k_dst + (long long)tok * d + (long long)(hh - n_heads) * dh + g * 8;
        *reinterpret_cast<uint4 *>(kd) = lo;
        *reinterpret_cast<uint4 *>(kd + half) = hi;
    }
}

// One launch for what follows the output projection of the recomputed rows: the split-K slabs of compact row j are added in
// slab order into the attention increment of its token (inc[rows[j]] = sum of slabs), and the MLP branch's input
// h[j] = bf16(RMSNorm(x[rows[j]] + inc[rows[j]]) * gain) is written to the compact buffer.
__global__ void __launch_bounds__(1024)
fold_norm_rows_kernel(const float *__restrict__ slabs, int n_slabs, long long slab_stride, const int32_t *__restrict__ rows,
                      const float *__restrict__ x, float *__restrict__ inc, const __nv_bfloat16 *__restrict__ gain,
                      __nv_bfloat16 *__restrict__ h, int d, float eps)
{
    pdl_wait();
    pdl_trigger();
    const int j = blockIdx.x, chunks = d / 4;
    const long long src = rows[j];
    const float4 *sp = reinterpret_cast<const float4 *>(slabs + (long long)j * d);
    const float4 *xr = reinterpret_cast<const float4 *>(x + src * d);
    float4 *ir = reinterpret_cast<float4 *>(inc + src * d);
    __shared__ float s_part[32];
    extern __shared__ float4 s_y[];                            // the row, kept between the two passes
    float ss = 0.f;
    for (int c = threadIdx.x; c < chunks; c += blockDim.x) {
        const float4 xv = xr[c], v = sum_slabs(sp + c, n_slabs, slab_stride / 4);
        ir[c] = v;
        const float4 y = make_float4(xv.x + v.x, xv.y + v.y, xv.z + v.z, xv.w + v.w);
        s_y[c] = y;
        ss += y.x * y.x + y.y * y.y + y.z * y.z + y.w * y.w;
    }
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
    for (int w = 0; w < ((int)blockDim.x >> 5); ++w) tot += s_part[w];
    const float inv = rsqrtf(tot / (float)d + eps);
    const uint2 *gp = reinterpret_cast<const uint2 *>(gain);
    uint2 *hp = reinterpret_cast<uint2 *>(h + (long long)j * d);
    for (int c = threadIdx.x; c < chunks; c += blockDim.x) {
        const float4 v = s_y[c];
        const uint2 g = gp[c];
        __nv_bfloat162 o0 = __floats2bfloat162_rn(v.x * inv * bf16_bits_to_f32(g.x & 0xFFFFu), v.y * inv * bf16_bits_to_f32(g.x >> 16));
        __nv_bfloat162 o1 = __floats2bfloat162_rn(v.z * inv * bf16_bits_to_f32(g.y & 0xFFFFu), v.w * inv * bf16_bits_to_f32(g.y >> 16));
        hp[c] = make_uint2(*reinterpret_cast<uint32_t *>(&o0), *reinterpret_cast<uint32_t *>(&o1));
    }
}

}  // namespace

int32_t launch_rope_scatter_kv(void *qk, long long ld, int n_rows, int S, int n_heads, int head_dim, const float2 *table, const int32_t *rows,
                               void *k_dst, const void *vt_src, long long ld_vt_src, void *vt_dst, long long ld_vt_dst, cudaStream_t s)
{
    if (n_rows <= 0) return SFS_OK;
    const long long total = (long long)n_rows * 2 * n_heads * (head_dim / 16);
    SFS_REQUIRE(total < (1LL << 31), SFS_ERR_INVALID_ARG, "rope: %lld items do not fit a 32-bit index", total);
    const int rope_blocks = (int)((total + 255) / 256), d = n_heads * head_dim;
    SFS_CUDA(launch_pdl(rope_scatter_kv_kernel, dim3((unsigned)(rope_blocks + (d + 7) / 8)), dim3((unsigned)(256)), (size_t)(0), s, reinterpret_cast<__nv_bfloat16 *>(qk), ld, n_rows, S, n_heads, head_dim, table, rows,
                                                                      reinterpret_cast<__nv_bfloat16 *>(k_dst), reinterpret_cast<const __nv_bfloat16 *>(vt_src),
                                                                      ld_vt_src, reinterpret_cast<__nv_bfloat16 *>(vt_dst), ld_vt_dst, rope_blocks));
    return SFS_OK;
}

int32_t launch_fold_norm_rows(const float *slabs, int n_slabs, long long slab_stride, const int32_t *rows, int n_rows, const float *x, float *inc,
                              const void *gain, void *h, int d, float eps, cudaStream_t s)
{
    if (n_rows <= 0) return SFS_OK;
    SFS_REQUIRE((size_t)d * 4 <= 96 * 1024, SFS_ERR_UNSUPPORTED, "d_model %d too wide for the fused fold + norm", d);
    const size_t smem = (size_t)d * 4;
    SFS_CUDA(allow_shared(fold_norm_rows_kernel, smem));
    SFS_CUDA(launch_pdl(fold_norm_rows_kernel, dim3((unsigned)(n_rows)), dim3((unsigned)(d >= 4096 ? 1024 : (d >= 2048 ? 512 : 256))), (size_t)(smem), s, slabs, n_slabs < 1 ? 1 : n_slabs, slab_stride, rows, x, inc, reinterpret_cast<const __nv_bfloat16 *>(gain),
                                                    reinterpret_cast<__nv_bfloat16 *>(h), d, eps));
    return SFS_OK;
}

int32_t launch_sim_partial(const void *vnew_t, long long ld_new, const void *vold_t, long long ld_old, int d, int t_first, int t_count, int T,
                           float *partial, cudaStream_t s)
{
    if (t_count <= 0) return SFS_OK;
    SFS_REQUIRE((t_first % 2) == 0 && (ld_new % 2) == 0 && (ld_old % 2) == 0, SFS_ERR_INVALID_ARG, "similarity: first token and row strides must be even");
    dim3 grid((unsigned)((t_count + 63) / 64), kSimSlices, 1);
    SFS_CUDA(launch_pdl(sim_partial_kernel, grid, dim3((unsigned)(256)), (size_t)(0), s, reinterpret_cast<const __nv_bfloat16 *>(vnew_t), ld_new,
                        reinterpret_cast<const __nv_bfloat16 *>(vold_t), ld_old, d, t_first, t_first + t_count, T, partial));
    return SFS_OK;
}

int32_t launch_cache_select(const CacheSelectArgs &a, cudaStream_t s)
{
    SFS_CUDA(allow_shared(cache_select_kernel, (size_t)a.L * 4));
    SFS_CUDA(launch_pdl(cache_select_kernel, dim3((unsigned)(a.B)), dim3(kChoiceThreads), (size_t)a.L * 4, s, a));
    return SFS_OK;
}

int32_t launch_gather_rows_bf16(const void *src, const int32_t *rows, int n_rows, int d, void *dst, cudaStream_t s)
{
    if (n_rows <= 0) return SFS_OK;
    SFS_CUDA(launch_pdl(gather_rows_bf16_kernel, dim3((unsigned)(n_rows)), dim3((unsigned)(128)), (size_t)(0), s, reinterpret_cast<const uint4 *>(src), rows, d / 8, reinterpret_cast<uint4 *>(dst)));
    return SFS_OK;
}

int32_t launch_scatter_rows_f32(const float *src, int n_slabs, long long slab_stride, const int32_t *rows, int n_rows, int d, float *dst,
                                cudaStream_t s)
{
    if (n_rows <= 0) return SFS_OK;
    SFS_CUDA(launch_pdl(scatter_rows_f32_kernel, dim3((unsigned)n_rows, 4, 1), dim3((unsigned)(256)), (size_t)(0), s, reinterpret_cast<const float4 *>(src), n_slabs < 1 ? 1 : n_slabs, slab_stride / 4, rows, d / 4,
                                                   reinterpret_cast<float4 *>(dst)));
    return SFS_OK;
}

}  // namespace sfs
