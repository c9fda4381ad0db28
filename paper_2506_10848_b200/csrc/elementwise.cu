// Memory-bound glue of the mask predictor's forward pass: embedding gather, RMSNorm (with optional row
// gather), rotary position embedding, and the RoPE table.  All of them move 16 bytes per thread per access.
#include "sfs_common.cuh"
#include "elementwise.cuh"
#include <type_traits>

namespace sfs {
namespace {

// h[r, :] = bf16( y * rsqrt(mean(y^2) + eps) * g ),  y = x[src(r), :] + sum_s partial[s][src(r), :],  src(r) = rows ? rows[r] : r.
// The partial products of a split-K projection are added in slab order (the sum does not depend on which CTA of the
// projection finished first); without a row list y is written back to x, so the residual stream is complete again.
// EMBED: y is the embedding of the row's token (bf16 -> fp32, written to x: the residual stream begins here).
// A thread keeps its part of the row in registers between the two passes (kNormRegChunks 16-byte chunks of it).
// NP bounds the number of slabs: all of a thread's loads are issued before the first addition (summed slab by slab in a loop,
// 512 rows of 4096 with four slabs took 8.5 us, four dependent round trips per chunk).
// Whatever NT is, the squares are added in the order of 256 threads that take every 256th chunk each: how many threads share a
// row depends on how many rows a launch has, and a row must not (a cached step compares the values of a few rows with those of a
// launch over all of them, where the last bit decides).  Blocks of more than 256 threads pass the chunks' sums through shared
// memory for that; narrower ones have a thread per chunk at least.  (A chunk's four squares are spelled out: contracted by the compiler,
// two instances rounded them differently.)
template <int NT, int NP, bool EMBED>
__global__ void __launch_bounds__(NT)
rmsnorm_kernel(float *__restrict__ x, const float *__restrict__ partial, int n_partial, long long partial_stride,
               const __nv_bfloat16 *__restrict__ gain, __nv_bfloat16 *__restrict__ h,
               const int32_t *__restrict__ rows, const int32_t *__restrict__ n_rows_ptr, int max_rows, int d, float eps,
               const int32_t *__restrict__ tokens, const __nv_bfloat16 *__restrict__ emb, int vocab, const int32_t *__restrict__ copy_src,
               int32_t *__restrict__ copy_dst, int copy_n)
{
    constexpr int kNormThreads = NT, kNormRegChunks = NT == 256 ? 4 : (NT == 512 ? 2 : 1), kSumThreads = NT < 256 ? NT : 256;
    extern __shared__ float s_sq[];                          // NT > 256: [chunks] sums of squares
    pdl_wait();
    pdl_trigger();
    if (EMBED && blockIdx.x == 0)
        for (int i = threadIdx.x; i < copy_n; i += kNormThreads) copy_dst[i] = copy_src[i];
    const int n_rows = n_rows_ptr ? min(*n_rows_ptr, max_rows) : max_rows;
    __shared__ float s_part[kSumThreads / 32];
    const int chunks = d / 4;
    for (int r = blockIdx.x; r < n_rows; r += gridDim.x) {
        const long long src = rows ? rows[r] : r;
        float4 *xr = reinterpret_cast<float4 *>(x + src * d);
        const float4 *pr = reinterpret_cast<const float4 *>(partial + src * d);
        const long long pstride4 = partial_stride / 4;
        const uint2 *er = nullptr;
        if (EMBED) {
            int id = tokens[src];
            id = id < 0 ? 0 : (id >= vocab ? vocab - 1 : id);  // out-of-range ids are clamped, never dereferenced
            er = reinterpret_cast<const uint2 *>(emb + (long long)id * d);
        }
        const bool write_x = EMBED || (n_partial > 0 && rows == nullptr);
        auto load = [&](int c) {                              // x + the partial products, slab by slab
            if (EMBED) {
                const uint2 e = er[c];
                return make_float4(bf16_bits_to_f32(e.x & 0xFFFFu), bf16_bits_to_f32(e.x >> 16), bf16_bits_to_f32(e.y & 0xFFFFu), bf16_bits_to_f32(e.y >> 16));
            }
            float4 v = xr[c], p[NP > 0 ? NP : 1];
#pragma unroll
            for (int s = 0; s < NP; ++s) if (s < n_partial) p[s] = pr[(long long)s * pstride4 + c];
#pragma unroll
            for (int s = 0; s < NP; ++s) if (s < n_partial) { v.x += p[s].x; v.y += p[s].y; v.z += p[s].z; v.w += p[s].w; }
            return v;
        };
        // the first kNormRegChunks chunks of a thread stay in registers (statically indexed); longer rows re-read the rest
        float4 keep[kNormRegChunks];
        float ss = 0.f;
        auto add = [&](int c, const float4 &v) {
            const float q = __fmaf_rn(v.w, v.w, __fmaf_rn(v.z, v.z, __fmaf_rn(v.y, v.y, __fmul_rn(v.x, v.x))));
            if (NT <= 256) ss += q;
            else if (c < chunks) s_sq[c] = q;
        };
        if (EMBED || NP == 0) {
#pragma unroll
            for (int k = 0; k < kNormRegChunks; ++k) {
                const int c = threadIdx.x + k * kNormThreads;
                keep[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (c < chunks) keep[k] = load(c);
            }
        } else {
            float4 p[NP > 0 ? NP : 1][kNormRegChunks];
#pragma unroll
            for (int k = 0; k < kNormRegChunks; ++k) {
                const int c = threadIdx.x + k * kNormThreads;
                keep[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (c < chunks) keep[k] = xr[c];
#pragma unroll
                for (int s = 0; s < NP; ++s) {
                    p[s][k] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (s < n_partial && c < chunks) p[s][k] = pr[(long long)s * pstride4 + c];
                }
            }
#pragma unroll
            for (int s = 0; s < NP; ++s)
#pragma unroll
                for (int k = 0; k < kNormRegChunks; ++k) { keep[k].x += p[s][k].x; keep[k].y += p[s][k].y; keep[k].z += p[s][k].z; keep[k].w += p[s][k].w; }
        }
#pragma unroll
        for (int k = 0; k < kNormRegChunks; ++k) {
            const int c = threadIdx.x + k * kNormThreads;
            const float4 v = keep[k];
            if (c < chunks && write_x) xr[c] = v;
            add(c, v);
        }
        for (int c = threadIdx.x + kNormRegChunks * kNormThreads; c < chunks; c += kNormThreads) {
            const float4 v = load(c);
            if (write_x) xr[c] = v;
            add(c, v);
        }
        if (NT > 256) {
            __syncthreads();
            if (threadIdx.x < 256) for (int c = threadIdx.x; c < chunks; c += 256) ss += s_sq[c];
        }
        if (threadIdx.x < kSumThreads) {
            ss = warp_sum(ss);
            if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = ss;
        }
        __syncthreads();
        float tot = 0.f;
#pragma unroll
        for (int w = 0; w < kSumThreads / 32; ++w) tot += s_part[w];
        const float inv = rsqrtf(tot / (float)d + eps);
        const uint2 *gp = reinterpret_cast<const uint2 *>(gain);
        uint2 *hp = reinterpret_cast<uint2 *>(h + (long long)r * d);
        auto emit = [&](int c, const float4 &v) {
            const uint2 g = gp[c];
            __nv_bfloat162 o0 = __floats2bfloat162_rn(v.x * inv * bf16_bits_to_f32(g.x & 0xFFFFu), v.y * inv * bf16_bits_to_f32(g.x >> 16));
            __nv_bfloat162 o1 = __floats2bfloat162_rn(v.z * inv * bf16_bits_to_f32(g.y & 0xFFFFu), v.w * inv * bf16_bits_to_f32(g.y >> 16));
            hp[c] = make_uint2(*reinterpret_cast<uint32_t *>(&o0), *reinterpret_cast<uint32_t *>(&o1));
        };
#pragma unroll
        for (int k = 0; k < kNormRegChunks; ++k) {
            const int c = threadIdx.x + k * kNormThreads;
            if (c < chunks) emit(c, keep[k]);
        }
        for (int c = threadIdx.x + kNormRegChunks * kNormThreads; c < chunks; c += kNormThreads) {
            // long rows: rebuild the value the first pass saw (x already holds it when it was written back)
            const float4 v = write_x ? xr[c] : load(c);
            emit(c, v);
        }
        __syncthreads();
    }
}

// table[pos, j] = (cos, sin)(pos * theta^(-2j/dh)), evaluated in double
__global__ void rope_table_kernel(float2 *table, int positions, int half, double theta)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= positions * half) return;
    const int pos = idx / half, j = idx % half;
    const double ang = (double)pos * pow(theta, -2.0 * (double)j / (double)(2 * half));
    table[idx] = make_float2((float)cos(ang), (float)sin(ang));
}

// in place on q, and in place on k or (k_dst given) into the K cache [T, n_heads * dh]: pairs (j, j + dh/2) of every head rotate by
// the angle of the token's position
__global__ void rope_kernel(__nv_bfloat16 *__restrict__ qk, long long ld, int T, int S, int n_heads, int dh,
                            const float2 *__restrict__ table, __nv_bfloat16 *__restrict__ k_dst)
{
    // one thread handles 8 consecutive j of one (token, q-or-k, head)
    pdl_wait();
    pdl_trigger();
    const int half = dh / 2, groups = half / 8;
    const unsigned idx = blockIdx.x * blockDim.x + threadIdx.x;   // the launcher checks that the item count fits 31 bits
    const unsigned total = (unsigned)T * 2u * (unsigned)n_heads * (unsigned)groups;
    if (idx >= total) return;
    const unsigned per_token = (unsigned)groups * 2u * (unsigned)n_heads;
    const int t = (int)(idx / per_token);
    const unsigned rem = idx - (unsigned)t * per_token;
    const int hh = (int)(rem / (unsigned)groups);              // q heads then k heads: contiguous columns
    const int g = (int)(rem - (unsigned)hh * (unsigned)groups);
    const int pos = t % S;
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
    if (k_dst != nullptr && hh >= n_heads) base = k_dst + (long long)t * n_heads * dh + (long long)(hh - n_heads) * dh + g * 8;
    *reinterpret_cast<uint4 *>(base) = lo;
    *reinterpret_cast<uint4 *>(base + half) = hi;
}

}  // namespace

// Threads per row: 256 while the rows fill the machine, up to one 16-byte chunk per thread when they do not (a row is then one
// round trip instead of four: 104 rows of 4096 with three slabs 6.8 -> 4.9 us), and no more threads than it takes.
static int norm_threads(int rows, int d)
{
    const int chunks = d / 4;
    if (rows > 2 * 148 || d > 32768) return 256;          // (wider rows: their sums would not fit the shared memory of a plain launch)
    return chunks >= 1024 ? 1024 : (chunks >= 512 ? 512 : (chunks > 128 ? 256 : (chunks > 64 ? 128 : 64)));
}

template <bool EMBED>
static int32_t launch_norm(float *x, const float *partial, int n_partial, long long partial_stride, const void *gain, void *h, const int32_t *rows,
                           const int32_t *n_rows, int max_rows, int d, float eps, const int32_t *tokens, const void *emb, int vocab, const int32_t *copy_src, int32_t *copy_dst, int copy_n,
                           cudaStream_t s)
{
    if (max_rows <= 0) return SFS_OK;
    const int grid = max_rows < 148 * 16 ? max_rows : 148 * 16, nt = norm_threads(max_rows, d);
    if (partial == nullptr) n_partial = 0;
    auto go = [&](auto kernel, int threads) {
        return launch_pdl(kernel, dim3(grid), dim3(threads), threads > 256 ? (size_t)d : 0, s, x, partial ? partial : x, n_partial, partial_stride,
                          reinterpret_cast<const __nv_bfloat16 *>(gain), reinterpret_cast<__nv_bfloat16 *>(h), rows, n_rows, max_rows, d, eps, tokens,
                          reinterpret_cast<const __nv_bfloat16 *>(emb), vocab, copy_src, copy_dst, copy_n);
    };
    auto pick = [&](auto np) {
        constexpr int NP = decltype(np)::value;
        return nt == 1024 ? go(rmsnorm_kernel<1024, NP, EMBED>, 1024) : (nt == 512 ? go(rmsnorm_kernel<512, NP, EMBED>, 512)
             : (nt == 256 ? go(rmsnorm_kernel<256, NP, EMBED>, 256) : (nt == 128 ? go(rmsnorm_kernel<128, NP, EMBED>, 128) : go(rmsnorm_kernel<64, NP, EMBED>, 64))));
    };
    SFS_REQUIRE(n_partial <= 6, SFS_ERR_UNSUPPORTED, "norm: %d slabs", n_partial);
    if (n_partial == 0) SFS_CUDA(pick(std::integral_constant<int, 0>()));
    else if (EMBED || n_partial <= 2) SFS_CUDA(pick(std::integral_constant<int, EMBED ? 0 : 2>()));
    else if (n_partial <= 4) SFS_CUDA(pick(std::integral_constant<int, EMBED ? 0 : 4>()));
    else SFS_CUDA(pick(std::integral_constant<int, EMBED ? 0 : 6>()));
    return SFS_OK;
}

int32_t launch_embed_norm(const int32_t *tokens, const void *emb, int vocab, float *x, const void *gain, void *h, int T, int d, float eps, const int32_t *copy_src,
                          int32_t *copy_dst, int copy_n, cudaStream_t s)
{
    return launch_norm<true>(x, nullptr, 0, 0, gain, h, nullptr, nullptr, T, d, eps, tokens, emb, vocab, copy_src, copy_dst, copy_n, s);
}

int32_t launch_rmsnorm(float *x, const float *partial, int n_partial, long long partial_stride, const void *gain, void *h,
                       const int32_t *rows, const int32_t *n_rows, int max_rows, int d, float eps, cudaStream_t s)
{
    return launch_norm<false>(x, partial, n_partial, partial_stride, gain, h, rows, n_rows, max_rows, d, eps, nullptr, nullptr, 0, nullptr, nullptr, 0, s);
}

int32_t launch_rope_table(float2 *table, int positions, int head_dim, float theta, cudaStream_t s)
{
    const int n = positions * (head_dim / 2);
    rope_table_kernel<<<(n + 255) / 256, 256, 0, s>>>(table, positions, head_dim / 2, (double)theta);
    SFS_LAUNCH_CHECK();
    return SFS_OK;
}

int32_t launch_rope(void *qk, int64_t ld, int T, int S, int n_heads, int head_dim, const float2 *table, void *k_dst, cudaStream_t s)
{
    const long long total = (long long)T * 2 * n_heads * (head_dim / 16);
    SFS_REQUIRE(total < (1LL << 31), SFS_ERR_INVALID_ARG, "rope: %lld items do not fit a 32-bit index", total);
    SFS_CUDA(launch_pdl(rope_kernel, dim3((unsigned)((total + 255) / 256)), dim3(256), 0, s, reinterpret_cast<__nv_bfloat16 *>(qk), (long long)ld, T, S,
                        n_heads, head_dim, table, reinterpret_cast<__nv_bfloat16 *>(k_dst)));
    return SFS_OK;
}

}  // namespace sfs
