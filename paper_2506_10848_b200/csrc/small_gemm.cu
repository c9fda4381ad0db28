// Projections of small models and few rows, where a step is bound by the number and the length of its launches: each kernel takes
// in the row-wise work before it (embedding, RMSNorm, row gather) and after it (rotary embedding, SwiGLU, residual add).
//
// A 64 x 256 x 256 product has 8 MFLOP; the tcgen05 kernel needs 4 us for it after its inputs are there (pair set-up, TMA round
// trip, tensor-memory hand-overs), its norm and its rotary kernel 1.5 to 1.7 each, and every launch in a chain 1.4 us on
// top.  Here a CTA of eight warps computes a 32 x 32 tile with mma.sync from shared memory that holds all of K at once: the weight
// rows are requested before the dependent-launch wait, the activation rows are normalised on the way in (every column tile
// repeats that for its 32 rows, from L2), and the accumulators of a warp pair up what the epilogue needs together (gate and up,
// the two halves of a rotary pair).  A layer is five launches instead of eight.
// Bound: the latency of one memory round trip, K / 32 dependent MMAs per warp and the launch: 2.0 to 2.6 us from wait to end at 64
// rows, 0.95 us from one kernel's end to the next one's wait.  2-layer d 256 step, before with the tensor-memory kernels / now: 64
// rows 70.6 / 34.8 us, 192 - / 43, 512 84 / 61.  All layers in one launch (a cluster of 16 CTAs per sequence, cluster barriers
// between the projections) took 54.8 us at 64 rows when this took 55.3, and twice this at 224: a barrier behind global stores and
// the first loads of lines that other SMs have just written cost as much as a launch.
#include "sfs_common.cuh"
#include "small_gemm.cuh"
#include "small_mma.cuh"

namespace sfs {
namespace {

using namespace small;

constexpr int TILE = 32, kThreads = 256, kWarps = kThreads / 32;

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// NCH: 16-byte chunks of a row per lane (SRC_NORM, SRC_EMBED: rows of up to NCH * 128 elements)
template <int SRC, int EPI, int NCH>
__global__ void __launch_bounds__(kThreads)
small_gemm_kernel(SmallGemmArgs g)
{
    extern __shared__ __align__(16) __nv_bfloat16 s_mem[];
    const int K = g.K, Kp = (K + 15) & ~15, ld = Kp + 8;          // rows 16 bytes apart modulo 128: ldmatrix is conflict-free
    __nv_bfloat16 *sA = s_mem, *sB = s_mem + TILE * ld;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockIdx.x, m0 = blockIdx.y * TILE;

    // ---- which weight rows: rows 0-15 and 16-31 of the tile are the two halves the epilogue combines
    const int half = g.head_dim / 2, tiles_per_map = g.n_per_map / TILE, per_head = g.head_dim / TILE;
    const int map = EPI == SMALL_QKV ? nt / tiles_per_map : 0, tt = EPI == SMALL_QKV ? nt - map * tiles_per_map : nt;
    const bool rotated = EPI == SMALL_QKV && map < 2;
    const int head = rotated ? tt / per_head : 0, j0 = rotated ? 16 * (tt - head * per_head) : 0;
    auto weight_row = [&](int r) -> const __nv_bfloat16 * {
        const int hi = r >> 4, q = r & 15;
        if (EPI == SMALL_SWIGLU) {
            const int n = nt * 16 + q;
            return n < g.N ? (hi ? g.B[1] : g.B[0]) + (long long)n * K : nullptr;
        }
        if (rotated) return (map ? g.B[1] : g.B[0]) + (long long)(head * g.head_dim + hi * half + j0 + q) * K;
        const int n = tt * TILE + r;
        return n < g.n_per_map ? (map == 2 ? g.B[2] : g.B[0]) + (long long)n * K : nullptr;
    };
    const int chunks = Kp / 8;
    const uint4 zero = make_uint4(0, 0, 0, 0);
    for (int r = warp; r < TILE; r += kWarps) {
        const __nv_bfloat16 *src = weight_row(r);
        for (int c = lane; c < chunks; c += 32)
            if (src != nullptr && c * 8 < K) cp_async16(sB + r * ld + c * 8, src + c * 8);
            else *reinterpret_cast<uint4 *>(sB + r * ld + c * 8) = zero;
    }

    // constant too: the gains of this lane's columns, the rotary angles of its rows
    const int wm = warp & 1, wn = (warp >> 1) & 1, wk = warp >> 2, em = m0 + wm * 16 + (lane >> 2), eq = wn * 8 + 2 * (lane & 3);      // epilogue: rows em and em + 8, columns eq, eq + 1 of both halves
    uint2 gain[NCH];
    float4 angle[2];
    if (SRC != SMALL_BF16)
#pragma unroll
        for (int k = 0; k < NCH; ++k) gain[k] = lane + 32 * k < K / 4 ? reinterpret_cast<const uint2 *>(g.gain)[lane + 32 * k] : make_uint2(0, 0);
    if (EPI == SMALL_QKV && rotated)
#pragma unroll
        for (int h = 0; h < 2; ++h) angle[h] = *reinterpret_cast<const float4 *>(g.table + (long long)((em + 8 * h) % g.S) * half + j0 + eq);       // two (cos, sin)

    pdl_wait();                                             // weights are constant; everything else may come from the kernel before
    pdl_trigger();                                          // (not earlier: see pdl_trigger)
    // the row count and the flag are used only after the loads below have been issued (which stay within g.M rows), but for a caller's
    // row list, which ends with the count
    const int M = g.d_m ? min(*g.d_m, g.M) : g.M;
    const bool active = g.d_active == nullptr || *g.d_active != 0;
    float2 xr[2][2];
    if (EPI == SMALL_RESIDUAL)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int n = nt * TILE + 16 * u + eq;
                xr[h][u] = (em + 8 * h < g.M && n < g.N) ? *reinterpret_cast<const float2 *>(g.x + (long long)(em + 8 * h) * g.N + n) : make_float2(0.f, 0.f);
            }

    // ---- activation rows
    if (SRC == SMALL_BF16) {
        for (int r = warp; r < TILE; r += kWarps)
            for (int c = lane; c < chunks; c += 32)
                if (m0 + r < g.M && c * 8 < K) cp_async16(sA + r * ld + c * 8, g.a + (long long)(m0 + r) * g.lda + c * 8);
                else *reinterpret_cast<uint4 *>(sA + r * ld + c * 8) = zero;
        if (!active || m0 >= M) { cp_async_wait(); return; }
    } else {
        constexpr int ROWS = TILE / kWarps;                 // rows of a warp, all in flight
        const int q4 = K / 4;
        float4 v[ROWS][NCH];
        int listed[ROWS] = {};                          // (all rows' entries at once: row by row, each would be a round trip)
        if (EPI == SMALL_STORE) {                       // only the LM head takes a row list
#pragma unroll
            for (int u = 0; u < ROWS; ++u) {
                const int e = list_entry_early(g, m0 + warp * ROWS + u);
                listed[u] = e >= 0 ? g.rows[e] : 0;
            }
            if (g.rows != nullptr && g.rows_known < M)
#pragma unroll
                for (int u = 0; u < ROWS; ++u) {
                    const int e = list_entry_late(g, m0 + warp * ROWS + u, M);
                    if (e >= 0) listed[u] = g.rows[e];
                }
        }
#pragma unroll
        for (int u = 0; u < ROWS; ++u) {
            const int m = m0 + warp * ROWS + u;
            const long long src = EPI == SMALL_STORE && g.rows ? (m < M ? listed[u] : 0) : (m < g.M ? m : 0);
            const float4 *xr = reinterpret_cast<const float4 *>(g.x + src * K);
            const uint2 *er = nullptr;
            if (SRC == SMALL_EMBED) {
                int id = g.tokens[src];
                id = id < 0 ? 0 : (id >= g.vocab ? g.vocab - 1 : id);     // out-of-range ids are clamped, never dereferenced
                er = reinterpret_cast<const uint2 *>(g.emb + (long long)id * K);
            }
#pragma unroll
            for (int k = 0; k < NCH; ++k) {
                const int c = lane + 32 * k;
                v[u][k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (m < g.M && c < q4) {
                    if (SRC == SMALL_EMBED) {
                        const uint2 e = er[c];
                        v[u][k] = make_float4(bf16_bits_to_f32(e.x & 0xFFFFu), bf16_bits_to_f32(e.x >> 16), bf16_bits_to_f32(e.y & 0xFFFFu),
                                              bf16_bits_to_f32(e.y >> 16));
                    } else v[u][k] = xr[c];
                }
            }
        }
        if (!active || m0 >= M) { cp_async_wait(); return; }
#pragma unroll
        for (int u = 0; u < ROWS; ++u) {
            const int r = warp * ROWS + u, m = m0 + r;
            float ss = 0.f;
#pragma unroll
            for (int k = 0; k < NCH; ++k) ss += v[u][k].x * v[u][k].x + v[u][k].y * v[u][k].y + v[u][k].z * v[u][k].z + v[u][k].w * v[u][k].w;
            const float inv = rsqrtf(warp_sum(ss) / (float)K + g.eps);
#pragma unroll
            for (int k = 0; k < NCH; ++k) {
                const int c = lane + 32 * k;
                if (c >= q4) continue;
                if (SRC == SMALL_EMBED && nt == 0 && m < M) reinterpret_cast<float4 *>(g.x)[(long long)m * q4 + c] = v[u][k];      // the residual stream begins
                const uint2 gn = gain[k];
                *reinterpret_cast<uint2 *>(sA + r * ld + 4 * c) =
                    make_uint2(pack2(v[u][k].x * inv * bf16_bits_to_f32(gn.x & 0xFFFFu), v[u][k].y * inv * bf16_bits_to_f32(gn.x >> 16)),
                               pack2(v[u][k].z * inv * bf16_bits_to_f32(gn.y & 0xFFFFu), v[u][k].w * inv * bf16_bits_to_f32(gn.y >> 16)));
            }
        }
        if (K < Kp) for (int r = tid; r < TILE; r += kThreads) *reinterpret_cast<uint4 *>(sA + r * ld + K) = zero;      // K is a multiple of 8
    }
    cp_async_wait();
    __syncthreads();

    // ---- 16 rows x (8 + 8) columns and half of k per warp; even and odd k-steps accumulate apart, which halves the chain again
    const uint32_t a_addr = smem_u32(sA + (wm * 16 + (lane & 15)) * ld + (lane >> 4) * 8);
    const uint32_t b_addr = smem_u32(sB + ((lane >> 4) * 16 + wn * 8 + (lane & 7)) * ld + ((lane >> 3) & 1) * 8);
    float acc[2][2][4] = {};
    const int steps = Kp / 16, mid = (steps + 1) / 2, end = wk ? steps : mid;
    int k = wk ? mid : 0;
#pragma unroll 2
    for (; k + 2 <= end; k += 2)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            uint32_t a[4], b[4];
            ldmatrix4(a, a_addr + (k + u) * 32); ldmatrix4(b, b_addr + (k + u) * 32);
            mma_16816(acc[u][0], a, b[0], b[1]);
            mma_16816(acc[u][1], a, b[2], b[3]);
        }
    if (k < end) {
        uint32_t a[4], b[4];
        ldmatrix4(a, a_addr + k * 32); ldmatrix4(b, b_addr + k * 32);
        mma_16816(acc[0][0], a, b[0], b[1]);
        mma_16816(acc[0][1], a, b[2], b[3]);
    }
    float4 sum[2];
#pragma unroll
    for (int u = 0; u < 2; ++u)
        sum[u] = make_float4(acc[0][u][0] + acc[1][u][0], acc[0][u][1] + acc[1][u][1], acc[0][u][2] + acc[1][u][2], acc[0][u][3] + acc[1][u][3]);
    __shared__ float4 s_half[2][kThreads / 2];
    if (wk) { s_half[0][tid - kThreads / 2] = sum[0]; s_half[1][tid - kThreads / 2] = sum[1]; }
    __syncthreads();
    if (wk) return;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const float4 o = s_half[u][tid];
        sum[u].x += o.x; sum[u].y += o.y; sum[u].z += o.z; sum[u].w += o.w;
    }

    // ---- epilogue: a thread holds, of both halves, rows lane / 4 and + 8, columns 2 (lane % 4) and + 1
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int m = em + 8 * h, q = eq;
        if (m >= M) continue;
        const float x0 = h ? sum[0].z : sum[0].x, x1 = h ? sum[0].w : sum[0].y, y0 = h ? sum[1].z : sum[1].x, y1 = h ? sum[1].w : sum[1].y;
        if (EPI == SMALL_SWIGLU) {
            const int n = nt * 16 + q;
            if (n < g.N) *reinterpret_cast<uint32_t *>(g.out + (long long)m * g.ldc + n) = pack2(silu(x0) * y0, silu(x1) * y1);       // N is even
        } else if (EPI == SMALL_RESIDUAL) {
            float2 *p0 = reinterpret_cast<float2 *>(g.x + (long long)m * g.N + nt * TILE + q), *p1 = p0 + 8;
            float2 *i0 = reinterpret_cast<float2 *>(g.inc + (long long)m * g.N + nt * TILE + q), *i1 = i0 + 8;
            if (nt * TILE + q < g.N) { *p0 = make_float2(xr[h][0].x + x0, xr[h][0].y + x1); if (g.inc) *i0 = make_float2(x0, x1); }
            if (nt * TILE + 16 + q < g.N) { *p1 = make_float2(xr[h][1].x + y0, xr[h][1].y + y1); if (g.inc) *i1 = make_float2(y0, y1); }
        } else if (EPI == SMALL_QKV) {
            if (rotated) {
                // the projection's result is rounded to bf16 and so is the rotated one, as when the two are kernels of their own
                const float a0 = round_bf16(x0), a1 = round_bf16(x1), b0 = round_bf16(y0), b1 = round_bf16(y1);
                const float4 cs = angle[h];
                const uint32_t lo = pack2(a0 * cs.x - b0 * cs.y, a1 * cs.z - b1 * cs.w), hi = pack2(b0 * cs.x + a0 * cs.y, b1 * cs.z + a1 * cs.w);
                const int col = head * g.head_dim + j0 + q;
                __nv_bfloat16 *dst = g.out + (long long)m * g.ldc + map * g.n_per_map + col;
                *reinterpret_cast<uint32_t *>(dst) = lo; *reinterpret_cast<uint32_t *>(dst + half) = hi;
                if (map && g.k_dst) {
                    dst = g.k_dst + (long long)m * g.n_per_map + col;
                    *reinterpret_cast<uint32_t *>(dst) = lo; *reinterpret_cast<uint32_t *>(dst + half) = hi;
                }
            } else {
                __nv_bfloat16 *dst = g.vt + (long long)(tt * TILE + q) * g.ldvt + m;       // values go out transposed
                dst[0] = __float2bfloat16_rn(x0); dst[g.ldvt] = __float2bfloat16_rn(x1);
                dst[16 * g.ldvt] = __float2bfloat16_rn(y0); dst[17 * g.ldvt] = __float2bfloat16_rn(y1);
            }
        } else {
            const float v[4] = {x0 * g.scale, x1 * g.scale, y0 * g.scale, y1 * g.scale};
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int n = nt * TILE + 16 * u + q;
                if (n >= g.N) continue;                     // N is even
                if (g.out_f32 != nullptr) *reinterpret_cast<float2 *>(g.out_f32 + (long long)m * g.ldc + n) = make_float2(v[2 * u], v[2 * u + 1]);
                else *reinterpret_cast<uint32_t *>(g.out + (long long)m * g.ldc + n) = pack2(v[2 * u], v[2 * u + 1]);
            }
        }
    }
}

size_t smem_bytes(int K) { return (size_t)2 * TILE * (((K + 15) & ~15) + 8) * 2; }

template <int SRC, int EPI, int NCH>
int32_t launch(const SmallGemmArgs &g, int n_tiles, cudaStream_t s)
{
    const size_t smem = smem_bytes(g.K);
    static size_t configured[kMaxDevices] = {};
    size_t &done = configured[current_device_slot()];
    if (smem > done) {
        SFS_CUDA(allow_shared(small_gemm_kernel<SRC, EPI, NCH>, smem));
        done = smem;
    }
    SFS_CUDA(launch_pdl(small_gemm_kernel<SRC, EPI, NCH>, dim3((unsigned)n_tiles, (unsigned)((g.M + TILE - 1) / TILE)), dim3(kThreads), smem, s, g));
    return SFS_OK;
}

}  // namespace

bool small_gemm_fits(int d_model, int d_ff, int head_dim) { return d_model <= 512 && smem_bytes(d_ff) <= 200 * 1024 && (d_model % 32) == 0 && (head_dim % 32) == 0; }

int32_t launch_small_gemm(int src, int epi, const SmallGemmArgs &g, cudaStream_t s)
{
    const int n_tiles = epi == SMALL_SWIGLU ? (g.N + 15) / 16 : (epi == SMALL_QKV ? 3 * (g.n_per_map / TILE) : (g.N + TILE - 1) / TILE);
    const bool wide = g.K > 256;
    if (src == SMALL_EMBED) return wide ? launch<SMALL_EMBED, SMALL_QKV, 4>(g, n_tiles, s) : launch<SMALL_EMBED, SMALL_QKV, 2>(g, n_tiles, s);
    if (src == SMALL_BF16) return launch<SMALL_BF16, SMALL_RESIDUAL, 2>(g, n_tiles, s);
    switch (epi) {
        case SMALL_QKV: return wide ? launch<SMALL_NORM, SMALL_QKV, 4>(g, n_tiles, s) : launch<SMALL_NORM, SMALL_QKV, 2>(g, n_tiles, s);
        case SMALL_SWIGLU: return wide ? launch<SMALL_NORM, SMALL_SWIGLU, 4>(g, n_tiles, s) : launch<SMALL_NORM, SMALL_SWIGLU, 2>(g, n_tiles, s);
        default: return wide ? launch<SMALL_NORM, SMALL_STORE, 4>(g, n_tiles, s) : launch<SMALL_NORM, SMALL_STORE, 2>(g, n_tiles, s);
    }
}

}  // namespace sfs
