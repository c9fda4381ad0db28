// Attention of short sequences with heads of 64, where what counts is the length of the chain.
//
// For a small model's step the tcgen05 kernel takes 5 us, most of them outside its key tiles: barriers and tensor memory set up,
// TMA round trips, the hand-overs of one tile.  Here four warps take 16 query rows of a head and divide the keys, 32 at a time,
// straight from L2 into registers as operands of mma.sync: within 32 columns both operands use the same order of k, in which a
// thread's fragments are 16 consecutive bytes.  A score tile's columns are assigned to keys such that the probabilities of a
// thread are those of eight consecutive keys, which is the operand order of V transposed.  The four partial results are merged in
// shared memory.  Bound: one L2 round trip, 32 dependent MMAs, the merge and the store; every 16 (or 32) query rows read all keys
// and values of the head again, which bounds the lengths this is good for.
#include "sfs_common.cuh"
#include "attention.cuh"
#include "gemm.cuh"

namespace sfs {
namespace {

constexpr int DH = 64, NB = DH / 32;         // head dimension, in 32-column blocks
constexpr int LD = DH + 4;                   // floats between rows of a partial result
constexpr size_t kWarpSmem = (16 * LD + 32) * sizeof(float);

__device__ __forceinline__ void mma_16816(float *c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// 32 columns of k: rows r (a) and r + 8 (b) of the thread's group against column lane / 4 (w)
__device__ __forceinline__ void mma_k32(float *c, const uint4 &a, const uint4 &b, const uint4 &w) {
    mma_16816(c, a.x, b.x, a.y, b.y, w.x, w.y);
    mma_16816(c, a.z, b.z, a.w, b.w, w.z, w.w);
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&h);
}
__device__ __forceinline__ float ex2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ uint4 ldg16(const __nv_bfloat16 *p) { return *reinterpret_cast<const uint4 *>(p); }
// PARTS warps divide the keys; grid: (query rows / (16 x tiles per CTA), heads, sequences); blockDim: 32 PARTS x tiles per CTA
template <int PARTS>
__global__ void __launch_bounds__(256, 1)
attention_short_kernel(AttnShort p, AttnArgs a)
{
    extern __shared__ __align__(16) float s_out[];       // per warp [16][LD], then per warp [32]: maxima, denominators
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3, part = warp & (PARTS - 1), n_warps = blockDim.x >> 5;
    const int S = a.S, head = blockIdx.y, b = blockIdx.z, r0 = (blockIdx.x * (n_warps / PARTS) + warp / PARTS) * 16;
    const long long tok0 = (long long)b * S;
    const float cs = a.scale_log2;
    float *ob = s_out + warp * 16 * LD, *s_ml = s_out + n_warps * 16 * LD + warp * 32;

    pdl_wait();
    pdl_trigger();
    const bool active = a.d_active == nullptr || *a.d_active != 0;      // (used only after the loads below)
    const int ra = min(r0 + g, a.kq - 1), rb = min(r0 + g + 8, a.kq - 1);
    uint4 qa[NB], qb[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        qa[i] = ldg16(p.q + ((long long)b * a.kq + ra) * p.ld_q + head * DH + i * 32 + c * 8);
        qb[i] = ldg16(p.q + ((long long)b * a.kq + rb) * p.ld_q + head * DH + i * 32 + c * 8);
    }
    float o[DH / 8][4];
#pragma unroll
    for (int f = 0; f < DH / 8; ++f) o[f][0] = o[f][1] = o[f][2] = o[f][3] = 0.f;
    float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
    for (int k0 = part * 32; k0 < S; k0 += 32 * PARTS) {
        const bool valid = k0 + c * 8 < S;               // this thread's eight keys (S is a multiple of 8)
        uint4 kf[4][NB], vf[DH / 8];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            // column n of score tile t is key 8 (n / 2) + 2 t + n % 2
            const int key = min(k0 + (g >> 1) * 8 + 2 * t + (g & 1), S - 1);
#pragma unroll
            for (int i = 0; i < NB; ++i) kf[t][i] = ldg16(p.k + (tok0 + key) * p.ld_k + head * DH + i * 32 + c * 8);
        }
#pragma unroll
        for (int f = 0; f < DH / 8; ++f)
            vf[f] = valid ? ldg16(p.vt + (long long)(head * DH + f * 8 + g) * p.ld_vt + tok0 + k0 + c * 8) : make_uint4(0, 0, 0, 0);
        float sc[4][4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            sc[t][0] = sc[t][1] = sc[t][2] = sc[t][3] = 0.f;
#pragma unroll
            for (int i = 0; i < NB; ++i) mma_k32(sc[t], qa[i], qb[i], kf[t][i]);
        }
        float x0 = -INFINITY, x1 = -INFINITY;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            if (!valid) sc[t][0] = sc[t][1] = sc[t][2] = sc[t][3] = -INFINITY;
            x0 = fmaxf(x0, fmaxf(sc[t][0], sc[t][1])); x1 = fmaxf(x1, fmaxf(sc[t][2], sc[t][3]));
        }
        x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, 1)); x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, 2));
        x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, 1)); x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, 2));
        const float n0 = fmaxf(m0, x0), n1 = fmaxf(m1, x1);               // every block has a valid key
        const float al0 = ex2((m0 - n0) * cs), al1 = ex2((m1 - n1) * cs);
        m0 = n0; m1 = n1; l0 *= al0; l1 *= al1;
        uint32_t pa[4], pb[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const float e0 = ex2(fmaf(sc[t][0], cs, -n0 * cs)), e1 = ex2(fmaf(sc[t][1], cs, -n0 * cs));
            const float e2 = ex2(fmaf(sc[t][2], cs, -n1 * cs)), e3 = ex2(fmaf(sc[t][3], cs, -n1 * cs));
            l0 += e0 + e1; l1 += e2 + e3;
            pa[t] = pack2(e0, e1); pb[t] = pack2(e2, e3);
        }
#pragma unroll
        for (int f = 0; f < DH / 8; ++f) {
            o[f][0] *= al0; o[f][1] *= al0; o[f][2] *= al1; o[f][3] *= al1;
            mma_16816(o[f], pa[0], pb[0], pa[1], pb[1], vf[f].x, vf[f].y);
            mma_16816(o[f], pa[2], pb[2], pa[3], pb[3], vf[f].z, vf[f].w);
        }
    }
    l0 += __shfl_xor_sync(0xffffffffu, l0, 1); l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
    l1 += __shfl_xor_sync(0xffffffffu, l1, 1); l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
#pragma unroll
    for (int f = 0; f < DH / 8; ++f) {
        *reinterpret_cast<float2 *>(ob + g * LD + f * 8 + 2 * c) = make_float2(o[f][0], o[f][1]);
        *reinterpret_cast<float2 *>(ob + (g + 8) * LD + f * 8 + 2 * c) = make_float2(o[f][2], o[f][3]);
    }
    if (!active) return;                                  // nothing left to decode
    if (c == 0) { s_ml[g] = m0; s_ml[g + 8] = m1; s_ml[16 + g] = l0; s_ml[24 + g] = l1; }
    __syncthreads();
    // the partial results of a tile: whole rows per warp, so that full lines are written
    constexpr int COLS = 32 / PARTS, LPR = DH / COLS;      // columns per lane, lanes per row
    const int r = part * (16 / PARTS) + lane / LPR, col = (lane % LPR) * COLS, first = warp & ~(PARTS - 1);
    const float *gml = s_out + n_warps * 16 * LD + first * 32, *go = s_out + first * 16 * LD + r * LD + col;
    float mm = -INFINITY, den = 0.f, f[PARTS];
#pragma unroll
    for (int i = 0; i < PARTS; ++i) mm = fmaxf(mm, gml[i * 32 + r]);
#pragma unroll
    for (int i = 0; i < PARTS; ++i) { f[i] = ex2((gml[i * 32 + r] - mm) * cs); den += f[i] * gml[i * 32 + 16 + r]; }      // (a warp without keys: factor 0)
    const float inv = 1.0f / den;
    if (r0 + r < a.kq) {
        __nv_bfloat16 *dst = a.out + ((long long)b * a.kq + r0 + r) * a.ld_out + head * DH + col;
#pragma unroll
        for (int k = 0; k < COLS / 4; ++k) {
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < PARTS; ++i) {
                const float4 v = *reinterpret_cast<const float4 *>(go + i * 16 * LD + 4 * k);
                acc.x += f[i] * v.x; acc.y += f[i] * v.y; acc.z += f[i] * v.z; acc.w += f[i] * v.w;
            }
            *reinterpret_cast<uint2 *>(dst + 4 * k) = make_uint2(pack2(acc.x * inv, acc.y * inv), pack2(acc.z * inv, acc.w * inv));
        }
    }
}

template <int PARTS>
int32_t launch(const AttnPlan &p, const AttnArgs &a, int mt, cudaStream_t s)
{
    const size_t smem = (size_t)mt * PARTS * kWarpSmem;
    static bool configured[kMaxDevices] = {};
    bool &done = configured[current_device_slot()];
    if (!done) {
        SFS_CUDA(cudaFuncSetAttribute(attention_short_kernel<PARTS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(8 * kWarpSmem)));
        done = true;
    }
    SFS_CUDA(launch_pdl(attention_short_kernel<PARTS>, dim3((unsigned)((a.kq + 16 * mt - 1) / (16 * mt)), (unsigned)a.n_heads, (unsigned)a.B), dim3((unsigned)(32 * PARTS * mt)),
                        smem, s, p.direct, a));
    return SFS_OK;
}

}  // namespace

// Heads of 64 and at most one wave of CTAs of two tiles.  4 heads, us per launch back to back, against the tcgen05 kernel: 64 tokens
// 2.6 / 4.6, 224 3.5 / 5.4, 4 x 224 4.4 / 5.6, 512 6.4 / 7.7, 3 x 512 (two waves) 10.9 / 7.8; in the chain of a step 192 tokens
// 2.4 / 6.0.  Heads of 128 gain nothing: 32 of them, 104 tokens 5.1 / 5.8, 192 tokens 11.5 / 6.8.
bool attn_is_short(const AttnPlan &p, int32_t kq)
{
    return p.head_dim == DH && p.args.S <= 512 && (long long)((kq + 31) / 32) * p.args.n_heads * p.args.B <= gemm_num_sms();
}

int32_t attn_launch_short(const AttnPlan &p, int32_t kq, const int32_t *d_active, cudaStream_t stream)
{
    AttnArgs a = p.args;
    a.d_active = d_active; a.kq = kq;
    const bool wave = (long long)((kq + 15) / 16) * a.n_heads * a.B <= gemm_num_sms();      // a CTA per tile leaves SMs free
    if (a.S <= 128) return launch<4>(p, a, wave ? 1 : 2, stream);
    return wave ? launch<8>(p, a, 1, stream) : launch<4>(p, a, 2, stream);
}

}  // namespace sfs
