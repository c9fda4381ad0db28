// What the kernels of small models share: mma.sync from shared memory, and the attention of 16 query rows by warps that divide the keys.
#pragma once
#include "sfs_common.cuh"
#include "attention.cuh"
#include "tc05.cuh"

namespace sfs {
namespace small {

using tc::smem_u32;
__device__ __forceinline__ void ldmatrix4(uint32_t *r, uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_16816(float *c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_16816(float *c, const uint32_t *a, uint32_t b0, uint32_t b1) { mma_16816(c, a[0], a[1], a[2], a[3], b0, b1); }
// the first eight columns of k
__device__ __forceinline__ void mma_1688(float *c, const uint32_t *a, uint32_t b) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(b));
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&h);
}
__device__ __forceinline__ float round_bf16(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float silu(float x) { return __fdividef(x, 1.0f + __expf(-x)); }
__device__ __forceinline__ float ex2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }

// ---- attention, heads of 64: PARTS warps take 16 query rows of a head and divide the keys, 32 at a time ------------------------
// Operands of mma.sync come straight from L2 into registers: within 32 columns both use the same order of k, in which a thread's
// fragments are 16 consecutive bytes.  A score tile's columns are assigned to keys such that the probabilities of a thread are
// those of eight consecutive keys, which is the operand order of V transposed.
constexpr int kHead = 64, kHeadBlocks = kHead / 32;      // head dimension, in 32-column blocks
constexpr int kPartLd = kHead + 4;                       // floats between rows of a partial result
constexpr size_t kPartBytes = (16 * kPartLd + 32) * sizeof(float);      // a warp's partial result, row maxima and denominators

// 32 columns of k: rows r (a) and r + 8 (b) of the thread's group against column lane / 4 (w)
__device__ __forceinline__ void mma_k32(float *c, const uint4 &a, const uint4 &b, const uint4 &w) {
    mma_16816(c, a.x, b.x, a.y, b.y, w.x, w.y);
    mma_16816(c, a.z, b.z, a.w, b.w, w.z, w.w);
}
__device__ __forceinline__ uint4 ldg16(const __nv_bfloat16 *p) { return *reinterpret_cast<const uint4 *>(p); }

// This warp's share (`part`) of the keys for query rows r0 .. r0 + 15 (clamped to kq) of sequence b: unnormalised rows into ob
// [16][kPartLd], their maxima and denominators into s_ml [32].
template <int PARTS>
__device__ __forceinline__ void attn_part(const AttnShort &p, int S, int kq, float cs, int head, int b, int r0, int part, int lane, float *ob, float *s_ml)
{
    const int g = lane >> 2, c = lane & 3;
    const long long tok0 = (long long)b * S;
    const int ra = min(r0 + g, kq - 1), rb = min(r0 + g + 8, kq - 1);
    uint4 qa[kHeadBlocks], qb[kHeadBlocks];
#pragma unroll
    for (int i = 0; i < kHeadBlocks; ++i) {
        qa[i] = ldg16(p.q + ((long long)b * kq + ra) * p.ld_q + head * kHead + i * 32 + c * 8);
        qb[i] = ldg16(p.q + ((long long)b * kq + rb) * p.ld_q + head * kHead + i * 32 + c * 8);
    }
    float o[kHead / 8][4];
#pragma unroll
    for (int f = 0; f < kHead / 8; ++f) o[f][0] = o[f][1] = o[f][2] = o[f][3] = 0.f;
    float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
    for (int k0 = part * 32; k0 < S; k0 += 32 * PARTS) {
        const bool valid = k0 + c * 8 < S;               // this thread's eight keys (S is a multiple of 8)
        uint4 kf[4][kHeadBlocks], vf[kHead / 8];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            // column n of score tile t is key 8 (n / 2) + 2 t + n % 2
            const int key = min(k0 + (g >> 1) * 8 + 2 * t + (g & 1), S - 1);
#pragma unroll
            for (int i = 0; i < kHeadBlocks; ++i) kf[t][i] = ldg16(p.k + (tok0 + key) * p.ld_k + head * kHead + i * 32 + c * 8);
        }
#pragma unroll
        for (int f = 0; f < kHead / 8; ++f)
            vf[f] = valid ? ldg16(p.vt + (long long)(head * kHead + f * 8 + g) * p.ld_vt + tok0 + k0 + c * 8) : make_uint4(0, 0, 0, 0);
        float sc[4][4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            sc[t][0] = sc[t][1] = sc[t][2] = sc[t][3] = 0.f;
#pragma unroll
            for (int i = 0; i < kHeadBlocks; ++i) mma_k32(sc[t], qa[i], qb[i], kf[t][i]);
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
        for (int f = 0; f < kHead / 8; ++f) {
            o[f][0] *= al0; o[f][1] *= al0; o[f][2] *= al1; o[f][3] *= al1;
            mma_16816(o[f], pa[0], pb[0], pa[1], pb[1], vf[f].x, vf[f].y);
            mma_16816(o[f], pa[2], pb[2], pa[3], pb[3], vf[f].z, vf[f].w);
        }
    }
    l0 += __shfl_xor_sync(0xffffffffu, l0, 1); l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
    l1 += __shfl_xor_sync(0xffffffffu, l1, 1); l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
#pragma unroll
    for (int f = 0; f < kHead / 8; ++f) {
        *reinterpret_cast<float2 *>(ob + g * kPartLd + f * 8 + 2 * c) = make_float2(o[f][0], o[f][1]);
        *reinterpret_cast<float2 *>(ob + (g + 8) * kPartLd + f * 8 + 2 * c) = make_float2(o[f][2], o[f][3]);
    }
    if (c == 0) { s_ml[g] = m0; s_ml[g + 8] = m1; s_ml[16 + g] = l0; s_ml[24 + g] = l1; }
}

// The partial results of a tile (go: [PARTS][16][kPartLd], gml: [PARTS][32]; the first `used` warps had keys) combined: lanes of warp
// `part` take whole rows, so that full lines are written; store(row, column, four bf16) receives them.
template <int PARTS, typename Store>
__device__ __forceinline__ void attn_merge(const float *go, const float *gml, int used, float cs, int part, int lane, Store &&store)
{
    constexpr int COLS = 32 / PARTS, LPR = kHead / COLS;      // columns per lane, lanes per row
    const int r = part * (16 / PARTS) + lane / LPR, col = (lane % LPR) * COLS;
    const float *row = go + r * kPartLd + col;
    float mm = -INFINITY, den = 0.f, f[PARTS];
#pragma unroll
    for (int i = 0; i < PARTS; ++i) mm = fmaxf(mm, i < used ? gml[i * 32 + r] : -INFINITY);
#pragma unroll
    for (int i = 0; i < PARTS; ++i) { f[i] = i < used ? ex2((gml[i * 32 + r] - mm) * cs) : 0.f; if (i < used) den += f[i] * gml[i * 32 + 16 + r]; }
    const float inv = 1.0f / den;
#pragma unroll
    for (int k = 0; k < COLS / 4; ++k) {
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < PARTS; ++i) {
            if (i >= used) continue;
            const float4 v = *reinterpret_cast<const float4 *>(row + i * 16 * kPartLd + 4 * k);
            acc.x += f[i] * v.x; acc.y += f[i] * v.y; acc.z += f[i] * v.z; acc.w += f[i] * v.w;
        }
        store(r, col + 4 * k, make_uint2(pack2(acc.x * inv, acc.y * inv), pack2(acc.z * inv, acc.w * inv)));
    }
}

}  // namespace small
}  // namespace sfs
