// The canonical softmax denominator S_q = sum_v trunc(2^28 exp(x_v - m)): the fixed-point exponential of a logit, evaluated two at
// a time, and the recomputation of listed rows that the selection step shares out over its warps.
#pragma once
#include "sfs_common.cuh"

namespace sfs {

constexpr float kLog2e = 0x1.715476p+0f;
constexpr float kLn2   = 0x1.62e430p-1f;
constexpr float kMagic = 12582912.0f;           // 1.5 * 2^23
constexpr float kC1 = 0x1.fffa48p-1f;
constexpr float kC2 = 0x1.fff8fcp-2f;
constexpr float kC3 = 0x1.57f67cp-3f;
constexpr float kC4 = 0x1.57de66p-5f;
constexpr uint32_t kShiftBase = 0x4B400003u;    // bits(kMagic) + 3

__device__ __forceinline__ uint32_t shr_clamp(uint32_t x, uint32_t s) {
    uint32_t r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));   // PTX semantics: shift >= 32 gives 0
    return r;
}

// ---- packed f32x2 arithmetic (two lanes per instruction) ----------------------------------------------
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi)); return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, uint32_t &lo, uint32_t &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r;
}

struct Consts2 { f32x2 negm, l2e, magic, negmagic, negln2, c1, c2, c3, c4, three; };

// the terms of two packed logits; returns e_lo + e_hi (each < 1.42 * 2^28)
__device__ __forceinline__ uint32_t canon2(f32x2 x, const Consts2 &k) {
    const f32x2 d = add2(x, k.negm);
    const f32x2 r = fma2(d, k.l2e, k.magic);
    const f32x2 n = add2(r, k.negmagic);
    const f32x2 f = fma2(n, k.negln2, d);
    f32x2 q = fma2(f, k.c4, k.c3);
    q = fma2(f, q, k.c2);
    q = fma2(f, q, k.c1);
    const f32x2 P = fma2(f, q, k.three);
    uint32_t r0, r1, p0, p1;
    unpack2(r, r0, r1);
    unpack2(P, p0, p1);
    return shr_clamp(p0 << 9, kShiftBase - r0) + shr_clamp(p1 << 9, kShiftBase - r1);
}

// the same from one 32-bit word holding two bf16 logits
__device__ __forceinline__ uint32_t canon_pair(uint32_t w, const Consts2 &k) {
    return canon2(pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u)), k);
}

__device__ __forceinline__ Consts2 canon_consts(float m) {
    Consts2 k;
    k.negm = pack2(-m, -m);           k.l2e = pack2(kLog2e, kLog2e);
    k.magic = pack2(kMagic, kMagic);  k.negmagic = pack2(-kMagic, -kMagic);
    k.negln2 = pack2(-kLn2, -kLn2);
    k.c1 = pack2(kC1, kC1); k.c2 = pack2(kC2, kC2); k.c3 = pack2(kC3, kC3); k.c4 = pack2(kC4, kC4);
    k.three = pack2(3.0f, 3.0f);
    return k;
}

// Canonical S_q of the listed positions' logits rows (bf16, 16-byte aligned, a multiple of 8 entries), by `n_warps` warps of which
// this one is `w`: a row is cut into items, and every item's integer sum is added to pos_sq of its position (which is zero before) —
// integer addition commutes, so the order of arrival does not matter.  The rows come from L2: the first pass has just streamed them,
// or the LM head wrote them.  An item is a round trip, a warp's reduction and an atomic, so it is as long as spreads all rows over all
// warps once (4 to 16 chunks a lane), with the loads of the next four chunks ahead of the terms of four: 53 rows of 126464 took 11000
// clocks as items of four chunks whose row number was another round trip.
constexpr int kOpenBatch = 4, kOpenMost = 4;                // chunks of a lane in a batch, batches in an item
__device__ __forceinline__ void recompute_rows(const LogitsRows &g, const int32_t *list, const int32_t *row_of, int n, const float *pos_max,
                                               unsigned long long *pos_sq, int w, int n_warps)
{
    const int lane = threadIdx.x & 31, batch = 32 * kOpenBatch, row_batches = (g.chunks + batch - 1) / batch;
    const int per = min(kOpenMost, max(1, (n * row_batches + n_warps - 1) / n_warps)), items = (row_batches + per - 1) / per;
    for (int it = w; it < n * items; it += n_warps) {
        const int r = it / items, first = (it - r * items) * per * batch + lane, end = min(g.chunks, first - lane + per * batch);
        const int pos = list[r];
        const uint4 *rp = g.base + (long long)row_of[r] * g.ld;
        uint4 v[2][kOpenBatch];
        auto fetch = [&](uint4 *q, int c) {
#pragma unroll
            for (int u = 0; u < kOpenBatch; ++u)
                q[u] = c + 32 * u < end ? __ldcg(rp + c + 32 * u) : make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);
        };
        fetch(v[0], first);
        const Consts2 k = canon_consts(__ldcg(&pos_max[pos]));
        unsigned long long acc = 0;
#pragma unroll
        for (int t = 0; t < kOpenMost; ++t) {
            if (t >= per) break;
            if (t + 1 < per) fetch(v[(t + 1) & 1], first + (t + 1) * batch);
#pragma unroll
            for (int u = 0; u < kOpenBatch; ++u)            // 8 terms < 8 * 1.42 * 2^28 < 2^32
                acc += canon_pair(v[t & 1][u].x, k) + canon_pair(v[t & 1][u].y, k) + canon_pair(v[t & 1][u].z, k) + canon_pair(v[t & 1][u].w, k);
        }
        acc = warp_sum_u64(acc);
        if (lane == 0) atomicAdd(&pos_sq[pos], acc);
    }
}

}  // namespace sfs
