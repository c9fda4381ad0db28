// Bidirectional (unmasked) multi-head attention of the mask predictor: out = softmax(q k^T / sqrt(dh)) v
// over all S positions of the same sequence.
//
// A CTA runs two streams of 128 query rows x 128-key tiles, so that the tensor core works on one while the softmax of the other
// runs.  With enough rows (PAIR) the streams are two query tiles of the same head that share every key and value tile; with few
// of them (cached steps, one short sequence) they are the even and the odd key tiles of one query tile, and the two partial
// results are combined at the end.
// Warp 0 streams K tiles [128 keys x dh] and V^T tiles [dh x 128 keys] through two two-stage TMA rings.  Warp 1 issues
// tcgen05.mma per stream: S = Q K_j^T into tensor memory, then O += P_j V_j with P read from tensor memory, followed at once by
// the next tile's S into the columns that P occupied (MMAs of a CTA execute in order, and P is written only after S was read).
// Warps 2-5 are the softmax of stream 0, warps 6-9 of stream 1, one thread per query row: it reads its 128 scores with
// tcgen05.ld, runs the online softmax in fp32 and writes the probabilities back as bf16 with tcgen05.st.  The exponentials
// use a reference maximum that is moved (with a rescale of O and of the denominator) only when the true running maximum has
// outgrown it by 2^8: the result is the same softmax, most tiles skip the pass over O.  V is consumed transposed (features x
// tokens); the QKV projection's epilogue writes it that way.
//
// Bound: a 128 x 128 tile needs 1024 clocks of the special-function unit and as many of the tensor core (dh = 128); the chain
// scores -> maximum -> exponentials -> P -> MMAs with its hand-overs takes ~4000 clocks for a pair of them, ~2500 of which remain
// without the exponentials and most of the MMAs, and a CTA spends 5.5 us outside its key tiles.  Measured, 32 heads of 128, us
// (before, with one stream per CTA and P through shared memory, in brackets): 512 tokens 9.8 [10.7], 1000 23 [32], 1536 51 [62],
// 2048 75 [103], 8 x 768 109 [142].  Score buffers of 64 keys, two per stream, hide the chain but double the hand-overs and
// the issue of MMAs at N = 64: 2048 tokens 88.
#include "sfs_common.cuh"
#include "tc05.cuh"
#include "attention.cuh"
#include "gemm.cuh"

namespace sfs {
namespace {

constexpr int kAttnThreads = 64 + 256;   // TMA warp, MMA warp, 2 x 4 softmax warps
constexpr int QT = 128;                 // query rows per stream
constexpr int KT = 128;                 // keys per tile
constexpr int KV_STAGES = 2;
constexpr int kAttnBars = 4 * KV_STAGES + 8;   // K full/empty, V full/empty, Q, S (two), P (two halves of two), exchange

template <int DH, bool PAIR>
__global__ void __launch_bounds__(kAttnThreads, 1)
attention_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmVt, AttnArgs a)
{
    constexpr int NQ = PAIR ? 2 : 1;                     // query tiles of this CTA
    constexpr int KB = DH / 64;                          // 64-element K-blocks along the head dimension
    constexpr int Q_BYTES = QT * DH * 2;
    constexpr int K_BYTES = KT * DH * 2;
    constexpr int V_BYTES = DH * KT * 2;
    constexpr uint32_t TMEM_COLS = 512;                  // S / P and O of each stream: 2 x (128 + DH) columns

    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *sQ = smem, *sK = smem + NQ * Q_BYTES, *sV = sK + KV_STAGES * K_BYTES;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sV + KV_STAGES * V_BYTES);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + kAttnBars);
    __shared__ int s_abort;
    __shared__ float s_max[2][QT], s_den[2][QT];           // key-split streams: what the combination needs

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q0 = blockIdx.x * (QT * NQ), h = blockIdx.y, b = blockIdx.z;
    const int S = a.S;
    const int tok0 = b * S;                                // first key / value token of this sequence
    const int qrow0 = b * a.kq + q0;                       // first query row of this CTA (queries may be a compact subset)
    const int nkv = (S + KT - 1) / KT;
    const int n_streams = PAIR ? (q0 + QT < a.kq ? 2 : 1) : (nkv > 1 ? 2 : 1);
    auto tiles_of = [&](int w) { return w >= n_streams ? 0 : (PAIR ? nkv : (nkv - w + 1) / 2); };     // key tiles of stream w
    auto key_tile = [&](int w, int i) { return PAIR ? i : 2 * i + w; };                               // its i-th one

    const uint32_t bar_kfull = tc::smem_u32(bars), bar_kempty = bar_kfull + 8 * KV_STAGES;
    const uint32_t bar_vfull = bar_kempty + 8 * KV_STAGES, bar_vempty = bar_vfull + 8 * KV_STAGES;
    const uint32_t bar_q = bar_vempty + 8 * KV_STAGES, bar_s = bar_q + 8 /* two */, bar_p = bar_q + 24 /* + 16 w + 8 half */, bar_x = bar_q + 56;

    if (threadIdx.x == 0) {
        for (int s = 0; s < KV_STAGES; ++s) {
            tc::mbar_init(bar_kfull + 8 * s, 1); tc::mbar_init(bar_kempty + 8 * s, 1);
            tc::mbar_init(bar_vfull + 8 * s, 1); tc::mbar_init(bar_vempty + 8 * s, 1);
        }
        tc::mbar_init(bar_q, 1);
        for (int w = 0; w < 2; ++w) { tc::mbar_init(bar_s + 8 * w, 1); tc::mbar_init(bar_p + 16 * w, QT); tc::mbar_init(bar_p + 16 * w + 8, QT); }
        tc::mbar_init(bar_x, 2 * QT);
        s_abort = 0;
        tc::mbar_init_fence();
    }
    if (warp == 0 && lane == 0) { tc::tma_prefetch_desc(&tmQ); tc::tma_prefetch_desc(&tmK); tc::tma_prefetch_desc(&tmVt); }
    if (warp == 1) { tc::tmem_alloc(tc::smem_u32(tmem_slot), TMEM_COLS); tc::tmem_relinquish(); }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t *>(tmem_slot);
    const uint32_t tmem_S = tmem_base, tmem_O = tmem_base + 2 * KT;      // stream w: + w * KT, + w * DH

    pdl_wait();                                          // the kernel before this one has completed: global memory from here on
    pdl_trigger();                                       // (not before the wait: see pdl_trigger)
    const bool live = !(a.d_active && *a.d_active == 0); // nothing left to decode: straight to the teardown (uniform)
    if (live) {
    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer: Q once, then K tiles and V^T tiles through their own rings (a K stage is free
            // again as soon as its last S = Q K^T has been computed, a V stage after its last P V)
            const int n_q = PAIR ? n_streams : 1;          // (a second tile that holds no queries is not loaded: 1024 heads of 128 over 64 tokens 35.1 us instead of 36.3)
            tc::mbar_expect_tx(bar_q, (uint32_t)(n_q * Q_BYTES));
            for (int t = 0; t < n_q; ++t)
#pragma unroll
                for (int kb = 0; kb < KB; ++kb)
                    tc::tma_load_2d(tc::smem_u32(sQ) + t * Q_BYTES + kb * (QT * 128), &tmQ, h * DH + kb * 64, qrow0 + t * QT, bar_q);
            int issued_k = 0, issued_v = 0;
            for (int j = 0; j < nkv; ++j) {
                const int s = j % KV_STAGES;
                const uint32_t ph = (uint32_t)(j / KV_STAGES) & 1u;
                if (!tc::mbar_wait(bar_kempty + 8 * s, ph ^ 1u, &s_abort)) break;
                const uint32_t sk = tc::smem_u32(sK) + s * K_BYTES;
                tc::mbar_expect_tx(bar_kfull + 8 * s, K_BYTES);
#pragma unroll
                for (int kb = 0; kb < KB; ++kb)
                    tc::tma_load_2d(sk + kb * (KT * 128), &tmK, a.k_col0 + h * DH + kb * 64, tok0 + j * KT, bar_kfull + 8 * s);
                issued_k = j + 1;
                if (!tc::mbar_wait(bar_vempty + 8 * s, ph ^ 1u, &s_abort)) break;
                const uint32_t sv = tc::smem_u32(sV) + s * V_BYTES;
                tc::mbar_expect_tx(bar_vfull + 8 * s, V_BYTES);
#pragma unroll
                for (int kb = 0; kb < KT / 64; ++kb)
                    tc::tma_load_2d(sv + kb * (DH * 128), &tmVt, tok0 + j * KT + kb * 64, h * DH, bar_vfull + 8 * s);
                issued_v = j + 1;
            }
            if (s_abort) {
                // give copies already in flight a bounded chance to land before the CTA retires
                for (int j = max(0, issued_k - KV_STAGES); j < issued_k; ++j) {
                    const uint32_t bar = bar_kfull + 8 * (j % KV_STAGES), ph = (uint32_t)(j / KV_STAGES) & 1u;
                    for (int i = 0; i < (1 << 16) && !tc::mbar_try(bar, ph); ++i) {}
                }
                for (int j = max(0, issued_v - KV_STAGES); j < issued_v; ++j) {
                    const uint32_t bar = bar_vfull + 8 * (j % KV_STAGES), ph = (uint32_t)(j / KV_STAGES) & 1u;
                    for (int i = 0; i < (1 << 16) && !tc::mbar_try(bar, ph); ++i) {}
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: the whole warp runs the loop with warp-uniform operands, one elected lane issues.
        constexpr uint32_t idesc_s = tc::idesc_bf16_f32(QT, KT);
        constexpr uint32_t idesc_o = tc::idesc_bf16_f32(QT, DH);
        const int last = n_streams - 1;
        // S of stream w on key tile j; bar_s of the stream completes when it, and every MMA before it, has completed
        auto issue_S = [&](int w, int j) {
            const int s = j % KV_STAGES;
            if (!__all_sync(0xffffffffu, tc::mbar_wait(bar_kfull + 8 * s, (uint32_t)(j / KV_STAGES) & 1u, &s_abort))) return false;
            tc::tc_fence_after();
            const uint32_t sk = tc::smem_u32(sK) + s * K_BYTES, sq = tc::smem_u32(sQ) + (PAIR ? w : 0) * Q_BYTES, d = tmem_S + (uint32_t)(w * KT);
#pragma unroll
            for (int kb = 0; kb < KB; ++kb) {
                const uint64_t dq = tc::smem_desc_sw128(sq + kb * (QT * 128));
                const uint64_t dk = tc::smem_desc_sw128(sk + kb * (KT * 128));
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    tc::mma_bf16_elect(d, dq + (uint64_t)(kk * 2), dk + (uint64_t)(kk * 2), idesc_s, (kb | kk) != 0 ? 1u : 0u);
            }
            tc::mma_commit_elect(bar_s + 8 * w);
            if (!PAIR || w == last) tc::mma_commit_elect(bar_kempty + 8 * s);
            return true;
        };
        bool ok = __all_sync(0xffffffffu, tc::mbar_wait(bar_q, 0, &s_abort));
        for (int w = 0; w < n_streams && ok; ++w) ok = issue_S(w, key_tile(w, 0));
        const int n0 = tiles_of(0);
        for (int i = 0; i < n0 && ok; ++i) {
            for (int w = 0; w < n_streams && ok; ++w) {
                if (i >= tiles_of(w)) continue;
                const int j = key_tile(w, i), s = j % KV_STAGES;
                ok = __all_sync(0xffffffffu, tc::mbar_wait(bar_vfull + 8 * s, (uint32_t)(j / KV_STAGES) & 1u, &s_abort));
                const uint32_t sv = tc::smem_u32(sV) + s * V_BYTES, tp = tmem_S + (uint32_t)(w * KT), d = tmem_O + (uint32_t)(w * DH);
#pragma unroll
                for (int kb = 0; kb < KT / 64; ++kb) {
                    // this half of P written (the first: O rescaled too); the softmax goes on with the second half meanwhile
                    ok = ok && __all_sync(0xffffffffu, tc::mbar_wait(bar_p + 16 * w + 8 * kb, (uint32_t)i & 1u, &s_abort));
                    if (!ok) break;
                    tc::tc_fence_after();
                    const uint64_t dv = tc::smem_desc_sw128(sv + kb * (DH * 128));
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)      // 16 keys are 8 columns of packed pairs
                        tc::mma_bf16_ts_elect(d, tp + (uint32_t)(kb * 32 + kk * 8), dv + (uint64_t)(kk * 2), idesc_o, (i | kb | kk) != 0 ? 1u : 0u);
                }
                if (!ok) break;
                if (!PAIR || w == last) tc::mma_commit_elect(bar_vempty + 8 * s);
                if (i + 1 < tiles_of(w)) ok = issue_S(w, key_tile(w, i + 1));
                else tc::mma_commit_elect(bar_s + 8 * w);                                   // O of the stream is complete
            }
        }
    } else {
        // ---------------- online softmax, one thread per query row.  O accumulates in tensor memory over the tiles; the
        // exponentials are taken against a reference maximum that follows the true running maximum lazily: it is moved (and
        // O and the denominator rescaled) only when the true one has risen by more than 2^8, so most tiles need no pass over O.
        constexpr float kLazy = 8.0f;                      // in log2 units: probabilities stay below 2^8
        const int w = (warp - 2) >> 2, row = (warp & 3) * 32 + lane;
        const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t ts = tmem_S + (uint32_t)(w * KT) + lane_off, to = tmem_O + (uint32_t)(w * DH) + lane_off;
        const float c = a.scale_log2;                      // log2(e) / sqrt(dh)
        const int n_tiles = tiles_of(w);
        float m = -INFINITY, l = 0.f;                      // reference maximum, denominator
        bool ok = true;
        for (int i = 0; i < n_tiles && ok; ++i) {
            ok = tc::mbar_wait(bar_s + 8 * w, (uint32_t)i & 1u, &s_abort);      // (P V of the tile before has finished too)
            if (!ok) break;
            tc::tc_fence_after();
            uint32_t v[64], pk[32];
            const int valid = S - key_tile(w, i) * KT;     // keys of this tile that belong to the sequence
            auto load = [&](int q) {                       // 64 scores, those beyond the sequence -inf
                tc::tmem_ld32(ts + q * 64, v); tc::tmem_ld32(ts + q * 64 + 32, v + 32);
                tc::tmem_ld_wait32(v); tc::tmem_ld_wait32(v + 32);
                if (valid < KT) {
#pragma unroll
                    for (int k = 0; k < 64; ++k)
                        if (q * 64 + k >= valid) v[k] = 0xFF800000u;    // probability 0
                }
            };
            auto row_max = [&]() {
                float mx[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) mx[k] = __uint_as_float(v[k]);
#pragma unroll
                for (int k = 4; k + 7 < 64; k += 8)
#pragma unroll
                    for (int e = 0; e < 4; ++e) mx[e] = tc::max3(mx[e], __uint_as_float(v[k + e]), __uint_as_float(v[k + 4 + e]));
#pragma unroll
                for (int e = 0; e < 4; ++e) mx[e] = fmaxf(mx[e], __uint_as_float(v[60 + e]));
                return fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
            };
            unsigned long long sum2[2];
            auto half = [&]() {                            // 64 keys: 32 columns of packed pairs
                const float mc = m * c;
                const unsigned long long c2 = tc::pack_f32x2(c, c), mc2 = tc::pack_f32x2(-mc, -mc);
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                    float e0, e1;
                    tc::unpack_f32x2(tc::fma_f32x2(tc::pack_f32x2(__uint_as_float(v[2 * k]), __uint_as_float(v[2 * k + 1])), c2, mc2), e0, e1);
                    const float p0 = tc::ex2_approx(e0), p1 = tc::ex2_approx(e1);
                    sum2[k & 1] = tc::add_f32x2(sum2[k & 1], tc::pack_f32x2(p0, p1));
                    __nv_bfloat162 hh = __floats2bfloat162_rn(p0, p1);
                    pk[k] = *reinterpret_cast<uint32_t *>(&hh);
                }
            };
            auto hand = [&](int q) {
                tc::tmem_st32(ts + q * 32, pk);
                tc::tmem_st_wait();
                tc::tc_fence_before();                     // S has been read, this half of P written, O rescaled
                tc::mbar_arrive(bar_p + 16 * w + 8 * q);
            };
            // the maximum of the second half first (the first half is then in registers for its exponentials)
            load(1);
            const float m_hi = row_max();
            load(0);
            sum2[0] = sum2[1] = 0ull;
            const float m_row = fmaxf(row_max(), m_hi);
            if (i == 0) {
                m = m_row;
            } else {
                const bool move = (m_row - m) * c > kLazy;
                if (__any_sync(0xffffffffu, move)) {
                    const float alpha = move ? tc::ex2_approx((m - m_row) * c) : 1.0f;
#pragma unroll 1
                    for (int q = 0; q < DH / 32; ++q) {
                        uint32_t o[32];
                        tc::tmem_ld32(to + q * 32, o);
                        tc::tmem_ld_wait32(o);
#pragma unroll
                        for (int k = 0; k < 32; ++k) o[k] = __float_as_uint(__uint_as_float(o[k]) * alpha);
                        tc::tmem_st32(to + q * 32, o);
                    }
                    if (move) { l *= alpha; m = m_row; }
                }
            }
            half();
            hand(0);
            load(1);
            half();
            hand(1);
            float s0, s1;
            tc::unpack_f32x2(tc::add_f32x2(sum2[0], sum2[1]), s0, s1);
            l += s0 + s1;
        }
        if (n_tiles > 0) ok = ok && tc::mbar_wait(bar_s + 8 * w, (uint32_t)n_tiles & 1u, &s_abort);       // the last P V
        // output columns of this thread, and the factors of the streams' accumulators
        constexpr int COLS = PAIR ? DH : DH / 2;
        float f0 = 0.f, f1 = 0.f;                          // PAIR: f0 of the own stream
        bool write = ok && !s_abort;
        if (PAIR) {
            f0 = 1.0f / l;
            write = write && n_tiles > 0;
        } else {
            s_max[w][row] = m; s_den[w][row] = l;
            tc::tc_fence_before();
            tc::mbar_arrive(bar_x);
            write = tc::mbar_wait(bar_x, 0, &s_abort) && write && !s_abort;
            const float m0 = s_max[0][row], m1 = s_max[1][row], mm = fmaxf(m0, m1);
            f0 = tc::ex2_approx((m0 - mm) * c); f1 = n_streams > 1 ? tc::ex2_approx((m1 - mm) * c) : 0.f;
            const float inv = 1.0f / (f0 * s_den[0][row] + f1 * s_den[1][row]);
            f0 *= inv; f1 *= inv;
        }
        if (write) {
            tc::tc_fence_after();
            const int r = q0 + (PAIR ? w * QT : 0) + row, col0 = PAIR ? 0 : w * COLS;
            const bool in = r < a.kq;
            const uint32_t t0 = tmem_O + lane_off + (uint32_t)(PAIR ? w * DH : col0);
            __nv_bfloat16 *dst = a.out + (long long)(b * a.kq + r) * a.ld_out + h * DH + col0;
#pragma unroll
            for (int q = 0; q < COLS / 32; ++q) {
                uint32_t o[32], o1[32];
                tc::tmem_ld32(t0 + q * 32, o);             // warp-collective: every lane takes part
                if (!PAIR && n_streams > 1) tc::tmem_ld32(t0 + DH + q * 32, o1);
                tc::tmem_ld_wait32(o);
                if (!PAIR && n_streams > 1) tc::tmem_ld_wait32(o1);
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                    float x = __uint_as_float(o[k]) * f0;
                    if (!PAIR && n_streams > 1) x = fmaf(__uint_as_float(o1[k]), f1, x);
                    o[k] = __float_as_uint(x);
                }
                if (in) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        uint32_t wd[4];
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            __nv_bfloat162 hh = __floats2bfloat162_rn(__uint_as_float(o[8 * i + 2 * t]), __uint_as_float(o[8 * i + 2 * t + 1]));
                            wd[t] = *reinterpret_cast<uint32_t *>(&hh);
                        }
                        reinterpret_cast<uint4 *>(dst)[q * 4 + i] = make_uint4(wd[0], wd[1], wd[2], wd[3]);
                    }
                }
            }
        }
    }
    }   // live

    tc::tc_fence_before();
    __syncthreads();
    if (warp == 1) { tc::tc_fence_after(); tc::tmem_dealloc(tmem_base, TMEM_COLS); }
    if (threadIdx.x == 0 && s_abort && a.err) atomicExch(a.err, SFS_ERR_TIMEOUT);
}

template <int DH, bool PAIR>
int32_t launch_dh(const AttnPlan &p, int kq, const int32_t *d_active, int32_t *err, cudaStream_t stream)
{
    constexpr int NQ = PAIR ? 2 : 1;
    constexpr size_t need = (size_t)NQ * QT * DH * 2 + KV_STAGES * (size_t)(KT * DH * 2 + DH * KT * 2) + kAttnBars * 8 + 16 + 1024;
    constexpr size_t smem = need < 120 * 1024 ? 120 * 1024 : need;      // one CTA per SM: all 512 tensor-memory columns are its own
    static bool configured[kMaxDevices] = {};
    bool &done = configured[current_device_slot()];
    if (!done) {
        SFS_CUDA(cudaFuncSetAttribute(attention_kernel<DH, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        done = true;
    }
    AttnArgs a = p.args;
    a.err = err; a.d_active = d_active;
    if (kq > 0) a.kq = kq;
    dim3 grid((unsigned)((a.kq + NQ * QT - 1) / (NQ * QT)), (unsigned)a.n_heads, (unsigned)a.B);
    SFS_CUDA(launch_pdl(attention_kernel<DH, PAIR>, grid, dim3(kAttnThreads), smem, stream, p.tmQ, p.tmK, p.tmVt, a));
    return SFS_OK;
}

}  // namespace

int32_t attn_plan_create_split(AttnPlan *p, const void *q, int64_t ld_q, const void *k, int64_t ld_k, int32_t k_cols, int32_t k_col0,
                               const void *vt, int64_t ld_vt, void *out, int64_t ld_out, int32_t B, int32_t S, int32_t n_heads, int32_t head_dim)
{
    SFS_REQUIRE(head_dim == 64 || head_dim == 128, SFS_ERR_UNSUPPORTED, "attention: head_dim %d (64 or 128 supported)", head_dim);
    SFS_REQUIRE((S % 8) == 0, SFS_ERR_UNSUPPORTED, "attention: sequence length %d must be a multiple of 8", S);
    SFS_REQUIRE(aligned_to(out, 16) && (ld_out % 8) == 0, SFS_ERR_INVALID_ARG, "attention: output must be 16-byte aligned");
    memset(p, 0, sizeof(*p));
    const int d = n_heads * head_dim;
    int32_t rc = make_tmap_bf16(&p->tmQ, q, (uint64_t)B * S, (uint64_t)d, (uint64_t)ld_q, 128);
    if (rc != SFS_OK) return rc;
    rc = make_tmap_bf16(&p->tmK, k, (uint64_t)B * S, (uint64_t)k_cols, (uint64_t)ld_k, 128);
    if (rc != SFS_OK) return rc;
    rc = make_tmap_bf16(&p->tmVt, vt, (uint64_t)d, (uint64_t)B * S, (uint64_t)ld_vt, (uint32_t)head_dim);
    if (rc != SFS_OK) return rc;
    AttnArgs &a = p->args;
    a.B = B; a.S = S; a.n_heads = n_heads; a.d_model = d; a.kq = S; a.k_col0 = k_col0;
    a.scale_log2 = 1.4426950408889634f / sqrtf((float)head_dim);
    a.out = reinterpret_cast<__nv_bfloat16 *>(out); a.ld_out = ld_out;
    p->head_dim = head_dim;
    p->direct = {reinterpret_cast<const __nv_bfloat16 *>(q), reinterpret_cast<const __nv_bfloat16 *>(k) + k_col0, reinterpret_cast<const __nv_bfloat16 *>(vt), ld_q, ld_k, ld_vt};
    return SFS_OK;
}

int32_t attn_plan_create(AttnPlan *p, const void *qkv, int64_t ld_qkv, const void *vt, int64_t ld_vt,
                         void *out, int64_t ld_out, int32_t B, int32_t S, int32_t n_heads, int32_t head_dim)
{
    const int d = n_heads * head_dim;
    return attn_plan_create_split(p, qkv, ld_qkv, qkv, ld_qkv, 2 * d, d, vt, ld_vt, out, ld_out, B, S, n_heads, head_dim);
}

int32_t attn_launch(const AttnPlan &p, const int32_t *d_active, int32_t *err, cudaStream_t stream)
{
    return attn_launch_queries(p, 0, d_active, err, stream);
}

int32_t attn_launch_queries(const AttnPlan &p, int32_t kq, const int32_t *d_active, int32_t *err, cudaStream_t stream)
{
    const int rows = kq > 0 ? kq : p.args.kq, nkv = (p.args.S + KT - 1) / KT;
    if (attn_is_short(p, rows)) return attn_launch_short(p, rows, d_active, stream);
    const long long heads = (long long)p.args.n_heads * p.args.B, sms = gemm_num_sms();
    // waves of CTAs x (tile pairs of a CTA + 3, about what its set-up, first loads and final store cost).  32 heads, pair against
    // split in us: 512 tokens 13.9 / 9.8, 1000 23.2 / 27.4, 1536 57.8 / 50.9, 2048 74.6 / 83.2, 8 x 768 108.7 / 124.4.
    const long long pair = ((((rows + 2 * QT - 1) / (2 * QT)) * heads + sms - 1) / sms) * (nkv + 3);
    const long long split = ((((rows + QT - 1) / QT) * heads + sms - 1) / sms) * ((nkv + 1) / 2 + 3);
    const bool use_pair = pair <= split;
    if (p.head_dim == 128) return use_pair ? launch_dh<128, true>(p, kq, d_active, err, stream) : launch_dh<128, false>(p, kq, d_active, err, stream);
    return use_pair ? launch_dh<64, true>(p, kq, d_active, err, stream) : launch_dh<64, false>(p, kq, d_active, err, stream);
}

}  // namespace sfs
