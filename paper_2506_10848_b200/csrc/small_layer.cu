// A small model's layer behind its QKV projection in one launch: attention, output projection, residual add, RMSNorm, gate / up
// with SwiGLU, down projection, residual add, and the next layer's RMSNorm, QKV projection and rotary embedding.
//
// After the attention every token is on its own, so a cluster of eight CTAs takes 16 or 32 tokens through all of it.  The weights are
// divided over the cluster (an eighth of each projection's output columns) and requested before the dependent-launch wait, one
// bulk copy per row.  What the next product needs of a CTA's columns goes into its seven peers' shared memory in one bulk copy each,
// whose bytes complete a barrier there:
//   attention   a CTA takes (head, 16 rows) units, its eight warps divide the keys       -> bf16 [head][rows][64]
//   output      rows x d/8 columns, k divided over the warps, + residual                  -> sums of squares [CTA][rows]
//   norm        of the same columns                                                       -> bf16 [CTA][rows][d/8]
//   gate, up    rows x ff/8 features, both products of a feature in one thread             -> bf16 [CTA][rows][ff/8]
//   down        rows x d/8 columns, k divided again, + residual                           -> x, sums of squares [CTA][rows]
//   norm        of the same columns                                                       -> bf16 [CTA][rows][d/8]
//   q, k, v     rows x d/8 columns of each, weights where gate's and up's were; a thread has both halves of its rotary pairs
// Bound: the chain of these exchanges: at 64 tokens, d 256, d_ff 688, 10600 clocks from the wait to the end, of which attention 3400, the
// four messages 3400, products 3500; four launches took 12 us.  A 2-layer step 33.3 -> 26.6 us, one of 2 x 224 tokens 53.5 -> 38.9, and
// 36.9 with the next QKV projection in it.  Between SMs of a cluster 20 bytes a clock leave a CTA, whatever carries them: 2 KB to each of
// seven peers are there after 970 clocks by bulk copies, 1400 by remote stores and a cluster barrier (417 of them the empty barrier),
// 1650 through L2 and 1830 by remote loads.  So the sums of squares go ahead and the rows follow normalised, as 16 bits (fp32 rows and a
// norm in every CTA: 3600 clocks), and no copy carries what its receiver has.
#include "sfs_common.cuh"
#include "small_layer.cuh"
#include "small_mma.cuh"
#include <type_traits>

namespace sfs {
namespace {

using namespace small;

constexpr int CL = 8, kThreads = 256, kWarps = kThreads / 32;
constexpr int kMaxTiles = 256;                              // 8-feature tiles of a model at most
constexpr int kHeadLd = kHead + 8;                           // attention rows in shared memory: 16 bytes apart modulo 128 (ldmatrix is conflict-free)

// ---- shared memory (bytes from the start) for RT tiles of 16 rows.  Where the peers later put their features lie the output
// projection's weights and partial sums, where they put their rows ends the attention's scratch, and the down projection's partial
// sums overwrite rows that have been read: each is dead by then, because a peer sends only after it has received this CTA's
// previous message, which leaves after the last access.
struct Layout {
    int rows, ldk, ldf, ldh;                 // rows of a tile; strides in elements: d-wide and ff-wide weight rows, a CTA's features
    int x_block, h_block;                    // bytes of a CTA's message: normalised rows, features
    int gu, down, hid, wo, red_o, xs, part, attn, red_d, sums, total;
    __host__ __device__ Layout(int d, int ff, int RT)
    {
        const int nc = d / CL, red = kWarps * 16 * (nc + 8) * 4, scratch = kWarps * (int)kPartBytes, tiles = (ff / 8 + CL - 1) / CL;
        rows = 16 * RT;
        ldk = d + 8; ldf = ((ff + 15) & ~15) + 8; ldh = 8 * (tiles | 1);      // an odd number of 16-byte chunks: conflict-free
        x_block = rows * nc * 2; h_block = rows * ldh * 2;
        gu = 0;                              // (later: the next QKV projection's rows)
        down = gu + (2 * 8 * tiles > 3 * nc ? 2 * 8 * tiles : 3 * nc) * ldk * 2;
        hid = down + nc * ldf * 2;
        wo = hid; red_o = wo + nc * ldk * 2;
        const int xs_bytes = CL * x_block, attn_bytes = d / kHead * rows * kHeadLd * 2;
        int hid_bytes = CL * h_block;        // (later: two tables of partial sums)
        if (hid_bytes < 2 * red) hid_bytes = 2 * red;
        if (hid_bytes < nc * ldk * 2 + red) hid_bytes = nc * ldk * 2 + red;
        if (hid_bytes < nc * ldk * 2 + scratch - xs_bytes) hid_bytes = nc * ldk * 2 + scratch - xs_bytes;
        xs = hid + hid_bytes;
        part = xs + xs_bytes - scratch;
        attn = xs + xs_bytes;
        red_d = xs;
        total = attn + attn_bytes;
        if (total < red_d + red) total = red_d + red;
        sums = total; total += CL * rows * 4;
    }
};

__device__ __forceinline__ void load_row(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// This CTA's `bytes` at `at` into the same place of its peers (called by all threads; what the CTA has written there is visible to the copy)
__device__ __forceinline__ void send(uint32_t at, uint32_t bytes, uint32_t bar, int rank, int tid) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid < CL - 1) {
        const int p = (rank + 1 + tid) % CL;
        asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(tc::mapa(at, p)), "r"(at), "r"(bytes), "r"(tc::mapa(bar, p)) : "memory");
    }
}
// (the lanes together again: ldmatrix and mma.sync follow)
__device__ __forceinline__ void await(uint32_t bar, int32_t *err) { tc::mbar_await(bar, err); __syncwarp(); }

enum { BAR_WO = 0, BAR_GU = 1, BAR_WD = 2, BAR_ATTN = 3, BAR_SUMS = 4, BAR_X = 5, BAR_HID = 6, BAR_QKV = 7, BAR_SUMS2 = 8, BAR_X2 = 9, N_BARS = 10 };

// NN: 8-column tiles of the output and down projections' columns in a CTA (d / 64); RT: tiles of 16 rows
template <int NN, int RT>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(kThreads, 1)
small_layer_kernel(SmallLayerArgs g)
{
    // columns of this CTA, stride of partial sums, float4s of a row, model width, rows, warps that divide k
    constexpr int NC = 8 * NN, RLD = NC + 8, Q = NC / 4, D = NC * CL, ROWS = 16 * RT, KP = kWarps / RT;
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ __align__(8) unsigned long long s_bar[N_BARS];
    const Layout L(D, g.ff, RT);
    __nv_bfloat16 *sG = reinterpret_cast<__nv_bfloat16 *>(smem + L.gu), *sD = reinterpret_cast<__nv_bfloat16 *>(smem + L.down);
    __nv_bfloat16 *sO = reinterpret_cast<__nv_bfloat16 *>(smem + L.wo), *sAt = reinterpret_cast<__nv_bfloat16 *>(smem + L.attn);
    float *sP = reinterpret_cast<float *>(smem + L.part);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rank = blockIdx.x % CL, tile = blockIdx.x / CL;
    const int per_seq = (g.S + ROWS - 1) / ROWS, b = tile / per_seq, row0 = (tile - b * per_seq) * ROWS, rows = min(ROWS, g.S - row0);
    const int ff8 = g.ff / 8, t0 = rank * ff8 / CL, nt = (rank + 1) * ff8 / CL - t0, tiles = (ff8 + CL - 1) / CL;      // 8-feature tiles: this CTA's, at most
    const uint32_t bar = smem_u32(s_bar);
    // attention: unit u = (head, tile of 16 rows) is CTA u % CL's
    const int units = g.n_heads * RT, my_units = units > rank ? (units - rank + CL - 1) / CL : 0;
    constexpr uint32_t kUnitBytes = 16 * kHeadLd * 2;

    if (tid == 0) {
        for (int i = 0; i < N_BARS; ++i) tc::mbar_init(bar + 8 * i, 1);
        tc::mbar_init_fence();
        tc::mbar_expect_tx(bar + 8 * BAR_WO, NC * D * 2); tc::mbar_expect_tx(bar + 8 * BAR_GU, 2 * nt * 8 * D * 2); tc::mbar_expect_tx(bar + 8 * BAR_WD, NC * g.ff * 2);
        tc::mbar_expect_tx(bar + 8 * BAR_ATTN, (units - my_units) * kUnitBytes);
        tc::mbar_expect_tx(bar + 8 * BAR_SUMS, (CL - 1) * ROWS * 4);
        tc::mbar_expect_tx(bar + 8 * BAR_X, (CL - 1) * L.x_block); tc::mbar_expect_tx(bar + 8 * BAR_HID, (CL - 1) * L.h_block);
        tc::mbar_expect_tx(bar + 8 * BAR_QKV, 3 * NC * D * 2);
        tc::mbar_expect_tx(bar + 8 * BAR_SUMS2, (CL - 1) * ROWS * 4); tc::mbar_expect_tx(bar + 8 * BAR_X2, (CL - 1) * L.x_block);
    }
    __syncthreads();
    tc::cluster_arrive();                                   // this CTA runs: its shared memory may be written by its peers
    // ---- weights: constant, so before the wait (rows of this CTA's columns, in the order they are needed)
    for (int r = tid; r < 2 * NC + 2 * nt * 8; r += kThreads) {
        if (r < NC) load_row(smem_u32(sO + r * L.ldk), g.wo + (long long)(rank * NC + r) * D, D * 2, bar + 8 * BAR_WO);
        else if (r < NC + 2 * nt * 8) {
            const int q = r - NC, up = q >= nt * 8 ? 1 : 0, f = q - up * nt * 8;
            load_row(smem_u32(sG + (up * 8 * tiles + f) * L.ldk), (up ? g.w_up : g.w_gate) + (long long)(t0 * 8 + f) * D, D * 2, bar + 8 * BAR_GU);
        } else {
            const int q = r - NC - 2 * nt * 8;
            load_row(smem_u32(sD + q * L.ldf), g.w_down + (long long)(rank * NC + q) * g.ff, (uint32_t)g.ff * 2, bar + 8 * BAR_WD);
        }
    }
    // where the down projection finds a tile of features: CTA q's begin at tile q ff8 / CL
    __shared__ uint16_t s_tile[kMaxTiles + 1];              // in 16 bytes from the first message; beyond the last tile, the last one again
    for (int i = tid; i <= ff8; i += kThreads) {
        const int q = min(i, ff8 - 1);
        int c = q * CL / ff8;
        while (c + 1 < CL && q >= (c + 1) * ff8 / CL) ++c;
        while (c > 0 && q < c * ff8 / CL) --c;
        s_tile[i] = (uint16_t)((c * L.h_block >> 4) + q - c * ff8 / CL);
    }
    // the (row, four columns) of x this thread owns
    constexpr int OWN = (ROWS * Q + kThreads - 1) / kThreads;
    const long long tok0 = (long long)b * g.S + row0;
    int own_row[OWN], own_col[OWN];
    uint2 gain[OWN], next_gain[OWN];
    float4 angle[OWN][2];                                   // (cos, sin) of this thread's four rotary pairs, if it has any
    const bool next = g.w_q != nullptr;
    constexpr int HALF = NC / 2;                            // rotary pairs of a CTA in each of q and k: pairs rank HALF .. of the d / 2
    const int pair_head = rank * HALF / (kHead / 2), pair_j = rank * HALF % (kHead / 2);
#pragma unroll
    for (int i = 0; i < OWN; ++i) {
        const int e = tid + i * kThreads;
        own_row[i] = e < ROWS * Q ? e / Q : ROWS; own_col[i] = 4 * (e % Q);
        gain[i] = *reinterpret_cast<const uint2 *>(g.gain + rank * NC + own_col[i]);
        if (next) {
            next_gain[i] = *reinterpret_cast<const uint2 *>(g.next_gain + rank * NC + own_col[i]);
            if (own_row[i] < rows && own_col[i] < HALF)
#pragma unroll
                for (int h = 0; h < 2; ++h) angle[i][h] = *reinterpret_cast<const float4 *>(g.table + (long long)(row0 + own_row[i]) * (kHead / 2) + pair_j + own_col[i] + 2 * h);
        }
    }

    pdl_wait();
    const bool active = g.d_active == nullptr || *g.d_active != 0;
    float4 xr[OWN];
#pragma unroll
    for (int i = 0; i < OWN; ++i)
        xr[i] = own_row[i] < rows ? *reinterpret_cast<const float4 *>(g.x + (tok0 + own_row[i]) * D + rank * NC + own_col[i]) : make_float4(0.f, 0.f, 0.f, 0.f);
    // ---- attention (rows that do not exist are computed as copies of the last one, and never stored)
    for (int u = rank; u < units; u += CL) {
        const int head = u / RT, r0 = 16 * (u % RT);
        attn_part<kWarps>(g.qkv, g.S, g.S, g.scale_log2, head, b, row0 + r0, warp, lane, sP + warp * 16 * kPartLd, sP + kWarps * 16 * kPartLd + warp * 32);
        if (!active) break;                                 // (the flag's load beside the others)
        __syncthreads();
        __nv_bfloat16 *dst = sAt + (head * ROWS + r0) * kHeadLd;
        attn_merge<kWarps>(sP, sP + kWarps * 16 * kPartLd, min(kWarps, (g.S + 31) / 32), g.scale_log2, warp, lane,
                           [&](int r, int col, uint2 v) { *reinterpret_cast<uint2 *>(dst + r * kHeadLd + col) = v; });
        if (u == rank) tc::cluster_wait();                  // (the peers run)
        send(smem_u32(dst), kUnitBytes, bar + 8 * BAR_ATTN, rank, tid);
    }
    if (my_units == 0 || !active) tc::cluster_wait();
    if (!active) {
        // nothing left to decode: the copies requested above are awaited, nobody reads them
        for (int i = BAR_WO; i <= BAR_WD; ++i) await(bar + 8 * i, g.err);
        return;
    }
    await(bar + 8 * BAR_WO, g.err);
    await(bar + 8 * BAR_ATTN, g.err);

    const int rt = warp % RT, kp = warp / RT, ra = rt * 16 + (lane & 15), hi = lane >> 4;      // ldmatrix of A: row, second half of a k-step
    float *red = reinterpret_cast<float *>(smem + L.red_o);
    // rows x this CTA's columns: k-steps [kp, kp + 1) / KP of `halves` / 2, A's 16 bytes of (step, half, row) where a_at says.  A last step
    // without a second half is an MMA of half its depth: there are no features to multiply, and what lies there may be NaN
    auto project = [&](auto &&a_at, const __nv_bfloat16 *sb, int ldb, int halves) {
        float acc[NN][4] = {};
        const uint32_t b_addr = smem_u32(sb + ((lane >> 4) * 8 + (lane & 7)) * ldb + ((lane >> 3) & 1) * 8);
        const int steps = (halves + 1) / 2, odd = kp == KP - 1 ? halves & 1 : 0, s1 = (kp + 1) * steps / KP - odd;
        auto step = [&](int s, auto whole) {
            uint32_t a[4];
            ldmatrix4(a, a_at(s));
#pragma unroll
            for (int t = 0; t < NN; t += 2) {
                uint32_t w[4];
                ldmatrix4(w, b_addr + (uint32_t)(t * 8 * ldb * 2) + s * 32);
                if constexpr (decltype(whole)::value) { mma_16816(acc[t], a, w[0], w[1]); mma_16816(acc[t + 1], a, w[2], w[3]); }
                else { mma_1688(acc[t], a, w[0]); mma_1688(acc[t + 1], a, w[2]); }
            }
        };
#pragma unroll 4
        for (int s = kp * steps / KP; s < s1; ++s) step(s, std::true_type{});
        if (odd) step(s1, std::false_type{});
        float *p = red + (kp * ROWS + rt * 16 + (lane >> 2)) * RLD + 2 * (lane & 3);
#pragma unroll
        for (int t = 0; t < NN; ++t) {
            *reinterpret_cast<float2 *>(p + 8 * t) = make_float2(acc[t][0], acc[t][1]);
            *reinterpret_cast<float2 *>(p + 8 * RLD + 8 * t) = make_float2(acc[t][2], acc[t][3]);
        }
        __syncthreads();
    };
    auto owned_sum = [&](int i) {
        const float *p = red + own_row[i] * RLD + own_col[i];
        float4 s = *reinterpret_cast<const float4 *>(p);
#pragma unroll
        for (int q = 1; q < KP; ++q) {
            const float4 v = *reinterpret_cast<const float4 *>(p + q * ROWS * RLD);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        return s;
    };

    // ---- output projection and residual, the norm's sums
    const uint32_t at_base = smem_u32(sAt + ra * kHeadLd) + 16 * hi;
    project([&](int s) { return at_base + (uint32_t)((s >> 2) * ROWS * kHeadLd * 2) + (s & 3) * 32; }, sO, L.ldk, D / 8);
    float *sums = reinterpret_cast<float *>(smem + L.sums);
    constexpr int CPR = NC / 8;                             // chunks of a message row; rows that share 128 bytes take other chunks
    auto chunk_at = [&](int r, int c) { return r * NC * 2 + ((c ^ ((r / (8 / CPR)) & (CPR - 1))) << 4); };
    // xr's norm: the sums of squares ahead, then the normalised rows' message, its 16-byte chunks XOR-swizzled by row
    auto send_normalised = [&](const uint2 *gn, int bar_sums, int bar_x) {
#pragma unroll
        for (int i = 0; i < OWN; ++i) {
            if (own_row[i] >= ROWS) continue;               // (whole warps: Q divides 32, and ROWS * Q is a multiple of 32)
            float ss = xr[i].x * xr[i].x + xr[i].y * xr[i].y + xr[i].z * xr[i].z + xr[i].w * xr[i].w;
#pragma unroll
            for (int o = Q / 2; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            if (own_col[i] == 0) sums[rank * ROWS + own_row[i]] = ss;
        }
        send(smem_u32(sums + rank * ROWS), ROWS * 4, bar + 8 * bar_sums, rank, tid);
        await(bar + 8 * bar_sums, g.err);
        uint8_t *mine = smem + L.xs + rank * L.x_block;
#pragma unroll
        for (int i = 0; i < OWN; ++i) {
            if (own_row[i] >= ROWS) continue;
            float ss = 0.f;
#pragma unroll
            for (int q = 0; q < CL; ++q) ss += sums[q * ROWS + own_row[i]];
            const float inv = rsqrtf(ss / (float)D + g.eps);
            *reinterpret_cast<uint2 *>(mine + chunk_at(own_row[i], own_col[i] >> 3) + 2 * (own_col[i] & 4)) =
                make_uint2(pack2(xr[i].x * inv * bf16_bits_to_f32(gn[i].x & 0xFFFFu), xr[i].y * inv * bf16_bits_to_f32(gn[i].x >> 16)),
                           pack2(xr[i].z * inv * bf16_bits_to_f32(gn[i].y & 0xFFFFu), xr[i].w * inv * bf16_bits_to_f32(gn[i].y >> 16)));
        }
        send(smem_u32(mine), (uint32_t)L.x_block, bar + 8 * bar_x, rank, tid);
    };
#pragma unroll
    for (int i = 0; i < OWN; ++i) {
        if (own_row[i] >= ROWS) continue;
        const float4 s = owned_sum(i);
        if (g.inc_attn && own_row[i] < rows) *reinterpret_cast<float4 *>(g.inc_attn + (tok0 + own_row[i]) * D + rank * NC + own_col[i]) = s;
        xr[i].x += s.x; xr[i].y += s.y; xr[i].z += s.z; xr[i].w += s.w;
    }
    send_normalised(gain, BAR_SUMS, BAR_X);
    await(bar + 8 * BAR_GU, g.err);
    await(bar + 8 * BAR_X, g.err);
    pdl_trigger();                                          // (the next launch has its own weights to request)

    const uint32_t x_base = smem_u32(smem + L.xs);
    constexpr int SPB = NC / 16;                            // k-steps of a message
    // ---- gate and up: the warps take the 8-feature tiles in turn, two at a time
    __nv_bfloat16 *own_h = reinterpret_cast<__nv_bfloat16 *>(smem + L.hid + rank * L.h_block);
    {
        const uint32_t b_addr = smem_u32(sG + ((lane >> 4) * 8 * tiles + (lane & 7)) * L.ldk + ((lane >> 3) & 1) * 8);      // lanes 0-15: gate, 16-31: up
        auto features = [&](auto many, int tb) {
            constexpr int T = decltype(many)::value;
            float ag[T][RT][4] = {}, au[T][RT][4] = {};
#pragma unroll 4
            for (int s = 0; s < D / 16; ++s) {
                uint32_t a[RT][4], w[T][4];
#pragma unroll
                for (int r = 0; r < RT; ++r) ldmatrix4(a[r], x_base + (s / SPB) * L.x_block + chunk_at(r * 16 + (lane & 15), (s % SPB) * 2 + hi));
#pragma unroll
                for (int t = 0; t < T; ++t) ldmatrix4(w[t], b_addr + (uint32_t)((tb + kWarps * t) * 8 * L.ldk * 2) + s * 32);
#pragma unroll
                for (int t = 0; t < T; ++t)
#pragma unroll
                    for (int r = 0; r < RT; ++r) { mma_16816(ag[t][r], a[r], w[t][0], w[t][1]); mma_16816(au[t][r], a[r], w[t][2], w[t][3]); }
            }
#pragma unroll
            for (int t = 0; t < T; ++t)
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    __nv_bfloat16 *p = own_h + (r * 16 + (lane >> 2)) * L.ldh + (tb + kWarps * t) * 8 + 2 * (lane & 3);
                    const float *u = ag[t][r], *v = au[t][r];
                    *reinterpret_cast<uint32_t *>(p) = pack2(silu(u[0]) * v[0], silu(u[1]) * v[1]);
                    *reinterpret_cast<uint32_t *>(p + 8 * L.ldh) = pack2(silu(u[2]) * v[2], silu(u[3]) * v[3]);
                }
        };
        int tb = warp;
        for (; tb + kWarps < nt; tb += 2 * kWarps) features(std::integral_constant<int, 2>{}, tb);
        if (tb < nt) features(std::integral_constant<int, 1>{}, tb);
    }
    send(smem_u32(own_h), (uint32_t)L.h_block, bar + 8 * BAR_HID, rank, tid);
    if (next)                                               // (gate's and up's rows have been read)
        for (int r = tid; r < 3 * NC; r += kThreads) {
            const int map = r / NC, q = r - map * NC;       // q and k: first halves of the CTA's pairs, then second halves
            const int row = map == 2 ? rank * NC + q : pair_head * kHead + pair_j + (q < HALF ? q : q - HALF + kHead / 2);
            load_row(smem_u32(sG + r * L.ldk), (map == 0 ? g.w_q : (map == 1 ? g.w_k : g.w_v)) + (long long)row * D, D * 2, bar + 8 * BAR_QKV);
        }
    await(bar + 8 * BAR_WD, g.err);
    await(bar + 8 * BAR_HID, g.err);
    if (!next) tc::cluster_arrive_relaxed();                // all messages have been received here: their senders may leave

    // ---- down projection and residual
    red = reinterpret_cast<float *>(smem + L.red_d);
    const uint32_t h_base = smem_u32(smem + L.hid) + ra * L.ldh * 2;
    project([&](int s) { return h_base + 16u * s_tile[2 * s + hi]; }, sD, L.ldf, ff8);
#pragma unroll
    for (int i = 0; i < OWN; ++i) {
        if (own_row[i] >= ROWS) continue;
        const float4 s = owned_sum(i);
        xr[i].x += s.x; xr[i].y += s.y; xr[i].z += s.z; xr[i].w += s.w;
        if (own_row[i] >= rows) continue;
        const long long at = (tok0 + own_row[i]) * D + rank * NC + own_col[i];
        if (g.inc_mlp) *reinterpret_cast<float4 *>(g.inc_mlp + at) = s;
        *reinterpret_cast<float4 *>(g.x + at) = xr[i];
    }
    if (next) {
        // ---- the next layer's norm and QKV projection, one matrix after the other
        send_normalised(next_gain, BAR_SUMS2, BAR_X2);
        await(bar + 8 * BAR_QKV, g.err);
        await(bar + 8 * BAR_X2, g.err);
        tc::cluster_arrive_relaxed();                       // (as above)
        auto x_at = [&](int s) { return x_base + (uint32_t)((s / SPB) * L.x_block + chunk_at(ra, (s % SPB) * 2 + hi)); };
#pragma unroll 1
        for (int map = 0; map < 3; ++map) {
            red = reinterpret_cast<float *>(smem + L.hid + (map & 1) * (kWarps * 16 * RLD * 4));      // (the other one may still be read)
            project(x_at, sG + map * NC * L.ldk, L.ldk, D / 8);
#pragma unroll
            for (int i = 0; i < OWN; ++i) {
                if (own_row[i] >= rows) continue;
                const long long tok = tok0 + own_row[i];
                const float4 lo = owned_sum(i);
                if (map == 2) {
                    const long long ld = (long long)g.B * g.S;
                    __nv_bfloat16 *dst = g.vt_out + (rank * NC + own_col[i]) * ld + tok;       // values go out transposed
                    dst[0] = __float2bfloat16_rn(lo.x); dst[ld] = __float2bfloat16_rn(lo.y);
                    dst[2 * ld] = __float2bfloat16_rn(lo.z); dst[3 * ld] = __float2bfloat16_rn(lo.w);
                } else if (own_col[i] < HALF) {
                    own_col[i] += HALF;
                    const float4 up = owned_sum(i);
                    own_col[i] -= HALF;
                    // the projection's result is rounded to bf16 and so is the rotated one, as when the two are kernels of their own
                    const float a0 = round_bf16(lo.x), a1 = round_bf16(lo.y), a2 = round_bf16(lo.z), a3 = round_bf16(lo.w);
                    const float b0 = round_bf16(up.x), b1 = round_bf16(up.y), b2 = round_bf16(up.z), b3 = round_bf16(up.w);
                    const float4 c = angle[i][0], e = angle[i][1];
                    const uint2 first = make_uint2(pack2(a0 * c.x - b0 * c.y, a1 * c.z - b1 * c.w), pack2(a2 * e.x - b2 * e.y, a3 * e.z - b3 * e.w));
                    const uint2 second = make_uint2(pack2(b0 * c.x + a0 * c.y, b1 * c.z + a1 * c.w), pack2(b2 * e.x + a2 * e.y, b3 * e.z + a3 * e.w));
                    const int col = pair_head * kHead + pair_j + own_col[i];
                    __nv_bfloat16 *dst = g.qk_out + tok * (2 * D) + map * D + col;
                    *reinterpret_cast<uint2 *>(dst) = first; *reinterpret_cast<uint2 *>(dst + kHead / 2) = second;
                    if (map == 1 && g.k_dst) {
                        dst = g.k_dst + tok * D + col;
                        *reinterpret_cast<uint2 *>(dst) = first; *reinterpret_cast<uint2 *>(dst + kHead / 2) = second;
                    }
                }
            }
        }
    }
    tc::cluster_wait();
}

constexpr int kSharedMost = 226 * 1024;                      // a CTA's most, minus the static arrays

template <int NN, int RT>
cudaError_t configure()
{
    static bool configured[kMaxDevices] = {};
    bool &done = configured[current_device_slot()];
    if (done) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(small_layer_kernel<NN, RT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSharedMost);
    done = e == cudaSuccess;
    return e;
}
template <int NN, int RT>
int32_t launch(const SmallLayerArgs &g, cudaStream_t s)
{
    SFS_CUDA((configure<NN, RT>()));
    SFS_CUDA(launch_pdl(small_layer_kernel<NN, RT>, dim3((unsigned)(CL * g.B * ((g.S + 16 * RT - 1) / (16 * RT)))), dim3(kThreads), (size_t)Layout(g.d, g.ff, RT).total, s, g));
    return SFS_OK;
}

// Clusters the device runs at once (one CTA per SM: registers): as many as it has groups of eight SMs, 0 if it does not say
int resident_clusters()
{
    static int known[kMaxDevices] = {};
    int &n = known[current_device_slot()];
    if (n > 0) return n;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CL); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = kSharedMost;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int c = 0;
    if (configure<4, 2>() != cudaSuccess || cudaOccupancyMaxActiveClusters(&c, small_layer_kernel<4, 2>, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
    return n = c;
}

int tiles(int B, int S, int RT) { return B * ((S + 16 * RT - 1) / (16 * RT)); }
// Tiles of 16 rows while their clusters are resident at once (a message is half as long, a product half as many MMAs), else of 32 (whose
// products divide k over four warps instead of eight: a sequence's last bits are not those it has in a smaller batch)
int row_tiles(int B, int S) { return tiles(B, S, 1) <= resident_clusters() ? 1 : 2; }

}  // namespace

// Widths whose weights and rows fit a cluster's shared memory, and one wave of clusters: the second costs as much as the separate kernels
// save.  A step of two layers, us, those kernels / this one: d 256, d_ff 688: 8 tokens 30.8 / 24.6, 64 34.8 / 26.6, 192 41.0 / 30.8, 256 43.0 / 32.8,
// 2 x 224 (14 clusters) 53.5 / 36.9, 512 (16 clusters, two waves) 59.4 / 57.4, 16 x 32 54.1 / 52.6; d_ff 256: 64 32.8 / 24.6, 512 49.2 / 49.3;
// d 128, d_ff 352: 64 30.8 / 22.6, 448 40.7 / 28.7, 512 43.0 / 45.1; d_ff 1024: 64 32.8 / 26.0, 512 51.2 / 55.3.
bool small_layer_fits(int d_model, int d_ff, int n_heads, int head_dim, int B, int S)
{
    if (!(d_model == 128 || d_model == 256) || n_heads * head_dim != d_model || head_dim != kHead || d_ff / 8 > kMaxTiles || (long long)B * S > 1 << 16) return false;
    const int RT = row_tiles(B, S);
    return Layout(d_model, d_ff, RT).total <= kSharedMost && tiles(B, S, RT) <= resident_clusters();
}

int32_t launch_small_layer(const SmallLayerArgs &g, cudaStream_t s)
{
    if (row_tiles(g.B, g.S) == 1) return g.d == 128 ? launch<2, 1>(g, s) : launch<4, 1>(g, s);
    return g.d == 128 ? launch<2, 2>(g, s) : launch<4, 2>(g, s);
}

}  // namespace sfs
