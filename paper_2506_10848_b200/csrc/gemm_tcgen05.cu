// Dense projections of the mask predictor (QKV / O / gate-up / down / LM head): C = A * B^T with bf16
// operands and fp32 accumulation in tensor memory.
//
// A pair of CTAs (a cluster of two, on the two SMs of a TPC) computes a (MB x 256) x BN output tile with
// tcgen05.mma.cta_group::2: each CTA stages its own 128 rows of every 256-row block of A and its own half of
// the BN weight rows, so a weight tile enters the pair once and the bytes an SM pulls through its L2 port per
// FLOP drop (the operand stream from L2, not the tensor core, bounds these shapes).  The pair walks a static
// list of tiles (persistent kernel).  In each CTA warp 0 streams 128-byte-swizzled operand tiles into a ring of
// shared-memory stages with TMA (completion is counted on the leader CTA's barrier), the leader's warp 1 issues
// the MMAs and releases stages in both CTAs with a multicast tcgen05.commit, and warps 2-9 read the accumulator
// back with tcgen05.ld and run the fused epilogue (scale / fp32 residual add / SwiGLU / transposed V store).
// When two accumulators fit tensor memory the epilogue of a tile overlaps the next tile's main loop.  The row
// count may live on the device, so the LM head can follow the shrinking set of masked rows without a host
// round trip.
#include "sfs_common.cuh"
#include "tc05.cuh"
#include "gemm.cuh"

namespace sfs {

// ---- host: tensor maps -------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

int32_t make_tmap_bf16(CUtensorMap *out, const void *base, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_rows)
{
    EncodeTiledFn enc = get_encode();
    SFS_REQUIRE(enc != nullptr, SFS_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    SFS_REQUIRE(aligned_to(base, 16) && (ld % 8) == 0 && rows >= 1 && cols >= 1 && box_rows >= 1 && box_rows <= 256,
                SFS_ERR_INVALID_ARG, "tensor map: base must be 16-byte aligned, ld a multiple of 8 (ld=%llu rows=%llu cols=%llu)",
                (unsigned long long)ld, (unsigned long long)rows, (unsigned long long)cols);
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {ld * 2};
    cuuint32_t box[2] = {64, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    SFS_REQUIRE(r == CUDA_SUCCESS, SFS_ERR_CUDA, "cuTensorMapEncodeTiled failed with %d", (int)r);
    return SFS_OK;
}

// A weight matrix for projections whose epilogue rotates pairs (j, j + half) of every head: the box's rows are, head by head, 16 rows of
// the first half and the same 16 of the second, so that 32 consecutive accumulator columns hold 16 whole pairs.  Dimensions: k, row of a
// half, half, head.  For a plain matrix half = 16.
static int32_t make_tmap_pairs(CUtensorMap *out, const void *base, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t half, uint32_t box_heads)
{
    EncodeTiledFn enc = get_encode();
    SFS_REQUIRE(enc != nullptr, SFS_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    SFS_REQUIRE(aligned_to(base, 16) && (ld % 8) == 0 && (rows % (2 * half)) == 0 && box_heads >= 1 && 32 * box_heads <= 256, SFS_ERR_INVALID_ARG, "tensor map of rotary pairs");
    cuuint64_t dims[4] = {cols, half, 2, rows / (2 * half)};
    cuuint64_t strides[3] = {ld * 2, (cuuint64_t)half * ld * 2, (cuuint64_t)2 * half * ld * 2};
    cuuint32_t box[4] = {64, 16, 2, box_heads};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    SFS_REQUIRE(r == CUDA_SUCCESS, SFS_ERR_CUDA, "cuTensorMapEncodeTiled failed with %d", (int)r);
    return SFS_OK;
}

namespace {

constexpr int BM = 128, BK = 64;         // rows per CTA of one 256-row MMA block; K elements per stage
constexpr int kEpiWarps = 8;
constexpr int kGemmThreads = 64 + 32 * kEpiWarps;
constexpr int A_BYTES = BM * BK * 2;
constexpr int FM = 64;                   // few-row tiles: rows per CTA of the pair's 128-row MMA
constexpr int kMaxStages = 12;
constexpr int kSmemBudget = 227 * 1024 - 64;      // the opt-in maximum minus the kernel's static shared memory
// barriers: full[kMaxStages], empty[kMaxStages], acc_full[2], acc_empty[2]; then the TMEM base slot
constexpr int kBarBytes = (2 * kMaxStages + 4) * 8 + 16;
constexpr int kTmemCols = 512;
constexpr int kEpiStageBytes = kEpiWarps * 32 * 128;   // one 32-row x 128-byte output unit per epilogue warp

// x * sigmoid(x) with the special-function unit's exponential and reciprocal (a few ulp: the result is rounded to bf16)
__device__ __forceinline__ float silu_f(float x) { return __fdividef(x, 1.0f + __expf(-x)); }

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&h);
}

// which output columns / weight rows a tile covers
struct TileCoord {
    int split;       // which range of k-blocks (split-K), 0 when K is not split
    int m0;          // first output row of the pair's tile
    int map_idx;     // which B matrix (concatenated outputs), 0 for SwiGLU
    int n_local;     // first row of that B matrix (SwiGLU: first gate row = first up row)
    int ncol0;       // first output column
    int ncols;       // valid output columns of the tile (<= BN, SwiGLU: <= BN/2)
    int j0;          // rotated tiles: the first of the 16 pairs the tile takes of each head (n_local: its first head), else -1
};

// (ROPE: the kernels of projections that rotate.  Asked of the arguments, the question and its divisions cost the other projections 0.2 us each: a
// layer of 10 heads of 64 at 8 rows, with a rotary kernel 36.4 us, without the question 35.7)
template <bool ROPE>
__device__ __forceinline__ TileCoord tile_coord(const GemmArgs &g, int tile, int m_groups)
{
    TileCoord t;
    // row groups fastest: pairs that share a weight tile run together (divisions only where there is something to divide)
    const int rest = m_groups == 1 ? tile : tile / m_groups;
    t.m0 = (tile - rest * m_groups) * g.tile_rows;
    const int n_tile = g.splits == 1 ? rest : rest / g.splits;
    t.split = rest - n_tile * g.splits;
    t.j0 = -1;
    if (ROPE) {
        // queries and keys: tiles of 16 pairs of tile_cols / 32 heads, the groups of a head's pairs fastest; then the values, plain
        if (n_tile < 2 * g.rope_tiles) {
            t.map_idx = n_tile >= g.rope_tiles ? 1 : 0;
            const int local = n_tile - t.map_idx * g.rope_tiles, hg = local / g.rope_groups;
            t.j0 = 16 * (local - hg * g.rope_groups);
            t.n_local = hg * (g.tile_cols / 32); t.ncol0 = t.map_idx * g.n_per_map; t.ncols = g.tile_cols;
        } else {
            t.map_idx = 2; t.n_local = (n_tile - 2 * g.rope_tiles) * g.tile_cols;
            t.ncol0 = 2 * g.n_per_map + t.n_local; t.ncols = min(g.tile_cols, g.n_per_map - t.n_local);
        }
    } else if (g.mode == GEMM_SWIGLU) {
        t.map_idx = 0; t.n_local = n_tile * g.tile_cols; t.ncol0 = t.n_local; t.ncols = min(g.tile_cols, g.N - t.ncol0);
    } else {
        t.map_idx = (n_tile >= g.tiles_per_map ? 1 : 0) + (n_tile >= 2 * g.tiles_per_map ? 1 : 0);      // at most three matrices
        t.n_local = (n_tile - t.map_idx * g.tiles_per_map) * g.tile_cols;
        t.ncol0 = t.map_idx * g.n_per_map + t.n_local;
        t.ncols = min(g.tile_cols, g.n_per_map - t.n_local);
    }
    return t;
}

// A k-block of a CTA's weight rows.  Projections that rotate: coordinates (k, row within a half, 0, head), plain rows as heads of 32.
template <bool ROPE>
__device__ __forceinline__ void load_weights(uint32_t dst, const CUtensorMap *map, int k, int row, int j0, uint32_t bar)
{
    if (ROPE) tc::tma_load_4d_2cta_elect(dst, map, k, j0, 0, row, bar);
    else tc::tma_load_2d_2cta_elect(dst, map, k, row, bar);
}
// its first row (ROPE: head) for CTA `rank` of the pair, whose share is `half` rows
template <bool ROPE>
__device__ __forceinline__ int weight_row0(const TileCoord &t, int rank, int half, bool shared_rows)
{
    if (ROPE) return (t.j0 >= 0 ? t.n_local : t.n_local / 32) + rank * (half / 32);
    return shared_rows ? t.n_local : t.n_local + rank * half;
}

// k-blocks of the pair's first tile whose weights are requested before the dependent-launch wait
__device__ __forceinline__ int early_weights(const GemmArgs &g, int pair, int stages)
{
    const int num_kb = (g.K + BK - 1) / BK;
    if (g.splits == 1) return min(stages, num_kb);
    const int kb0 = tile_coord<false>(g, pair, (g.M + g.tile_rows - 1) / g.tile_rows).split * g.kb_per_split;
    return min(stages, min(num_kb, kb0 + g.kb_per_split) - kb0);
}

// ---- epilogue --------------------------------------------------------------------------------------------
// tcgen05.ld hands every lane one accumulator ROW, so storing from those registers makes each store instruction
// touch 32 different lines.  Instead a warp parks a 32-row x 128-byte unit of output in shared memory (16-byte
// chunks XOR-swizzled by row, so both directions are conflict-free) and writes it out as 4 rows x 128 contiguous
// bytes per instruction.  A unit is 32 fp32 or 64 bf16 output columns.
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void red_add_v4_f32(float *p, uint4 v) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};"
                 ::"l"(p), "f"(__uint_as_float(v.x)), "f"(__uint_as_float(v.y)), "f"(__uint_as_float(v.z)), "f"(__uint_as_float(v.w)) : "memory");
}
// lane = row: park 4 consecutive 16-byte chunks (chunk0 .. chunk0+3) of this lane's row
__device__ __forceinline__ void park16(uint32_t stage, int lane, int chunk0, const uint32_t *w) {
#pragma unroll
    for (int c = 0; c < 4; ++c)
        st_shared_v4(stage + lane * 128 + (((chunk0 + c) ^ (lane & 7)) << 4), w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
}

// Writes the parked unit out.  Row r of the unit is output row grow0 + r; its 128 bytes start at output column col0.
// ELEM = bytes per output element (2 or 4); columns at or beyond `lim` and rows at or beyond M are skipped.
// Every output element belongs to exactly one tile, so the residual add (one vector red per chunk) is deterministic.
template <int ELEM, bool RESIDUAL>
__device__ __forceinline__ void flush_unit(const GemmArgs &g, long long slab, uint32_t stage, int lane, int grow0, int M, int col0, int lim)
{
    constexpr int PER = 16 / ELEM;                       // elements per 16-byte chunk
    const int c = lane & 7, col = col0 + c * PER;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = 4 * i + (lane >> 3), grow = grow0 + r;
        if (grow >= M || col >= lim) continue;
        const uint4 v = ld_shared_v4(stage + r * 128 + ((c ^ (r & 7)) << 4));
        uint8_t *dst = reinterpret_cast<uint8_t *>(g.C) + (slab + (long long)grow * g.ldc + col) * ELEM;
        if (col + PER <= lim) {
            if (RESIDUAL) red_add_v4_f32(reinterpret_cast<float *>(dst), v);
            else *reinterpret_cast<uint4 *>(dst) = v;
        } else {                                         // ragged last chunk of the matrix: element by element
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
            for (int e = 0; e < PER && col + e < lim; ++e) {
                if (RESIDUAL) atomicAdd(reinterpret_cast<float *>(dst) + e, __uint_as_float(w[e]));
                else if (ELEM == 4) reinterpret_cast<uint32_t *>(dst)[e] = w[e];
                else reinterpret_cast<uint16_t *>(dst)[e] = (uint16_t)(w[e >> 1] >> ((e & 1) * 16));
            }
        }
    }
}

// Where one warp's share of a tile's accumulators lies: `blocks` blocks of `seg` output columns each (the pair kernel: 256-row
// blocks under one another; the few-row kernel: N-blocks beside one another).
struct EpiShare {
    uint32_t tmem, tmem_block;   // tensor-memory address of block 0 (with the warp's lane quarter), columns between blocks
    uint32_t up;                 // SwiGLU: columns from a gate accumulator to its up accumulator
    int row0, row_block;         // output row of lane 0 in block 0, rows between blocks
    int col0, col_block;         // output column of the first accumulator column in block 0, columns between blocks
    int blocks, seg;             // number of blocks (1 or 2), accumulator columns of each that may be valid
    int col_end;                 // columns at or beyond this belong to another tile or matrix
    int rec, rec_block;          // fused row statistics: record of block 0, records between blocks
    int head0, j0;               // rotated tiles: head of the first 32 accumulator columns, first of the 16 pairs
    __device__ __forceinline__ int lim(int b) const { return min(col_end, col0 + b * col_block + seg); }
};

// V columns of the QKV projection go out transposed: the 32 lanes hold 32 consecutive tokens of a feature (LISTED: of the row list's)
template <bool LISTED>
__device__ __forceinline__ void epilogue_values(const GemmArgs &g, const EpiShare &e, int par, int lane, int M)
{
    const int upb = (e.seg + 31) / 32;
    const int n_pieces = (e.blocks * upb - par + 1) / 2;
    auto piece_col = [&](int pc, int *b) { const int u = par + 2 * pc; *b = u >= upb ? 1 : 0; return 32 * (u - *b * upb); };
    uint32_t v[32];
    int b0;
    if (n_pieces > 0) { const int c = piece_col(0, &b0); tc::tmem_ld32(e.tmem + (uint32_t)b0 * e.tmem_block + (uint32_t)c, v); }
    for (int pc = 0; pc < n_pieces; ++pc) {
        int b;
        const int c = piece_col(pc, &b);
        uint16_t h[32];
        tc::tmem_ld_wait32(v);
#pragma unroll
        for (int j = 0; j < 32; ++j) { __nv_bfloat16 r = __float2bfloat16_rn(__uint_as_float(v[j]) * g.scale); h[j] = *reinterpret_cast<uint16_t *>(&r); }
        if (pc + 1 < n_pieces) { int bn2; const int c2 = piece_col(pc + 1, &bn2); tc::tmem_ld32(e.tmem + (uint32_t)bn2 * e.tmem_block + (uint32_t)c2, v); }
        const int grow = e.row0 + b * e.row_block + lane, col0 = e.col0 + b * e.col_block + c;
        if (grow < M) {
            uint16_t *dst = reinterpret_cast<uint16_t *>(g.vt) + (long long)(col0 - g.vt_col0) * g.ldvt + (LISTED && g.rope.rows ? g.rope.rows[grow] : grow);
            const int nv = e.lim(b) - col0;                            // valid features of this piece
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (j < nv) dst[(long long)j * g.ldvt] = h[j];
        }
    }
}

// The parked unit of a rotated tile: 16-byte chunks 4 p .. 4 p + 3 are pairs j0 .. j0 + 15 of head `head` + p, first halves then second
// halves; `heads` of them are this share's.  `tok`: this lane's row's token (a row of the list: keys go to their token's row).
__device__ __forceinline__ void flush_pairs(const GemmArgs &g, uint32_t stage, int lane, int grow0, int M, int ncol0, int head, int heads, int j0, int tok)
{
    const int c = lane & 7, dh = g.rope.head_dim, h = head + (c >> 2), col = h * dh + ((c >> 1) & 1) * (dh / 2) + j0 + 8 * (c & 1);
    const bool key = ncol0 != 0 && g.rope.k_dst != nullptr;
    __nv_bfloat16 *base = key ? g.rope.k_dst : reinterpret_cast<__nv_bfloat16 *>(g.C) + ncol0;
    const long long ld = key ? g.n_per_map : g.ldc;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = 4 * i + (lane >> 3), grow = grow0 + r, t = __shfl_sync(0xffffffffu, tok, r);
        if (grow >= M || (c >> 2) >= heads || col >= g.n_per_map) continue;
        *reinterpret_cast<uint4 *>(base + (long long)(key ? t : grow) * ld + col) = ld_shared_v4(stage + r * 128 + ((c ^ (r & 7)) << 4));
    }
}

// A rotated tile: of every 32 accumulator columns (a head's), j and 16 + j are a pair.  The projection is rounded to bf16 and so is
// its rotation, as two kernels would.  A function of its own: beside the other epilogues its angles spilled (664 bytes), and the
// epilogue of 512 x 192 took 32 us instead of 11.
__device__ __forceinline__ void epilogue_pairs(const GemmArgs &g, const EpiShare &e, uint32_t stage, int par, int lane, int M)
{
    const int upb = (e.seg + 63) / 64;                       // units of 64 columns per block: those of all blocks, numbered on, alternate between the parities
    for (int b = 0; b < e.blocks; ++b) {
        int u = (par + b * upb) & 1;
        if (u >= upb) continue;
        // every row's 128 bytes of the table by eight lanes, through the stage; they serve every head of the tile
        const int grow = e.row0 + b * e.row_block + lane;
        const int tok = grow < M ? (g.rope.rows ? g.rope.rows[grow] : grow) : 0, pos = tok % g.rope.S;
        float2 cs[16];
        {
            uint4 v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                v[i] = reinterpret_cast<const uint4 *>(g.rope.table + (long long)__shfl_sync(0xffffffffu, pos, 4 * i + (lane >> 3)) * (g.rope.head_dim / 2) + e.j0)[lane & 7];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int r = 4 * i + (lane >> 3);
                st_shared_v4(stage + r * 128 + (((lane & 7) ^ (r & 7)) << 4), v[i].x, v[i].y, v[i].z, v[i].w);
            }
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint4 w = ld_shared_v4(stage + lane * 128 + ((j ^ (lane & 7)) << 4));
                cs[2 * j] = make_float2(__uint_as_float(w.x), __uint_as_float(w.y)); cs[2 * j + 1] = make_float2(__uint_as_float(w.z), __uint_as_float(w.w));
            }
            __syncwarp();
        }
        const uint32_t t0 = e.tmem + (uint32_t)b * e.tmem_block;
        uint32_t x[32];
        tc::tmem_ld32(t0 + 64u * u, x);
        for (; u < upb; u += 2) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {                    // two heads to a parked unit
                uint32_t o[16];
                tc::tmem_ld_wait32(x);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t p = pack_bf16(__uint_as_float(x[2 * j]), __uint_as_float(x[2 * j + 1])), q = pack_bf16(__uint_as_float(x[16 + 2 * j]), __uint_as_float(x[17 + 2 * j]));
                    const float p0 = __uint_as_float(p << 16), p1 = __uint_as_float(p & 0xFFFF0000u), q0 = __uint_as_float(q << 16), q1 = __uint_as_float(q & 0xFFFF0000u);
                    const float2 a = cs[2 * j], c = cs[2 * j + 1];
                    o[j] = pack_bf16(p0 * a.x - q0 * a.y, p1 * c.x - q1 * c.y);
                    o[8 + j] = pack_bf16(q0 * a.x + p0 * a.y, q1 * c.x + p1 * c.y);
                }
                if (h == 0) tc::tmem_ld32(t0 + 64u * u + 32u, x);
                else if (u + 2 < upb) tc::tmem_ld32(t0 + 64u * (u + 2), x);
                park16(stage, lane, 4 * h, o);
            }
            __syncwarp();
            flush_pairs(g, stage, lane, e.row0 + b * e.row_block, M, e.col0, e.head0 + 2 * u, e.seg / 32 - 2 * u, e.j0, tok);
            __syncwarp();
        }
    }
}

// One warp's share of a tile's epilogue: 32 rows of every block, the 64-column (fp32: 32-column) units of parity `par`.
// A unit may reach past the block's valid columns: those accumulator columns exist (inside the 256-column buffer) and
// are never stored.  The tensor-memory loads of the next piece are issued as soon as the current piece has been
// converted, so their latency hides behind the parking and the stores of the current one.
template <bool STATS>
__device__ __forceinline__ void epilogue_tile(const GemmArgs &g, const EpiShare &e, int split, uint32_t stage, int par, int lane, int M)
{
    if (g.mode == GEMM_SWIGLU || (g.mode == GEMM_STORE && !g.out_f32 && !(g.vt != nullptr && e.col0 >= g.vt_col0))) {
        // ---- bf16 output (plain or SwiGLU): units of 64 output columns, handled as two pieces of 32
        const bool swiglu = (g.mode == GEMM_SWIGLU);
        // the units of all blocks, numbered block by block, alternate between the two warps of a lane quarter
        const int upb = (e.seg + 63) / 64;                                // units per block
        const int n_pieces = 2 * ((e.blocks * upb - par + 1) / 2);
        auto piece_addr = [&](int pc) {                                   // tensor-memory column of piece pc
            const int u = par + 2 * (pc >> 1), b = u >= upb ? 1 : 0, c = 64 * (u - b * upb);
            return e.tmem + (uint32_t)b * e.tmem_block + (uint32_t)(c + 32 * (pc & 1));
        };
        uint32_t x0[32], x1[32];
        if (n_pieces > 0) {
            tc::tmem_ld32(piece_addr(0), x0);
            if (swiglu) tc::tmem_ld32(piece_addr(0) + e.up, x1);
        }
        // fused row statistics (LM head): this lane's row of the current block
        const bool stats_on = STATS && (g.stats != nullptr) && !swiglu;
        float st_mx = -INFINITY, st_ref = 0.f, st_nref = 0.f, st_sum = 0.f;
        int st_arg = 0x7FFFFFFF, st_b = -1;
        auto stats_flush = [&]() {
            if (st_b < 0) return;
            const int grow = e.row0 + st_b * e.row_block + lane;
            if (grow < M) g.stats[(long long)grow * g.stats_ld + e.rec + st_b * e.rec_block + par] = make_float4(st_mx, st_ref, st_sum, __int_as_float(st_arg));
        };
        for (int pc = 0; pc < n_pieces; ++pc) {
            const int u = par + 2 * (pc >> 1), b = u >= upb ? 1 : 0, col0 = e.col0 + b * e.col_block + 64 * (u - b * upb);
            uint32_t o[16];
            tc::tmem_ld_wait32(x0);
            if (swiglu) tc::tmem_ld_wait32(x1);
            if (swiglu) {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    o[j] = pack_bf16(silu_f(__uint_as_float(x0[2 * j])) * __uint_as_float(x1[2 * j]),
                                     silu_f(__uint_as_float(x0[2 * j + 1])) * __uint_as_float(x1[2 * j + 1]));
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) o[j] = pack_bf16(__uint_as_float(x0[2 * j]) * g.scale, __uint_as_float(x0[2 * j + 1]) * g.scale);
            }
            if (pc + 1 < n_pieces) {
                tc::tmem_ld32(piece_addr(pc + 1), x0);
                if (swiglu) tc::tmem_ld32(piece_addr(pc + 1) + e.up, x1);
            }
            if (stats_on) {
                // statistics of the ROUNDED values, as a reader of the stored logits would see them
                const int c0 = col0 + 32 * (pc & 1);
                if (b != st_b) { stats_flush(); st_b = b; st_mx = -INFINITY; st_sum = 0.f; st_arg = 0x7FFFFFFF; st_ref = 0.f; st_nref = 0.f; }
                const int nvalid = min(32, e.lim(b) - c0);               // columns of this piece inside the matrix (warp-uniform)
                float pm = -INFINITY;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float lo = __uint_as_float(o[j] << 16), hi = __uint_as_float(o[j] & 0xFFFF0000u);
                    if (2 * j < nvalid) pm = fmaxf(pm, lo);
                    if (2 * j + 1 < nvalid) pm = fmaxf(pm, hi);
                }
                if (st_mx == -INFINITY && st_sum == 0.f) {               // first piece of this row: it gives the reference
                    st_ref = (fabsf(pm) <= 3.0e38f) ? pm : 0.f;
                    st_nref = -st_ref * 1.4426950408889634f;
                }
                if (pm > st_mx) {                                        // strict: the first position of the maximum
                    st_mx = pm;
#pragma unroll
                    for (int j = 15; j >= 0; --j) {
                        const float lo = __uint_as_float(o[j] << 16), hi = __uint_as_float(o[j] & 0xFFFF0000u);
                        if (2 * j + 1 < nvalid && hi == pm) st_arg = c0 + 2 * j + 1;
                        if (2 * j < nvalid && lo == pm) st_arg = c0 + 2 * j;
                    }
                }
                float s0 = 0.f, s1 = 0.f;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float lo = __uint_as_float(o[j] << 16), hi = __uint_as_float(o[j] & 0xFFFF0000u);
                    const float e0 = tc::ex2_approx(__fmaf_rn(lo, 1.4426950408889634f, st_nref));
                    const float e1 = tc::ex2_approx(__fmaf_rn(hi, 1.4426950408889634f, st_nref));
                    s0 += (2 * j < nvalid) ? e0 : 0.f;
                    s1 += (2 * j + 1 < nvalid) ? e1 : 0.f;
                }
                st_sum += s0 + s1;
            }
            park16(stage, lane, 4 * (pc & 1), o);
            if (pc & 1) {
                __syncwarp();
                flush_unit<2, false>(g, 0, stage, lane, e.row0 + b * e.row_block, M, col0, e.lim(b));
                __syncwarp();
            }
        }
        if (stats_on) stats_flush();
    } else if (g.vt != nullptr && e.col0 >= g.vt_col0) {
        epilogue_values<false>(g, e, par, lane, M);
    } else {
        // ---- fp32 output (residual add, split-K slab, or fp32 logits): units of 32 columns
        const int upb = (e.seg + 31) / 32;
        const int n_pieces = (e.blocks * upb - par + 1) / 2;
        auto piece_col = [&](int pc, int *b) { const int u = par + 2 * pc; *b = u >= upb ? 1 : 0; return 32 * (u - *b * upb); };
        const bool scale = (g.mode != GEMM_RESIDUAL_F32 && g.scale != 1.0f);
        uint32_t v[32];
        int b0;
        if (n_pieces > 0) { const int c = piece_col(0, &b0); tc::tmem_ld32(e.tmem + (uint32_t)b0 * e.tmem_block + (uint32_t)c, v); }
        for (int pc = 0; pc < n_pieces; ++pc) {
            int b;
            const int c = piece_col(pc, &b);
            uint32_t o[32];
            tc::tmem_ld_wait32(v);
#pragma unroll
            for (int j = 0; j < 32; ++j) o[j] = scale ? __float_as_uint(__uint_as_float(v[j]) * g.scale) : v[j];
            if (pc + 1 < n_pieces) { int bn2; const int c2 = piece_col(pc + 1, &bn2); tc::tmem_ld32(e.tmem + (uint32_t)bn2 * e.tmem_block + (uint32_t)c2, v); }
            park16(stage, lane, 0, o);
            park16(stage, lane, 4, o + 16);
            __syncwarp();
            const int row = e.row0 + b * e.row_block, col0 = e.col0 + b * e.col_block + c;
            if (g.mode == GEMM_RESIDUAL_F32 && g.splits == 1) flush_unit<4, true>(g, 0, stage, lane, row, M, col0, e.lim(b));
            else flush_unit<4, false>(g, (long long)split * g.split_stride, stage, lane, row, M, col0, e.lim(b));
            __syncwarp();
        }
    }
}

template <bool STATS, bool ROPE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1)
gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB0,
            const __grid_constant__ CUtensorMap tmB1, const __grid_constant__ CUtensorMap tmB2, GemmArgs g)
{
    // This kernel may have been scheduled while the one before it in the stream still runs (programmatic dependent launch):
    // everything up to pdl_wait() touches only this CTA's shared and tensor memory.
    const int MB = g.mb;
    const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
    // uniform over the pair, before any barrier or allocation: pairs beyond the tiles of even the largest row count
    if (pair >= ((g.M + MB * 2 * BM - 1) / (MB * 2 * BM)) * g.n_col_tiles * g.splits) return;

    const int BN = g.bn, HALF = BN >> 1;
    int STAGES = g.stages, STAGE_BYTES = MB * A_BYTES + HALF * BK * 2;      // per CTA: MB blocks of 128 A rows, half of the weight rows
    const int ring_bytes = STAGES * STAGE_BYTES;
    const uint32_t rank = tc::cluster_ctarank();            // 0 = leader (issues the MMAs), 1 = peer

    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + ring_bytes);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * kMaxStages + 4);
    __shared__ int s_abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int num_kb = (g.K + BK - 1) / BK;
    const uint32_t smem_base = tc::smem_u32(smem);
    const uint32_t bar_full = tc::smem_u32(bars), bar_empty = bar_full + 8 * kMaxStages;
    const uint32_t bar_acc_full = bar_full + 16 * kMaxStages, bar_acc_empty = bar_acc_full + 16;
    // the leader's copies of the barriers both CTAs signal
    const uint32_t lead_full = tc::mapa(bar_full, 0), lead_acc_empty = tc::mapa(bar_acc_empty, 0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxStages; ++s) { tc::mbar_init(bar_full + 8 * s, 1); tc::mbar_init(bar_empty + 8 * s, 1); }
        for (int b = 0; b < 2; ++b) { tc::mbar_init(bar_acc_full + 8 * b, 1); tc::mbar_init(bar_acc_empty + 8 * b, 2 * kEpiWarps); }
        s_abort = 0;
        tc::mbar_init_fence();
    }
    if (threadIdx.x == 64) {                                // descriptors on their way while the kernel before this one runs
        tc::tma_prefetch_desc(&tmA); tc::tma_prefetch_desc(&tmB0);
        if (g.mode == GEMM_SWIGLU || g.n_per_map < g.N) { tc::tma_prefetch_desc(&tmB1); tc::tma_prefetch_desc(&tmB2); }
    }
    __syncwarp();
    if (warp == 1) { tc::tmem_alloc_2cta(tc::smem_u32(tmem_slot), kTmemCols); tc::tmem_relinquish_2cta(); }
    tc::tc_fence_before();
    tc::cluster_sync();                                     // barriers of both CTAs are initialised, TMEM is allocated
    tc::tc_fence_after();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t *>(tmem_slot);
    const uint32_t bn_pad = (uint32_t)((BN + 31) & ~31);
    const uint32_t buf_stride = 256;
    const bool swiglu = (g.mode == GEMM_SWIGLU);

    // Model weights do not depend on the kernel before this one: the first tile's weight rows are requested at once, as many
    // k-blocks as the ring holds; their activation rows follow after the wait.
    const int pre = (g.b_static && g.d_m == nullptr) ? early_weights(g, pair, STAGES) : 0;
    // 256-row blocks of a tile that hold rows at all: the last one of an odd number of blocks, and every tile when the device's
    // row count is below the planned one, is half as high (an LM head planned for 512 rows and given 256 took 370 us, 1.9x)
    auto blocks_of = [&](const TileCoord &t, int rows) { return MB == 2 && t.m0 + 2 * BM < rows ? 2 : 1; };
    if (warp == 0 && pre > 0) {
        const TileCoord t = tile_coord<ROPE>(g, pair, (g.M + MB * 2 * BM - 1) / (MB * 2 * BM));
        const CUtensorMap *mb = swiglu ? (rank == 0 ? &tmB0 : &tmB1) : (t.map_idx == 0 ? &tmB0 : (t.map_idx == 1 ? &tmB1 : &tmB2));
        const int brow = weight_row0<ROPE>(t, (int)rank, HALF, swiglu), j0 = max(t.j0, 0), kb0 = t.split * g.kb_per_split;
        for (int j = 0; j < pre; ++j) {
            if (rank == 0) tc::mbar_expect_tx_elect(bar_full + 8 * j, 2u * (uint32_t)(STAGE_BYTES - (MB - blocks_of(t, g.M)) * A_BYTES));
            load_weights<ROPE>(smem_base + j * STAGE_BYTES + MB * A_BYTES, mb, (kb0 + j) * BK, brow, j0, lead_full + 8 * j);
        }
    }
    pdl_wait();                                             // the kernel before this one has completed: global memory from here on
    // nothing left to decode, or fewer rows than planned: the loops below find no tile (same values in both CTAs of the pair)
    const bool live = !(g.d_active && *g.d_active == 0);
    const int M = g.d_m ? min(*g.d_m, g.M) : g.M;
    const int m_groups = (M + MB * 2 * BM - 1) / (MB * 2 * BM);
    const int num_tiles = live ? m_groups * g.n_col_tiles * g.splits : 0;
    // Fewer rows than planned, one block in use: two accumulators fit tensor memory, and the ring holds more, smaller stages
    // (256 rows of an LM head planned for 512: 250 us with the four stages of two blocks).
    const bool one_block = g.d_m != nullptr && M <= 2 * BM;
    const uint32_t n_bufs = one_block ? 2u : (uint32_t)g.acc_bufs;
    const int MBS = one_block ? 1 : MB;                     // blocks a stage has room for
    if (one_block) { STAGE_BYTES = A_BYTES + HALF * BK * 2; STAGES = min(kMaxStages, ring_bytes / STAGE_BYTES); }

    // The producer and MMA loops are run by all 32 lanes of their warp with warp-uniform operands; one elected lane
    // issues each asynchronous instruction.  (Issued from a single-lane branch, every tcgen05.mma cost the thread
    // about 90 cycles and an already-complete mbarrier wait about 200: the loop, not the tensor core, set the pace.)
    // The readiness of the next stage is polled (without blocking) before the current stage's instructions are
    // issued, so the latency of that poll overlaps the issue.
    if (warp == 0) {
        // ---------------- TMA producer (both CTAs; completion bytes are counted on the leader's barrier)
        uint32_t it = 0, s = 0, ph = 0;                     // stage and phase are counted along: dividing by STAGES in both loops cost 256 + 256 tokens 6 %
        bool ok = true;
        bool ready = tc::mbar_test(bar_empty, 1u);
        for (int tile = pair; tile < num_tiles && ok; tile += num_pairs) {
            const TileCoord t = tile_coord<ROPE>(g, tile, m_groups);
            // leader: first half of the weight rows (SwiGLU: the gate rows); peer: second half (the up rows)
            const CUtensorMap *mb = swiglu ? (rank == 0 ? &tmB0 : &tmB1)
                                           : (t.map_idx == 0 ? &tmB0 : (t.map_idx == 1 ? &tmB1 : &tmB2));
            const int brow = weight_row0<ROPE>(t, (int)rank, HALF, swiglu), j0 = max(t.j0, 0);
            const int arow = t.m0 + (int)rank * BM, mbt = blocks_of(t, M);
            const int kb0 = t.split * g.kb_per_split, kb1 = min(num_kb, kb0 + g.kb_per_split);
            for (int kb = kb0; kb < kb1; ++kb, ++it) {
                if (!ready) ready = tc::mbar_wait(bar_empty + 8 * s, ph ^ 1u, &s_abort);
                ok = __all_sync(0xffffffffu, ready);
                if (!ok) break;
                const uint32_t ns = s + 1u == (uint32_t)STAGES ? 0u : s + 1u, nph = ns == 0u ? ph ^ 1u : ph;
                ready = tc::mbar_test(bar_empty + 8 * ns, nph ^ 1u);
                const uint32_t sa = smem_base + s * STAGE_BYTES;
                const bool early = it < (uint32_t)pre;
                if (rank == 0 && !early) tc::mbar_expect_tx_elect(bar_full + 8 * s, 2u * (uint32_t)(STAGE_BYTES - (MBS - mbt) * A_BYTES));
                tc::tma_load_2d_2cta_elect(sa, &tmA, kb * BK, arow, lead_full + 8 * s);
                if (mbt == 2) tc::tma_load_2d_2cta_elect(sa + A_BYTES, &tmA, kb * BK, arow + 2 * BM, lead_full + 8 * s);
                if (!early) load_weights<ROPE>(sa + MBS * A_BYTES, mb, kb * BK, brow, j0, lead_full + 8 * s);
                s = ns; ph = nph;
            }
        }
        if (!live && pre > 0) {
            // nothing left to decode: the stages requested above are completed and awaited, nobody reads them
            const int mbt = blocks_of(tile_coord<ROPE>(g, pair, m_groups), g.M);
            for (int j = 0; j < pre; ++j) {
                const uint32_t sa = smem_base + j * STAGE_BYTES;
                tc::tma_load_2d_2cta_elect(sa, &tmA, 0, 0, lead_full + 8 * j);
                if (mbt == 2) tc::tma_load_2d_2cta_elect(sa + A_BYTES, &tmA, 0, 0, lead_full + 8 * j);
            }
            if (rank == 0) for (int j = 0; j < pre && tc::mbar_wait(bar_full + 8 * j, 0u, &s_abort); ++j) {}
        }
        // every stage has been released (by both CTAs' MMAs): no signal of the tensor core is on its way to this CTA when it leaves
        if (ok)
            for (uint32_t j = it > (uint32_t)STAGES ? it - (uint32_t)STAGES : 0u; j < it && tc::mbar_wait(bar_empty + 8 * (j % (uint32_t)STAGES), (j / (uint32_t)STAGES) & 1u, &s_abort); ++j) {}
        if (s_abort && rank == 0 && lane == 0) {
            // give copies already in flight (both CTAs') a bounded chance to land before the pair retires
            const uint32_t first = it > (uint32_t)STAGES ? it - (uint32_t)STAGES : 0u;
            for (uint32_t j = first; j < it; ++j) {
                const uint32_t bar = bar_full + 8 * (j % (uint32_t)STAGES), ph = (j / (uint32_t)STAGES) & 1u;
                for (int i = 0; i < (1 << 16) && !tc::mbar_try(bar, ph); ++i) {}
            }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            // ---------------- MMA issuer (leader CTA only)
            const uint32_t idesc = tc::idesc_bf16_f32(2 * BM, BN);
            uint32_t s = 0, ph = 0, lt = 0;
            bool ok = true;
            bool ready = tc::mbar_test(bar_full, 0u);
            for (int tile = pair; tile < num_tiles && ok; tile += num_pairs, ++lt) {
                const uint32_t buf = lt % n_bufs, use = lt / n_bufs;
                // both CTAs' epilogues have drained this accumulator buffer
                ok = __all_sync(0xffffffffu, tc::mbar_wait(bar_acc_empty + 8 * buf, (use & 1u) ^ 1u, &s_abort));
                if (!ok) break;
                tc::tc_fence_after();
                const uint32_t d_tmem = tmem_base + buf * buf_stride;
                const TileCoord t = tile_coord<ROPE>(g, tile, m_groups);
                const bool second = blocks_of(t, M) == 2;
                const int kb0 = t.split * g.kb_per_split, kb1 = min(num_kb, kb0 + g.kb_per_split);
                for (int kb = kb0; kb < kb1; ++kb) {
                    if (!ready) ready = tc::mbar_wait(bar_full + 8 * s, ph, &s_abort);
                    ok = __all_sync(0xffffffffu, ready);
                    if (!ok) break;
                    tc::tc_fence_after();
                    const uint32_t ns = s + 1u == (uint32_t)STAGES ? 0u : s + 1u, nph = ns == 0u ? ph ^ 1u : ph;
                    ready = tc::mbar_test(bar_full + 8 * ns, nph);
                    const uint32_t sa = smem_base + s * STAGE_BYTES;
                    const uint64_t da = tc::smem_desc_sw128(sa), db = tc::smem_desc_sw128(sa + MBS * A_BYTES);
                    const uint32_t acc = kb != kb0 ? 1u : 0u;
                    tc::mma_bf16_2cta_elect(d_tmem, da, db, idesc, acc);
#pragma unroll
                    for (int kk = 1; kk < BK / 16; ++kk) tc::mma_bf16_2cta_elect(d_tmem, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, 1u);
                    if (second) {
                        const uint64_t da1 = tc::smem_desc_sw128(sa + A_BYTES);
                        tc::mma_bf16_2cta_elect(d_tmem + bn_pad, da1, db, idesc, acc);
#pragma unroll
                        for (int kk = 1; kk < BK / 16; ++kk) tc::mma_bf16_2cta_elect(d_tmem + bn_pad, da1 + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, 1u);
                    }
                    tc::mma_commit_2cta_elect(bar_empty + 8 * s);     // frees the stage in both CTAs once these MMAs have read it
                    s = ns; ph = nph;
                }
                tc::mma_commit_2cta_elect(bar_acc_full + 8 * buf);    // accumulator complete (or abandoned), both CTAs
            }
        }
    } else {
        // ---------------- epilogue: 8 warps; warp w reads TMEM lanes 32*(w%4).., the column units of parity (w-2)/4
        const int q = warp & 3, par = (warp - 2) >> 2;
        const uint32_t stage = smem_base + ring_bytes + kBarBytes + (uint32_t)(warp - 2) * (32 * 128);
        uint32_t lt = 0;
        bool ok = true;
        for (int tile = pair; tile < num_tiles && ok; tile += num_pairs, ++lt) {
            const TileCoord t = tile_coord<ROPE>(g, tile, m_groups);
            const uint32_t buf = lt % n_bufs, use = lt / n_bufs;
            ok = tc::mbar_wait(bar_acc_full + 8 * buf, use & 1u, &s_abort) && !s_abort;
            if (!ok) break;
            tc::tc_fence_after();
            if (tile + num_pairs >= num_tiles) pdl_trigger();   // the rest takes about as long as a launch (see pdl_trigger)
            EpiShare e;
            e.tmem = tmem_base + buf * buf_stride + ((uint32_t)(q * 32) << 16); e.tmem_block = bn_pad; e.up = (uint32_t)HALF;
            e.row0 = t.m0 + (int)rank * BM + q * 32; e.row_block = 2 * BM;
            e.col0 = t.ncol0; e.col_block = 0; e.blocks = blocks_of(t, M); e.seg = STATS ? BN : t.ncols;      // (every record is written)
            e.col_end = min(t.ncol0 + t.ncols, g.N);
            e.rec = 2 * (t.ncol0 / BN); e.rec_block = 0;
            e.head0 = t.n_local; e.j0 = t.j0;
            if constexpr (ROPE) {
                if (t.j0 >= 0) epilogue_pairs(g, e, stage, par, lane, M);
                else epilogue_values<true>(g, e, par, lane, M);
            } else epilogue_tile<STATS>(g, e, t.split, stage, par, lane, M);
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0 && tile + (int)n_bufs * num_pairs < num_tiles) tc::mbar_arrive_cluster(lead_acc_empty + 8 * buf);     // (if it is used again)
        }
    }

    // ---------------- teardown: no CTA of the pair leaves while the other may still signal its barriers
    // (whatever one CTA signals the other has been waited for by then, unless a wait gave up: the barrier orders execution only)
    __syncwarp();                                           // the diverged roles rejoin their warps
    tc::tc_fence_before();
    if (s_abort) tc::cluster_sync(); else tc::cluster_sync_relaxed();
    if (warp == 1) { tc::tc_fence_after(); tc::tmem_dealloc_2cta(tmem_base, kTmemCols); }
    if (threadIdx.x == 0 && s_abort && g.err) atomicExch(g.err, SFS_ERR_TIMEOUT);
}

// ---- few rows (M <= 128): weights stream through all SMs ---------------------------------------------------------
// With at most 128 rows the projection is bound by streaming its weights: from HBM once, and from L2 into the SMs together
// with the activation rows that every tile needs again.  A pair of CTAs computes a 128 x (NB x BN) tile with
// tcgen05.mma.cta_group::2, M = 128: each CTA stages 64 activation rows and half of the weight rows of every N-block, so per
// k-block an SM pulls 64 + NB * BN / 2 rows and the ring holds up to nine k-blocks of wide tiles.  Measured at 128 rows, 8B
// widths, weights from HBM, QKV / O / gate-up / down in us: 24.8 / 12.0 / 40.2 / 24.0 (the HBM floor at 6458 GB/s: 15.6 / 5.2 /
// 31.2 / 15.6); single-CTA 128 x BN tiles, which pull 128 + BN rows for BN weight rows, took 29.1 / 12.0 / 42.3 / 24.7.
// In a step, where the first weights arrive while the kernel ahead still runs: 20.7 / 10.4 / 36.5 / 19.5 from wait to end.  Two
// k-blocks per stage with the epilogue parked in the idle ring (fewer hand-overs): 8 layers 1142 -> 1209 us, not taken.
// SwiGLU: N-block 0
// holds gate rows, N-block 1 the up rows of the same features.  Of an N-block's accumulators every CTA holds its 64 rows:
// tensor-memory lanes 0-63 the columns [0, BN/2), lanes 64-127 the columns [BN/2, BN), in BN/2 tensor-memory columns.
// Warp roles, ring, hand-over and bounded waits are those of the pair kernel above.
template <bool STATS, bool ROPE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1)
gemm_few_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB0,
                const __grid_constant__ CUtensorMap tmB1, const __grid_constant__ CUtensorMap tmB2, GemmArgs g)
{
    const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
    if (pair >= ((g.M + 2 * FM - 1) / (2 * FM)) * g.n_col_tiles * g.splits) return;      // beyond the tiles of even the largest row count

    const int BN = g.bn, NB = g.nb, STAGES = g.stages, HALF = BN >> 1;
    const int B_BYTES = HALF * BK * 2, STAGE_BYTES = FM * BK * 2 + NB * B_BYTES;
    const uint32_t rank = tc::cluster_ctarank();
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + STAGES * STAGE_BYTES);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * kMaxStages + 4);
    __shared__ int s_abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int num_kb = (g.K + BK - 1) / BK;
    const uint32_t smem_base = tc::smem_u32(smem);
    const uint32_t bar_full = tc::smem_u32(bars), bar_empty = bar_full + 8 * kMaxStages;
    const uint32_t bar_acc_full = bar_full + 16 * kMaxStages, bar_acc_empty = bar_acc_full + 16;
    const uint32_t lead_full = tc::mapa(bar_full, 0), lead_acc_empty = tc::mapa(bar_acc_empty, 0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { tc::mbar_init(bar_full + 8 * s, 1); tc::mbar_init(bar_empty + 8 * s, 1); }
        for (int b = 0; b < 2; ++b) { tc::mbar_init(bar_acc_full + 8 * b, 1); tc::mbar_init(bar_acc_empty + 8 * b, 2 * kEpiWarps); }
        s_abort = 0;
        tc::mbar_init_fence();
    }
    if (threadIdx.x == 64) {                                // descriptors on their way while the kernel before this one runs
        tc::tma_prefetch_desc(&tmA); tc::tma_prefetch_desc(&tmB0);
        if (g.mode == GEMM_SWIGLU || g.n_per_map < g.N) { tc::tma_prefetch_desc(&tmB1); tc::tma_prefetch_desc(&tmB2); }
    }
    __syncwarp();
    if (warp == 1) { tc::tmem_alloc_2cta(tc::smem_u32(tmem_slot), kTmemCols); tc::tmem_relinquish_2cta(); }
    tc::tc_fence_before();
    tc::cluster_sync();
    tc::tc_fence_after();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t *>(tmem_slot);
    const bool swiglu = (g.mode == GEMM_SWIGLU);

    // the first tile's weight rows are requested before the wait (see the pair kernel)
    const int pre = (g.b_static && g.d_m == nullptr) ? early_weights(g, pair, STAGES) : 0;
    if (warp == 0 && pre > 0) {
        const TileCoord t = tile_coord<ROPE>(g, pair, (g.M + 2 * FM - 1) / (2 * FM));
        const CUtensorMap *m0 = swiglu ? &tmB0 : (t.map_idx == 0 ? &tmB0 : (t.map_idx == 1 ? &tmB1 : &tmB2));
        const CUtensorMap *m1 = swiglu ? &tmB1 : m0;
        const int brow0 = weight_row0<ROPE>(t, (int)rank, HALF, false), brow1 = swiglu ? brow0 : brow0 + BN, j0 = max(t.j0, 0), kb0 = t.split * g.kb_per_split;
        for (int j = 0; j < pre; ++j) {
            const uint32_t sa = smem_base + j * STAGE_BYTES;
            if (rank == 0) tc::mbar_expect_tx_elect(bar_full + 8 * j, 2u * (uint32_t)STAGE_BYTES);
            load_weights<ROPE>(sa + FM * BK * 2, m0, (kb0 + j) * BK, brow0, j0, lead_full + 8 * j);
            if (!ROPE && NB == 2) tc::tma_load_2d_2cta_elect(sa + FM * BK * 2 + B_BYTES, m1, (kb0 + j) * BK, brow1, lead_full + 8 * j);
        }
    }
    pdl_wait();                                             // the kernel before this one has completed: global memory from here on
    const bool live = !(g.d_active && *g.d_active == 0);    // nothing left to decode: the loops below find no tile
    const int M = g.d_m ? min(*g.d_m, g.M) : g.M;
    const int m_groups = (M + 2 * FM - 1) / (2 * FM);
    const int num_tiles = live ? m_groups * g.n_col_tiles * g.splits : 0;

    if (warp == 0) {
        // ---------------- TMA producer (both CTAs; completion bytes are counted on the leader's barrier)
        uint32_t it = 0, s = 0, ph = 0;
        bool ok = true;
        bool ready = tc::mbar_test(bar_empty, 1u);
        for (int tile = pair; tile < num_tiles && ok; tile += num_pairs) {
            const TileCoord t = tile_coord<ROPE>(g, tile, m_groups);
            const CUtensorMap *m0 = swiglu ? &tmB0 : (t.map_idx == 0 ? &tmB0 : (t.map_idx == 1 ? &tmB1 : &tmB2));
            const CUtensorMap *m1 = swiglu ? &tmB1 : m0;
            const int brow0 = weight_row0<ROPE>(t, (int)rank, HALF, false), brow1 = swiglu ? brow0 : brow0 + BN, j0 = max(t.j0, 0);
            const int arow = t.m0 + (int)rank * FM;
            const int kb0 = t.split * g.kb_per_split, kb1 = min(num_kb, kb0 + g.kb_per_split);
            for (int kb = kb0; kb < kb1; ++kb, ++it) {
                if (!ready) ready = tc::mbar_wait(bar_empty + 8 * s, ph ^ 1u, &s_abort);
                ok = __all_sync(0xffffffffu, ready);
                if (!ok) break;
                const uint32_t ns = s + 1u == (uint32_t)STAGES ? 0u : s + 1u, nph = ns == 0u ? ph ^ 1u : ph;
                ready = tc::mbar_test(bar_empty + 8 * ns, nph ^ 1u);
                const uint32_t sa = smem_base + s * STAGE_BYTES;
                if (it >= (uint32_t)pre) {
                    if (rank == 0) tc::mbar_expect_tx_elect(bar_full + 8 * s, 2u * (uint32_t)STAGE_BYTES);
                    load_weights<ROPE>(sa + FM * BK * 2, m0, kb * BK, brow0, j0, lead_full + 8 * s);
                    if (!ROPE && NB == 2) tc::tma_load_2d_2cta_elect(sa + FM * BK * 2 + B_BYTES, m1, kb * BK, brow1, lead_full + 8 * s);
                }
                tc::tma_load_2d_2cta_elect(sa, &tmA, kb * BK, arow, lead_full + 8 * s);
                s = ns; ph = nph;
            }
        }
        if (!live && pre > 0) {
            // nothing left to decode: the stages requested above are completed and awaited, nobody reads them
            for (int j = 0; j < pre; ++j) tc::tma_load_2d_2cta_elect(smem_base + j * STAGE_BYTES, &tmA, 0, 0, lead_full + 8 * j);
            if (rank == 0) for (int j = 0; j < pre && tc::mbar_wait(bar_full + 8 * j, 0u, &s_abort); ++j) {}
        }
        // every stage has been released (by both CTAs' MMAs): no signal of the tensor core is on its way to this CTA when it leaves
        if (ok)
            for (uint32_t j = it > (uint32_t)STAGES ? it - (uint32_t)STAGES : 0u; j < it && tc::mbar_wait(bar_empty + 8 * (j % (uint32_t)STAGES), (j / (uint32_t)STAGES) & 1u, &s_abort); ++j) {}
        if (s_abort && rank == 0 && lane == 0) {
            // give copies already in flight (both CTAs') a bounded chance to land before the pair retires
            const uint32_t first = it > (uint32_t)STAGES ? it - (uint32_t)STAGES : 0u;
            for (uint32_t j = first; j < it; ++j) {
                const uint32_t bar = bar_full + 8 * (j % (uint32_t)STAGES), pj = (j / (uint32_t)STAGES) & 1u;
                for (int i = 0; i < (1 << 16) && !tc::mbar_try(bar, pj); ++i) {}
            }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            // ---------------- MMA issuer (leader CTA only)
            const uint32_t idesc = tc::idesc_bf16_f32(2 * FM, BN);
            uint32_t lt = 0, s = 0, ph = 0;
            bool ok = true;
            bool ready = tc::mbar_test(bar_full, 0u);
            for (int tile = pair; tile < num_tiles && ok; tile += num_pairs, ++lt) {
                const uint32_t buf = lt & 1u, use = lt >> 1;
                // both CTAs' epilogues have drained this accumulator buffer
                ok = __all_sync(0xffffffffu, tc::mbar_wait(bar_acc_empty + 8 * buf, (use & 1u) ^ 1u, &s_abort));
                if (!ok) break;
                tc::tc_fence_after();
                const uint32_t d_tmem = tmem_base + buf * 256u;
                const int kb0 = tile_coord<ROPE>(g, tile, m_groups).split * g.kb_per_split, kb1 = min(num_kb, kb0 + g.kb_per_split);
                for (int kb = kb0; kb < kb1; ++kb) {
                    if (!ready) ready = tc::mbar_wait(bar_full + 8 * s, ph, &s_abort);
                    ok = __all_sync(0xffffffffu, ready);
                    if (!ok) break;
                    tc::tc_fence_after();
                    const uint32_t ns = s + 1u == (uint32_t)STAGES ? 0u : s + 1u, nph = ns == 0u ? ph ^ 1u : ph;
                    ready = tc::mbar_test(bar_full + 8 * ns, nph);
                    const uint32_t sa = smem_base + s * STAGE_BYTES;
                    const uint64_t da = tc::smem_desc_sw128(sa), db = tc::smem_desc_sw128(sa + FM * BK * 2);
                    const uint32_t acc = kb != kb0 ? 1u : 0u;
                    tc::mma_bf16_2cta_elect(d_tmem, da, db, idesc, acc);
#pragma unroll
                    for (int kk = 1; kk < BK / 16; ++kk) tc::mma_bf16_2cta_elect(d_tmem, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, 1u);
                    if (NB == 2) {
                        const uint64_t db1 = tc::smem_desc_sw128(sa + FM * BK * 2 + B_BYTES);
                        tc::mma_bf16_2cta_elect(d_tmem + (uint32_t)HALF, da, db1, idesc, acc);
#pragma unroll
                        for (int kk = 1; kk < BK / 16; ++kk) tc::mma_bf16_2cta_elect(d_tmem + (uint32_t)HALF, da + (uint64_t)(kk * 2), db1 + (uint64_t)(kk * 2), idesc, 1u);
                    }
                    tc::mma_commit_2cta_elect(bar_empty + 8 * s);     // frees the stage in both CTAs once these MMAs have read it
                    s = ns; ph = nph;
                }
                tc::mma_commit_2cta_elect(bar_acc_full + 8 * buf);    // accumulator complete (or abandoned), both CTAs
            }
        }
    } else {
        // ---------------- epilogue: 8 warps; warp w reads TMEM lanes 32*(w%4).. (rows 32*(w%2).. of this CTA, column half (w%4)/2)
        const int q = warp & 3, par = (warp - 2) >> 2, hq = q >> 1;
        const uint32_t stage = smem_base + STAGES * STAGE_BYTES + kBarBytes + (uint32_t)(warp - 2) * (32 * 128);
        uint32_t lt = 0;
        bool ok = true;
        for (int tile = pair; tile < num_tiles && ok; tile += num_pairs, ++lt) {
            const TileCoord t = tile_coord<ROPE>(g, tile, m_groups);
            const uint32_t buf = lt & 1u, use = lt >> 1;
            ok = tc::mbar_wait(bar_acc_full + 8 * buf, use & 1u, &s_abort) && !s_abort;
            if (!ok) break;
            tc::tc_fence_after();
            if (tile + num_pairs >= num_tiles) pdl_trigger();   // the rest takes about as long as a launch (see pdl_trigger)
            EpiShare e;
            e.tmem = tmem_base + buf * 256u + ((uint32_t)(q * 32) << 16); e.tmem_block = (uint32_t)HALF; e.up = (uint32_t)HALF;
            e.row0 = t.m0 + (int)rank * FM + (q & 1) * 32; e.row_block = 0;
            e.col0 = t.ncol0 + hq * HALF; e.col_block = BN; e.blocks = swiglu ? 1 : NB; e.seg = HALF;
            e.col_end = min(t.ncol0 + t.ncols, g.N);
            e.rec = 4 * NB * (t.ncol0 / (NB * BN)) + 2 * hq; e.rec_block = 4;
            e.head0 = t.n_local + hq * (HALF / 32); e.j0 = t.j0;
            if (ROPE && t.j0 >= 0) e.col0 = t.ncol0;        // (which matrix: the columns follow from the heads)
            if constexpr (ROPE) {
                if (t.j0 >= 0) epilogue_pairs(g, e, stage, par, lane, M);
                else epilogue_values<true>(g, e, par, lane, M);
            } else epilogue_tile<STATS>(g, e, t.split, stage, par, lane, M);
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0 && tile + 2 * num_pairs < num_tiles) tc::mbar_arrive_cluster(lead_acc_empty + 8 * buf);
        }
    }

    // ---------------- teardown: no CTA of the pair leaves while the other may still signal its barriers
    __syncwarp();
    tc::tc_fence_before();
    if (s_abort) tc::cluster_sync(); else tc::cluster_sync_relaxed();
    if (warp == 1) { tc::tc_fence_after(); tc::tmem_dealloc_2cta(tmem_base, kTmemCols); }
    if (threadIdx.x == 0 && s_abort && g.err) atomicExch(g.err, SFS_ERR_TIMEOUT);
}

int num_sms()
{
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
            n = 148;
    }
    return n;
}

// column tiles of a problem at `tile_cols` output columns per tile
int col_tiles(int mode, int n_maps, int n_per_map, int tile_cols, int rope_dim = 0)
{
    if (rope_dim) {                                          // two rotated matrices (16 pairs of tile_cols / 32 heads a tile) and a plain one
        const int heads = n_per_map / rope_dim, per_tile = tile_cols / 32;
        return 2 * (rope_dim / 32) * ((heads + per_tile - 1) / per_tile) + (n_per_map + tile_cols - 1) / tile_cols;
    }
    const int per_map = (n_per_map + tile_cols - 1) / tile_cols;
    return mode == GEMM_SWIGLU ? per_map : n_maps * per_map;
}

int stages_for(int mb, int bn)
{
    const int stage_bytes = mb * A_BYTES + (bn / 2) * BK * 2;
    const int s = (kSmemBudget - 1024 - kBarBytes - kEpiStageBytes) / stage_bytes;
    return s > kMaxStages ? kMaxStages : s;
}

// Modelled clocks of one candidate: waves x (k-blocks x clocks per k-block + exposed epilogue), per pair of SMs.
// Per k-block and CTA the tensor core needs MB*bn*2 clocks (8192 FLOP/clk/SM) and some 80 pass between k-blocks; the operand
// stream is (MB*128 + bn/2) rows x 128 B at the ~54 B/clk an SM sustains from L2 when every SM streams; below 540 (MB = 1) or 980
// clocks the k-block time stops shrinking with the tile.  Fitted to sweeps of MB, bn and the split at 512 to 2048 rows with operands
// that do not heat the part; what it changed against the calibration before (40 B/clk, 750 clocks), us: down 512 rows 40.7 -> 37.1
// (240 x 2 ranges instead of 512 x 240 x 4), QKV 1000 rows 70.4 -> 61.9, 1536 rows 90.8 -> 82.9, gate / up 1536 rows 168 -> 153.
// The epilogue hides behind the next tile when two accumulators fit tensor memory, except for a pair's last tile.
// Splitting K pays for few rows only: the slabs grow with M, the idle pairs they avoid do not.
long long model_clocks(int M, int K, int mode, int n_maps, int n_per_map, int rope_dim, int pairs, int mb, int bn, int splits)
{
    const long long num_kb = (K + BK - 1) / BK, kbps = (num_kb + splits - 1) / splits;
    const int m_groups = (M + mb * 2 * BM - 1) / (mb * 2 * BM);
    const long long tiles = (long long)m_groups * col_tiles(mode, n_maps, n_per_map, mode == GEMM_SWIGLU ? bn / 2 : bn, rope_dim) * ((num_kb + kbps - 1) / kbps);
    const long long waves = (tiles + pairs - 1) / pairs;
    const long long mma = (long long)mb * bn * 2 + 80, load = (long long)(mb * BM + bn / 2) * 128 / 54, least = mb == 1 ? 540 : 980;
    long long kb_clk = mma > load ? mma : load;
    if (kb_clk < least) kb_clk = least;
    const long long epi = (long long)mb * bn * 16 + 3000;
    const bool hidden = mb * ((bn + 31) & ~31) <= 256;
    // a split K also costs the fp32 slab that the next RMSNorm reads back: M x N x 4 bytes, measured at ~1.2e-3 clocks per element
    const long long n_out = (mode == GEMM_SWIGLU) ? n_per_map : (long long)n_maps * n_per_map;
    const long long slab = 1500 + (long long)((double)M * (double)n_out * 1.2e-3);
    return waves * kbps * kb_clk + (hidden ? 1 : waves) * epi + (splits > 1 ? slab * splits : 0);
}

// Tile shape (MB blocks of 256 rows, width bn) and number of K ranges with the smallest modelled time.  Wide, tall tiles
// win when there are many tiles; narrower or shorter ones, or a split K, when a big tile would leave most pairs idle.
void pick_tile(int M, int K, int mode, int n_maps, int n_per_map, int rope_dim, int pairs, int max_splits, int *mb_out, int *bn_out, int *splits_out)
{
    const int step = rope_dim ? 64 : (mode == GEMM_SWIGLU ? 32 : 16);      // (a CTA's half of a rotating tile: whole groups of 16 pairs)
    long long best_cost = -1;
    for (int mb = (M > 2 * BM ? 2 : 1); mb >= 1; --mb)
        for (int bn = 256; bn >= 32; bn -= step)
            for (int sp = 1; sp <= max_splits; ++sp) {
                if (rope_dim && (n_per_map / rope_dim) % (bn / 32) != 0 && bn > 64) continue;      // (see gemm_rotates)
                const long long cost = model_clocks(M, K, mode, n_maps, n_per_map, rope_dim, pairs, mb, bn, sp);
                if (best_cost < 0 || cost < best_cost) { best_cost = cost; *mb_out = mb; *bn_out = bn; *splits_out = sp; }
            }
}

// Few rows: 128 x (nb x bn) tiles of CTA pairs.  Measured: a k-block costs the issuing warp 255 + 165 nb clocks, an SM's L2
// port ~40 B/clk for its 64 + nb * bn / 2 rows of 128 B, and HBM 3370 B/clk over all pairs; the largest sets the pace.  A slab
// of a split K costs its reader ~600 clocks and 1.2e-3 per element.  At 128 rows, 8B widths this picks QKV 192 x 1 (24.8 us; the
// next best 224: 25.4, nb = 2: 28.1), O 192 x 1 in 3 ranges of K (12.0; 2 ranges of 128: 13.0), gate / up 192 (40.2; 224: 40.8),
// down 256 x 1 in 4 ranges (24.0; 192 in 3: 24.8).
long long model_clocks_few(int M, int K, int mode, int n_maps, int n_per_map, int rope_dim, int pairs, int bn, int nb, int splits)
{
    const long long num_kb = (K + BK - 1) / BK, kbps = (num_kb + splits - 1) / splits;
    const int tile_cols = mode == GEMM_SWIGLU ? bn : nb * bn;
    const long long tiles = (long long)col_tiles(mode, n_maps, n_per_map, tile_cols, rope_dim) * ((num_kb + kbps - 1) / kbps);
    const long long waves = (tiles + pairs - 1) / pairs;
    const long long issue = 255 + 165 * nb, port = (long long)(FM + nb * bn / 2) * 128 / 40;
    const long long hbm = (tiles < pairs ? tiles : pairs) * (long long)nb * bn * 128 / 3370;
    long long kb_clk = issue > port ? issue : port;
    if (kb_clk < hbm) kb_clk = hbm;
    const long long epi = (long long)nb * bn * 8 + 3000;
    const long long n_out = (mode == GEMM_SWIGLU) ? n_per_map : (long long)n_maps * n_per_map;
    const long long slab = 600 + (long long)((double)M * (double)n_out * 1.2e-3);
    return waves * kbps * kb_clk + epi + (splits > 1 ? slab * splits : 0);
}

void pick_tile_few(int M, int K, int mode, int n_maps, int n_per_map, int rope_dim, int pairs, int max_splits, int *bn_out, int *nb_out, int *splits_out)
{
    long long best_cost = -1;
    for (int nb = (mode == GEMM_SWIGLU ? 2 : 1); nb <= (rope_dim ? 1 : 2); ++nb)
        for (int bn = 256; bn >= 32; bn -= rope_dim ? 64 : 32)
            for (int sp = 1; sp <= max_splits; ++sp) {
                const long long cost = model_clocks_few(M, K, mode, n_maps, n_per_map, rope_dim, pairs, bn, nb, sp);
                if (best_cost < 0 || cost < best_cost) { best_cost = cost; *bn_out = bn; *nb_out = nb; *splits_out = sp; }
            }
}

// Clocks of the rotary kernel that a rotating epilogue does without: 104 rows of 2 x 4096 4.0 us with its hand-over, 512 6.3, 1536 12, 2048 17
// (of the 4.0, 2 are left when the epilogue has done the work: see gemm_rotates).
long long rope_kernel_clocks(int M, int n_per_map) { return 6600 + (long long)((double)M * n_per_map * 3e-3); }

int stages_for_few(int bn, int nb)
{
    const int stage_bytes = FM * BK * 2 + nb * (bn / 2) * BK * 2;
    const int s = (kSmemBudget - 1024 - kBarBytes - kEpiStageBytes) / stage_bytes;
    return s > kMaxStages ? kMaxStages : s;
}

}  // namespace

int gemm_num_sms() { return num_sms(); }

// A rotating tile takes 16 pairs of each of bn / 32 heads.  Where tiles stream weights (128 rows) a last one of fewer heads costs nothing;
// otherwise whole tiles only (512 rows of 32 heads: 192 columns, a tenth of them padding, 58 us where 176 plain ones take 52).  And only where
// the projection is faster by more than the model's error than a plain one and the rotary kernel: beyond 48 heads of 128 it is not at up to
// 128 rows, whose plain tiles then take two weight blocks each, in one wave instead of two.
// us a layer in the chain (d_ff 3 d), with the rotary kernel / rotating; forward passes of 8, 64, 128 tokens, then 128 rows of a cached 1024 + 512 (where a
// scatter of keys and values goes too): 8 heads of 128 44.2 / 43.3, 44.6 / 44.7, 47.6 / 46.3, 86.3 / 84.6; 16 59.8 / 59.8, 62.6 / 61.3, 65.8 / 64.1,
// 111.8 / 108.9; 24 81.6 / 79.3, 84.0 / 82.3, 89.0 / 85.9, 143.9 / 139.4; 32 110.0 / 109.2, 114.1 / 112.0, 119.6 / 117.9, 180.2 / 175.5 (spreads 0.02 to 0.2, at 32
// heads up to 1.6); 49 219.9 / 229.5, 230.7 / 237.5, 249.2 / 253.9, 329 / 334; 64 351 / 358, 371 / 379, 394 / 400, 499 / 505 (spreads 1 to 12).
// 384 and 1536 rows: 8 heads 59.4 / 56.1 and 88.3 / 84.6, 16 92.1 / 89.8 and 192 / 187 (5).
bool gemm_rotates(int32_t M, int32_t K, int32_t n_per_map, int32_t head_dim)
{
    const bool few = M <= 2 * FM;
    const int pairs = num_sms() / 2;
    int mb = 1, bn = 256, nb = 1, sp = 1;
    auto clocks = [&](int rope_dim) {
        if (few) pick_tile_few(M, K, GEMM_STORE, 3, n_per_map, rope_dim, pairs, 1, &bn, &nb, &sp);
        else pick_tile(M, K, GEMM_STORE, 3, n_per_map, rope_dim, pairs, 1, &mb, &bn, &sp);
        return few ? model_clocks_few(M, K, GEMM_STORE, 3, n_per_map, rope_dim, pairs, bn, nb, 1) : model_clocks(M, K, GEMM_STORE, 3, n_per_map, rope_dim, pairs, mb, bn, 1);
    };
    const long long plain = clocks(0) + rope_kernel_clocks(M, n_per_map), rotating = clocks(head_dim);
    return (few || (n_per_map / head_dim) % (bn / 32) == 0) && rotating * 100 < plain * 97;
}

int32_t gemm_plan_create(GemmPlan *p, const void *A, int64_t lda, int32_t M, int32_t K,
                         const void *const *Bs, int32_t n_maps, int32_t n_per_map, int64_t ldb,
                         int32_t mode, void *C, int64_t ldc, int32_t out_f32, float scale,
                         __nv_bfloat16 *vt, int64_t ldvt, int32_t vt_col0, const GemmTune *tune, const GemmRope *rope)
{
    SFS_REQUIRE(M >= 1 && K >= 1 && n_per_map >= 1 && n_maps >= 1 && n_maps <= 3, SFS_ERR_INVALID_ARG, "gemm: bad sizes");
    SFS_REQUIRE((K % 8) == 0 && (lda % 8) == 0 && (ldb % 8) == 0, SFS_ERR_INVALID_ARG, "gemm: K, lda, ldb must be multiples of 8");
    SFS_REQUIRE(mode != GEMM_SWIGLU || n_maps == 2, SFS_ERR_INVALID_ARG, "gemm: SwiGLU takes two B matrices");
    memset(p, 0, sizeof(*p));
    const int N = (mode == GEMM_SWIGLU) ? n_per_map : n_per_map * n_maps;
    SFS_REQUIRE(aligned_to(C, 16) && (ldc % 8) == 0, SFS_ERR_INVALID_ARG, "gemm: C must be 16-byte aligned, ldc a multiple of 8");
    int mb = 1, bn = 256, nb = 1;
    int sp_unused = 1;
    // at most 128 rows: few-row tiles (a pair's 256-row MMA would be half padding); tune->mb = 1 or 2 forces the pair kernel
    const bool few = (M <= 2 * FM) && !(tune && (tune->mb == 1 || tune->mb == 2));
    const int rope_dim = rope ? rope->head_dim : 0;
    SFS_REQUIRE(!rope || (mode == GEMM_STORE && !out_f32 && n_maps == 3 && vt != nullptr && vt_col0 == 2 * n_per_map && scale == 1.0f && (rope_dim % 32) == 0 &&
                          (n_per_map % rope_dim) == 0 && (n_per_map % 32) == 0), SFS_ERR_INVALID_ARG, "gemm: rotary epilogue takes the QKV projection of whole heads");
    const int step = rope ? 64 : (few ? 32 : ((mode == GEMM_SWIGLU) ? 32 : 16));
    if (few) pick_tile_few(M, K, mode, n_maps, n_per_map, rope_dim, num_sms() / 2, 1, &bn, &nb, &sp_unused);
    else pick_tile(M, K, mode, n_maps, n_per_map, rope_dim, num_sms() / 2, 1, &mb, &bn, &sp_unused);
    if (tune) {                                              // measurement overrides; invalid values are ignored
        if (tune->mb == 1 || tune->mb == 2) mb = tune->mb;
        if (tune->bn >= 32 && tune->bn <= 256 && (tune->bn % step) == 0) bn = tune->bn;
        if (few && (tune->nb == 1 || tune->nb == 2) && mode != GEMM_SWIGLU && !rope) nb = tune->nb;
    }
    p->bn = bn; p->n_maps = n_maps; p->n_per_map = n_per_map;
    int32_t rc = make_tmap_bf16(&p->tmA, A, (uint64_t)M, (uint64_t)K, (uint64_t)lda, few ? FM : BM);
    if (rc != SFS_OK) return rc;
    for (int i = 0; i < 3; ++i) {
        const void *b = Bs[i < n_maps ? i : 0];
        if (rope) rc = make_tmap_pairs(&p->tmB[i], b, (uint64_t)n_per_map, (uint64_t)K, (uint64_t)ldb, i < 2 ? (uint32_t)rope_dim / 2 : 16, (uint32_t)bn / 64);
        else rc = make_tmap_bf16(&p->tmB[i], b, (uint64_t)n_per_map, (uint64_t)K, (uint64_t)ldb, (uint32_t)(bn / 2));
        if (rc != SFS_OK) return rc;
    }
    GemmArgs &g = p->args;
    g.M = M; g.N = N; g.K = K; g.mode = mode; g.out_f32 = out_f32; g.scale = scale;
    g.C = C; g.ldc = ldc; g.vt = vt; g.ldvt = ldvt; g.vt_col0 = vt_col0;
    g.bn = bn; g.mb = few ? 1 : mb; g.nb = few ? nb : 1; g.n_per_map = n_per_map;
    g.few = few ? 1 : 0; g.tile_rows = few ? 2 * FM : mb * 2 * BM;
    g.tile_cols = (mode == GEMM_SWIGLU) ? (few ? bn : bn / 2) : (few ? nb * bn : bn);
    g.tiles_per_map = (mode == GEMM_SWIGLU) ? 0x3FFFFFFF : (n_per_map + g.tile_cols - 1) / g.tile_cols;
    g.n_col_tiles = col_tiles(mode, n_maps, n_per_map, g.tile_cols, rope_dim);
    if (rope) { g.rope = *rope; g.rope_groups = rope_dim / 32; g.rope_tiles = (g.n_col_tiles - (n_per_map + g.tile_cols - 1) / g.tile_cols) / 2; }
    g.stages = few ? stages_for_few(bn, nb) : stages_for(mb, bn);
    if (tune && tune->stages >= 1 && tune->stages <= g.stages) g.stages = tune->stages;
    g.acc_bufs = few || (g.mb * ((bn + 31) & ~31) <= 256) ? 2 : 1;
    // records of the fused row statistics per row; both epilogue-warp parities must own columns of every block
    g.stats_parts = few ? (bn / 2 > 64 ? 4 * nb * g.n_col_tiles : 0) : (bn > 64 ? 2 * g.n_col_tiles : 0);
    g.splits = 1; g.kb_per_split = (K + BK - 1) / BK; g.split_stride = 0;
    p->A = A; p->lda = lda; p->ldb = ldb;
    for (int i = 0; i < 3; ++i) p->Bs[i] = Bs[i < n_maps ? i : 0];
    return SFS_OK;
}

int32_t gemm_plan_enable_split(GemmPlan *p, float *ws, int32_t max_splits, const GemmTune *tune)
{
    GemmArgs &g = p->args;
    const bool f32_out = g.mode == GEMM_RESIDUAL_F32 || (g.mode == GEMM_STORE && g.out_f32 && g.vt == nullptr);
    if (!f32_out || ws == nullptr || max_splits < 2) return SFS_OK;
    int mb = g.mb, bn = g.bn, nb = g.nb, sp = 1;
    const bool few = g.few != 0;
    if (few) pick_tile_few(g.M, g.K, g.mode, p->n_maps, p->n_per_map, 0, num_sms() / 2, max_splits, &bn, &nb, &sp);
    else pick_tile(g.M, g.K, g.mode, p->n_maps, p->n_per_map, 0, num_sms() / 2, max_splits, &mb, &bn, &sp);
    if (tune) {
        if (tune->mb == 1 || tune->mb == 2) mb = tune->mb;
        if (tune->bn >= 32 && tune->bn <= 256 && (tune->bn % 16) == 0) bn = tune->bn;
        if (tune->nb == 1 || tune->nb == 2) nb = tune->nb;
        if (tune->splits >= 1 && tune->splits <= max_splits) sp = tune->splits;
    }
    if (sp <= 1 && !tune) return SFS_OK;
    // rebuild the plan at the new tile shape, then cut K
    GemmPlan q;
    GemmTune t2 = {few ? 0 : mb, bn, tune ? tune->stages : 0, 0, nb};
    int32_t rc = gemm_plan_create(&q, p->A, p->lda, g.M, g.K, p->Bs, p->n_maps, p->n_per_map, p->ldb, g.mode, g.C, g.ldc, g.out_f32,
                                  g.scale, g.vt, g.ldvt, g.vt_col0, &t2);
    if (rc != SFS_OK) return rc;
    q.args.b_static = g.b_static;
    *p = q;
    GemmArgs &h = p->args;
    const int num_kb = (h.K + BK - 1) / BK;
    if (sp > num_kb) sp = num_kb;
    if (sp > 1) {
        h.kb_per_split = (num_kb + sp - 1) / sp;
        h.splits = (num_kb + h.kb_per_split - 1) / h.kb_per_split;
        h.split_stride = (long long)h.M * h.ldc;
        h.C = ws;
    }
    return SFS_OK;
}

int32_t gemm_launch(const GemmPlan &p, const int32_t *d_m, const int32_t *d_active, int32_t *err, cudaStream_t stream)
{
    GemmArgs g = p.args;
    g.d_m = d_m; g.err = err; g.d_active = d_active;
    const int pairs = num_sms() / 2;
    auto launch = [&](auto kernel, bool *configured, size_t smem, long long tiles) -> int32_t {
        bool &done = configured[current_device_slot()];
        if (!done) {
            SFS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget));
            done = true;
        }
        // always ask for more than half of an SM's shared memory: one CTA per SM, so the allocation of all 512
        // tensor-memory columns can never wait for a co-resident CTA
        if (smem < 120 * 1024) smem = 120 * 1024;
        SFS_CUDA(launch_pdl(kernel, dim3((unsigned)(2 * (tiles < pairs ? tiles : pairs))), dim3(kGemmThreads), smem, stream, p.tmA, p.tmB[0], p.tmB[1], p.tmB[2], g));
        return SFS_OK;
    };
    static bool configured[6][kMaxDevices] = {};
    const size_t fixed = kBarBytes + kEpiStageBytes + 1024, b_bytes = (size_t)(g.bn / 2) * BK * 2;
    const long long tiles = (long long)((g.M + g.tile_rows - 1) / g.tile_rows) * g.n_col_tiles * g.splits;
    if (g.few) {
        const size_t smem = (size_t)g.stages * (FM * BK * 2 + g.nb * b_bytes) + fixed;
        if (g.rope.table) return launch(gemm_few_kernel<false, true>, configured[0], smem, tiles);
        return g.stats ? launch(gemm_few_kernel<true, false>, configured[1], smem, tiles) : launch(gemm_few_kernel<false, false>, configured[2], smem, tiles);
    }
    const size_t smem = (size_t)g.stages * (g.mb * A_BYTES + b_bytes) + fixed;
    if (g.rope.table) return launch(gemm_kernel<false, true>, configured[3], smem, tiles);
    return g.stats ? launch(gemm_kernel<true, false>, configured[4], smem, tiles) : launch(gemm_kernel<false, false>, configured[5], smem, tiles);
}

}  // namespace sfs
