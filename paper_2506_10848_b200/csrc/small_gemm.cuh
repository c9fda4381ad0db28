// Internal interface of the projections of small models (norm / embedding in front, rotary / SwiGLU / residual behind, one launch).
#pragma once
#include "sfs_common.cuh"

namespace sfs {

enum { SMALL_BF16 = 0, SMALL_NORM = 1, SMALL_EMBED = 2 };                              // where the activation rows come from
enum { SMALL_QKV = 0, SMALL_RESIDUAL = 1, SMALL_SWIGLU = 2, SMALL_STORE = 3 };         // what becomes of the product

struct SmallGemmArgs {
    int M, N, K;                             // N: output columns (SMALL_QKV: unused)
    const int32_t *d_m, *d_active;           // optional device-side row count; nothing is done when *d_active == 0
    const __nv_bfloat16 *a; long long lda;   // SMALL_BF16: activation rows
    float *x;                                // fp32 residual stream [., K] (read by SMALL_NORM, written by SMALL_EMBED), [., N] for SMALL_RESIDUAL
    const __nv_bfloat16 *gain; float eps;
    const int32_t *rows;                     // SMALL_STORE, optional: row m is row rows[m] of x, for m below the row count
    int rows_known;                          // entries of `rows` that are there whatever *d_m says
    const int32_t *tokens; const __nv_bfloat16 *emb; int vocab;      // SMALL_EMBED
    const __nv_bfloat16 *B[3]; int n_per_map;                        // weights [n_per_map, K] each (model weights: constant)
    __nv_bfloat16 *out; float *out_f32; long long ldc; float scale;
    float *inc;                              // SMALL_RESIDUAL, optional [M, N]: receives what is added to x
    __nv_bfloat16 *vt; long long ldvt;       // SMALL_QKV: q and k rotated into out [M, 2 n_per_map], v transposed into vt [n_per_map, M]
    __nv_bfloat16 *k_dst;                    // SMALL_QKV, optional [M, n_per_map]: k goes there as well
    const float2 *table; int S, head_dim;    // rotary table, tokens per sequence
};
// The entry of the row list that output row m reads before the device's row count has arrived, and the one it reads after it (M);
// -1: none.  A caller's list ends with the count, so nothing beyond it may be touched, not even to throw the value away.
__host__ __device__ inline int list_entry_early(const SmallGemmArgs &g, int m) { return g.rows != nullptr && m < g.rows_known ? m : -1; }
__host__ __device__ inline int list_entry_late(const SmallGemmArgs &g, int m, int M) { return g.rows != nullptr && m >= g.rows_known && m < M ? m : -1; }
// combinations: (EMBED | NORM, QKV), (BF16, RESIDUAL), (NORM, SWIGLU), (NORM, STORE)
int32_t launch_small_gemm(int src, int epi, const SmallGemmArgs &g, cudaStream_t s);
// whether a model's widths fit these kernels (all of K in shared memory, a row's norm in a warp's registers)
bool small_gemm_fits(int d_model, int d_ff, int head_dim);

}  // namespace sfs
