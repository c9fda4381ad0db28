// Both forms of the QKV projection for tests/test_gpu_qkv_rotation.py: queries and keys rotated in the projection's epilogue, and a plain
// projection with the rotary kernel behind it.  Compiled by the test against the library's internal headers; which form a forward pass
// takes is the library's own choice.
#include "cache.cuh"
#include "elementwise.cuh"
#include "gemm.cuh"

using namespace sfs;

extern "C" int32_t qkv_table(float2 *table, int32_t positions, int32_t head_dim, float theta) { return launch_rope_table(table, positions, head_dim, theta, nullptr); }

extern "C" int32_t qkv_rotates(int32_t M, int32_t K, int32_t heads, int32_t head_dim) { return gemm_rotates(M, K, heads * head_dim, head_dim) ? 1 : 0; }

// h [M, K], w [3][heads * head_dim, K], qk [M, 2 n], vt [n, T].  rows != NULL: the tokens of the M rows, keys to k_dst [T, n] and values to vt at
// their tokens' places, by way of vt_compact [n, T] in the plain form.  mb, bn: tile of the rotating form (0: the planner's)
extern "C" int32_t qkv_project(const void *h, const void *const *w, int32_t M, int32_t K, int32_t heads, int32_t head_dim, int32_t S, int32_t T, const float2 *table,
                               const int32_t *rows, void *k_dst, void *qk, void *vt, void *vt_compact, int32_t rotate, int32_t mb, int32_t bn)
{
    const int32_t n = heads * head_dim;
    const GemmTune tune = {mb, bn, 0, 0, 0};
    const GemmRope rope = {table, S, head_dim, rows, static_cast<__nv_bfloat16 *>(k_dst)};
    void *const values = !rotate && rows ? vt_compact : vt;
    GemmPlan p;
    int32_t rc = gemm_plan_create(&p, h, K, M, K, w, 3, n, K, GEMM_STORE, qk, 2 * n, 0, 1.0f, static_cast<__nv_bfloat16 *>(values), T, 2 * n, rotate ? &tune : nullptr,
                                  rotate ? &rope : nullptr);
    if (rc == SFS_OK) rc = gemm_launch(p, nullptr, nullptr, device_status_word(), nullptr);
    if (rc != SFS_OK || rotate) return rc;
    if (rows) return launch_rope_scatter_kv(qk, 2 * n, M, S, heads, head_dim, table, rows, k_dst, vt_compact, T, vt, T, nullptr);
    return launch_rope(qk, 2 * n, M, S, heads, head_dim, table, k_dst, nullptr);
}
