// Internal launchers of the memory-bound forward kernels.
#pragma once
#include "sfs_common.cuh"

namespace sfs {
// the start of a forward pass: x[t,:] = the embedding of tokens[t] as fp32, h[t,:] = bf16(RMSNorm(x[t,:]) * gain) of the first layer;
// copy_n integers are copied from copy_src to copy_dst on the way
int32_t launch_embed_norm(const int32_t *tokens, const void *emb, int vocab, float *x, const void *gain, void *h, int T, int d, float eps, const int32_t *copy_src,
                          int32_t *copy_dst, int copy_n, cudaStream_t s);
// h[r,:] = bf16(RMSNorm(y[rows ? rows[r] : r, :]) * gain) with y = x + the n_partial slabs of `partial` (partial_stride
// floats apart, added in slab order; may be NULL).  Without a row list y is written back to x.  The row count may
// come from the device (n_rows).
int32_t launch_rmsnorm(float *x, const float *partial, int n_partial, long long partial_stride, const void *gain, void *h,
                       const int32_t *rows, const int32_t *n_rows, int max_rows, int d, float eps, cudaStream_t s);
int32_t launch_rope_table(float2 *table, int positions, int head_dim, float theta, cudaStream_t s);
// rotates q and k (the first 2*n_heads*head_dim columns of each row) by position = token index mod S: q in place, k in place or,
// when k_dst is given, into k_dst [T, n_heads*head_dim]
int32_t launch_rope(void *qk, int64_t ld, int T, int S, int n_heads, int head_dim, const float2 *table, void *k_dst, cudaStream_t s);
}  // namespace sfs
