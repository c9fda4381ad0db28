// Internal interface of the kernel that takes a small model's layer from its rotated queries, keys and values to the next layer's.
#pragma once
#include "sfs_common.cuh"
#include "attention.cuh"

namespace sfs {

struct SmallLayerArgs {
    AttnShort qkv; float scale_log2;         // rotated q and k rows, values transposed (as attention_short reads them)
    int B, S, n_heads, d, ff;
    const __nv_bfloat16 *wo, *w_gate, *w_up, *w_down, *gain; float eps;      // model weights: constant
    float *x;                                // [B * S, d] fp32 residual stream, updated in place
    float *inc_attn, *inc_mlp;               // optional [B * S, d]: receive the two increments
    // the next layer's QKV projection (w_q == NULL: none): q and k rotated into qk_out [B * S, 2 d], v transposed into vt_out [d, B * S].  Not the
    // buffers `qkv` reads: other tokens' attention may still be reading them
    const __nv_bfloat16 *w_q, *w_k, *w_v, *next_gain;
    __nv_bfloat16 *qk_out, *vt_out, *k_dst;  // k_dst: optional [B * S, d], the keys go there as well
    const float2 *table;                     // rotary table [positions, 32]
    const int32_t *d_active; int32_t *err;
};
// whether a model's widths and B sequences of S tokens take this kernel
bool small_layer_fits(int d_model, int d_ff, int n_heads, int head_dim, int B, int S);
int32_t launch_small_layer(const SmallLayerArgs &g, cudaStream_t s);

}  // namespace sfs
