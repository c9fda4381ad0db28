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
#include "small_mma.cuh"

namespace sfs {
namespace {

using namespace small;

// PARTS warps divide the keys; grid: (query rows / (16 x tiles per CTA), heads, sequences); blockDim: 32 PARTS x tiles per CTA
template <int PARTS>
__global__ void __launch_bounds__(256, 1)
attention_short_kernel(AttnShort p, AttnArgs a)
{
    extern __shared__ __align__(16) float s_out[];       // per warp [16][kPartLd], then per warp [32]: maxima, denominators
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, part = warp & (PARTS - 1), n_warps = blockDim.x >> 5, first = warp & ~(PARTS - 1);
    const int head = blockIdx.y, b = blockIdx.z, r0 = (blockIdx.x * (n_warps / PARTS) + warp / PARTS) * 16;
    float *s_ml = s_out + n_warps * 16 * kPartLd;

    pdl_wait();
    pdl_trigger();
    const bool active = a.d_active == nullptr || *a.d_active != 0;      // (used only after the loads below)
    attn_part<PARTS>(p, a.S, a.kq, a.scale_log2, head, b, r0, part, lane, s_out + warp * 16 * kPartLd, s_ml + warp * 32);
    if (!active) return;                                  // nothing left to decode
    __syncthreads();
    attn_merge<PARTS>(s_out + first * 16 * kPartLd, s_ml + first * 32, min(PARTS, (a.S + 31) / 32), a.scale_log2, part, lane, [&](int r, int col, uint2 v) {
        if (r0 + r < a.kq) *reinterpret_cast<uint2 *>(a.out + ((long long)b * a.kq + r0 + r) * a.ld_out + head * kHead + col) = v;
    });
}

template <int PARTS>
int32_t launch(const AttnPlan &p, const AttnArgs &a, int mt, cudaStream_t s)
{
    const size_t smem = (size_t)mt * PARTS * kPartBytes;
    static bool configured[kMaxDevices] = {};
    bool &done = configured[current_device_slot()];
    if (!done) {
        SFS_CUDA(cudaFuncSetAttribute(attention_short_kernel<PARTS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(8 * kPartBytes)));
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
    return p.head_dim == kHead && p.args.S <= 512 && (long long)((kq + 31) / 32) * p.args.n_heads * p.args.B <= gemm_num_sms();
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
