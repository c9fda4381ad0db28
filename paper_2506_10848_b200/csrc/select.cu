// The transition rule S of one denoising step, on the device: the SlowFast rule (paper Section 3.3, Algorithm 1) or one of
// the LLaDA strategies of Section 3.1 (low-confidence / random remasking, optionally block by block).
// One CTA per sequence (with two-pass statistics a group of them, of which the last to finish goes on alone) reads the row
// statistics scattered by token position, applies the exploratory (slow) or accelerated (fast) rule, unmasks the chosen
// positions in place, advances the per-sequence state (k, s_cycle, e_cycle, H_W, phase) and lists the rows the next step needs.
// The last CTA to finish concatenates the per-sequence row lists (sequence-major, positions ascending) so that the next forward
// pass gets one deterministic row list without a host round trip.
#include "sfs_common.cuh"
#include "canonical.cuh"
#include "tc05.cuh"

namespace sfs {
namespace {

constexpr int kSelThreads = 256;
constexpr unsigned long long kNoKey = ~0ull;
constexpr int kGoesOn = 1 << 30;             // beside a sequence's row count: its next step will hardly be its last
constexpr int kMostCluster = 8;               // sequences whose CTAs are one cluster at most
constexpr int kPosBits = 17;                 // key = S_q << 17 | position  (S_q < 2^47, position < 2^17)

struct BlockRed {
    int n_cand, n_high, max_above, min_cand, n_masked, missing;      // (counts: at most 22755, see select_fits)
    unsigned long long kmin;                                // smallest key
};

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
    const uint32_t hi = __reduce_min_sync(0xffffffffu, (uint32_t)(v >> 32));
    const uint32_t lo = __reduce_min_sync(0xffffffffu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : ~0u);
    return (unsigned long long)hi << 32 | lo;
}

// One barrier: each warp leaves its result, then every warp reduces the eight of them.  The chain of these block-wide steps is what
// bounds a selection, so counts travel in pairs and minima of 64 bits as two instructions (ten shuffles before); the caller gives
// each reduction tables of its own.
constexpr int kSelWarps = kSelThreads / 32;
__device__ BlockRed block_reduce(BlockRed v, int4 *s_int /* [8] */, unsigned long long *s_min /* [8] */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int4 e = make_int4(warp_sum_i32(v.n_cand | v.n_high << 16), warp_sum_i32(v.n_masked | v.missing << 16), warp_max_i32(v.max_above), warp_min_i32(v.min_cand));
    v.kmin = warp_min_u64(v.kmin);
    if (lane == 0) { s_int[warp] = e; s_min[warp] = v.kmin; }
    __syncthreads();
    e = s_int[lane & (kSelWarps - 1)];
    const bool mine = lane < kSelWarps;                     // (maxima and minima do not mind the copies)
    const int a = warp_sum_i32(mine ? e.x : 0), b = warp_sum_i32(mine ? e.y : 0);
    return BlockRed{a & 0xFFFF, a >> 16, warp_max_i32(e.z), warp_min_i32(e.w), b & 0xFFFF, b >> 16, warp_min_u64(s_min[lane & (kSelWarps - 1)])};
}
// count (two of 16 bits at most) of all warps, and of those before this one; one barrier, the caller alternates between tables
__device__ __forceinline__ int block_count(int warp_count, int *s_cnt /* [8] */, int *before) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) s_cnt[warp] = warp_count;
    __syncthreads();
    const int c = lane < kSelWarps ? s_cnt[lane] : 0;
    if (before) *before = warp_sum_i32(lane < warp ? c : 0);
    return warp_sum_i32(c);
}

enum { MODE_ALL = 0, MODE_TOPK = 1, MODE_HIGH = 2, MODE_RANDOM = 3 };

// Philox-4x32-10 (Salmon et al., SC'11): ten rounds of multiply / xor on a 128-bit counter under a 64-bit key; the first
// output word is returned.  Random remasking draws one word per (position, step, sequence).
__device__ __forceinline__ uint32_t philox_first_word(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t h0 = __umulhi(0xD2511F53u, c0), l0 = 0xD2511F53u * c0;
        const uint32_t h1 = __umulhi(0xCD9E8D57u, c2), l1 = 0xCD9E8D57u * c2;
        c0 = h1 ^ c1 ^ k0; c1 = l1; c2 = h0 ^ c3 ^ k1; c3 = l0;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    return c0;
}

// what the whole step leaves: the size of the next row list, the number of sequences still decoding and, in a generation, the
// host's mirror of it (host_active[0]: sequences still decoding; host_active[1]: denoising steps finished; one 8-byte write, so
// that who sees the step sees whether it was the last, without a system-wide fence between two; kMayEnd is set in the step count when
// the next step may well be the last, and the host then waits for it instead of enqueueing another one behind it)
__device__ __forceinline__ void finish_step(const SelectArgs &a, int n_next, int n_active, int steps_before, bool may_end)
{
    if (a.next_n_rows) *a.next_n_rows = n_next;
    if (a.n_active) *a.n_active = n_active;
    if (a.host_active) {
        *reinterpret_cast<volatile unsigned long long *>(a.host_active) = (unsigned long long)(uint32_t)n_active | (unsigned long long)(uint32_t)((steps_before + 1) | (may_end ? kMayEnd : 0)) << 32;
        *a.step_count = steps_before + 1;
    }
}

// flags of a response position
enum { F_MASKED = 1, F_HIGH = 2, F_SEL = 4, F_OPEN = 8 };

// Which candidate rows of a step must be recomputed canonically (two-pass statistics): flags them F_OPEN and lists their logits
// rows, in position order, in s_list; returns how many.  Every other candidate row's enclosure [lo, hi] answers what the step's
// rule asks, and its lower bound stands for it:
//   * a row whose enclosure is one value is never open;
//   * a threshold is open when lo and hi fall on different sides of it;
//   * the ranking (k most confident candidates, smallest S_q first) is open for every candidate whose lo does not exceed
//     U = the k-th smallest hi among the candidates: the k rows with the smallest hi all have S_q <= U, so a row with
//     lo > U is not among the k most confident, and its lower bound (still > U) orders it behind them.  Only k = 1 is
//     evaluated this way (U = the smallest hi); for k > 1 every candidate is recomputed.
// Positions go to s_list, their logits rows to s_row.  m0 / lo0 / hi0 / row0: mask, enclosure and row of position threadIdx.x, loaded
// by the caller beside the state.
__device__ int list_open_rows(const SelectArgs &a, const sfs_state &st, int b, uint8_t m0, unsigned long long lo0, unsigned long long hi0, int32_t row0, uint8_t *s_fl,
                              int32_t *s_list, int32_t *s_row, int4 *s_int, unsigned long long *s_min, int (*s_cnt)[kSelWarps])
{
    const int tid = threadIdx.x, lane = tid & 31, L = a.L;
    const StepAsk ask = step_ask(a.params, st, L);
    const long long base = (long long)b * a.S + a.P;
    const uint8_t *msk = a.mask + base;
    const unsigned long long *plo = a.pos_lo + base, *phi = a.pos_hi + base;
    int k_top = 0;
    unsigned long long U = ~0ull;
    if (ask.rank_needed) {
        BlockRed r{0, 0, -1, 0x7FFFFFFF, 0, 0, ~0ull};
        for (int i = tid; i < ask.hi && i < L; i += kSelThreads) {
            const bool first = i == tid;
            if (i < ask.lo || !(first ? m0 : msk[i])) continue;
            r.n_cand++;
            if ((first ? lo0 : plo[i]) != 0) r.kmin = min(r.kmin, first ? hi0 : phi[i]);
        }
        r = block_reduce(r, s_int, s_min);
        U = r.kmin;
        if (a.params.sampler == SFS_SAMPLER_LOW_CONFIDENCE) {
            const BlockStep blk = block_step(a.params, L, st.steps_done);
            const long long Lb = ask.hi - ask.lo, Nb = blk.steps_per_block;
            k_top = (int)max(0ll, (Lb * (Nb - blk.k_b + 1)) / Nb - (Lb - r.n_cand));
        } else {
            k_top = (st.phase == SFS_PHASE_SLOW) ? a.params.k_slow : a.params.k_fast;
        }
        if (k_top >= r.n_cand) k_top = 0;                   // everything is chosen: no ranking
    }
    int n_open = 0;
    for (int i0 = 0; i0 < L; i0 += kSelThreads) {
        const int i = i0 + tid;
        bool open = false;
        if (i >= ask.lo && i < ask.hi && i < L && (i0 == 0 ? m0 : msk[i])) {
            const unsigned long long lo = i0 == 0 ? lo0 : plo[i], hi = i0 == 0 ? hi0 : phi[i];
            if (lo != 0 && lo != hi) {                      // 0: no row supplied for this candidate
                if (ask.tau > 0.f) open = conf_exceeds(lo, ask.tau) && !conf_exceeds(hi, ask.tau);
                if (k_top > 1) open = true;
                else if (k_top == 1) open = open || lo <= U;
            }
        }
        const unsigned bal = __ballot_sync(0xffffffffu, open);
        int before;
        const int total = block_count(__popc(bal), s_cnt[(i0 / kSelThreads) & 1], &before);
        if (i < L) s_fl[i] = open ? F_OPEN : 0;
        if (open) {
            const int at = n_open + before + __popc(bal & ((1u << lane) - 1u));
            s_list[at] = i; s_row[at] = i0 == 0 ? row0 : __ldcg(&a.pos_row[base + i]);
        }
        n_open += total;
    }
    __syncthreads();
    return n_open;
}

// One step of the transition rule.  `groups` CTAs per sequence: with two-pass row statistics (pos_lo given) every one of them
// first lists the rows whose enclosure leaves the step's question open (the same list in each), they share the canonical
// recomputation of those rows, warp by warp, adding integer partial sums to pos_sq, and the CTA that finishes last (a ticket)
// goes on alone.  So the list, the recomputation and the choice are one launch: on 256 rows of 126464 logits the three kernels
// they were took 6 + 9 + 11 us of a 45 us sfs_select call; DRAM has no part in it, the chain of block-wide steps bounds it.
// Without two-pass statistics there is one CTA per sequence; those of up to eight sequences are a cluster (CLUSTER), whose CTAs tell
// each other the lengths of their row lists instead of leaving them to the last one (2 sequences: 3500 of 9200 clocks).
// State that follows from the step is worked out by every thread, from the same values: no thread waits for another's arithmetic.
// dynamic shared memory: keys u64[L] (before: the list of open rows and their logits rows; after: the next step's rows) | flags u8[L]
template <bool CLUSTER>
__global__ void __launch_bounds__(kSelThreads) select_kernel(SelectArgs a)
{
    extern __shared__ unsigned long long s_keys[];
    const int L = a.L, S = a.S, P = a.P, b = CLUSTER ? blockIdx.x : blockIdx.x / a.groups, part = CLUSTER ? 0 : blockIdx.x - b * a.groups;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint8_t *s_fl = reinterpret_cast<uint8_t *>(s_keys + L);
    __shared__ int4 s_int[2][kSelWarps];
    __shared__ unsigned long long s_min[2][kSelWarps];
    __shared__ int s_cnt[4][kSelWarps];
    __shared__ sfs_state st;
    __shared__ int s_last;
    __shared__ int2 s_seq[kMostCluster];                    // CLUSTER: (rows and flag, still decoding) of every sequence

    const long long base = (long long)b * S + P;
    int32_t *tok = a.tokens + base;
    uint8_t *msk = a.mask + base;
    unsigned long long *psq = a.pos_sq + base;
    const int32_t *parg = a.pos_arg + base;
    const sfs_params &p = a.params;
    const bool two_pass = !CLUSTER && a.pos_lo != nullptr, vanilla = p.sampler != SFS_SAMPLER_SLOWFAST;

    if (CLUSTER) tc::cluster_arrive();      // this CTA runs
    pdl_wait();
    pdl_trigger();
    const int steps_before = tid == 0 && a.step_count ? *a.step_count : 0;      // (of the whole generation)
    // the state and everything about position tid (all of a sequence, usually) in one round trip
    uint8_t m0 = 0;
    int32_t arg0 = 0, row0 = 0;
    unsigned long long lo0 = 0, hi0 = 0;                    // two-pass: the enclosure; else lo0 = S_q
    if (tid < L) {
        m0 = msk[tid]; arg0 = parg[tid];
        if (two_pass) { lo0 = __ldcg(&a.pos_lo[base + tid]); hi0 = a.pos_hi[base + tid]; row0 = __ldcg(&a.pos_row[base + tid]); }
        else lo0 = psq[tid];
    }
    if (tid < (int)(sizeof(sfs_state) / 4)) reinterpret_cast<int *>(&st)[tid] = reinterpret_cast<const int *>(a.state + b)[tid];
    __syncthreads();

    const bool active = !st.done && st.status == SFS_OK;
    const int phase0 = st.phase, s0 = st.s_cycle, hi_fast = st.hi, steps0 = st.steps_done;
    const bool forced = !vanilla && (st.k_remaining == 1);
    if (a.groups > 1 && !active && part != 0) return;
    if (two_pass && active) {
        int32_t *s_list = reinterpret_cast<int32_t *>(s_keys), *s_row = s_list + L;
        const int n_open = list_open_rows(a, st, b, m0, lo0, hi0, row0, s_fl, s_list, s_row, s_int[0], s_min[0], s_cnt);
        recompute_rows(a.lrows, s_list, s_row, n_open, a.pos_max + base, psq, part * kSelWarps + warp, a.groups * kSelWarps);
        if (a.groups > 1) {
            __syncthreads();
            if (tid == 0) {                                 // (releases the whole CTA's sums, and acquires the others')
                int before;
                asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(before) : "l"(&a.seq_ticket[b]) : "memory");
                s_last = before == a.groups - 1 ? 1 : 0;
                if (s_last) a.seq_ticket[b] = 0;
            }
            __syncthreads();
            if (!s_last) return;
        } else {
            __threadfence();
            __syncthreads();
        }
    }

    int n_sel = 0, e_cand = -1, stable = 0, n_sure = 0;    // n_sure: candidates above the high threshold
    int rec_phase = phase0, rec_s = s0;
    int rec_hi = (phase0 == SFS_PHASE_SLOW) ? L : hi_fast;
    // the state after this step (of the history only its length)
    int phase1 = phase0, s1 = s0, hi1 = hi_fast, count1 = st.step_count, hist1 = st.hist_len, k1 = st.k_remaining, masked1 = st.n_masked, done1 = st.done, status1 = st.status;
    const int hist0 = hist1;
    bool stepped = false, slow_step = false, fell_back = false, new_cycle = false;
    BlockStep blk{};
    if (vanilla) { blk = block_step(p, L, steps0); rec_phase = blk.j; rec_s = blk.lo; rec_hi = blk.hi; e_cand = blk.k_b; }

    if (active) {
        const int lo = vanilla ? blk.lo : (forced ? 0 : s0);
        const int hi = vanilla ? blk.hi : (forced ? L : ((phase0 == SFS_PHASE_SLOW) ? L : hi_fast));

        // ---- candidates of this step and their statistics (consumed: a later step must bring its own)
        BlockRed r{0, 0, -1, 0x7FFFFFFF, 0, 0, kNoKey};
        for (int i = tid; i < L; i += kSelThreads) {
            const bool m = (i == tid ? m0 : msk[i]) != 0;
            const bool cand = m && i >= lo && i < hi;
            unsigned long long key = kNoKey, sq;
            if (two_pass) {
                if (s_fl[i] & F_OPEN) sq = __ldcg(&psq[i]);
                else sq = i == tid ? lo0 : __ldcg(&a.pos_lo[base + i]);
                a.pos_lo[base + i] = 0;
            } else {
                sq = i == tid ? lo0 : psq[i];
            }
            psq[i] = 0;
            uint8_t fl = m ? F_MASKED : 0;
            if (cand) {
                if (sq == 0) r.missing++;
                key = (sq << kPosBits) | (unsigned long long)i;
                r.n_cand++;
                r.min_cand = min(r.min_cand, i);
                if (conf_exceeds(sq, p.tau_min_conf)) r.max_above = max(r.max_above, i);
                if (conf_exceeds(sq, p.tau_high_conf)) { fl |= F_HIGH; r.n_high++; }
            }
            r.kmin = min(r.kmin, key);
            r.n_masked += m ? 1 : 0;
            s_keys[i] = key; s_fl[i] = fl;
        }
        r = block_reduce(r, s_int[1], s_min[1]);
        n_sure = r.n_high;

        if (r.missing > 0 || (r.n_cand == 0 && !vanilla)) {
            status1 = SFS_ERR_MISSING_ROW;                  // a needed row was not supplied (or the state is inconsistent): report, change nothing
        } else {
            int mode, k_top = 0;
            if (p.sampler == SFS_SAMPLER_LOW_CONFIDENCE) {
                // Section 3.1: after this step floor(L_b (1 - (k_b - 1) / N_b)) positions of the block are unmasked
                const long long Lb = hi - lo, Nb = blk.steps_per_block;
                const long long target = (Lb * (Nb - blk.k_b + 1)) / Nb;
                mode = MODE_TOPK; k_top = (int)max(0ll, target - (Lb - r.n_cand));
            } else if (p.sampler == SFS_SAMPLER_RANDOM) mode = MODE_RANDOM;
            else if (forced) mode = MODE_ALL;
            else if (phase0 == SFS_PHASE_SLOW) { mode = MODE_TOPK; k_top = p.k_slow; }
            else if (r.n_high >= p.min_high_count) mode = MODE_HIGH;
            else { mode = MODE_TOPK; k_top = p.k_fast; }

            // ---- scheduler state (Algorithm 1): what does not depend on the choice
            stepped = true;
            k1 = forced ? 0 : k1 - 1;
            if (!vanilla && !forced && phase0 == SFS_PHASE_SLOW) {
                slow_step = true;
                e_cand = (r.max_above >= 0) ? r.max_above : r.min_cand;
                const bool full = hist0 >= p.w_hist;        // the history with e_cand in it: appended, or the oldest dropped
                hist1 = full ? hist0 : hist0 + 1;
                int sum = 0;                                              // (at most 8 positions below 2^17)
                long long sum2 = 0;
                for (int h = 0; h < hist1; ++h) {
                    const int e = full ? (h < p.w_hist - 1 ? st.hist[h + 1] : (h == p.w_hist - 1 ? e_cand : st.hist[h])) : (h < hist0 ? st.hist[h] : e_cand);
                    sum += e; sum2 += (long long)e * e;
                }
                count1++;
                const int n = hist1;
                const long long num = n * sum2 - (long long)sum * sum;               // n^2 * population variance, exact
                if (n >= p.w_hist && (double)num < (double)p.sigma2_stable * (double)((long long)n * n)) {
                    stable = 1;
                    phase1 = SFS_PHASE_FAST; hi1 = sum / n + 1;       // floor(mean(H_W)) + 1
                } else if (count1 >= p.k_max) {
                    phase1 = SFS_PHASE_FAST; hi1 = e_cand + 1;
                }
            } else if (!vanilla && !forced) fell_back = mode == MODE_TOPK;
            // is the span clean after this step?  (decides whether the next cycle starts)
            const bool span = !vanilla && !forced && phase1 == SFS_PHASE_FAST;

            // ---- choose
            const bool ranked = mode == MODE_TOPK && k_top > 1 && k_top < r.n_cand;      // (one or all: no ranking)
            int my_sel = 0, my_left = 0;
            for (int i = tid; i < L; i += kSelThreads) {
                const unsigned long long key = s_keys[i];
                uint8_t fl = s_fl[i];
                bool sel = false;
                if (key != kNoKey) {
                    if (mode == MODE_ALL) sel = true;
                    else if (mode == MODE_HIGH) sel = (fl & F_HIGH) != 0;
                    else if (mode == MODE_RANDOM)
                        sel = (unsigned long long)philox_first_word((uint32_t)i, (uint32_t)steps0, (uint32_t)b, 0u, p.seed_lo, p.seed_hi)
                              * (unsigned long long)blk.k_b < (1ull << 32);
                    else if (k_top == 1) sel = key == r.kmin;
                    else if (!ranked) sel = k_top > 0;
                    else {
                        int rank = 0;                           // candidates that are more confident (ties: smaller position)
                        for (int j = 0; j < L; ++j) rank += (s_keys[j] < key) ? 1 : 0;
                        sel = rank < k_top;
                    }
                }
                if (sel) { fl = (uint8_t)((fl | F_SEL) & ~F_MASKED); s_fl[i] = fl; my_sel++; tok[i] = i == tid ? arg0 : parg[i]; msk[i] = 0; }
                if ((fl & F_MASKED) && i >= s0 && i < hi1) my_left++;
            }
            const int chosen = block_count(warp_sum_i32(my_sel | my_left << 16), s_cnt[2], nullptr), left = chosen >> 16;
            n_sel = chosen & 0xFFFF;
            masked1 = r.n_masked - n_sel;
            if (span && left == 0 && masked1 > 0) { new_cycle = true; s1 = hi1; phase1 = SFS_PHASE_SLOW; hist1 = 0; count1 = 0; }
            if (masked1 == 0 || k1 == 0) { done1 = 1; if (masked1 > 0) status1 = SFS_ERR_STEP_LIMIT; }
        }
    } else {
        // a finished (or stopped) sequence consumes the statistics supplied for it as well: nothing stale is left for a
        // later generation that reuses the scratch
        for (int i = tid; i < L; i += kSelThreads) { s_fl[i] = 0; psq[i] = 0; if (two_pass) a.pos_lo[base + i] = 0; }
    }

    // ---- ordered outputs (ballots and per-warp counts): selected positions, and the rows of the next step
    const bool next_active = !done1 && status1 == SFS_OK;
    // a single sequence's list is the whole list; a cluster's wait in shared memory for their place (the keys
    // have been ranked: the counts' barrier lies between)
    int32_t *const next = CLUSTER ? reinterpret_cast<int32_t *>(s_keys) : (a.B == 1 ? a.next_rows : a.seq_rows + (long long)b * L);
    int n_out = 0, n_next = 0;
    {
        const bool nforced = !vanilla && k1 == 1;
        BlockStep nblk{};
        if (vanilla) nblk = block_step(p, L, steps0 + (stepped ? 1 : 0));
        const int nlo = vanilla ? nblk.lo : (nforced ? 0 : s1);
        const int nhi = vanilla ? nblk.hi : (nforced ? L : ((phase1 == SFS_PHASE_SLOW) ? L : hi1));
        for (int i0 = 0; i0 < L; i0 += kSelThreads) {
            const int i = i0 + tid;
            const uint8_t fl = i < L ? s_fl[i] : 0;
            const bool sel = (fl & F_SEL) != 0, need = next_active && (fl & F_MASKED) && i >= nlo && i < nhi;
            const unsigned bs = __ballot_sync(0xffffffffu, sel), bn = __ballot_sync(0xffffffffu, need);
            int before;
            const int total = block_count(__popc(bs) | (__popc(bn) << 16), s_cnt[(i0 / kSelThreads) & 1], &before);
            const unsigned lt = (1u << lane) - 1u;
            if (sel && a.sel_pos) {
                const int o = n_out + (before & 0xFFFF) + __popc(bs & lt);
                a.sel_pos[(long long)b * L + o] = i;
                a.sel_tok[(long long)b * L + o] = i == tid ? arg0 : parg[i];
            }
            if (need && next) next[n_next + (before >> 16) + __popc(bn & lt)] = b * S + P + i;
            n_out += total & 0xFFFF; n_next += total >> 16;
        }
    }
    // May the next step finish the sequence?  It does when the budget ends.  Before that (SlowFast) its rows must be all that
    // is masked, and no more than its ranking unmasks or, in the fast phase, twice what has just been unmasked or was sure.
    const int reach = phase1 == SFS_PHASE_SLOW ? p.k_slow : max(p.k_fast, 2 * max(n_sel, n_sure));
    const bool may_end = k1 <= 1 || (!vanilla && n_next == masked1 && reach >= masked1);
    const bool goes_on = next_active && !may_end;
    const int2 seq = make_int2(n_next | (goes_on ? kGoesOn : 0), next_active ? 1 : 0);
    if (tid == 0) {
        if (a.sel_count) a.sel_count[b] = n_out;
        if (!CLUSTER) a.seq_row_count[b] = seq.x;
        if (a.trace) {
            int32_t *t = a.trace + (long long)b * SFS_TRACE_INTS;
            t[0] = rec_phase; t[1] = rec_s; t[2] = rec_hi; t[3] = e_cand; t[4] = stable; t[5] = n_sel;
            t[6] = masked1; t[7] = k1;
        }
        if (a.B == 1) finish_step(a, n_next, next_active ? 1 : 0, steps_before, !goes_on);
        if (slow_step) {                                    // (nobody reads the old history any more: a barrier lies behind the choice)
            if (hist0 < p.w_hist) st.hist[hist0] = e_cand;
            else { for (int h = 1; h < p.w_hist; ++h) st.hist[h - 1] = st.hist[h]; st.hist[p.w_hist - 1] = e_cand; }
            st.n_slow++;
        } else if (stepped && !vanilla && !forced) st.n_fast++;
        st.phase = phase1; st.s_cycle = s1; st.hi = hi1; st.step_count = count1; st.hist_len = hist1; st.k_remaining = k1; st.n_masked = masked1;
        st.steps_done = steps0 + (stepped ? 1 : 0); st.n_cycles += new_cycle ? 1 : 0; st.n_fallback += fell_back ? 1 : 0; st.done = done1; st.status = status1;
    }
    __syncwarp();
    if (tid < (int)(sizeof(sfs_state) / 4)) reinterpret_cast<int *>(a.state + b)[tid] = reinterpret_cast<const int *>(&st)[tid];
    if (CLUSTER) {
        // every sequence its numbers to all, then its rows to their place (sequence-major)
        tc::cluster_wait();                                 // all run
        if (tid < a.B) {
            const uint32_t at = tc::mapa(tc::smem_u32(&s_seq[b]), (uint32_t)tid);
            asm volatile("st.shared::cluster.v2.b32 [%0], {%1, %2};" ::"r"(at), "r"(seq.x), "r"(seq.y) : "memory");
        }
        tc::cluster_sync();
        const int2 o = lane < a.B ? s_seq[lane] : make_int2(0, 0);
        const int c = o.x & ~kGoesOn, off = warp_sum_i32(lane < b ? c : 0), all = warp_sum_i32(c), act = warp_sum_i32(o.y);
        const bool on = __any_sync(0xffffffffu, (o.x & kGoesOn) != 0);
        if (a.next_rows) for (int i = tid; i < n_next; i += kSelThreads) a.next_rows[off + i] = next[i];
        if (b == 0 && tid == 0) finish_step(a, all, act, steps_before, !on);
        return;
    }
    if (a.B == 1) return;

    // ---- last sequence: concatenate the row lists, count the active sequences
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(a.ticket, 1) == a.B - 1) ? 1 : 0;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    int off = 0, act = 0, on = 0;
    for (int q0 = 0; q0 < a.B; q0 += 32) {                  // every warp: offsets of 32 sequences; then each warp copies every 8th list
        const int q = q0 + lane;
        const int cw = q < a.B ? __ldcg(&a.seq_row_count[q]) : 0, c = cw & ~kGoesOn;
        on |= cw & kGoesOn;
        act += (q < a.B && __ldcg(&a.state[q].done) == 0 && __ldcg(&a.state[q].status) == SFS_OK) ? 1 : 0;
        int pre = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, pre, o); if (lane >= o) pre += t; }
        for (int k = warp; k < 32 && q0 + k < a.B; k += kSelWarps) {
            const int ck = __shfl_sync(0xffffffffu, c, k), ok = off + __shfl_sync(0xffffffffu, pre, k) - ck;
            if (a.next_rows)
                for (int i = lane; i < ck; i += 32) a.next_rows[ok + i] = __ldcg(&a.seq_rows[(long long)(q0 + k) * L + i]);
        }
        off += __shfl_sync(0xffffffffu, pre, 31);
    }
    act = warp_sum_i32(act);
    on = __any_sync(0xffffffffu, on != 0);
    if (tid == 0) {
        finish_step(a, off, act, steps_before, !on);
        *a.ticket = 0;
    }
}

__global__ void state_init_kernel(sfs_state *state, int B, int L, sfs_params p)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    state[b] = initial_state(L, p.max_steps);
}

}  // namespace

static size_t select_shared(int32_t L) { return (size_t)L * (sizeof(unsigned long long) + 1); }
int32_t select_fits(int32_t L)
{
    SFS_REQUIRE(select_shared(L) <= 200 * 1024, SFS_ERR_UNSUPPORTED, "gen_len %d too long for the selection kernel", L);
    return SFS_OK;
}

int32_t launch_select(const SelectArgs &args, cudaStream_t stream)
{
    SelectArgs a = args;
    const size_t smem = select_shared(a.L);
    const int32_t rc = select_fits(a.L);
    if (rc != SFS_OK) return rc;
    // two-pass statistics: two CTAs per SM over all sequences share the recomputation (k > 1 can ask for every row)
    a.groups = 1;
    if (a.pos_lo != nullptr) a.groups = a.B < 148 ? 296 / a.B : 1;
    else if (a.B > 1 && a.B <= kMostCluster) {
        SFS_CUDA(allow_shared(select_kernel<true>, smem));
        SFS_CUDA(launch_pdl_cluster(select_kernel<true>, a.B, dim3((unsigned)a.B), dim3(kSelThreads), smem, stream, a));
        return SFS_OK;
    }
    SFS_CUDA(allow_shared(select_kernel<false>, smem));
    SFS_CUDA(launch_pdl(select_kernel<false>, dim3((unsigned)(a.B * a.groups)), dim3((unsigned)(kSelThreads)), (size_t)(smem), stream, a));
    return SFS_OK;
}

int32_t launch_state_init(sfs_state *d_state, int32_t B, int32_t L, const sfs_params &p, cudaStream_t stream)
{
    state_init_kernel<<<(B + 63) / 64, 64, 0, stream>>>(d_state, B, L, p);
    SFS_LAUNCH_CHECK();
    return SFS_OK;
}

}  // namespace sfs
