// Acceptance / freeze update of one denoising step: one CTA per sequence.
// Section 4.1 of the paper: confidence ratio (Eq. 4), spatial weight over a window of radius D (Eq. 5),
// softening factor (Eq. 6), adaptive threshold (Eq. 7), early-exit test (Eq. 8); then the transfer
// schedule (k highest max-probability candidates), the logical OR of both masks, and the write of
// the argmax token into every chosen position (Algorithm 1).
#pragma once
#include <cuda_runtime.h>
#include <limits.h>
#include <stdint.h>

#include "pdl.cuh"

namespace jot {

constexpr int kAcceptThreads = 256;
constexpr int kMaxD = 32;

struct AcceptParamsDev {     // mirrors jot_params
    float tau_max, tau_min, gamma;
    int32_t D;
    float eps;
    int32_t schedule_after_exit;
    int32_t gate;                // 0: ratio r >= tau (Eq. 8); 1: fixed probability gate p1 >= prob_threshold;
    float prob_threshold;        // 2: global early commit, mean top-2 logit gap of the candidates >= gap_threshold
    float gap_threshold;
    int32_t schedule;            // 0: fixed per-block table; 1: ceil(still masked / steps the block has left)
};

// Per-sequence loop state used by the generate loop (device resident).
struct SeqState {
    int32_t blk;          // current semi-autoregressive block
    int32_t s;            // step inside the block
    int32_t steps_used;   // denoising steps this sequence has run
    int32_t n_masked;     // candidates still masked in the current block after the last update
};

struct AcceptArgs {
    AcceptParamsDev uniform;         // used when params == nullptr
    const AcceptParamsDev* params;   // device: 1 or B entries (nullable)
    int per_seq_params;
    int32_t mask_id;
    int32_t* tokens;                 // [B, L], updated in place
    int B, L;
    int blk_lo, blk_hi, k_transfer;  // used when state == nullptr
    const float* top1;
    const float* top2;
    const float* sumexp;
    const int32_t* argmax;
    int32_t* n_masked;               // [B] nullable
    uint8_t* exit_reason;            // [B, L] nullable
    int16_t* exit_step;              // [B, L] nullable
    int step_index;
    // generate mode: block pointer / step per sequence, schedule table from (block_len, steps_per_block)
    SeqState* state;                 // [B] nullable
    int P, block_len, n_blocks, steps_per_block;
    int32_t* n_unfinished;           // device counter: += 1 per sequence that still has work (nullable)
    int lockstep;                    // generate mode under a block-wise KV cache: every sequence works on the block
                                     // [blk_lo, blk_hi) with k_transfer; the host moves all of them on together
    int lockstep_s;                  // ... and this is the block's step index (the fractional schedule needs it)
    // generate mode, optional trace (Appendix "Confidence Dynamics"): row = the sequence's own 0-based step
    float* mean_ratio;               // [steps, B]: mean of r over the step's candidates
    int32_t* n_candidates;           // [steps, B]
};

// Per-sequence parameter sets handed over as kernel arguments (the single-step entry point has no device
// memory of its own to put them in): at most this many sequences per launch.
constexpr int kAcceptInlineParams = 64;
struct AcceptParamsInline {
    AcceptParamsDev p[kAcceptInlineParams];
};
struct AcceptParamsNone {};

template <bool INLINE> struct AcceptInlineArg { using type = AcceptParamsNone; };
template <> struct AcceptInlineArg<true> { using type = AcceptParamsInline; };

__device__ __forceinline__ AcceptParamsDev accept_pick_params(const AcceptArgs& a, const AcceptParamsInline& inl, int b) {
    return inl.p[b];
}
__device__ __forceinline__ AcceptParamsDev accept_pick_params(const AcceptArgs& a, const AcceptParamsNone&, int b) {
    return a.params ? a.params[a.per_seq_params ? b : 0] : a.uniform;
}

// The kernel is a chain of memory round trips and barriers over a few hundred numbers, so it is kept short: everything a
// decision reads is requested before the canvas has arrived, thread t looks after position lo + t of the block, and the ranks
// are counted by all threads together.  What is ranked stands in a list of its own: a long block with few positions left must
// not pay for the ones that are decided.  Call after call in a graph, with 5 % / all of the positions masked: 2.8 / 2.8 us for a
// block of 32 in a canvas of 384, 3.8 / 11.3 for 512 in 704, 31 / 1937 for 8192 (comparing with every position of the block: 3.9 /
// 3.9, 16 / 16, 2281 / 2675).
// Dynamic shared memory: resolved bitmap words; the list of (sum-exp, position) to rank; per position of the block its flags.
template <bool INLINE>
__global__ void __launch_bounds__(kAcceptThreads)
accept_freeze_kernel(const AcceptArgs a, const __grid_constant__ typename AcceptInlineArg<INLINE>::type inl) {
    extern __shared__ uint32_t sh[];
    grid_launch_dependents();
    grid_dependency_wait();
    const int L = a.L, b = blockIdx.x, tid = threadIdx.x;
    const int n_words = (L + 31) / 32;
    uint32_t* res_bits = sh;                                   // [n_words + 2] resolved bitmap (padded)
    const int L4 = (L + 3) & ~3;
    uint64_t* keys = reinterpret_cast<uint64_t*>(sh + ((n_words + 2 + 3) & ~3));  // [L4] 16-byte aligned, in any order
    uint8_t* flag = reinterpret_cast<uint8_t*>(keys + L4);                        // [L4] bit0 exit, bit1 schedule, bit2 ranks first
    __shared__ float gpow[kMaxD + 1];
    __shared__ int rank[kAcceptThreads];                       // of the positions of a block no longer than this
    __shared__ uint32_t counts_sh;                             // entries of the list; candidates in the upper half (both below 2^15)
    __shared__ int n_final_sh;
    __shared__ float inv_wmax;
    __shared__ float ratio_sums[kAcceptThreads / 32], gap_sums[kAcceptThreads / 32];

    const AcceptParamsDev prm = accept_pick_params(a, inl, b);
    int32_t* x = a.tokens + (size_t)b * L;

    int lo = a.blk_lo, hi = a.blk_hi, k = a.k_transfer;
    SeqState st = {0, 0, 0, 0};
    if (a.state) st = a.state[b];
    if (a.state && !a.lockstep) {
        if (st.blk >= a.n_blocks) return;                      // finished sequence idles (uniform exit)
        lo = a.P + st.blk * a.block_len;
        hi = lo + a.block_len;
        int base = a.block_len / a.steps_per_block, rem = a.block_len % a.steps_per_block;
        k = base + (st.s < rem ? 1 : 0);
    }

    const int n_pos = hi - lo;
    const size_t row = (size_t)b * L;
    // the first 256 positions' statistics and the first part of the canvas are on their way together
    float m1_0 = 0.f, m2_0 = 0.f, S_0 = 0.f;
    int32_t arg_0 = 0;
    if (tid < n_pos) {
        m1_0 = a.top1[row + lo + tid];
        m2_0 = a.top2[row + lo + tid];
        S_0 = a.sumexp[row + lo + tid];
        arg_0 = a.argmax[row + lo + tid];
    }
    constexpr int AHEAD = 3;
    int32_t x_0[AHEAD];
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
        const int i = k * kAcceptThreads + tid;
        x_0[k] = i < L ? x[i] : a.mask_id;
    }
    if (tid == 0) {
        // gamma^d by repeated multiplication, and w_max = 2 * sum_{d=1..D} gamma^d  (Eq. 6)
        float g = 1.f, sum = 0.f;
        gpow[0] = 0.f;
        for (int d = 1; d <= prm.D; ++d) {
            g *= prm.gamma;
            gpow[d] = g;
            sum += g;
        }
        inv_wmax = 1.f / (2.f * sum);
        counts_sh = 0;
        n_final_sh = 0;
    }
    for (int w = n_words + tid; w < n_words + 2; w += blockDim.x) res_bits[w] = 0;
    // resolved bitmap: bit i set iff x_i != mask_id (prompt tokens count as resolved)
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
        const int i = k * kAcceptThreads + tid;
        const uint32_t bal = __ballot_sync(0xffffffffu, i < L && x_0[k] != a.mask_id);
        if ((tid & 31) == 0 && (i >> 5) < n_words) res_bits[i >> 5] = bal;
    }
    for (int base = AHEAD * kAcceptThreads; base < L; base += kAcceptThreads) {
        const int i = base + tid;
        const uint32_t bal = __ballot_sync(0xffffffffu, i < L && x[i] != a.mask_id);
        if ((tid & 31) == 0 && (i >> 5) < n_words) res_bits[i >> 5] = bal;
    }
    __syncthreads();

    // per candidate (masked position of the block): ratio, threshold, early-exit decision
    float r_sum = 0.f, gap_sum = 0.f;
    float m1_next = m1_0, m2_next = m2_0, S_next = S_0;
    for (int base = 0; base < n_pos; base += kAcceptThreads) {
        const int c = base + tid, i = lo + c;
        const float m1 = m1_next, m2 = m2_next, S = S_next;
        if (c + kAcceptThreads < n_pos) {                      // the next 256 positions' statistics are on their way meanwhile
            m1_next = a.top1[row + i + kAcceptThreads];
            m2_next = a.top2[row + i + kAcceptThreads];
            S_next = a.sumexp[row + i + kAcceptThreads];
        }
        const bool cand = c < n_pos && !((res_bits[i >> 5] >> (i & 31)) & 1u);
        bool listed = false;
        uint8_t f = 0;
        if (cand) {
            // Eq. 4 with p1 = 1/S, p2 = exp(m2 - m1)/S:  r = 1 / (exp(m2 - m1) + eps * S)
            const float r = 1.f / (expf(m2 - m1) + prm.eps * S);
            // Eq. 5: resolved neighbours at distance 1..D <= 32 on both sides, 32 bits of the bitmap each (zero past its ends)
            const int iw = i >> 5, rw = (i + 1) >> 5;
            const uint32_t left = __funnelshift_r(iw ? res_bits[iw - 1] : 0u, res_bits[iw], i & 31);      // bit 32 - d: i - d
            const uint32_t right = __funnelshift_r(res_bits[rw], res_bits[rw + 1], (i + 1) & 31);         // bit d - 1: i + d
            float w = 0.f;
#pragma unroll 4
            for (int d = 1; d <= prm.D; ++d) {
                const float g = gpow[d];
                w += (left >> (32 - d)) & 1u ? g : 0.f;
                w += (right >> (d - 1)) & 1u ? g : 0.f;
            }
            const float phi = fminf(1.f, w * inv_wmax);                        // Eq. 6
            const float tau = prm.tau_max - (prm.tau_max - prm.tau_min) * phi; // Eq. 7
            r_sum += r;
            gap_sum += m1 - m2;
            // Eq. 8; or the fixed probability gate the paper contrasts it with (p1 = 1/S, no spatial modulation)
            // (the global early-commit gate decides for all candidates together, after the sum below)
            f = (prm.gate == 1 ? (1.f / S >= prm.prob_threshold) : (prm.gate == 2 ? false : r >= tau)) ? 1 : 0;
            listed = !(prm.schedule_after_exit && f);                            // the schedule ranks what is left
            if (listed && !(S == S)) {                                           // a sum that is no number ranks first, ahead of no one
                f |= 4;
                listed = false;
            }
        }
        if (base == 0) rank[tid] = listed ? 0 : INT_MAX;
        if (c < n_pos) flag[c] = f;
        const uint32_t in_list = __ballot_sync(0xffffffffu, listed), all = __ballot_sync(0xffffffffu, cand);
        uint32_t at = 0;
        if ((tid & 31) == 0 && all) at = atomicAdd(&counts_sh, (uint32_t)__popc(all) << 16 | (uint32_t)__popc(in_list));
        at = (__shfl_sync(0xffffffffu, at, 0) & 0xffffu) + __popc(in_list & ((1u << (tid & 31)) - 1u));
        if (listed) {
            // ordered like (S, position); -0 counts as 0
            const uint32_t bits = __float_as_uint(S + 0.f);
            keys[at] = (uint64_t)(bits ^ ((bits >> 31) ? 0xffffffffu : 0x80000000u)) << 32 | (uint32_t)c;
        }
    }
    if (prm.gate == 2) {                                       // fixed-order tree: the same sum on every run
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) gap_sum += __shfl_xor_sync(0xffffffffu, gap_sum, o);
        if ((tid & 31) == 0) gap_sums[tid >> 5] = gap_sum;
    }
    if (a.mean_ratio) {                                        // fixed-order tree: the same sum on every run
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r_sum += __shfl_xor_sync(0xffffffffu, r_sum, o);
        if ((tid & 31) == 0) ratio_sums[tid >> 5] = r_sum;
    }
    __syncthreads();
    const int n_cand = counts_sh >> 16, n_list = counts_sh & 0xffffu;
    auto is_cand = [&](int c) { return !((res_bits[(lo + c) >> 5] >> ((lo + c) & 31)) & 1u); };
    if (a.state && prm.schedule == 1) {
        // adaptive schedule: the share of what is still masked that keeps the block on pace to end with its last step
        const int steps_left = max(1, a.steps_per_block - (a.lockstep ? a.lockstep_s : st.s));
        k = (n_cand + steps_left - 1) / steps_left;
    }

    bool all_exit = false;
    if (prm.gate == 2 && n_cand > 0) {
        // global early commit: every candidate exits when the mean top-2 logit gap clears the threshold
        float t = 0.f;
        for (int w = 0; w < kAcceptThreads / 32; ++w) t += gap_sums[w];
        all_exit = t / (float)n_cand >= prm.gap_threshold;
    }

    // transfer schedule: the k candidates with the largest p1 = 1/S, i.e. the smallest S; equal S
    // resolves to the lower position.  Rank by counting: W threads take an entry each, 256 / W of them share its
    // comparisons.
    const int k_eff = all_exit && prm.schedule_after_exit ? 0 : min(k, n_cand);
    const bool short_block = n_pos <= kAcceptThreads;
    if (k_eff > 0) {
        int W = 32;
        while (W < (short_block ? n_list : kAcceptThreads) && W < kAcceptThreads) W <<= 1;
        const int share = kAcceptThreads / W, q = tid / W, pairs = n_list >> 1;
        const int o_lo = pairs * q / share, o_hi = pairs * (q + 1) / share;
        for (int e = tid % W; e < n_list; e += W) {
            const uint64_t key = keys[e];
            int before = 0;
            for (int o = o_lo; o < o_hi; ++o) {
                const ulonglong2 v = reinterpret_cast<const ulonglong2*>(keys)[o];
                before += (v.x < key) + (v.y < key);
            }
            if ((n_list & 1) && q == share - 1) before += keys[n_list - 1] < key;
            const int c = (int)(uint32_t)key;
            if (short_block) atomicAdd(&rank[c], before);
            else if (before < k_eff) flag[c] |= 2;
        }
        __syncthreads();
    }

    // freeze: chosen candidates receive their argmax; everything else is left untouched
    int my_final = 0;
    for (int c = tid; c < n_pos; c += blockDim.x) {
        uint8_t f = flag[c] | (all_exit && is_cand(c) ? 1 : 0);
        if (k_eff > 0 && ((f & 4) || (short_block && rank[c] < k_eff))) f |= 2;
        f &= 3;
        if (f) {
            const int i = lo + c;
            const size_t gi = row + i;
            x[i] = c < kAcceptThreads ? arg_0 : a.argmax[gi];
            if (a.exit_reason) a.exit_reason[gi] = f;
            if (a.exit_step) a.exit_step[gi] = (int16_t)(a.state ? st.steps_used + 1 : a.step_index);
            ++my_final;
        }
    }
    if (my_final) atomicAdd(&n_final_sh, my_final);
    __syncthreads();
    if (tid == 0) {
        const int left = n_cand - n_final_sh;
        if (a.n_masked) a.n_masked[b] = left;
        if (a.state) {
            if (n_cand > 0 && a.mean_ratio) {
                float t = 0.f;
                for (int w = 0; w < kAcceptThreads / 32; ++w) t += ratio_sums[w];
                a.mean_ratio[(size_t)st.steps_used * a.B + b] = t / (float)n_cand;
            }
            if (n_cand > 0 && a.n_candidates) a.n_candidates[(size_t)st.steps_used * a.B + b] = n_cand;
            if (n_cand > 0) st.steps_used += 1;
            st.n_masked = left;
            if (a.lockstep) {                                  // the host advances the block for everyone
                a.state[b] = st;
                if (a.n_unfinished && left > 0) atomicAdd(a.n_unfinished, 1);
            } else {
                if (left == 0) { st.blk += 1; st.s = 0; } else { st.s += 1; }
                a.state[b] = st;
                if (a.n_unfinished && st.blk < a.n_blocks) atomicAdd(a.n_unfinished, 1);
            }
        }
    }
}

// The longest canvas taken: 9 bytes a position and a bit in 200 KB.
inline bool accept_length_ok(int L) {
    return (size_t)((L + 31) / 32 + 2) * 4 + (size_t)L * 8 + (size_t)((L + 3) / 4) * 4 + 16 <= 200 * 1024;
}
inline size_t accept_smem_bytes(int L) {
    const size_t words = ((size_t)(L + 31) / 32 + 2 + 3) / 4 * 4, L4 = (size_t)(L + 3) / 4 * 4;
    return words * 4 + L4 * 9 + 16;
}

}  // namespace jot
