// Projections of small canvases (at most 256 rows) as one stream of weights against a few tokens.
//
//   D^T[feature, token] = W[feature, :] . X[token, :]^T      (fp32 in tensor memory, bf16 operands, both K-major)
//
// The weight rows are the MMA's M side and ALL tokens its N side, so every byte of W enters one SM, once.  What bounds these
// kernels is HBM, and next to it whatever makes the stream pause, so:
//   - W and X have a ring of shared-memory slots and a producer warp each.  W comes from HBM (2.2 us away when HBM is busy: the chip wants
//     14 MB in flight), X from L2 (under 1 us); in common stages the X tiles take the memory that W's depth needs.  The W producer
//     never waits for the preceding kernel: weights are nobody's output.
//   - k-block i of a CTA's whole run is one barrier pair, full[i % D] (both operands have landed) and done[i % D] (its products have
//     retired: both its slots are free), so that the issuing thread spends one wait and one commit per k-block however many rings there are.
//   - the epilogue behind the last product is spread thin: 16 warps, eight tokens at a time (a thread holds one feature of them), straight
//     from the registers.
#pragma once
#include "gemm.cuh"

namespace jot {

constexpr int kStreamThreads = 640;        // warp 0 W producer, warp 1 MMA issuer, warp 2 X producer, warps 4..19 epilogue
constexpr int kStreamRing = 12;            // barrier pairs, and the most slots a ring can have
constexpr int kStreamSmem = 226 * 1024;    // dynamic part; the static barriers take the rest of the 227 KB
constexpr int kStreamMaxTokens = 256;      // beyond, the accumulators of gate and up no longer fit tensor memory side by side

struct StreamGeom {
    int n;              // token columns of the accumulators: a multiple of 16
    int acc_cols;       // ... rounded to 32
    int w_bytes, x_bytes;
    int nw, nx;         // ring slots
    int x_off, smem_bytes;
};
// `w_rows` rows of W and `x_rows` of X per slot.  An MMA reads 128 rows of W from wherever a tile begins: past a tile of fewer rows it reads
// the next slot or the X ring (16 KB or more behind the last slot), and nobody takes what comes of that.
__host__ __device__ inline StreamGeom stream_geom(int M, int w_rows, int x_rows) {
    StreamGeom g;
    g.n = (M + 15) / 16 * 16;
    g.acc_cols = (M + 31) / 32 * 32;
    g.w_bytes = w_rows * 128;
    g.x_bytes = x_rows * 128;
    g.nx = g.x_bytes > 8 * 1024 ? 4 : 8;
    const int room = kStreamSmem - 1024 - g.nx * g.x_bytes;
    g.nw = room / g.w_bytes < kStreamRing ? room / g.w_bytes : kStreamRing;
    g.x_off = g.nw * g.w_bytes;
    g.smem_bytes = g.x_off + g.nx * g.x_bytes + 1024;
    return g;
}

// Which k-block of a CTA's run it is, as ring positions.
struct StreamPos {
    int slot = 0, bar = 0;
    uint32_t bar_phase = 0;
    __device__ __forceinline__ void next(int slots) {
        if (++slot == slots) slot = 0;
        if (++bar == kStreamRing) { bar = 0; bar_phase ^= 1; }
    }
};
// A producer's view of its ring: where k-block i goes, and the barrier of k-block i - slots, whose products free the slot.
struct StreamProducer {
    StreamPos at;
    int ahead = 0, freed = 0;
    uint32_t freed_phase = 0;
    __device__ __forceinline__ bool wait_free(uint64_t* done, int slots, volatile int* abortp) {
        if (ahead < slots) { ++ahead; return true; }
        const bool ok = mbar_wait(&done[freed], freed_phase, abortp);
        if (++freed == kStreamRing) { freed = 0; freed_phase ^= 1; }
        return ok;
    }
};

// ---------------------------------------------------------------- O and down: K ranges over CTA pairs, fp32 partial sums
// A unit is (256 weight rows, one of split_k K ranges), one per CTA pair (tcgen05 cta_group::2, UMMA M = 256: 128 rows and half of the
// tokens per CTA).  The sums leave as fp32, a warp store 32 features of a token, one 128-byte line; splitk_reduce_norm_kernel, which is
// there for the RMSNorm anyway, adds the ranges.  An exchange between the pairs of a cluster (gemm_slab.cuh) in its place took 4 to 8 us
// after the last product.  Projection and norm of a layer, between events: 32 rows of the LLaDA-8B shape O 25.4 -> 19.4 us, down 35.8 ->
// 29.0; 133 rows of the Dream-7B shape 30.6 -> 21.8 and 47.5 -> 40.1.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kStreamThreads, 1)
gemm_stream_partial_kernel(const GemmParams p, const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[kStreamRing], done[kStreamRing], acc_full;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_ctarank();
    const bool leader = rank == 0;
    const int half = (p.M + 15) / 16 * 8;                       // this CTA's share of the tokens
    const StreamGeom g = stream_geom(p.M, 128, half);
    const int num_kb = (p.K + kBK - 1) / kBK;
    const int n_slabs = (p.N + 255) / 256, unit = (int)(blockIdx.x >> 1);
    const int ks = unit / n_slabs, slab = unit - ks * n_slabs, f0 = (2 * slab + rank) * 128;
    const int kb0 = (int)((long long)ks * num_kb / p.split_k), kb1 = (int)((long long)(ks + 1) * num_kb / p.split_k);
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < g.acc_cols) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < kStreamRing; ++s) {
            mbar_init(&full[s], 2);                   // the leader's two producers
            mbar_init(&done[s], 1);
        }
        mbar_init(&acc_full, 1);
        fence_barrier_init();
        fence_proxy_async_smem();
        tma_prefetch_desc(&tmW);
        tma_prefetch_desc(&tmX);
    }
    if (warp == 1) {
        tmem_alloc_pair(&tmem_base_slot, tmem_cols);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    cluster_sync_all();                       // both CTAs' barriers exist before anyone signals across
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    volatile int* abortp = &abort_flag;
    grid_launch_dependents();

    if (warp == 0 || warp == 2) {
        // ================= producers (whole warps run the loop, one lane issues) =================
        const bool is_w = warp == 0, elected = elect_one();
        const uint64_t once = l2_evict_first();     // every W byte is read once
        const int slots = is_w ? g.nw : g.nx;
        if (!is_w) grid_dependency_wait();
        StreamProducer pr;
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!pr.wait_free(done, slots, abortp)) break;
            uint64_t* bar = &full[pr.at.bar];
            const uint32_t leader_bar = mapa_u32(bar, 0);
            const int k = kb * kBK;
            if (elected) {
                if (leader) mbar_arrive_expect_tx(bar, 2 * (uint32_t)(is_w ? g.w_bytes : g.x_bytes));
                if (is_w) tma_load_2d_pair_hint(smem + pr.at.slot * g.w_bytes, &tmW, leader_bar, k, f0, once);
                else tma_load_2d_pair(smem + g.x_off + pr.at.slot * g.x_bytes, &tmX, leader_bar, k, rank * half);
            }
            __syncwarp();
            pr.at.next(slots);
        }
    } else if (warp == 1) {
        // ================= MMA issuer (even CTA of the pair; the whole warp runs the loop, one lane issues) ======
        if (leader) {
            const bool elected = elect_one();
            const uint32_t idesc = umma_idesc_bf16(256, g.n);
            // descriptors of a slot: those of slot 0 advanced in the 16-byte-granular address field, which never carries
            const uint64_t wd0 = umma_desc_k128(smem_u32(smem)), xd0 = umma_desc_k128(smem_u32(smem + g.x_off));
            const uint32_t w_units = (uint32_t)g.w_bytes >> 4, x_units = (uint32_t)g.x_bytes >> 4;
            StreamPos w, x;
            uint64_t wd = wd0, xd = xd0;
            uint32_t accum = 0;
            bool ok = true;
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!mbar_wait(&full[w.bar], w.bar_phase, abortp)) { ok = false; break; }
                tc_fence_after();
                if (elected) {
#pragma unroll
                    for (int k = 0; k < kBK / 16; ++k) umma_bf16_pair(tmem_base, wd + 2 * k, xd + 2 * k, idesc, accum | k);
                    umma_commit_pair(&done[w.bar], 0x3);
                }
                __syncwarp();
                accum = 1;
                w.next(g.nw);
                x.next(g.nx);
                wd = w.slot ? wd + w_units : wd0;
                xd = x.slot ? xd + x_units : xd0;
            }
            if (ok && elected) umma_commit_pair(&acc_full, 0x3);
        }
        __syncwarp();
    } else if (warp >= 4) {
        // ================= epilogue: a lane is an output FEATURE, four warps per TMEM lane quadrant =================
        grid_dependency_wait();                   // what is written here, earlier kernels may still be reading
        const int quad = warp & 3, grp = (warp - 4) >> 2;
        const uint32_t lane_base = tmem_base + (uint32_t(quad * 32) << 16);
        const int f = f0 + quad * 32 + lane;
        // (the tensor-memory loads below are warp-wide: a warp gives up as one)
        if (__all_sync(0xffffffffu, mbar_wait(&acc_full, 0, abortp))) {
            tc_fence_after();
            // (two chunks of 8 tokens at a time: their loads and stores overlap)
            for (int t0 = grp * 16; t0 < p.M; t0 += 64) {
                float v[16];
                tmem_ld8(lane_base + t0, v);
                tmem_ld8(lane_base + t0 + 8, v + 8);
                tmem_ld8_wait(v);
                tmem_ld8_wait(v + 8);
                float* dst = p.partial + ((size_t)ks * p.M + t0) * p.N + f;
                const int n_here = p.M - t0;
                if (f < p.N) {
#pragma unroll
                    for (int j = 0; j < 16; ++j, dst += p.N)
                        if (j < n_here) *dst = v[j];
                }
            }
        }
    }
    __syncwarp();

    // ---- teardown: nobody leaves while the other CTA of the pair may still signal or read across ----
    tc_fence_before();
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, tmem_cols);
    }
    if (threadIdx.x == 0 && abort_flag && p.status) atomicExch(p.status, 6);
}

// ---------------------------------------------------------------- gate/up + SwiGLU
// Each CTA takes `rows` gate rows and the matching up rows, a multiple of 8 that deals all output features evenly over the SMs (88 of
// 12288, 128 of 18944 on 148 SMs; more than 128 a CTA: several units one after the other, with the accumulators double-buffered where
// tensor memory has room).  Gate and up rows are two UMMAs of M = 128 into two accumulators: feature f's gate and up products sit in the
// same TMEM lane, so SwiGLU needs no exchange and a warp writes 32 consecutive outputs of a token.  Against 96 token-major tiles (32
// rows, LLaDA-8B shape) 44.6 -> 43.0 us between events, and the step 3575 -> 3425; against two waves of slabs (133 rows, Dream-7B shape)
// 62.5 -> 55.5, 3810 -> 3645.  Which passes come here: stream_gateup_pays (jot.cu).
__host__ __device__ inline int stream_gateup_rows(int n_out, int ctas) {
    const int groups = (n_out + 7) / 8, waves = (groups + 16 * ctas - 1) / (16 * ctas);
    return 8 * ((groups + waves * ctas - 1) / (waves * ctas));
}

__global__ void __launch_bounds__(kStreamThreads, 1)
gemm_stream_gateup_kernel(const GemmParams p, const int rows, const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[kStreamRing], done[kStreamRing], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const StreamGeom g = stream_geom(p.M, 2 * rows, (p.M + 15) / 16 * 16);
    const int num_kb = (p.K + kBK - 1) / kBK, n_out = p.N / 2, n_units = (n_out + rows - 1) / rows;
    const int n_acc = 4 * g.acc_cols <= 512 ? 2 : 1;
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < 2 * n_acc * g.acc_cols) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < kStreamRing; ++s) {
            mbar_init(&full[s], 2);                   // the two producers
            mbar_init(&done[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&acc_full[a], 1);
            mbar_init(&acc_empty[a], 16);             // the epilogue warps
        }
        fence_barrier_init();
        fence_proxy_async_smem();
        tma_prefetch_desc(&tmW);
        tma_prefetch_desc(&tmX);
    }
    if (warp == 1) {
        tmem_alloc(&tmem_base_slot, tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    volatile int* abortp = &abort_flag;
    grid_launch_dependents();

    if (warp == 0 || warp == 2) {
        // ================= producers (whole warps run the loop, one lane issues) =================
        const bool is_w = warp == 0, elected = elect_one();
        const uint64_t once = l2_evict_first();     // every W byte is read once
        const int slots = is_w ? g.nw : g.nx;
        if (!is_w) grid_dependency_wait();
        StreamProducer pr;
        bool ok = true;
        for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x) {
            for (int kb = 0; kb < num_kb; ++kb) {
                if (!pr.wait_free(done, slots, abortp)) { ok = false; break; }
                const int k = kb * kBK;
                uint64_t* bar = &full[pr.at.bar];
                if (elected) {
                    mbar_arrive_expect_tx(bar, (uint32_t)(is_w ? g.w_bytes : g.x_bytes));
                    if (is_w) {
                        uint8_t* sW = smem + pr.at.slot * g.w_bytes;
                        tma_load_2d_hint(sW, &tmW, bar, k, u * rows, once);
                        tma_load_2d_hint(sW + rows * 128, &tmW, bar, k, n_out + u * rows, once);
                    } else {
                        tma_load_2d(smem + g.x_off + pr.at.slot * g.x_bytes, &tmX, bar, k, 0);
                    }
                }
                __syncwarp();
                pr.at.next(slots);
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer (the whole warp runs the loop, one lane issues) ======
        const bool elected = elect_one();
        const uint32_t idesc = umma_idesc_bf16(128, g.n);
        const uint64_t wd0 = umma_desc_k128(smem_u32(smem)), xd0 = umma_desc_k128(smem_u32(smem + g.x_off));
        const uint32_t w_units = (uint32_t)g.w_bytes >> 4, x_units = (uint32_t)g.x_bytes >> 4, up_units = (uint32_t)(rows * 128) >> 4;
        StreamPos w, x;
        uint64_t wd = wd0, xd = xd0;
        int acc = 0;
        uint32_t acc_phase = 0;
        bool ok = true;
        for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x) {
            if (!mbar_wait(&acc_empty[acc], acc_phase ^ 1, abortp)) break;
            tc_fence_after();
            const uint32_t d_gate = tmem_base + 2 * acc * g.acc_cols, d_up = d_gate + g.acc_cols;
            uint32_t accum = 0;
            for (int kb = 0; kb < num_kb; ++kb) {
                if (!mbar_wait(&full[w.bar], w.bar_phase, abortp)) { ok = false; break; }
                tc_fence_after();
                if (elected) {
#pragma unroll
                    for (int k = 0; k < kBK / 16; ++k) {
                        umma_bf16(d_gate, wd + 2 * k, xd + 2 * k, idesc, accum | k);
                        umma_bf16(d_up, wd + up_units + 2 * k, xd + 2 * k, idesc, accum | k);
                    }
                    umma_commit(&done[w.bar]);
                }
                __syncwarp();
                accum = 1;
                w.next(g.nw);
                x.next(g.nx);
                wd = w.slot ? wd + w_units : wd0;
                xd = x.slot ? xd + x_units : xd0;
            }
            if (!ok) break;
            if (elected) umma_commit(&acc_full[acc]);
            __syncwarp();
            if (++acc == n_acc) { acc = 0; acc_phase ^= 1; }
        }
        __syncwarp();
    } else if (warp >= 4) {
        // ================= epilogue: a lane is an output FEATURE, four warps per TMEM lane quadrant =================
        grid_dependency_wait();                   // what is written here, earlier kernels may still be reading
        const int quad = warp & 3, grp = (warp - 4) >> 2;
        const int f_in = quad * 32 + lane;
        const uint32_t lane_base = tmem_base + (uint32_t(quad * 32) << 16);
        int acc = 0;
        uint32_t acc_phase = 0;
        for (int u = blockIdx.x; u < n_units; u += gridDim.x) {
            // (the tensor-memory loads below are warp-wide: a warp gives up as one)
            if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[acc], acc_phase, abortp))) break;
            tc_fence_after();
            const uint32_t a_gate = lane_base + 2 * acc * g.acc_cols;
            const bool mine = f_in < rows && u * rows + f_in < n_out;
            if (quad * 32 < rows)
                for (int t0 = grp * 8; t0 < p.M; t0 += 32) {
                    float gate[8], up[8];
                    tmem_ld8(a_gate + t0, gate);
                    tmem_ld8(a_gate + g.acc_cols + t0, up);
                    tmem_ld8_wait(gate);
                    tmem_ld8_wait(up);
                    __nv_bfloat16* dst = p.C + (size_t)t0 * p.ldc + u * rows + f_in;
                    const int n_here = p.M - t0;
                    if (mine) {
#pragma unroll
                        for (int j = 0; j < 8; ++j, dst += p.ldc)
                            if (j < n_here) *dst = __float2bfloat16_rn(silu_mul(gate[j], up[j]));
                    }
                }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[acc]);
            if (++acc == n_acc) { acc = 0; acc_phase ^= 1; }
        }
    }
    __syncwarp();

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, tmem_cols);
    }
    if (threadIdx.x == 0 && abort_flag && p.status) atomicExch(p.status, 7);
}

}  // namespace jot
