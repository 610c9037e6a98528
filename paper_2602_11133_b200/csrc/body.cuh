// The whole transformer body of a small canvas (at most 37 rows on 148 SMs) as ONE persistent kernel.
//
// With few rows a pass is a stream of the weights, and as separate launches every projection pays a launch, a pipeline
// fill, a drain and an epilogue that nothing overlaps (7-10 us each at 32 rows, seven launches a layer; 132 us a layer of the LLaDA-8B shape, 66 us for the bytes; here 107 us).  Here one CTA per
// SM stays for the whole pass; the steps of a layer follow each other through a grid-wide barrier (1.3-1.8 us), and the
// producer requests the first weight tiles of the next projection while the other roles are still in the steps before it
// (weights are nobody's output; only the token tiles wait for the barrier).
//
//   warp 0       TMA producer: per stage two 128 x 64 tiles of W (256 weight rows) and every token's 64 columns
//   warp 1       tcgen05.mma issuer: two UMMA 128 x tokens x 16 per k-step (weight rows are the M side)
//   warp 2       requests into L2 what the workers will need from HBM
//   warps 4..11  workers: projection epilogues (a thread owns a weight row), and the steps between the projections
//
// Steps of a layer (| is a grid barrier):
//   QKV: fp32 partial sums of K ranges | sum, bf16, rotary embedding, V transposed | attention | O: partial sums |
//   sum + residual + RMSNorm | gate/up with SwiGLU | down: partial sums | sum + residual + next RMSNorm |
// Before the first layer: embedding + RMSNorm, and one CTA lists the active rows; after the last one only the active
// rows are normalised (with the final gain) into the head's input.
//
// Partial sums [range][row][column] are added in the order of the ranges: the same bits on every run.
// Every wait is bounded; on expiry the CTA reports through the status word, which the other CTAs watch, and leaves.
//
// The pipeline takes nearly all of shared memory, so there is next to no L1: a register spilled in a step costs an L2 round
// trip (a spilling build took 6 us for a 1 us epilogue).  Hence the steps are functions of their own that read their
// parameters from shared memory, and the loops that run once per layer stay rolled (their instructions come from L2 too).
#pragma once
#include "glue.cuh"
#include "pdl.cuh"
#include "ptx.cuh"

namespace jot {

constexpr int kBodyThreads = 384;
constexpr int kBodyWorkers = 256;
constexpr int kBodyMaxTokens = 64;         // what tensor memory is laid out for; body_applies stops earlier
constexpr int kBodyMaxStages = 8;
constexpr int kBodyMaxSmem = 226 * 1024;   // dynamic part; the static barriers take the rest of the 227 KB
constexpr int kBodyWTile = 256 * 128;      // bytes of W per stage: 256 rows x 64 bf16
constexpr int kBodyMaxSplit = 8;           // K ranges of a projection
constexpr int kBodyQT = 16;                // queries per attention item
constexpr int kBodyPad = 8;                // floats of padding per row of the attention exchange
constexpr int kBodyMaxParts = 4;           // CTAs that share a row in the reduction steps
constexpr int kBodyMaxCtas = 256;
constexpr int kBodyStatus = 6;             // status word: a wait of this kernel expired

struct BodyLayer {                         // one layer's weights, in device memory
    CUtensorMap wqkv, wo, wgu, wdown;      // boxes of 128 rows x 64 columns (gate/up: as many rows as its tiles have)
    const __nv_bfloat16 *attn_norm, *mlp_norm;
    uint64_t pad[14];
};
static_assert(sizeof(BodyLayer) % 128 == 0, "tensor maps stay aligned in an array");

struct BodyParams {
    const BodyLayer* layers;
    int n_layers;
    int M, n_tok;                          // rows of the pass; the same rounded up to 16 (UMMA N)
    int B, L, Lp, rows_per_seq, pos0;      // row r = (r / rows_per_seq, pos0 + r % rows_per_seq)
    int d, ff, nq, nkv, hd, vocab;
    float eps, scale_log2e;
    int stages, stage_bytes;
    int s_qkv, s_o, s_down;                // K ranges per 256-row tile
    int gu_rows;                           // gate rows (and as many up rows) per tile of the gate/up projection: 8 .. 128
    int attn_pairs;                        // two attention items side by side in a CTA
    __nv_bfloat16 *h, *a, *attn, *act, *hsel;
    __nv_bfloat16 *qkv, *vt;               // layer 0's; the next layer's `*_stride` elements further (0: one scratch buffer)
    size_t qkv_stride, vt_stride;
    const float2* rope_cs;
    float* partial;
    const int32_t* tokens;
    const __nv_bfloat16 *embed, *final_norm;
    const int32_t* seq_map;
    // active rows: as build_rows_kernel
    int32_t mask_id;
    int blk_lo, blk_hi;
    const SeqState* state;
    int P, block_len, n_blocks;
    int32_t *rows, *rows_out, *d_R;
    int parts;                             // CTAs that share a row in the reduction steps: rows x parts <= CTAs unless 1
    unsigned long long* row_sums;          // [CTAs / parts][kBodyMaxParts] (tag, sum of squares)
    unsigned long long* barrier;           // arrivals so far: a multiple of the grid size between launches
    int32_t* status;
};

// Shared memory of the workers: the attention exchange (and Q), or one row as bf16.
__host__ __device__ inline int body_work_bytes(int hd, int d) {
    const int exchange = 4 * kBodyQT * (hd + kBodyPad) * 4 + 8 * kBodyQT * 2 * 4 + 2 * kBodyQT * hd * 2;
    return ((exchange > 2 * d ? exchange : 2 * d) + 127) / 128 * 128;
}

__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void l2_prefetch_line(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// ---- grid barrier: arrivals are counted in one 64-bit word that never goes back ----
__device__ __forceinline__ void grid_arrive(unsigned long long* bar) {
    asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(bar) : "memory");
}
__device__ __forceinline__ unsigned long long grid_count(const unsigned long long* bar) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(bar) : "memory");
    return v;
}
__device__ __forceinline__ bool grid_wait(const BodyParams& p, unsigned long long target, volatile int* abort_flag) {
    if (grid_count(p.barrier) >= target) return true;
    const unsigned long long t0 = global_ns();
    uint32_t spins = 0;
    while (grid_count(p.barrier) < target) {
        if ((++spins & 0xFFu) == 0) {
            const int32_t s = *reinterpret_cast<volatile int32_t*>(p.status);
            if (*abort_flag || (s != 0 && s != kStatusBadToken) || global_ns() - t0 > kWaitLimitNs) {
                *abort_flag = 1;
                return false;
            }
        }
    }
    return true;
}

__device__ __forceinline__ void mma_16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float x, float y) {
    __nv_bfloat162 v = __floats2bfloat162_rn(x, y);
    return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float2 unpack_bf16(uint32_t v) { return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v)); }

// What another CTA wrote earlier in this launch is read through L2 (never the read-only path).
__device__ __forceinline__ float4 ld_l2f(const float* p) { return __ldcg(reinterpret_cast<const float4*>(p)); }
// ... by an instruction the compiler leaves where it stands: the attention step places its loads by hand.
__device__ __forceinline__ uint4 ld_l2_here(const void* p) {
    uint4 v;
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

#define BODY_SYNC_WORKERS() asm volatile("bar.sync 1, 256;" ::: "memory")

// Sum of v over the 256 workers, in every one of them.
__device__ __forceinline__ float body_block_sum(float v, float* scratch /* 8 floats */, int wid, int lane) {
    v = warp_sum(v);
    if (lane == 0) scratch[wid] = v;
    BODY_SYNC_WORKERS();
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) t += scratch[i];
    BODY_SYNC_WORKERS();
    return t;
}

// out[c0 .. c1) = bf16(x * inv * gain) of a row whose columns from c0 on are staged as bf16 in shared memory; `gv` is the
// gain of this thread's first four columns.
__device__ __forceinline__ void body_norm_out(const __nv_bfloat16* row_sh, const __nv_bfloat16* gain, uint2 gv, __nv_bfloat16* out,
                                              int c0, int c1, float inv, int tid) {
    for (int i = c0 + tid * 4; i < c1; i += kBodyWorkers * 4) {
        const uint2 xv = *reinterpret_cast<const uint2*>(row_sh + i - c0);
        const float2 x0 = unpack_bf16(xv.x), x1 = unpack_bf16(xv.y), g0 = unpack_bf16(gv.x), g1 = unpack_bf16(gv.y);
        const int next = i + kBodyWorkers * 4;
        if (next < c1) gv = *reinterpret_cast<const uint2*>(gain + next);
        *reinterpret_cast<uint2*>(out + i) =
            make_uint2(pack_bf16(x0.x * inv * g0.x, x0.y * inv * g0.y), pack_bf16(x1.x * inv * g1.x, x1.y * inv * g1.y));
    }
}

// One row, or one of `parts` equal parts of it: h += sum of the partial sums (rounded once), then out = RMSNorm(h) * gain.
// With few rows several CTAs share one: each publishes its part's sum of squares as one 64-bit word (tag, value) and
// picks up the others' (the tag is this step's number, never used before, so no word has to be reset); the parts are
// added in order.  Columns of a part: a multiple of 16.
__device__ __noinline__ bool body_reduce_norm(const BodyParams& p, int row, int slot, int part, int parts, uint32_t tag, int split,
                                              const __nv_bfloat16* gain, __nv_bfloat16* out, __nv_bfloat16* row_sh,
                                              float* scratch, volatile int* abort_flag, int tid) {
    const int d = p.d, c0 = part * (d / parts), c1 = c0 + d / parts;
    const size_t total = (size_t)p.M * d;
    const float* sums = p.partial + (size_t)row * d;
    __nv_bfloat16* hrow = p.h + (size_t)row * d;
    const int first = c0 + tid * 4;
    const uint2 gv = first < c1 ? *reinterpret_cast<const uint2*>(gain + first) : make_uint2(0u, 0u);
    float ss = 0.f;
#pragma unroll 2
    for (int i = first; i < c1; i += kBodyWorkers * 4) {
        const uint2 rv = __ldcg(reinterpret_cast<const uint2*>(hrow + i));
        float4 v[kBodyMaxSplit];
#pragma unroll
        for (int s = 0; s < kBodyMaxSplit; ++s)
            if (s < split) v[s] = ld_l2f(sums + s * total + i);
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int s = 0; s < kBodyMaxSplit; ++s)
            if (s < split) { x.x += v[s].x; x.y += v[s].y; x.z += v[s].z; x.w += v[s].w; }
        const float2 r0 = unpack_bf16(rv.x), r1 = unpack_bf16(rv.y);
        const uint2 hv = make_uint2(pack_bf16(x.x + r0.x, x.y + r0.y), pack_bf16(x.z + r1.x, x.w + r1.y));
        const float2 h0 = unpack_bf16(hv.x), h1 = unpack_bf16(hv.y);
        ss += h0.x * h0.x + h0.y * h0.y + h1.x * h1.x + h1.y * h1.y;
        *reinterpret_cast<uint2*>(hrow + i) = hv;
        *reinterpret_cast<uint2*>(row_sh + i - c0) = hv;
    }
    ss = body_block_sum(ss, scratch, tid >> 5, tid & 31);
    bool ok = true;
    if (parts > 1) {
        unsigned long long* words = p.row_sums + (size_t)slot * kBodyMaxParts;
        if (tid == 0) {
            const unsigned long long w = ((unsigned long long)tag << 32) | __float_as_uint(ss);
            // (an atomic acts where the word lives; a plain store took up to 4 us to be seen from the other die)
            atomicExch(words + part, w);
        }
        if (tid < parts) {
            unsigned long long w = 0, t0 = 0;
            uint32_t spins = 0;
            while (true) {
                asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(words + tid) : "memory");
                if ((uint32_t)(w >> 32) == tag) break;
                if ((++spins & 0xFFu) == 0) {
                    if (t0 == 0) t0 = global_ns();
                    if (*abort_flag || global_ns() - t0 > kWaitLimitNs) { *abort_flag = 1; break; }
                }
            }
            scratch[tid] = __uint_as_float((uint32_t)w);
        }
        BODY_SYNC_WORKERS();
        ok = *abort_flag == 0;
        ss = 0.f;
        for (int i = 0; i < parts; ++i) ss += scratch[i];
    }
    if (ok) body_norm_out(row_sh, gain, gv, out, c0, c1, rsqrtf(ss / (float)d + p.eps), tid);
    BODY_SYNC_WORKERS();                   // row_sh and scratch are free again
    return ok;
}

// One row of the embedding and its first RMSNorm.
__device__ __noinline__ void body_embed_norm(const BodyParams& p, int row, const __nv_bfloat16* gain, __nv_bfloat16* row_sh,
                                             float* scratch, int tid) {
    int b = row / p.rows_per_seq;
    const int pos = p.pos0 + row - b * p.rows_per_seq;
    if (p.seq_map) {
        b = p.seq_map[b];
        b = b < 0 ? 0 : b;                 // unused slots of a compacted batch compute on sequence 0; nobody reads them
    }
    int tok = p.tokens[(size_t)b * p.L + pos];
    if ((unsigned)tok >= (unsigned)p.vocab) {
        if (tid == 0) atomicCAS(p.status, 0, kStatusBadToken);
        tok = 0;
    }
    const int d = p.d;
    const __nv_bfloat16* src = p.embed + (size_t)tok * d;
    __nv_bfloat16* hrow = p.h + (size_t)row * d;
    const uint2 gv = tid * 4 < d ? *reinterpret_cast<const uint2*>(gain + tid * 4) : make_uint2(0u, 0u);
    float ss = 0.f;
    for (int i = tid * 4; i < d; i += kBodyWorkers * 4) {
        const uint2 xv = *reinterpret_cast<const uint2*>(src + i);
        const float2 x0 = unpack_bf16(xv.x), x1 = unpack_bf16(xv.y);
        ss += x0.x * x0.x + x0.y * x0.y + x1.x * x1.x + x1.y * x1.y;
        *reinterpret_cast<uint2*>(hrow + i) = xv;
        *reinterpret_cast<uint2*>(row_sh + i) = xv;
    }
    ss = body_block_sum(ss, scratch, tid >> 5, tid & 31);
    body_norm_out(row_sh, gain, gv, p.a + (size_t)row * d, 0, d, rsqrtf(ss / (float)d + p.eps), tid);
    BODY_SYNC_WORKERS();
}

// The active rows, by one CTA: every position of its block that holds mask_id, in (slot, position) order.
__device__ __noinline__ void body_active_rows(const BodyParams& p, int* count /* 9 words */, int tid) {
    const int wid = tid >> 5, lane = tid & 31;
    if (tid == 0) count[8] = 0;
    BODY_SYNC_WORKERS();
    for (int slot = 0; slot < p.B; ++slot) {
        const int b = p.seq_map ? p.seq_map[slot] : slot;
        if (b < 0) continue;                                     // unused slot of a compacted batch
        int lo = p.blk_lo, hi = p.blk_hi;
        if (p.state) {
            const int blk = p.state[b].blk;
            if (blk >= p.n_blocks) continue;
            lo = p.P + blk * p.block_len;
            hi = lo + p.block_len;
        }
        for (int at = lo; at < hi; at += kBodyWorkers) {
            const int i = at + tid;
            const bool c = i < hi && p.tokens[(size_t)b * p.L + i] == p.mask_id;
            const uint32_t bal = __ballot_sync(0xffffffffu, c);
            if (lane == 0) count[wid] = __popc(bal);
            BODY_SYNC_WORKERS();
            int off = count[8], all = 0;
            for (int k = 0; k < 8; ++k) {
                if (k < wid) off += count[k];
                all += count[k];
            }
            if (c) {
                const int r = off + __popc(bal & ((1u << lane) - 1u));
                p.rows[r] = slot * p.rows_per_seq + (i - p.pos0);
                p.rows_out[r] = b * p.L + i;
            }
            BODY_SYNC_WORKERS();
            if (tid == 0) count[8] += all;
            BODY_SYNC_WORKERS();
        }
    }
    if (tid == 0) *p.d_R = count[8];
}

// QKV: add the K ranges, round to bf16, rotate Q and K, transpose V.
__device__ __noinline__ void body_qkv_finish(const BodyParams& p, __nv_bfloat16* qkv, __nv_bfloat16* vt, int tid) {
    const int hd = p.hd, half = hd >> 1, N = (p.nq + 2 * p.nkv) * hd, split = p.s_qkv, qk_heads = p.nq + p.nkv;
    const int Lr = p.rows_per_seq, L = p.L, Lp = p.Lp, pos0 = p.pos0;
    const float* partial = p.partial;
    const float2* rope_cs = p.rope_cs;
    const size_t total = (size_t)p.M * N;
    const int per_row = qk_heads * (half / 4), qk_items = p.M * per_row;
    const int tg = (Lr + 3) / 4, v_cols = p.nkv * hd, v_items = p.B * tg * v_cols;
    for (int it = blockIdx.x * kBodyWorkers + tid; it < qk_items + v_items; it += gridDim.x * kBodyWorkers) {
        if (it < qk_items) {
            // four rotation pairs (j, j + hd/2) of one head of one row
            const int row = it / per_row, rem = it - row * per_row, head = rem / (half / 4), j = (rem - head * (half / 4)) * 4;
            const int seq = row / Lr, pos = pos0 + row - seq * Lr;
            const float* src = partial + (size_t)row * N + head * hd + j;
            const float4* cs4 = reinterpret_cast<const float4*>(rope_cs + (size_t)pos * half + j);
            const float4 k0 = cs4[0], k1 = cs4[1];               // (cos, sin) of pairs j, j + 1 and j + 2, j + 3
            float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
#pragma unroll 1
            for (int s0 = 0; s0 < split; s0 += 4, src += 4 * total) {
                float4 a[4], b[4];
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    if (s0 + s < split) { a[s] = ld_l2f(src + s * total); b[s] = ld_l2f(src + s * total + half); }
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    if (s0 + s < split) {
                        lo.x += a[s].x; lo.y += a[s].y; lo.z += a[s].z; lo.w += a[s].w;
                        hi.x += b[s].x; hi.y += b[s].y; hi.z += b[s].z; hi.w += b[s].w;
                    }
            }
            // the projection's output is bf16; the rotation acts on the rounded values
            const float2 l0 = unpack_bf16(pack_bf16(lo.x, lo.y)), l1 = unpack_bf16(pack_bf16(lo.z, lo.w));
            const float2 h0 = unpack_bf16(pack_bf16(hi.x, hi.y)), h1 = unpack_bf16(pack_bf16(hi.z, hi.w));
            __nv_bfloat16* dst = qkv + ((size_t)seq * L + pos) * N + head * hd + j;
            *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16(l0.x * k0.x - h0.x * k0.y, l0.y * k0.z - h0.y * k0.w),
                                                        pack_bf16(l1.x * k1.x - h1.x * k1.y, l1.y * k1.z - h1.y * k1.w));
            *reinterpret_cast<uint2*>(dst + half) = make_uint2(pack_bf16(h0.x * k0.x + l0.x * k0.y, h0.y * k0.z + l0.y * k0.w),
                                                               pack_bf16(h1.x * k1.x + l1.x * k1.y, h1.y * k1.z + l1.y * k1.w));
        } else {
            // four consecutive positions of one V column: neighbouring threads read neighbouring columns
            const int v = it - qk_items, col = v % v_cols, grp = v / v_cols, seq = grp / tg, i0 = (grp - seq * tg) * 4;
            const int n = min(4, Lr - i0);
            const float* src = partial + ((size_t)seq * Lr + i0) * N + qk_heads * hd + col;
            float x[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
            for (int s0 = 0; s0 < split; s0 += 4, src += 4 * total) {
                float y[4][4];
#pragma unroll
                for (int s = 0; s < 4; ++s)
#pragma unroll
                    for (int j = 0; j < 4; ++j) y[s][j] = (s0 + s < split && j < n) ? __ldcg(src + s * total + (size_t)j * N) : 0.f;
#pragma unroll
                for (int s = 0; s < 4; ++s)
#pragma unroll
                    for (int j = 0; j < 4; ++j) x[j] += y[s][j];
            }
            __nv_bfloat16* dst = vt + ((size_t)seq * v_cols + col) * Lp + pos0 + i0;
            if (n == 4 && ((pos0 + i0) & 3) == 0) {
                *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]));
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j < n) dst[j] = __float2bfloat16_rn(x[j]);
            }
        }
    }
}

// Attention of 16 queries of one head by a group of GW warps (all 8, or 4 when there are more items than CTAs and the
// keys are few: two items side by side): the warps take blocks of 32 keys each with their own running maximum, row sum and
// output, and meet in shared memory.  Few queries leave nothing for a 128-row tcgen05 tile to do, and this way K and V
// do not pass through shared memory: contraction indices may be permuted as long as both operands agree, so a thread's
// 16-byte load of 8 consecutive elements serves as its fragment of two k-steps.
//   scores: thread q4 = lane % 4 holds elements 32 s + 8 q4 .. + 7 of the head dimension
//   keys:   column c of 8-key tile t is key 8 (c / 2) + 2 t + c % 2 of the block, so that a thread's eight probabilities
//           of a row belong to 8 consecutive keys, 16 bytes of V^T
template <int HD, int GW>
__device__ __noinline__ void body_attention(const BodyParams& p, const __nv_bfloat16* qkv, const __nv_bfloat16* vt, uint8_t* work,
                                            int tid) {
    constexpr int KS = HD / 32;            // 16-byte loads per row and thread
    constexpr int NT = HD / 8;             // 8-column tiles of the output
    constexpr int LDO = HD + kBodyPad;
    constexpr int VB = 8;                  // V tiles on their way ahead of their products
    constexpr int HW = GW / 2, GROUPS = 8 / GW;
    const int grp = (tid >> 5) / GW, w = (tid >> 5) % GW, lane = tid & 31, r = lane >> 2, q4 = lane & 3;
    float* sO = reinterpret_cast<float*>(work) + grp * HW * kBodyQT * LDO;                  // [HW][16 rows][LDO]
    float* sM = reinterpret_cast<float*>(work) + 4 * kBodyQT * LDO + grp * GW * kBodyQT;     // [GW][16] maximum (base-2 exponent)
    float* sL = sM + 8 * kBodyQT;                                                           // ... and row sum
    uint4* sQ = reinterpret_cast<uint4*>(reinterpret_cast<float*>(work) + 4 * kBodyQT * LDO + 16 * kBodyQT) + grp * KS * 64;    // [2 KS][32]
    auto sync_group = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + (GROUPS > 1 ? 1 + grp : 0)), "n"(GW * 32) : "memory"); };
    const int Lr = p.rows_per_seq, L = p.L, Lp = p.Lp, pos0 = p.pos0, nq = p.nq, nkv = p.nkv, group = nq / nkv;
    const int N = (nq + 2 * nkv) * HD;
    const int nqt = (Lr + kBodyQT - 1) / kBodyQT, nkb = (L + 31) / 32, items = p.B * nq * nqt;
    __nv_bfloat16* attn = p.attn;
    const float c = p.scale_log2e;
    for (int item = blockIdx.x + grp * gridDim.x; item < items; item += GROUPS * gridDim.x) {
        const int qt = item % nqt, hb = item / nqt, h = hb % nq, b = hb / nq, kvh = h / group;
        const __nv_bfloat16* seq = qkv + (size_t)b * L * N;
        const __nv_bfloat16* vrow = vt + ((size_t)b * nkv + kvh) * HD * Lp;
        float O[NT][4];
#pragma unroll
        for (int n = 0; n < NT; ++n) O[n][0] = O[n][1] = O[n][2] = O[n][3] = 0.f;
        float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
        // Q as fragments in shared memory: [k-step pair][row half][lane]
#pragma unroll
        for (int f = w; f < 2 * KS; f += GW) {
            const int i = min(qt * kBodyQT + r + 8 * (f & 1), Lr - 1);
            sQ[f * 32 + lane] = ld_l2_here(seq + (size_t)(pos0 + i) * N + h * HD + (f >> 1) * 32 + q4 * 8);
        }
        sync_group();
#pragma unroll 1
        for (int j = w; j < nkb; j += GW) {
            const int k0 = j * 32;
            float S[4][4];
#pragma unroll
            for (int t = 0; t < 4; ++t) S[t][0] = S[t][1] = S[t][2] = S[t][3] = 0.f;
            {
                // two k-step pairs of all four tiles at a time (more at once would spill); tile t's key is 2 t rows further on
                const __nv_bfloat16* kp = seq + (size_t)min(k0 + 8 * (r >> 1) + (r & 1), L - 1) * N + (nq + kvh) * HD + q4 * 8;
                const int k_room = L - 1 - (k0 + 8 * (r >> 1) + (r & 1));       // rows left below this one
                uint4 kk[4][2];
                auto load_k = [&](int s) {
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        kk[t][s & 1] = ld_l2_here(kp + (size_t)max(min(2 * t, k_room), 0) * N + s * 32);
                };
                load_k(0);
                load_k(1);
#pragma unroll
                for (int s = 0; s < KS; ++s) {
                    const uint4 qa = sQ[(2 * s) * 32 + lane], qb = sQ[(2 * s + 1) * 32 + lane];
                    const uint32_t a0[4] = {qa.x, qb.x, qa.y, qb.y}, a1[4] = {qa.z, qb.z, qa.w, qb.w};
#pragma unroll
                    for (int t = 0; t < 4; ++t) mma_16816(S[t], a0, kk[t][s & 1].x, kk[t][s & 1].y);
#pragma unroll
                    for (int t = 0; t < 4; ++t) mma_16816(S[t], a1, kk[t][s & 1].z, kk[t][s & 1].w);
                    if (s + 2 < KS) load_k(s + 2);
                }
            }
            const int kq = k0 + 8 * q4;                                // this thread's keys: kq .. kq + 7
            uint4 vv[VB];
            const __nv_bfloat16* vp = vrow + (size_t)r * Lp + kq;
            uint32_t v_step = (uint32_t)Lp * 8;
            auto load_v = [&](int n) {
                uint4 v = make_uint4(0u, 0u, 0u, 0u);                  // keys past the canvas: nothing is read, zero counts
                if (kq < L) v = ld_l2_here(vp);                        // (Lp is L rounded up to 8)
                asm volatile("" : "+r"(v_step));                       // one running pointer, not sixteen kept ones
                vp += v_step;
                if (kq + 8 > L) {
                    v.x &= kq < L ? (kq + 1 < L ? ~0u : 0xffffu) : 0u;
                    v.y &= kq + 2 < L ? (kq + 3 < L ? ~0u : 0xffffu) : 0u;
                    v.z &= kq + 4 < L ? (kq + 5 < L ? ~0u : 0xffffu) : 0u;
                    v.w &= kq + 6 < L ? (kq + 7 < L ? ~0u : 0xffffu) : 0u;
                }
                vv[n % VB] = v;
            };
#pragma unroll
            for (int n = 0; n < VB; ++n) load_v(n);
            float bm0 = -INFINITY, bm1 = -INFINITY;
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const bool in = kq + 2 * t + e < L;
                    S[t][e] = in ? S[t][e] * c : -INFINITY;
                    S[t][2 + e] = in ? S[t][2 + e] * c : -INFINITY;
                    bm0 = fmaxf(bm0, S[t][e]);
                    bm1 = fmaxf(bm1, S[t][2 + e]);
                }
            bm0 = fmaxf(bm0, __shfl_xor_sync(0xffffffffu, bm0, 1));
            bm1 = fmaxf(bm1, __shfl_xor_sync(0xffffffffu, bm1, 1));
            bm0 = fmaxf(bm0, __shfl_xor_sync(0xffffffffu, bm0, 2));
            bm1 = fmaxf(bm1, __shfl_xor_sync(0xffffffffu, bm1, 2));
            const float n0 = fmaxf(m0, bm0), n1 = fmaxf(m1, bm1);       // finite: every block has a key below L
            if (j != w) {
                const float f0 = ex2_approx(m0 - n0), f1 = ex2_approx(m1 - n1);
                l0 *= f0;
                l1 *= f1;
#pragma unroll
                for (int n = 0; n < NT; ++n) { O[n][0] *= f0; O[n][1] *= f0; O[n][2] *= f1; O[n][3] *= f1; }
            }
            m0 = n0;
            m1 = n1;
            uint32_t P0[4], P1[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const float x0 = ex2_approx(S[t][0] - m0), x1 = ex2_approx(S[t][1] - m0);
                const float y0 = ex2_approx(S[t][2] - m1), y1 = ex2_approx(S[t][3] - m1);
                l0 += x0 + x1;
                l1 += y0 + y1;
                P0[t] = pack_bf16(x0, x1);
                P1[t] = pack_bf16(y0, y1);
            }
            const uint32_t a0[4] = {P0[0], P1[0], P0[1], P1[1]}, a1[4] = {P0[2], P1[2], P0[3], P1[3]};
#pragma unroll
            for (int n0t = 0; n0t < NT; n0t += 4) {
#pragma unroll
                for (int n = n0t; n < n0t + 4; ++n) mma_16816(O[n], a0, vv[n % VB].x, vv[n % VB].y);
#pragma unroll
                for (int n = n0t; n < n0t + 4; ++n) {
                    mma_16816(O[n], a1, vv[n % VB].z, vv[n % VB].w);
                    if (n + VB < NT) load_v(n + VB);
                }
            }
        }
        l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
        l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
        l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
        l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
        // two rounds: the upper half of the warps hand over to the lower half, whose results are combined below
        float* o0 = sO + ((w % HW) * kBodyQT + r) * LDO + 2 * q4;
        auto put = [&]() {
            if (q4 == 0) {
                sM[w * kBodyQT + r] = m0; sM[w * kBodyQT + r + 8] = m1;
                sL[w * kBodyQT + r] = l0; sL[w * kBodyQT + r + 8] = l1;
            }
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                *reinterpret_cast<float2*>(o0 + n * 8) = make_float2(O[n][0], O[n][1]);
                *reinterpret_cast<float2*>(o0 + 8 * LDO + n * 8) = make_float2(O[n][2], O[n][3]);
            }
        };
        if (nkb > HW) {
            if (w >= HW) put();
            sync_group();
            if (w < HW) {                                               // (these warps have keys here: m0 and m1 are finite)
                const float p0 = sM[(w + HW) * kBodyQT + r], p1 = sM[(w + HW) * kBodyQT + r + 8];
                const float x0 = fmaxf(m0, p0), x1 = fmaxf(m1, p1);
                const float f0 = ex2_approx(m0 - x0), f1 = ex2_approx(m1 - x1), g0 = ex2_approx(p0 - x0), g1 = ex2_approx(p1 - x1);
                l0 = l0 * f0 + sL[(w + HW) * kBodyQT + r] * g0;
                l1 = l1 * f1 + sL[(w + HW) * kBodyQT + r + 8] * g1;
                m0 = x0;
                m1 = x1;
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    const float2 a = *reinterpret_cast<const float2*>(o0 + n * 8), e = *reinterpret_cast<const float2*>(o0 + 8 * LDO + n * 8);
                    O[n][0] = O[n][0] * f0 + a.x * g0; O[n][1] = O[n][1] * f0 + a.y * g0;
                    O[n][2] = O[n][2] * f1 + e.x * g1; O[n][3] = O[n][3] * f1 + e.y * g1;
                }
            }
            sync_group();
        }
        if (w < HW) put();
        sync_group();
        {
            constexpr int PER = HD / (2 * GW);                          // output columns per thread: 2 GW threads a row
            const int tg = tid % (GW * 32), row = tg / (2 * GW), c0 = tg % (2 * GW) * PER, i = qt * kBodyQT + row;
            float m = -INFINITY;
#pragma unroll
            for (int s = 0; s < HW; ++s) m = fmaxf(m, sM[s * kBodyQT + row]);
            float l = 0.f, x[PER];
#pragma unroll
            for (int e = 0; e < PER; ++e) x[e] = 0.f;
#pragma unroll
            for (int s = 0; s < HW; ++s) {
                const float f = ex2_approx(sM[s * kBodyQT + row] - m);    // 0 for a warp that had no keys
                l += sL[s * kBodyQT + row] * f;
#pragma unroll
                for (int e = 0; e < PER; e += 4) {
                    const float4 v = *reinterpret_cast<const float4*>(sO + (s * kBodyQT + row) * LDO + c0 + e);
                    x[e] += v.x * f; x[e + 1] += v.y * f; x[e + 2] += v.z * f; x[e + 3] += v.w * f;
                }
            }
            const float inv = 1.f / l;
            if (i < Lr) {
                __nv_bfloat16* dst = attn + ((size_t)b * Lr + i) * (size_t)(nq * HD) + h * HD + c0;
#pragma unroll
                for (int e = 0; e < PER; e += 4)
                    *reinterpret_cast<uint2*>(dst + e) = make_uint2(pack_bf16(x[e] * inv, x[e + 1] * inv), pack_bf16(x[e + 2] * inv, x[e + 3] * inv));
            }
        }
        sync_group();               // the exchange area is free again
    }
}

__global__ void __launch_bounds__(kBodyThreads, 1)
body_kernel(const __grid_constant__ BodyParams kp, const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmAttn,
            const __grid_constant__ CUtensorMap tmAct) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ BodyParams p;
    __shared__ uint64_t full_bar[kBodyMaxStages], empty_bar[kBodyMaxStages], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag, leave_flag, count_sh[9];
    __shared__ float scratch[8];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int G = gridDim.x, cta = blockIdx.x;
    if (threadIdx.x == 0) {
        p = kp;
        abort_flag = 0;
        leave_flag = 0;
        for (int s = 0; s < kp.stages; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&acc_full[i], 1);
            mbar_init(&acc_empty[i], 8);
        }
        fence_barrier_init();
        fence_proxy_async_smem();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmAttn);
        tma_prefetch_desc(&tmAct);
    }
    if (warp == 1) {
        tmem_alloc(&tmem_base_slot, 256);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    uint8_t* work = smem + p.stages * p.stage_bytes;
    const uint32_t tmem_base = tmem_base_slot;
    volatile int* abortp = &abort_flag;
    // This CTA has not arrived at the first barrier, so the count is less than one full round past the launch's start.
    const unsigned long long seen = grid_count(p.barrier), base = seen - seen % (unsigned long long)G;
    auto target = [&](int n_done) { return base + (unsigned long long)n_done * G; };       // n_done barriers complete
    const uint32_t acc_cols = (uint32_t)(p.n_tok + 31) & ~31u;                              // one accumulator of 128 weight rows
    constexpr int n_buf = 2, TMEM_COLS = 256;                                               // two pairs of accumulators
    static_assert(2 * n_buf * kBodyMaxTokens <= TMEM_COLS, "accumulators fit");

    // ---- the four projections (0 QKV, 1 O, 2 gate/up, 3 down): tiles of weight rows, K ranges per tile, k-blocks ----
    const int qkv_cols = (p.nq + 2 * p.nkv) * p.hd, kd = (p.d + 63) / 64, ko = (p.nq * p.hd + 63) / 64, kf = (p.ff + 63) / 64;
    auto split_of = [&](int i) { return i == 0 ? p.s_qkv : (i == 1 ? p.s_o : (i == 2 ? 1 : p.s_down)); };
    auto kb_of = [&](int i) { return i == 1 ? ko : (i == 3 ? kf : kd); };
    auto units_of = [&](int i) {
        return i == 2 ? (p.ff + p.gu_rows - 1) / p.gu_rows : ((i == 0 ? qkv_cols : p.d) + 255) / 256 * split_of(i);
    };
    // barriers complete before the token operand of projection i of layer l may be read; 8 barriers a layer after the first
    auto ready = [](int l, int i) { return 1 + 8 * l + (i == 0 ? 0 : (i == 1 ? 3 : (i == 2 ? 5 : 6))); };

    if (warp == 0) {
        // ================= TMA producer =================
        const bool elected = elect_one();
        const uint64_t once = l2_evict_first();
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int l = 0; ok && l < p.n_layers; ++l) {
            const BodyLayer* ly = p.layers + l;
            for (int i = 0; ok && i < 4; ++i) {
                const int units = units_of(i), split = split_of(i), num_kb = kb_of(i);
                const CUtensorMap* tw = i == 0 ? &ly->wqkv : (i == 1 ? &ly->wo : (i == 2 ? &ly->wgu : &ly->wdown));
                const CUtensorMap* tx_map = i == 1 ? &tmAttn : (i == 3 ? &tmAct : &tmA);
                const uint32_t tx = (uint32_t)((i == 2 ? p.gu_rows : 128) * 256 + p.n_tok * 128);
                bool waited = false;
                for (int u = cta; ok && u < units; u += G) {
                    const int tile = u / split, ks = u - tile * split;
                    const int kb0 = ks * num_kb / split, kb1 = (ks + 1) * num_kb / split;
                    const int row0 = tile * (i == 2 ? p.gu_rows : 256), row1 = i == 2 ? p.ff + row0 : row0 + 128;
                    auto load_w = [&](int st, int kb) {
                        uint8_t* s = smem + st * p.stage_bytes;
                        mbar_arrive_expect_tx(&full_bar[st], tx);
                        tma_load_2d_hint(s, tw, &full_bar[st], kb * 64, row0, once);
                        tma_load_2d_hint(s + 128 * 128, tw, &full_bar[st], kb * 64, row1, once);
                    };
                    auto load_x = [&](int st, int kb) {
                        tma_load_2d(smem + st * p.stage_bytes + kBodyWTile, tx_map, &full_bar[st], kb * 64, 0);
                    };
                    int kb = kb0;
                    if (!waited) {
                        // weights first, as far as the pipeline reaches; the tokens once the barrier is through
                        const int n_pre = min(p.stages, kb1 - kb0), st0 = stage;
                        for (int n = 0; n < n_pre; ++n) {
                            if (!mbar_wait(&empty_bar[stage], phase ^ 1, abortp)) { ok = false; break; }
                            if (elected) load_w(stage, kb0 + n);
                            __syncwarp();
                            if (++stage == p.stages) { stage = 0; phase ^= 1; }
                        }
                        if (!ok) break;
                        ok = __all_sync(0xffffffffu, grid_wait(p, target(ready(l, i)), abortp));
                        if (!ok) break;
                        waited = true;
                        if (elected) {
                            fence_proxy_async_all();
                            for (int n = 0, st = st0; n < n_pre; ++n) {
                                load_x(st, kb0 + n);
                                if (++st == p.stages) st = 0;
                            }
                        }
                        __syncwarp();
                        kb = kb0 + n_pre;
                    }
                    for (; kb < kb1; ++kb) {
                        if (!mbar_wait(&empty_bar[stage], phase ^ 1, abortp)) { ok = false; break; }
                        if (elected) {
                            load_w(stage, kb);
                            load_x(stage, kb);
                        }
                        __syncwarp();
                        if (++stage == p.stages) { stage = 0; phase ^= 1; }
                    }
                }
            }
        }
        if (!ok)                               // copies in flight land before the shared memory is given up
            for (int n = 0; n < 100; ++n) __nanosleep(1000);
    } else if (warp == 1) {
        // ================= MMA issuer =================
        const bool elected = elect_one();
        const uint32_t idesc = umma_idesc_bf16(128, p.n_tok);
        const uint64_t wd0 = umma_desc_k128(smem_u32(smem)), xd0 = wd0 + (kBodyWTile >> 4);
        const uint32_t stage_units = (uint32_t)p.stage_bytes >> 4;
        const int stages = p.stages;
        int stage = 0, acc = 0;
        uint32_t phase = 0, acc_phase = 0;
        uint64_t wd = wd0, xd = xd0;
        bool ok = true;
        for (int l = 0; ok && l < p.n_layers; ++l)
            for (int i = 0; ok && i < 4; ++i) {
                const int units = units_of(i), split = split_of(i), num_kb = kb_of(i);
                for (int u = cta; ok && u < units; u += G) {
                    const int ks = u % split, kb0 = ks * num_kb / split, kb1 = (ks + 1) * num_kb / split;
                    if (!mbar_wait(&acc_empty[acc], acc_phase ^ 1, abortp)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t d0 = tmem_base + acc * 2 * acc_cols, d1 = d0 + acc_cols;
                    uint32_t accum = 0;
                    for (int kb = kb0; kb < kb1; ++kb) {
                        if (!mbar_wait(&full_bar[stage], phase, abortp)) { ok = false; break; }
                        tc_fence_after();
                        if (elected) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                umma_bf16(d0, wd + 2 * k, xd + 2 * k, idesc, accum | k);
                                umma_bf16(d1, wd + (128 * 128 >> 4) + 2 * k, xd + 2 * k, idesc, accum | k);
                            }
                            umma_commit(&empty_bar[stage]);
                        }
                        __syncwarp();
                        accum = 1;
                        wd += stage_units;
                        xd += stage_units;
                        if (++stage == stages) { stage = 0; phase ^= 1; wd = wd0; xd = xd0; }
                    }
                    if (!ok) break;
                    if (elected) umma_commit(&acc_full[acc]);
                    __syncwarp();
                    if (++acc == n_buf) { acc = 0; acc_phase ^= 1; }
                }
            }
        __syncwarp();
    } else if (warp == 2) {
        // ================= what the workers will read from HBM, requested into L2 while they wait =================
        // Their own loads would queue behind the weight tiles in flight (2-3 us each).  Nothing waits for this warp.
        const int k_bytes = p.nkv * p.hd * 2, vt_bytes = k_bytes * p.Lp;
        auto reached = [&](int n_done) -> bool {
            const unsigned long long t0 = global_ns(), go = target(n_done);
            bool in_time = true;
            while (in_time && grid_count(p.barrier) < go) {
                __nanosleep(200);
                in_time = !*abortp && global_ns() - t0 <= kWaitLimitNs;
            }
            return __all_sync(0xffffffffu, in_time);
        };
        auto prefetch = [&](const void* at, int bytes) {
            for (int i = lane * 128; i < bytes; i += 32 * 128) l2_prefetch_line(static_cast<const uint8_t*>(at) + i);
        };
        for (int l = 0; l < p.n_layers; ++l) {
            const BodyLayer* ly = p.layers + l;
            if (!reached(8 * l)) break;
            if (l + 1 < p.n_layers && lane < 4) tma_prefetch_desc(&ly[1].wqkv + lane);
            if (cta < p.rows_per_seq)
                for (int pos = p.pos0 + cta; pos < p.pos0 + p.rows_per_seq; pos += G) prefetch(p.rope_cs + (size_t)pos * (p.hd / 2), p.hd * 4);
            if (!reached(8 * l + 2)) break;                        // the QKV weights are through
            if (cta == G - 1) prefetch(ly->mlp_norm, p.d * 2);
            if (p.qkv_stride && p.rows_per_seq < p.L) {
                const int qkv_row = (p.nq + 2 * p.nkv) * p.hd;
                const __nv_bfloat16* k0 = p.qkv + l * p.qkv_stride + p.nq * p.hd;
                for (int row = cta; row < p.B * p.L; row += G) prefetch(k0 + (size_t)row * qkv_row, k_bytes);
                const uint8_t* v0 = reinterpret_cast<const uint8_t*>(p.vt + l * p.vt_stride);
                for (size_t i = ((size_t)cta * 32 + lane) * 128; i < (size_t)p.B * vt_bytes; i += (size_t)G * 32 * 128)
                    l2_prefetch_line(v0 + i);
            }
            if (!reached(8 * l + 6)) break;                        // gate/up is streaming
            if (cta == G - 1) prefetch(l + 1 < p.n_layers ? ly[1].attn_norm : p.final_norm, p.d * 2);
        }
    } else if (warp >= 4) {
        // ================= workers =================
        const int tid = threadIdx.x - 128, wid = warp - 4;
        const int quad = warp & 3, grp = wid >> 2;               // TMEM lane quadrant; warp group 0 / 1
        const uint32_t lane_base = tmem_base + (uint32_t(quad * 32) << 16);
        int acc = 0;
        uint32_t acc_phase = 0;
        int done = 0;                                            // barriers this CTA has arrived at
        __nv_bfloat16* row_sh = reinterpret_cast<__nv_bfloat16*>(work);

        // the step's writes are out (for_tma: TMA fetches them next): arrive, then wait for everyone
        auto step_end = [&](bool for_tma) -> bool {
            if (for_tma) fence_proxy_async_all();
            BODY_SYNC_WORKERS();
            ++done;
            if (tid == 0) {
                grid_arrive(p.barrier);
                if (!grid_wait(p, target(done), abortp)) leave_flag = 1;
            }
            BODY_SYNC_WORKERS();
            return leave_flag == 0;
        };
        // epilogues of this CTA's units of projection i
        auto epilogue = [&](int i) {
            const int units = units_of(i), split = split_of(i);
            const int M = p.M, n_tok = p.n_tok, ff = p.ff, t_rows = p.gu_rows;
            const int N = i == 0 ? qkv_cols : p.d;
            for (int u = cta; u < units; u += G) {
                const int tile = u / split, ks = u - tile * split;
                const bool w = mbar_wait(&acc_full[acc], acc_phase, abortp);
                if (!__all_sync(0xffffffffu, w)) { leave_flag = 1; return; }
                tc_fence_after();
                const uint32_t t0 = lane_base + acc * 2 * acc_cols, t1 = t0 + acc_cols;
                if (i == 2) {
                    const int r = quad * 32 + lane, f = tile * t_rows + r;
                    const bool mine = r < t_rows && f < ff, odd = lane & 1;     // t_rows and ff are even: a pair of lanes agrees
                    __nv_bfloat16* dst = p.act + (f & ~1);
#pragma unroll 1
                    for (int c = grp * 8; c < n_tok; c += 16) {
                        float g[8], up[8];
                        tmem_ld8(t0 + c, g);
                        tmem_ld8(t1 + c, up);
                        tmem_ld_wait_regs8(g);
                        tmem_ld_wait_regs8(up);
                        // neighbouring lanes trade one of two tokens, so that each stores two neighbouring columns
#pragma unroll
                        for (int j = 0; j < 8; j += 2) {
                            const float y0 = silu_mul(g[j], up[j]), y1 = silu_mul(g[j + 1], up[j + 1]);
                            const float got = __shfl_xor_sync(0xffffffffu, odd ? y0 : y1, 1);
                            const int t = c + j + (odd ? 1 : 0);
                            if (mine && t < M)
                                *reinterpret_cast<uint32_t*>(dst + (size_t)t * ff) = odd ? pack_bf16(got, y1) : pack_bf16(y0, got);
                        }
                    }
                } else {
                    // a warp's store covers 32 consecutive columns of one row
                    const int f = tile * 256 + grp * 128 + quad * 32 + lane;
                    float* dst = p.partial + (size_t)ks * M * N + f;
                    const uint32_t src = grp ? t1 : t0;
#pragma unroll 1
                    for (int c = 0; c < n_tok; c += 16) {
                        float v[16];
                        tmem_ld8(src + c, v);
                        tmem_ld8(src + c + 8, v + 8);
                        tmem_ld_wait_regs8(v);
                        tmem_ld_wait_regs8(v + 8);
                        if (f < N) {
                            float* to = dst + (size_t)c * N;
#pragma unroll
                            for (int j = 0; j < 16; ++j, to += N)
                                if (c + j < M) __stcg(to, v[j]);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[acc]);
                if (++acc == n_buf) { acc = 0; acc_phase ^= 1; }
            }
        };
        // n rows (row r, or rows[r]) -> row r of `out`
        auto reduce_norm = [&](int n, const int32_t* rows, int split, const __nv_bfloat16* gain, __nv_bfloat16* out) {
            const uint32_t tag = (uint32_t)(base / (unsigned long long)G) + (uint32_t)done;     // barriers before this step, ever
            const int parts = p.parts;
            for (int r = cta / parts; r < n && cta < G / parts * parts; r += G / parts)
                if (!body_reduce_norm(p, rows ? __ldcg(rows + r) : r, r, cta % parts, parts, tag, split, gain, out + (size_t)r * p.d,
                                      row_sh, scratch, abortp, tid))
                    leave_flag = 1;
        };

        // ---- embedding, first norm; the last CTA lists the active rows ----
        for (int row = cta; row < p.M; row += G) body_embed_norm(p, row, p.layers[0].attn_norm, row_sh, scratch, tid);
        if (cta == G - 1) body_active_rows(p, count_sh, tid);
        bool ok = step_end(true);
        for (int l = 0; ok && l < p.n_layers; ++l) {
            const BodyLayer* ly = p.layers + l;
            __nv_bfloat16* qkv = p.qkv + l * p.qkv_stride;
            __nv_bfloat16* vt = p.vt + l * p.vt_stride;
            const bool last = l + 1 == p.n_layers;
            const __nv_bfloat16 *mlp_gain = ly->mlp_norm, *next_gain = last ? p.final_norm : ly[1].attn_norm;   // long before their use
            epilogue(0);
            if (!(ok = step_end(false))) break;
            body_qkv_finish(p, qkv, vt, tid);
            if (!(ok = step_end(false))) break;
            if (p.hd == 128) {
                if (p.attn_pairs) body_attention<128, 4>(p, qkv, vt, work, tid);
                else body_attention<128, 8>(p, qkv, vt, work, tid);
            } else {
                if (p.attn_pairs) body_attention<64, 4>(p, qkv, vt, work, tid);
                else body_attention<64, 8>(p, qkv, vt, work, tid);
            }
            if (!(ok = step_end(true))) break;
            epilogue(1);
            if (!(ok = step_end(false))) break;
            reduce_norm(p.M, nullptr, p.s_o, mlp_gain, p.a);
            if (!(ok = step_end(true))) break;
            epilogue(2);
            if (!(ok = step_end(true))) break;
            epilogue(3);
            if (!(ok = step_end(false))) break;
            if (last) reduce_norm(__ldcg(p.d_R), p.rows, p.s_down, next_gain, p.hsel);
            else reduce_norm(p.M, nullptr, p.s_down, next_gain, p.a);
            if (!last) ok = step_end(true);
        }
        if (!ok) {
            if (tid == 0) *abortp = 1;
        } else if (tid == 0) {
            grid_arrive(p.barrier);            // nobody waits any more: this keeps the count a multiple of the grid size
        }
    }

    // ---- teardown ----
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
    if (threadIdx.x == 0 && abort_flag) atomicExch(p.status, kBodyStatus);
}

}  // namespace jot
