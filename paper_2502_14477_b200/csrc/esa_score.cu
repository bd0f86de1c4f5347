// Eq. 6 + Eq. 4 (+ Eq. 8) for a single query per sequence (decode), and the choice between this kernel and those of
// esa_score_tc.cu, which take every other chunk.
#include "esa_internal.h"
#include "esa_umma.cuh"

namespace esa {

// ---------------------------------------------------------------------------
// l_C = 1: S[m] = q' . k'_m as a streaming matrix-vector product, with the front half of the
// selection fused in.  With a single query, Eq. 4 is s_m = S_m - r (r = max_m S_m), and the
// proximity pooling of Eq. 8 commutes with subtracting r (x -> fl(x - r) is monotone), so the
// kernel pools the raw scores: P_j = max of S over [j - eps, j + eps] clipped to M.  It leaves
//   * pkey[m]  = order-preserving key of P_m,
//   * rkey[b]  = key of r (atomic max),
// and the selection kernel subtracts r from the scores as it reads them.
// Bound: the read of the compressed keys.  Every warp owns consecutive middle tokens (and computes eps neighbours on
// each side again, so that the window maxima need no other warp) and streams their rows, which are contiguous, through a
// ring of its own, filled by bulk copies: up to 192 KB in flight per SM, no barrier across warps, and no use of L1, so
// that the SM can stay set up for shared memory like the selection and the attention that follow (an SM is set up anew
// only when it is idle; with loads through L1, which want the opposite split, the attention's CTAs could not start beside
// the selection).  The keys are older than the preceding kernel (see launch_score_tc): the rings are filled ahead of the
// wait for it.  (8 x 129k tokens: 44 us of streaming, 6 TB/s, against 52 for loads through L1 into registers; 16 ragged
// sequences of 10k to 40k: the selection 52 -> 36 us, since the shares are equal whatever the lengths.)
// ---------------------------------------------------------------------------
constexpr int SD_WARPS = 8;
constexpr int SD_STAGES = 3;
constexpr int SD_STAGE_BYTES = 8192;
constexpr int SD_UNROLL = SD_STAGE_BYTES / 512;      // 16-byte loads of a lane per stage
constexpr int SD_MIN_SHARE = 8;                      // middle tokens per warp

struct ScoreDecodeParams {
    const __nv_bfloat16* kc;
    const __nv_bfloat16* qc;    // [B, DC]
    uint32_t* rkey;             // [B]
    uint32_t* pkey;             // [B, max_tokens] keys of the pooled raw scores
    int* status;
    int64_t max_tokens;
    int eps;
    int B;
    int share;                  // middle tokens per warp
    int n_warps;
    int first_warp[kMaxBatch];  // first warp of each sequence
    SeqMeta meta;
};

template <int DC>
__global__ void __launch_bounds__(SD_WARPS * 32)
score_decode_kernel(ScoreDecodeParams p) {
    constexpr int LPR = DC / 8;         // lanes per key row (16 bytes each)
    constexpr int RPW = 32 / LPR;       // rows per warp access
    constexpr int TILE = RPW * SD_UNROLL;                    // rows per stage
    constexpr int RING = 2 * TILE;      // scores kept: this tile and the one before
    static_assert(TILE >= 32, "the ring holds a window");
    extern __shared__ __align__(128) uint8_t sd_smem[];
    __shared__ float ring_all[SD_WARPS][RING];
    __shared__ uint64_t bars[SD_WARPS][SD_STAGES];
    __shared__ int abort_flag;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int w_id = blockIdx.x * SD_WARPS + warp;
    // the sequence of this warp: the last one that starts at or before it
    int b = -1;
    for (int s0 = 0; s0 < p.B; s0 += 32)
        b += __popc(__ballot_sync(0xffffffffu, s0 + lane < p.B && p.first_warp[min(s0 + lane, kMaxBatch - 1)] <= w_id));
    const int i_end = p.meta.i_end[b];
    const int l_M = p.meta.m_end[b] - i_end;
    const int eps = p.eps;
    const int a = min(l_M, (w_id - p.first_warp[b]) * p.share);     // first middle token of this warp
    const int own_end = min(l_M, a + p.share);
    const int s0 = max(0, a - eps), s1 = min(l_M, own_end + eps);   // tokens whose scores it computes
    const int n_tiles = own_end > a ? (s1 - s0 + TILE - 1) / TILE : 0;
    const __nv_bfloat16* kc = p.kc + ((int64_t)b * p.max_tokens + i_end + s0) * DC;
    uint8_t* stages = sd_smem + warp * (SD_STAGES * SD_STAGE_BYTES);
    float* ring = ring_all[warp];
    WaitCtx wc{&abort_flag, p.status};
    auto bar = [&](int i) { return smem_u32(&bars[warp][i]); };
    auto fetch = [&](int i) {                                       // lane 0
        const uint32_t bytes = (uint32_t)min(TILE, s1 - s0 - i * TILE) * (DC * 2);
        const int st = i % SD_STAGES;
        mbar_arrive_expect_tx(bar(st), bytes);
        bulk_load(smem_u32(stages + st * SD_STAGE_BYTES), kc + (int64_t)i * TILE * DC, bytes, bar(st));
    };
    if (tid == 0) abort_flag = 0;
    if (lane == 0) {
        for (int i = 0; i < SD_STAGES; ++i) mbar_init(bar(i), 1);
        mbar_init_fence();
        for (int i = 0; i < min(n_tiles, SD_STAGES); ++i) fetch(i);
    }
    __syncthreads();
    pdl_wait();
    pdl_launch_dependents();

    float q[8];
    {
        const uint4 v = __ldcg(reinterpret_cast<const uint4*>(p.qc + (int64_t)b * DC) + lane % LPR);
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float2 f = __bfloat1622float2(h[i]);
            q[2 * i] = f.x;
            q[2 * i + 1] = f.y;
        }
    }
    uint32_t* pk = p.pkey + (int64_t)b * p.max_tokens;
    float vmax = -INFINITY;
    int done = a;                                                   // outputs written so far end here
    for (int t = 0; t < n_tiles; ++t) {
        const int st = t % SD_STAGES;
        mbar_wait(bar(st), (t / SD_STAGES) & 1, wc);
        const uint4* src = reinterpret_cast<const uint4*>(stages + st * SD_STAGE_BYTES) + lane;
        uint4 v[SD_UNROLL];
#pragma unroll
        for (int u = 0; u < SD_UNROLL; ++u) v[u] = src[u * 32];
        __syncwarp();
        if (lane == 0 && t + SD_STAGES < n_tiles) fetch(t + SD_STAGES);
        float acc[SD_UNROLL];
#pragma unroll
        for (int u = 0; u < SD_UNROLL; ++u) {
            const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v[u]);
            float x = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 f = __bfloat1622float2(h[i]);
                x = fmaf(q[2 * i], f.x, x);
                x = fmaf(q[2 * i + 1], f.y, x);
            }
            acc[u] = x;
        }
        // sums over the LPR lanes of a row; every step hands half of the rows to the partner lane
        int n = SD_UNROLL, row = 0;
#pragma unroll
        for (int o = LPR / 2; o >= 1; o >>= 1) {
            n >>= 1;
            const bool up = lane & o;
            row += up ? n : 0;
#pragma unroll
            for (int i = 0; i < n; ++i) {
                const float keep = up ? acc[i + n] : acc[i], give = up ? acc[i] : acc[i + n];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
        }
#pragma unroll
        for (int i = 0; i < SD_UNROLL / LPR; ++i) {
            const int u = t * TILE + (row + i) * RPW + lane / LPR;
            if (u < s1 - s0) {
                ring[u & (RING - 1)] = acc[i];
                vmax = fmaxf(vmax, acc[i]);
            }
        }
        __syncwarp();
        // Eq. 8 on the raw scores for every token whose window is complete
        const int ready = t == n_tiles - 1 ? own_end : min(own_end, s0 + (t + 1) * TILE - eps);
        for (int m = done + lane; m < ready; m += 32) {
            float best = -INFINITY;                                 // (clamped positions are positions of the window)
#pragma unroll 4
            for (int w = -eps; w <= eps; ++w) best = fmaxf(best, ring[(min(max(m + w, 0), l_M - 1) - s0) & (RING - 1)]);
            pk[m] = f32_to_key(best);
        }
        done = max(done, ready);
        __syncwarp();
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
    if (lane == 0 && vmax > -INFINITY) atomicMax(p.rkey + b, f32_to_key(vmax));
}

template <int DC>
static cudaError_t launch_score_t(esa_ctx* ctx, int B, int l_C, const __nv_bfloat16* kc_cache,
                                  const SeqMeta& meta, int max_lM, bool rkey_cleared, cudaStream_t st,
                                  bool* pooled_ready) {
    cudaError_t e = cudaSuccess;
    *pooled_ready = false;
    if (!rkey_cleared) e = cudaMemsetAsync(ctx->rkey, 0, sizeof(uint32_t) * (size_t)B * l_C, st);
    if (e != cudaSuccess) return e;
    if (l_C == 1) {
        ScoreDecodeParams p;
        p.kc = kc_cache; p.qc = ctx->Qc; p.rkey = ctx->rkey;
        p.pkey = ctx->pkey; p.status = ctx->status; p.B = B;
        p.max_tokens = ctx->cfg.max_tokens; p.eps = ctx->cfg.eps; p.meta = meta;
        // One CTA per SM, all sequences dealt out to the warps in equal shares: the smallest share that needs no more
        // warps than there are.
        const int warps = ctx->num_sms * SD_WARPS;
        int64_t total = 0;
        for (int b = 0; b < B; ++b) total += meta.m_end[b] - meta.i_end[b];
        int share = (int)((total + warps - 1) / warps);
        if (share < SD_MIN_SHARE) share = SD_MIN_SHARE;
        while (true) {
            p.n_warps = 0;
            for (int b = 0; b < B; ++b) {
                p.first_warp[b] = p.n_warps;
                p.n_warps += (meta.m_end[b] - meta.i_end[b] + share - 1) / share;
            }
            if (p.n_warps <= warps || share > max_lM) break;
            share += 1 + share / 64;
        }
        p.share = share;
        constexpr int smem = SD_WARPS * SD_STAGES * SD_STAGE_BYTES;
        static KernelMemo memo;
        e = allow_smem(score_decode_kernel<DC>, ctx->device, smem, memo, true);
        if (e != cudaSuccess) return e;
        ProfScope prof(ctx, KC_SCORE_DECODE, st);
        e = launch_pdl(score_decode_kernel<DC>, dim3((p.n_warps + SD_WARPS - 1) / SD_WARPS), dim3(SD_WARPS * 32), smem, st, p);
        ctx->launches += 1;
        *pooled_ready = true;
        return e;
    }
    return launch_score_tc(ctx, B, l_C, kc_cache, meta, max_lM, st, pooled_ready);
}

cudaError_t launch_score(esa_ctx* ctx, int B, int l_C, const __nv_bfloat16* kc_cache, const SeqMeta& meta,
                         int max_lM, bool rkey_cleared, cudaStream_t st, bool* pooled_ready) {
    switch (ctx->dc) {
        case 32: return launch_score_t<32>(ctx, B, l_C, kc_cache, meta, max_lM, rkey_cleared, st, pooled_ready);
        case 64: return launch_score_t<64>(ctx, B, l_C, kc_cache, meta, max_lM, rkey_cleared, st, pooled_ready);
        case 128: return launch_score_t<128>(ctx, B, l_C, kc_cache, meta, max_lM, rkey_cleared, st, pooled_ready);
    }
    return cudaErrorInvalidValue;
}

}  // namespace esa
