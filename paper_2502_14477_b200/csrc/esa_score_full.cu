// Eq. 3 + Eq. 4 on the full-dimension queries and keys (no compression), and the per-head vote of
// Section 4.3 -- the two scoring variants the paper compares its compressed scores against.
//
//   uniform    f_s(m; c) = sum_h q_{h,c} . k_{h,m}          (Eq. 3; head h reads key/value head h / G)
//              s_m = max_c ( f_s(m; c) - max_m' f_s(m'; c) )  (Eq. 4)
//   per head   every head h scores by itself, s_m^h = max_c ( q_{h,c} . k_{h,m} - max_m' q_{h,c} . k_{h,m'} ),
//              and s_m = max_h s_m^h
//
// Per head, a head is a scoring problem of the compressed kind with d' = d: it runs on the kernels of
// esa_score_tc.cu, one group of CTAs per head.  This file holds the uniform variant, a product with a long
// reduction, on tcgen05:
//
//   * The G heads of a group meet the same keys, so their queries can be added first: q_g = sum of G bf16 rows, an
//     fp32 number, cut into three bf16 pieces (24 bits: as exact as the fp32 sums that follow).  Three pieces in place
//     of G heads: fewer products from G = 4 on (below that the heads are taken one by one, same kernel).
//   * Two passes as for the compressed scores: pass 1 keeps the row maxima r_c, pass 2 forms the scores again and
//     folds max_c (S - r_c).  The operands swap sides between the passes (pass 1: queries on the tensor-memory lanes;
//     pass 2: keys), so both maxima run along a thread's own columns.  Every S is the same sum of the same products in
//     the same order in both passes: the score of a query's arg-max is exactly 0.
//   * A CTA owns one tile of up to 256 x 256 scores (two 128-row blocks, all 512 columns of tensor memory) and streams
//     the reduction in 64-column chunks: a chunk of keys stays in shared memory while the pieces (or heads) of the
//     queries that meet it pass through a ring of their own, so a chunk of 4096 products a score moves 42 bytes per
//     clock into the SM instead of 64.  The accumulators are not double-buffered: a tile's products take 26 us at
//     d_G = 1024, its epilogue 2.
//   Bound: tensor core.  512 queries, 32/8 heads of 128, both passes: 84 us at 18304 keys, 312 us at 63360 keys (mma.sync
//   kernels without folding: 563 and 1929 us); per head 150 and 424 us (739 and 2514).
#include "esa_internal.h"
#include "esa_umma.cuh"

namespace esa {

namespace {

constexpr int FT_THREADS = 320;    // TMA warp, MMA warp, eight epilogue warps
constexpr int FT_RING_BYTES = 200 * 1024;
constexpr int FT_MAX_SLOTS = 8;

struct FullTcParams {
    uint32_t* rkey;     // [B, l_C] ordered keys of r_c
    uint32_t* skey;     // [B, max_tokens] ordered keys of s_m (index = m - i_end)
    int* status;
    int64_t max_tokens;
    int l_C;
    int blocks;         // 128-row blocks on the lane side: 1 or 2
    int n;              // rows on the column side: 64, 128 or 256
    int k_slots, q_slots;
    int k_chunks;       // 64-column chunks of a key row
    int pieces;         // query chunks that meet one key chunk
    int folded;         // 1: piece p of chunk i is column p * d_G + 64 i of the folded queries; 0: a head of the group
    int d, G, dG;
    SeqMeta meta;
};

enum { FB_K_FULL = 0, FB_K_EMPTY = FB_K_FULL + FT_MAX_SLOTS, FB_Q_FULL = FB_K_EMPTY + FT_MAX_SLOTS,
       FB_Q_EMPTY = FB_Q_FULL + FT_MAX_SLOTS, FB_ACC = FB_Q_EMPTY + FT_MAX_SLOTS, FB_COUNT };

__device__ __forceinline__ float max3_full(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;\n" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// grid: (key tiles, query tiles, B)
template <int PASS>
__global__ void __launch_bounds__(FT_THREADS, 1)
score_full_tc_kernel(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap qmap, FullTcParams p) {
    extern __shared__ uint8_t smem_dyn[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t bars[FB_COUNT];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ __align__(16) float sR[256];                 // pass 2: r_c of this tile's queries

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int b = blockIdx.z;
    const int i_end = p.meta.i_end[b], l_M = p.meta.m_end[b] - i_end;
    const int x_rows = p.blocks * 128;                      // lane side
    const int key_rows = PASS == 1 ? p.n : x_rows, q_rows = PASS == 1 ? x_rows : p.n;
    const int key0 = blockIdx.x * key_rows, q0 = blockIdx.y * q_rows;
    const bool work = key0 < l_M;
    const uint32_t k_bytes = key_rows * 128, q_bytes = q_rows * 128;
    uint8_t* sK = smem;
    uint8_t* sQ = smem + p.k_slots * k_bytes;

    WaitCtx wc{&abort_flag, p.status};
    auto bar = [&](int i) { return smem_u32(&bars[i]); };
    if (tid == 0) {
        abort_flag = 0;
        for (int i = 0; i < FB_COUNT; ++i) mbar_init(bar(i), 1);
        mbar_init_fence();
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_slot), 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_slot;

    if (warp == 0) {
        if (lane == 0 && work) {
            tma_prefetch_desc(&kmap);
            tma_prefetch_desc(&qmap);
            const int krow = i_end + key0, qrow = b * p.l_C + q0;
            const int k_box = min(128, key_rows), q_box = min(128, q_rows);
            int qi = 0;
            // the queries may come from the preceding kernel; the keys are older (see launch_score_full)
            bool waited = false;
            for (int i = 0; i < p.k_chunks; ++i) {
                const int s = i % p.k_slots;
                mbar_wait(bar(FB_K_EMPTY + s), ((i / p.k_slots) & 1) ^ 1, wc);
                mbar_arrive_expect_tx(bar(FB_K_FULL + s), k_bytes);
                for (int r = 0; r < key_rows; r += k_box)
                    tma_load_3d(smem_u32(sK + s * k_bytes + r * 128), &kmap, i * 64, krow + r, b, bar(FB_K_FULL + s));
                if (!waited) {
                    pdl_wait();
                    waited = true;
                }
                for (int j = 0; j < p.pieces; ++j, ++qi) {
                    const int col = p.folded ? (p.pieces - 1 - j) * p.dG + i * 64
                                             : ((i * 64) / p.d * p.G + j) * p.d + (i * 64) % p.d;
                    const int t = qi % p.q_slots;
                    mbar_wait(bar(FB_Q_EMPTY + t), ((qi / p.q_slots) & 1) ^ 1, wc);
                    mbar_arrive_expect_tx(bar(FB_Q_FULL + t), q_bytes);
                    for (int r = 0; r < q_rows; r += q_box)
                        tma_load_2d(smem_u32(sQ + t * q_bytes + r * 128), &qmap, col, qrow + r, bar(FB_Q_FULL + t));
                }
            }
        }
    } else if (warp == 1) {
        if (work) {
            const uint32_t lead = lane == 0, hi = desc_hi_sw128();
            const uint32_t idesc = idesc_bf16(128, p.n, false, false);
            const uint32_t klo = desc_lo_kmajor(smem_u32(sK)), qlo = desc_lo_kmajor(smem_u32(sQ));
            int qi = 0;
            for (int i = 0; i < p.k_chunks; ++i) {
                const int s = i % p.k_slots;
                mbar_wait(bar(FB_K_FULL + s), (i / p.k_slots) & 1, wc);
                const uint32_t k0 = klo + ((s * k_bytes) >> 4);
                for (int j = 0; j < p.pieces; ++j, ++qi) {
                    const int t = qi % p.q_slots;
                    mbar_wait(bar(FB_Q_FULL + t), (qi / p.q_slots) & 1, wc);
                    tc_fence_after_sync();
                    const uint32_t qq = qlo + ((t * q_bytes) >> 4);
                    for (int mb = 0; mb < p.blocks; ++mb) {
                        const uint32_t a = (PASS == 1 ? qq : k0) + mb * ((128 * 128) >> 4), c = PASS == 1 ? k0 : qq;
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            umma_ss(tmem + mb * p.n, a + ks * 2, c + ks * 2, hi, idesc, qi | ks, lead);
                    }
                    umma_commit(bar(FB_Q_EMPTY + t), lead);
                }
                umma_commit(bar(FB_K_EMPTY + s), lead);
            }
            umma_commit(bar(FB_ACC), lead);
        }
    } else {
        // ------------------------------------------------------------ epilogue: two groups of four warps
        const int quarter = warp & 3, grp = (warp - 2) >> 2;
        const int et = quarter * 32 + lane;
        pdl_wait();
        pdl_launch_dependents();
        if (PASS == 2) {
            const int c = (warp - 2) * 32 + lane;
            sR[c] = (c < p.n && q0 + c < p.l_C) ? key_to_f32(__ldcg(p.rkey + (int64_t)b * p.l_C + q0 + c)) : INFINITY;
            asm volatile("bar.sync 1, 256;\n" ::: "memory");
        }
        if (work) {
            // two blocks: one group each; one block: half of the columns each
            const int mb = p.blocks == 2 ? grp : 0;
            const int ncol = p.blocks == 2 ? p.n : p.n / 2, c_lo = p.blocks == 2 ? 0 : grp * ncol;
            const uint32_t t0 = tmem_addr(tmem, quarter * 32, mb * p.n + c_lo);
            mbar_wait(bar(FB_ACC), 0, wc);
            tc_fence_after_sync();
            float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
            for (int c = 0; c < ncol; c += 32) {
                uint32_t v[32];
                tmem_ld32(t0 + c, v);
                tmem_wait_ld();
                if (PASS == 1) {
                    const int first = key0 + c_lo + c;               // keys of these columns; those past M never win
                    if (first + 32 > l_M) {
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (first + j >= l_M) v[j] = 0xff800000u;
                    }
#pragma unroll
                    for (int j = 0; j < 32; j += 8) {
                        m0 = max3_full(m0, __uint_as_float(v[j]), __uint_as_float(v[j + 1]));
                        m1 = max3_full(m1, __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
                        m2 = max3_full(m2, __uint_as_float(v[j + 4]), __uint_as_float(v[j + 5]));
                        m3 = max3_full(m3, __uint_as_float(v[j + 6]), __uint_as_float(v[j + 7]));
                    }
                } else {
                    const float4* r4 = reinterpret_cast<const float4*>(sR + c_lo + c);
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        const float4 r = r4[j / 4];
                        m0 = fmaxf(m0, __uint_as_float(v[j]) - r.x);
                        m1 = fmaxf(m1, __uint_as_float(v[j + 1]) - r.y);
                        m2 = fmaxf(m2, __uint_as_float(v[j + 2]) - r.z);
                        m3 = fmaxf(m3, __uint_as_float(v[j + 3]) - r.w);
                    }
                }
            }
            const float mx = fmaxf(max3_full(m0, m1, m2), m3);
            const int row = mb * 128 + et;
            if (PASS == 1) {
                if (q0 + row < p.l_C) atomicMax(p.rkey + (int64_t)b * p.l_C + q0 + row, f32_to_key(mx));
            } else {
                if (key0 + row < l_M) atomicMax(p.skey + (int64_t)b * p.max_tokens + key0 + row, f32_to_key(mx));
            }
        }
    }
    // (every thread passes the wait for the preceding kernel before the CTA ends: a CTA's exit also releases the
    // dependents, and they must not start ahead of the kernels before this one)
    pdl_wait();
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, 512);
}

// First launch of a call: clears what the passes accumulate into, and (fold) writes the group sums of the queries as
// three bf16 pieces, Qf [rows, 3 d_G], piece p of the sum in columns p d_G ...
__global__ void __launch_bounds__(256)
full_prepare_kernel(const __nv_bfloat16* __restrict__ Q, __nv_bfloat16* __restrict__ Qf, int64_t rows, int dG, int d, int G, int fold,
                    uint32_t* __restrict__ rkey, int64_t n_rkey, uint32_t* __restrict__ skey, int64_t max_tokens, int clear_keys,
                    int B) {
    pdl_wait();
    pdl_launch_dependents();
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = i0; i < n_rkey; i += step) rkey[i] = 0u;
    for (int64_t i = i0; i < (int64_t)B * clear_keys; i += step) skey[i / clear_keys * max_tokens + i % clear_keys] = 0u;
    if (!fold) return;
    const int per_row = dG / 2;
    for (int64_t i = i0; i < rows * per_row; i += step) {
        const int64_t row = i / per_row;
        const int col = (int)(i % per_row) * 2, g = col / d, c = col % d;
        const __nv_bfloat16* q = Q + (row * dG + (int64_t)g * d) * G + c;      // head g G of the row
        float2 s = make_float2(0.f, 0.f);
        for (int h = 0; h < G; ++h) {
            const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(q + h * d));
            s.x += x.x;
            s.y += x.y;
        }
#pragma unroll
        for (int pc = 0; pc < 3; ++pc) {
            const uint32_t w = pack_bf16(s.x, s.y);
            *reinterpret_cast<uint32_t*>(Qf + (row * 3 + pc) * dG + col) = w;
            s.x -= __uint_as_float(w << 16);
            s.y -= __uint_as_float(w & 0xffff0000u);
        }
    }
}

// Tile of one pass: rows on the lane side (blocks x 128) and on the column side (n).  Large tiles read least, small
// ones give a short chunk or a short context enough CTAs; the choice minimises waves x (cycles of a tile's products or
// of its loads, whichever is longer, + a fixed 6000 for start-up and epilogue).  86 cycles: what one issuing warp needs
// per instruction of 128 columns or fewer; 56 bytes per clock: what an SM was seen to load here.
struct FullTile { int blocks, n, k_slots, q_slots, key_rows, q_rows; };
FullTile pick_tile(int pass, int l_C, int max_lM, int B, int k_chunks, int pieces, int num_sms) {
    FullTile best = {};
    double best_cost = -1;
    for (int blocks = 1; blocks <= 2; ++blocks)
        for (int n = 64; n <= 256; n *= 2) {
            const int kr = pass == 1 ? n : blocks * 128, qr = pass == 1 ? blocks * 128 : n;
            const int64_t tiles = (int64_t)((max_lM + kr - 1) / kr) * ((l_C + qr - 1) / qr) * B;
            const double mma = (double)blocks * 4 * (n / 2 > 86 ? n / 2 : 86) * pieces;
            const double load = (kr + (double)pieces * qr) * 128 / 56;
            const double cost = (double)((tiles + num_sms - 1) / num_sms) * (k_chunks * (mma > load ? mma : load) + 6000);
            if (best_cost < 0 || cost < best_cost) {
                best_cost = cost;
                best.blocks = blocks; best.n = n; best.key_rows = kr; best.q_rows = qr;
                best.k_slots = kr <= 128 ? 4 : 2;
                int qs = (FT_RING_BYTES - best.k_slots * kr * 128) / (qr * 128);
                best.q_slots = qs < FT_MAX_SLOTS ? qs : FT_MAX_SLOTS;
            }
        }
    return best;
}

template <int PASS>
cudaError_t launch_pass(esa_ctx* ctx, FullTcParams p, const FullTile& t, const CUtensorMap& kmap, const CUtensorMap& qmap, int B,
                        int max_lM, cudaStream_t st) {
    static KernelMemo memo;
    cudaError_t e = allow_smem(score_full_tc_kernel<PASS>, ctx->device, FT_RING_BYTES + 1024, memo);
    if (e != cudaSuccess) return e;
    p.blocks = t.blocks; p.n = t.n; p.k_slots = t.k_slots; p.q_slots = t.q_slots;
    const dim3 grid((max_lM + t.key_rows - 1) / t.key_rows, (p.l_C + t.q_rows - 1) / t.q_rows, B);
    const size_t smem = (size_t)t.k_slots * t.key_rows * 128 + (size_t)t.q_slots * t.q_rows * 128 + 1024;
    e = launch_pdl(score_full_tc_kernel<PASS>, grid, dim3(FT_THREADS), smem, st, kmap, qmap, p);
    ctx->launches += 1;
    return e;
}

}  // namespace

// The folded queries go to the attention's scratch (written and read within the attention kernel, idle here).
// Three pieces beat the heads of a group from four heads on.
bool score_full_folds(const esa_ctx* ctx, int64_t rows, bool per_head) {
    return !per_head && ctx->G > 3 && (size_t)rows * 3 * ctx->dG * 2 <= ctx->att_part_elems * sizeof(float);
}

// Fills ctx->skey with the unpooled full-dimension scores (ordered keys).
// The keys of M may be loaded ahead of a pass's wait for the kernel before it: everything enqueued ahead of the call
// has completed when the first launch below lets its dependents start, and M ends before the current chunk.
cudaError_t launch_score_full(esa_ctx* ctx, int B, int l_C, const __nv_bfloat16* Q, const __nv_bfloat16* K, const SeqMeta& meta,
                              int max_lM, bool per_head, cudaStream_t st) {
    const int64_t rows = (int64_t)B * l_C;
    const bool fold = score_full_folds(ctx, rows, per_head);
    __nv_bfloat16* Qf = reinterpret_cast<__nv_bfloat16*>(ctx->att_part);
    const int64_t n_rkey = rows * (per_head ? ctx->H : 1);
    int gx = (int)((rows * (fold ? ctx->dG / 2 : 0) + (int64_t)B * max_lM + 511) / 512);
    if (gx > 4 * ctx->num_sms) gx = 4 * ctx->num_sms;
    if (gx < 1) gx = 1;
    ProfScope prof(ctx, KC_SCORE_FULL, st);
    cudaError_t e = launch_pdl(full_prepare_kernel, dim3(gx), dim3(256), 0, st, Q, Qf, rows, ctx->dG, ctx->d, ctx->G, fold ? 1 : 0,
                               ctx->rkey_heads, n_rkey, ctx->skey, ctx->cfg.max_tokens, per_head ? 0 : max_lM, B);
    if (e != cudaSuccess) return e;
    ctx->launches += 1;
    if (per_head) return launch_score_tc_heads(ctx, B, l_C, Q, K, meta, max_lM, st);

    FullTcParams p;
    p.rkey = ctx->rkey_heads; p.skey = ctx->skey; p.status = ctx->status;
    p.max_tokens = ctx->cfg.max_tokens; p.l_C = l_C; p.meta = meta;
    p.k_chunks = ctx->dG / 64; p.pieces = fold ? 3 : ctx->G; p.folded = fold ? 1 : 0;
    p.d = ctx->d; p.G = ctx->G; p.dG = ctx->dG;
    const FullTile t1 = pick_tile(1, l_C, max_lM, B, p.k_chunks, p.pieces, ctx->num_sms);
    const FullTile t2 = pick_tile(2, l_C, max_lM, B, p.k_chunks, p.pieces, ctx->num_sms);
    const __nv_bfloat16* qbase = fold ? Qf : Q;
    const uint64_t qcols = fold ? 3 * (uint64_t)ctx->dG : (uint64_t)ctx->dH, krows = ctx->cfg.max_tokens;
    CUtensorMap k1, q1, k2, q2;
    auto box = [](int r) { return (uint32_t)(r < 128 ? r : 128); };
    if (!make_tensor_map_cache(&k1, K, B, krows, ctx->dG, box(t1.key_rows)) || !make_tensor_map_bf16(&q1, qbase, rows, qcols, box(t1.q_rows)) ||
        !make_tensor_map_cache(&k2, K, B, krows, ctx->dG, box(t2.key_rows)) || !make_tensor_map_bf16(&q2, qbase, rows, qcols, box(t2.q_rows)))
        return cudaErrorInvalidValue;
    e = launch_pass<1>(ctx, p, t1, k1, q1, B, max_lM, st);
    if (e == cudaSuccess) e = launch_pass<2>(ctx, p, t2, k2, q2, B, max_lM, st);
    return e;
}

}  // namespace esa
