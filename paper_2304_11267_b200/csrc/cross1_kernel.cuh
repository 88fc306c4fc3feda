// Cross-attention with every key of a (batch, head) in ONE shared-memory tile (Nk <= 128): the softmax of Eq. 3 needs no
// running rescale.  One CTA per tile of 128 query rows, two to four of them resident per SM; one launch serves up to
// X1_GROUP_MAX problems of one shape.
//
// Bound: latency.  A call of the UNet is 16 to 512 tiles, so what counts is the length of ONE tile's chain -- fetch, scores,
// softmax, product, output -- and most of it used to be the instructions of single threads.  Measured on 64 tokens at
// d = 160, in clocks: nine tiled copies issued one after another 1300 (and 900 of latency), the MMAs in a run-time loop 1300,
// a row of 64 weights per thread 950, and 40 row-strided stores of it 1900.  Hence three warps issue the copies of Q, K and V,
// S of a 64-column chunk starts when that chunk has landed, both products come from unrolled code of threads of their own,
// a row's output columns are fetched from tensor memory together (a load and its wait are 130 clocks), and leave through
// shared memory as whole lines.  (Fetching by 16-byte asynchronous copies of all threads, straight into the swizzled layout, was
// slower, 6.8 us a call against 5.0; so were two threads per row, 5.4.)
// DENSE: a tiled copy costs the copy engine about 7 clocks per 80-byte row, 2000 for a tile of d = 40, which queues behind
// the SM's other CTAs.  Rows of a head-major tensor are one contiguous run, so at d <= 48 Q, K and V come as three untiled
// copies, and all threads move the rows into the swizzled layout, in place: every thread holds its two rows in registers across
// one barrier.  (At d = 80 the rows take longer to move than to fetch: 7.0 us against 5.5.)
// Tiles of 64 rows, when that many CTAs still fit the GPU at once: the products are 128 rows high all the same, but fetch,
// output and bank traffic of a tile halve (256 x 77, d = 160, B = 2: 5.8 -> 5.2 us; 32 rows gain nothing more).
// Measured against the persistent kernel (cross2) and the one-tile kernel before it: 4096 x 77 d = 40 7.3 -> 6.1 us, 1024 x 77
// d = 80 5.7 -> 5.0, 256 x 77 d = 160 6.2 -> 5.2, 64 x 64 d = 160 5.3 -> 4.4 (CUDA graphs).
// The maximum as anchor, where a weight above it needs no second look, against an anchor at the first score (CUDA graphs, us):
// 64 keys 4.4 -> 4.4 (16 x 64 rows, d = 160), 17.1 -> 17.4 (64 x 4096, d = 40); 16 keys 4.55 -> 4.7; 128 keys 5.35 -> 5.4, 35.1 ->
// 37.2.  The largest weight is then exact; the error that the weights' rounding leaves in the result falls from 2.0e-4 to 1.6e-4 for
// logits of deviation 1, from 1.8e-4 to 6.8e-5 for 4 (64 keys, binary16, simulated).
// Tensor memory: S takes KN columns; the weights P (packed 16-bit) go over its first KN / 2 and O behind them, over scores
// that sit in registers.
#pragma once
#include <cuda.h>

#include "cross_common.cuh"   // TILE_M, CHUNK_COLS, CHUNK_ROW_BYTES
#include "softmax_math.cuh"
#include "tc_common.cuh"

namespace sd_attn {

constexpr int X1_THREADS = 192;            // four softmax warps (thread = query row), two MMA issuers
constexpr int X1_GROUP_MAX = 5;            // problems of one shape per launch
constexpr float X1_HEADROOM_LOG2 = 8.0f;   // 65..80 keys: exponents are anchored 2^8 above the first key's weight (see cross2_kernel.cuh)
constexpr float X1_SUM_LIMIT = 4096.0f;    // no weight above 2^12 reaches the 16-bit pack
enum { SITE_X1_QK = 90, SITE_X1_V = 91, SITE_X1_S = 92, SITE_X1_P = 93, SITE_X1_O = 94 };

struct Cross1Problem {
    CUtensorMap tq, tk, tv;            // (not used by DENSE)
    const __half *q, *k, *v;           // (DENSE)
    __half* out;
    float scale_log2e;  // |scale| * log2(e)
    int negate;         // scale < 0: the MMA negates Q
};
template <int NP>       // NP = 1: a launch of one problem; else X1_GROUP_MAX
struct Cross1ArgsT {
    HeadLayout lay;     // heads of q and out
    int Nq, Nk, d;
    int tile_rows;      // query rows per CTA: 128 or 64
    int tmem_cols;      // see x1_tmem_cols
    int* status;
    Cross1Problem prob[NP];
};

// Columns of tensor memory: S (KN), or P and behind it O; a power of two.
__host__ inline int x1_tmem_cols(int kn, int dpad) {
    const int need = kn > kn / 2 + dpad ? kn : kn / 2 + dpad;
    return need <= 64 ? 64 : need <= 128 ? 128 : 256;
}
// Keys of a tile: the instances there are (80: the 77 text tokens).
__host__ inline int x1_key_tile(int Nk) { return Nk <= 64 ? 64 : Nk <= 80 ? 80 : 128; }
constexpr int X1_DENSE_PIECES = 6;         // 16-byte pieces of a row DENSE holds in registers: d <= 48
__host__ inline bool x1_dense(int d, int kn, bool head_major) { return head_major && kn <= 80 && d <= 8 * X1_DENSE_PIECES; }
__host__ inline size_t x1_smem_bytes(int nch, int kn) { return (size_t)nch * (TILE_M + 2 * kn) * CHUNK_ROW_BYTES + 1024; }

// KN: keys rounded up (a multiple of 16: the N of S, the contraction of P V).  NCH: 64-column chunks of a row.  BF: bfloat16.
template <int KN, int NCH, bool DENSE, bool BF, int NP>
__global__ void __launch_bounds__(X1_THREADS)
cross1_attention_kernel(const __grid_constant__ Cross1ArgsT<NP> args) {
    extern __shared__ uint8_t x1_smem_raw[];
    __shared__ __align__(8) uint64_t bars[4 + NCH];   // V landed | S ready | P ready | O ready | chunks of Q and K landed
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int tile = blockIdx.x, bh = blockIdx.y, row0 = tile * args.tile_rows, d = args.d;
    const Cross1Problem& pr = args.prob[NP == 1 ? 0 : blockIdx.z];
    constexpr uint32_t Q_BYTES = NCH * TILE_M * CHUNK_ROW_BYTES, KV_BYTES = NCH * KN * CHUNK_ROW_BYTES;
    const uint32_t q_smem = (smem_u32(x1_smem_raw) + 1023u) & ~1023u, k_smem = q_smem + Q_BYTES, v_smem = k_smem + KV_BYTES;
    const uint32_t bar_v = smem_u32(&bars[0]), bar_s = smem_u32(&bars[1]), bar_p = smem_u32(&bars[2]), bar_o = smem_u32(&bars[3]),
                   bar_qk = smem_u32(&bars[4]);
    volatile int* abort_p = &abort_flag;
    if (tid == 0) {
        pdl_launch_dependents();
        abort_flag = 0;
        for (int ch = 0; ch < NCH; ++ch) mbar_init(bar_qk + ch * 8, DENSE ? 1 : 2);
        mbar_init(bar_v, 1);
        mbar_init(bar_s, 1);
        mbar_init(bar_p, args.tile_rows >> 5);
        mbar_init(bar_o, 1);
        mbar_init_fence();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&tmem_base_slot), (uint32_t)args.tmem_cols);
        tmem_relinquish();
    }
    if (!DENSE) {
        if (warp == 4 && elect_one()) tma_prefetch_desc(&pr.tq);
        if (warp == 5 && elect_one()) tma_prefetch_desc(&pr.tk);
        if (warp == 2 && elect_one()) tma_prefetch_desc(&pr.tv);
    }
    int bz, hz;
    split_head(args.lay, bh, bz, hz);
    // what the roles read of the parameters, whose first touch misses the constant cache
    asm volatile("" ::"l"(pr.out), "f"(pr.scale_log2e), "r"(pr.negate), "r"(args.lay.ld), "l"(args.lay.head_stride), "l"(args.lay.batch_stride),
                 "r"(args.Nq), "r"(args.Nk), "r"(bz), "r"(hz));
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    pdl_wait();   // set-up overlapped the tail of the stream's previous kernel
    const uint32_t tmem_s = tmem_base_slot, tmem_o = tmem_s + KN / 2;   // P over the first KN / 2 columns of S

    bool fetched = true;
    if (DENSE) {
        const uint32_t row_bytes = (uint32_t)d * 2, raw_k = q_smem + TILE_M * row_bytes, raw_v = raw_k + KN * row_bytes;
        const int q_rows = min(args.tile_rows, args.Nq - row0), kv_rows = args.Nk;
        if (tid == 0) {
            mbar_arrive_expect_tx(bar_qk, (uint32_t)(q_rows + 2 * kv_rows) * row_bytes);
            bulk_load(q_smem, pr.q + ((size_t)bh * args.Nq + row0) * d, (uint32_t)q_rows * row_bytes, bar_qk);
            bulk_load(raw_k, pr.k + (size_t)bh * kv_rows * d, (uint32_t)kv_rows * row_bytes, bar_qk);
            bulk_load(raw_v, pr.v + (size_t)bh * kv_rows * d, (uint32_t)kv_rows * row_bytes, bar_qk);
        }
        // rows 0..127 are Q's, then KN of K, KN of V; thread t moves rows t and t + 192 (rows past the end become zeros)
        constexpr int ROWS = TILE_M + 2 * KN, PP = X1_DENSE_PIECES;
        static_assert(ROWS <= 2 * X1_THREADS, "two rows per thread");
        const int pieces = d >> 3, padded = (d + 15) >> 4 << 1;
        fetched = mbar_wait_eager(bar_qk, 0, abort_p, args.status, SITE_X1_QK, tile);
        uint4 v[2][PP];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int r = tid + u * X1_THREADS;
            const bool there = fetched && (r < TILE_M ? r < q_rows : r < TILE_M + KN ? r - TILE_M < kv_rows : r < ROWS && r - TILE_M - KN < kv_rows);
            const uint32_t src = q_smem + (uint32_t)r * row_bytes;   // (raw K and V lie behind raw Q, KN rows each)
#pragma unroll
            for (int p = 0; p < PP; ++p) v[u][p] = there && p < pieces ? ld_shared_v4(src + p * 16) : make_uint4(0u, 0u, 0u, 0u);
        }
        fetched = __syncthreads_and(fetched);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int r = tid + u * X1_THREADS;
            const int k = r - TILE_M, rr = r < TILE_M ? r : k < KN ? k : k - KN;                       // row inside its operand
            const uint32_t base = r < TILE_M ? q_smem : k < KN ? k_smem : v_smem, chunk = (r < TILE_M ? TILE_M : KN) * CHUNK_ROW_BYTES;
            if (fetched && r < ROWS) {
#pragma unroll
                for (int p = 0; p < PP; ++p)
                    if (p < padded) st_shared_v4(base + (p >> 3) * chunk + rr * CHUNK_ROW_BYTES + (((p & 7) ^ (rr & 7)) << 4), v[u][p]);
            }
        }
        fence_proxy_async_smem();   // generic-proxy stores before the tensor core reads them
        __syncthreads();
    }

    if (warp == 4) {
        if (fetched && elect_one()) {
            const uint32_t idesc = idesc_f16(TILE_M, KN, false, false, pr.negate != 0, BF);
            const int ksteps = (d + 15) >> 4;
            const uint64_t q_desc = smem_desc_sw128(q_smem, 16, 1024), k_desc = smem_desc_sw128(k_smem, 16, 1024);
            if (!DENSE) {
#pragma unroll
                for (int ch = 0; ch < NCH; ++ch) {
                    mbar_arrive_expect_tx(bar_qk + ch * 8, (uint32_t)(args.tile_rows * CHUNK_ROW_BYTES));
                    tma_load_4d(q_smem + ch * TILE_M * CHUNK_ROW_BYTES, &pr.tq, bar_qk + ch * 8, ch * CHUNK_COLS, row0, hz, bz);
                }
            }
            bool landed = true;
#pragma unroll
            for (int ch = 0; ch < NCH; ++ch) {
                if (!DENSE) landed = landed && mbar_wait_eager(bar_qk + ch * 8, 0, abort_p, args.status, SITE_X1_QK, tile);
                if (!landed) break;
                tc_fence_after_sync();
#pragma unroll
                for (int kk = 4 * ch; kk < 4 * ch + 4; ++kk)
                    if (kk < ksteps)
                        mma_f16_ss(tmem_s, q_desc + (uint64_t)(((kk >> 2) * TILE_M * CHUNK_ROW_BYTES + (kk & 3) * 32) >> 4),
                                   k_desc + (uint64_t)(((kk >> 2) * KN * CHUNK_ROW_BYTES + (kk & 3) * 32) >> 4), idesc, kk > 0);
            }
            if (landed) tc_commit(bar_s);
        }
    } else if (warp == 5) {
        if (fetched && elect_one()) {
            if (!DENSE) {
#pragma unroll
                for (int ch = 0; ch < NCH; ++ch) {
                    mbar_arrive_expect_tx(bar_qk + ch * 8, KV_BYTES / NCH);
                    tma_load_4d(k_smem + ch * KN * CHUNK_ROW_BYTES, &pr.tk, bar_qk + ch * 8, ch * CHUNK_COLS, 0, hz, bz);
                }
                // V behind K: the copy engine takes rows one after the other, and the scores wait for K's
                mbar_arrive_expect_tx(bar_v, KV_BYTES);
#pragma unroll
                for (int ch = 0; ch < NCH; ++ch)
                    tma_load_4d(v_smem + ch * KN * CHUNK_ROW_BYTES, &pr.tv, bar_v, ch * CHUNK_COLS, 0, hz, bz);
            }
            const uint32_t idesc = idesc_f16(TILE_M, (d + 15) >> 4 << 4, false, true, false, BF);
            const uint64_t v_desc = smem_desc_sw128(v_smem, KN * CHUNK_ROW_BYTES, 1024);
            if ((DENSE || mbar_wait(bar_v, 0, abort_p, args.status, SITE_X1_V, tile)) &&
                mbar_wait_eager(bar_p, 0, abort_p, args.status, SITE_X1_P, tile)) {
                tc_fence_after_sync();
#pragma unroll
                for (int kk = 0; kk < KN / 16; ++kk)
                    mma_f16_ts(tmem_o, tmem_s + kk * 8, v_desc + (uint64_t)((kk * 16 * CHUNK_ROW_BYTES) >> 4), idesc, kk > 0);
                tc_commit(bar_o);
            }
        }
    } else {
        // ---- softmax: thread = query row = TMEM lane; the weights stay in registers
        const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
        const int valid = args.Nk;
        const float c2 = pr.scale_log2e;
        uint32_t packed[KN / 2];
        float row_sum = 0.f, anchor = 0.f;
        // (a tile of fewer rows leaves the other warps without)
        bool ok = fetched && warp * 32 < args.tile_rows && mbar_wait_eager(bar_s, 0, abort_p, args.status, SITE_X1_S, tile);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) {
            tc_fence_after_sync();
            uint64_t acc[2] = {0ull, 0ull};
            float tail = 0.f;
            auto load_32 = [&](int c, uint32_t* s) {   // scores c .. c + 31 (fewer at the end of 80)
                if (c + 32 <= KN) tmem_ld32(tmem_s + lane_off + c, *reinterpret_cast<uint32_t(*)[32]>(s));
                else tmem_ld16(tmem_s + lane_off + c, *reinterpret_cast<uint32_t(*)[16]>(s));
            };
            auto weights_32 = [&](int c, const uint32_t* s) {   // their weights, packed, and the weights' sum
                const float neg_mc = -anchor;
                const uint64_t c2c2 = pack_b64(__float_as_uint(c2), __float_as_uint(c2));
                const uint64_t nmnm = pack_b64(__float_as_uint(neg_mc), __float_as_uint(neg_mc));
                if (c + 32 > KN) exp2_pack_32_masked<8, BF>(s, c2, neg_mc, c, valid, &packed[c / 2], tail);
                else if (valid >= c + 32) exp2_pack_32<0, 16, BF>(s, c2c2, nmnm, &packed[c / 2], acc);
                else exp2_pack_32_masked<16, BF>(s, c2, neg_mc, c, valid, &packed[c / 2], tail);   // (keys past Nk: zeros)
            };
            if constexpr (KN != 80) {
                // Anchored at the maximum, L_i of Eq. 4: the largest weight is 1, which 16 bits hold exactly.  A block of scores is
                // held in registers (DENSE: of 32, so that a fourth CTA fits); only 128 keys, and DENSE, fetch one again.
                constexpr int HELD = DENSE ? 32 : 64;
                uint32_t s[HELD];
                float row_max = -INFINITY;
#pragma unroll
                for (int c = 0; c < KN; c += HELD) {
#pragma unroll
                    for (int u = 0; u < HELD; u += 32) load_32(c + u, &s[u]);
                    tmem_wait_ld();
                    row_max = fmaxf(row_max, valid >= c + HELD ? row_max_3<HELD>(s) : row_max_first<HELD>(s, valid - c));
                }
                anchor = row_max * c2;
#pragma unroll
                for (int c = KN - HELD; c >= 0; c -= HELD) {   // (from the end: the last block is there)
                    if (c < KN - HELD) {
#pragma unroll
                        for (int u = 0; u < HELD; u += 32) load_32(c + u, &s[u]);
                        tmem_wait_ld();
                    }
#pragma unroll
                    for (int u = HELD - 32; u >= 0; u -= 32) weights_32(c + u, &s[u]);
                }
                row_sum = sum_f32x2(acc[0], acc[1]) + tail;   // S_i of Eq. 4, relative to the anchor
            } else {
                // as the persistent kernel anchors them, so that the two give the same bits
#pragma unroll 1
                for (int attempt = 0; attempt < 2; ++attempt) {
                    acc[0] = acc[1] = 0ull;
                    tail = 0.f;
#pragma unroll
                    for (int c = 0; c < KN; c += 32) {
                        uint32_t s[32];
                        load_32(c, s);
                        tmem_wait_ld();
                        if (c == 0 && attempt == 0) anchor = __uint_as_float(s[0]) * c2 + X1_HEADROOM_LOG2;
                        weights_32(c, s);
                    }
                    row_sum = sum_f32x2(acc[0], acc[1]) + tail;
                    const bool over = !(row_sum <= X1_SUM_LIMIT);
                    if (attempt == 1 || !__any_sync(0xffffffffu, over)) break;
                    // rare: the row maximum lies far above the first score.  Nothing has been stored yet: take the maximum
                    // from the scores and redo the row.
                    float row_max = -INFINITY;
                    for (int c = 0; c < KN; c += 16) {
                        uint32_t s[16];
                        tmem_ld16(tmem_s + lane_off + c, s);
                        tmem_wait_ld();
                        row_max = fmaxf(row_max, row_max_masked<16>(s, valid - c));
                    }
                    anchor = row_max * c2;
                }
            }
#pragma unroll
            for (int c = 0; c < KN / 2; c += 8) tmem_st8(tmem_s + lane_off + c, *reinterpret_cast<uint32_t(*)[8]>(&packed[c]));
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_p);
            ok = mbar_wait_eager(bar_o, 0, abort_p, args.status, SITE_X1_O, tile);
            ok = __all_sync(0xffffffffu, ok);
        }
        if (ok) {
            // ---- output: O / S_i -> 16 bits -> this warp's rows in shared memory (Q's, which S has consumed) -> whole lines
            tc_fence_after_sync();
            const float inv = 1.f / row_sum;
            const int pieces = d >> 3, swz = stage_swizzle(lane, pieces);
            const uint32_t rows = q_smem + warp * 32 * pieces * 16, own = rows + lane * pieces * 16;
            constexpr int CW = NCH == 1 ? 64 : 80;   // columns fetched together
#pragma unroll
            for (int c0 = 0; c0 < (NCH == 3 ? 160 : DENSE ? 8 * X1_DENSE_PIECES : NCH * CHUNK_COLS); c0 += CW) {
                if (c0 < d) {
                    uint32_t x[CW];
#pragma unroll
                    for (int c = 0; c < CW; c += 16)
                        if (c0 + c < d) tmem_ld16(tmem_o + lane_off + c0 + c, *reinterpret_cast<uint32_t(*)[16]>(&x[c]));
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < CW; c += 8) {
                        uint4 v8;
                        v8.x = pack_16x2<BF>(__uint_as_float(x[c + 0]) * inv, __uint_as_float(x[c + 1]) * inv);
                        v8.y = pack_16x2<BF>(__uint_as_float(x[c + 2]) * inv, __uint_as_float(x[c + 3]) * inv);
                        v8.z = pack_16x2<BF>(__uint_as_float(x[c + 4]) * inv, __uint_as_float(x[c + 5]) * inv);
                        v8.w = pack_16x2<BF>(__uint_as_float(x[c + 6]) * inv, __uint_as_float(x[c + 7]) * inv);
                        if (c0 + c < d) st_shared_v4(own + ((((c0 + c) >> 3) ^ swz) << 4), v8);
                    }
                }
            }
            __syncwarp();
            const int at = row0 + warp * 32;
            store_staged_rows(head_row(pr.out, args.lay, bh, at), args.lay, rows, pieces, min(32, args.Nq - at), lane);
        }
    }
    __syncwarp();
    if (tid == 0 && abort_flag) {   // gave up: let the copies that may still be in flight land before shared memory is released
        for (int ch = 0; ch < (DENSE ? 1 : NCH); ++ch) mbar_drain(bar_qk + ch * 8, 0);
        if (!DENSE) mbar_drain(bar_v, 0);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_s, (uint32_t)args.tmem_cols);
}

}  // namespace sd_attn
