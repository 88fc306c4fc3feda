// Single-pass attention of binary32 tensors on the bf16 tensor cores, at binary32 precision.
//
// A binary32 value is the sum of three bfloat16 values, h = bf16(x), m = bf16(x - h), l = bf16(x - h - m): 3 x 8 bits hold
// its 24-bit significand exactly.  A product of two such sums is taken as the six of its nine terms that reach its last
// bits, h h + h m + m h + m m + h l + l h; the three left out are below 2^-24 of the product (r.m.s. 2^-27).  Each term
// is exact in the tensor core's binary32 accumulator input, so what remains is the rounding of the accumulation.  The tensor
// core truncates there, which over thousands of keys would add up to a bias: the product P V of every key tile therefore
// goes into a fresh accumulator and is added to the running output on the CUDA cores, rounded to nearest -- and inside a
// tile the small terms are issued first.  (4096 tokens, d = 40: relative error 2.9e-7, with plain binary32 FMAs 1.2e-6.)
//
// Eight columns left behind the whole 16-column steps of Q K^T (d = 40: 32 and 8) do not take six half-empty steps but share three: what
// they contribute is l h + h l, m m + m h and h m + h h, two terms a step, with [l | h], [m | m], [h | h] of Q against [h | l], [m | h],
// [m | h] of K.
//
// Bound: the softmax warps.  A key tile of two query tiles takes about 3900 clocks, of which a sweep is 2500 (clock stamps: exponentials,
// and on the half-rate integer pipe the splitting of the weights, with four warps a scheduler in it at once) and the rest waits and the
// addition of the product; six bf16 products per binary32 one are 960 tensor clocks per 128 x 64 tile of scores at d = 40.
//
// One CTA: T query tiles of 128 rows.  Warpgroups (four warps each):
//   softmax     two per query tile, thread = half a query row: its scores from tensor memory into registers, exp2, row sum; the
//               weights are split into three packed bf16 operands and stored over the scores.  Two such slots per query tile:
//               the next key tile's scores are computed meanwhile.  The same threads hold the row's output columns, half
//               each, and add the product of the previous key tile to them: O = O + P V.
//               (One thread per row and a warpgroup of its own for the addition took 3500 clocks per key tile for the
//               softmax alone, against 2900 of the tensor core for two query tiles.)
//   convert     K, V: binary32 rows from global memory (fetched a tile ahead into registers), split, stored in the 64-byte
//               swizzled layout (Q is converted by the softmax warps, which have nothing else to do yet)
//   issue       one thread per query tile and product: S_t = Q_t K^T, O_t = P_t V
// The exponents are anchored at the row maximum of the FIRST key tile: bf16 parts have binary32's range, so a later score may
// lie 2^64 above it before anything overflows; only then (the sum of a tile's weights says so) is the row re-anchored and the
// tile redone.
// The ends of binary32's range: a value above the largest bfloat16 (or an infinity) has no three parts, and weights of up to 2^64 may
// overflow a product whose result is finite.  Either leaves an infinity or a NaN in the row's output, never a wrong finite value:
// rows whose output is not finite are computed once more by the warp that holds them, with plain FMAs.  Values below 2^-109 lose
// their lowest bits (the parts end at bfloat16's smallest subnormal, 2^-133).
// Operands in shared memory are [part h, m, l][32-column chunk][row][64 bytes].  V is used as it lies (MN-major).  Where one
// query tile leaves room in tensor memory, its Q goes there: read from shared memory, 128 rows for each product of 32 or 64 keys
// were most of the product's time.
// us a call, half-empty steps, steps counted at run time, parts taken out with masks -> now: 16 x 4096 x 4096, d = 40 291 -> 271, 3000
// 196 -> 176; 16 x 1024, d = 64 29.8 -> 29.0, d = 80 35.9 -> 35.0; 16 x 600, d = 120 50.0 -> 40.8; 16 x 256, d = 160 27.6 -> 24.5.
// Every wait is bounded and reports to the status block.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "cross_common.cuh"  // TILE_M
#include "softmax_math.cuh"
#include "tc_common.cuh"

namespace sd_attn {

constexpr int F3_CHUNK = 32;        // columns per 64-byte swizzled row
constexpr int F3_MAX_TILES = 2;
enum { SITE_F_Q = 70, SITE_F_K = 71, SITE_F_KEMPTY = 72, SITE_F_V = 73, SITE_F_VEMPTY = 74, SITE_F_S = 75, SITE_F_SLOT = 76,
       SITE_F_P = 77, SITE_F_PV = 78, SITE_F_OFREE = 79 };

struct F32Args {
    const float *q, *k, *v;
    float* out;
    HeadLayout lq, lk;      // heads of q and out (Nq rows each), of k and v (Nk rows)
    int Nq, Nk, d;
    int units_per_head;     // ceil(query tiles of a head / T)
    float scale;
    float scale_log2e;      // |scale| * log2(e)
    int negate;             // scale < 0: the tensor core negates Q
    FastDiv by_pieces;      // division by the eight-column pieces of a row
    int* status;
};

// NC: 32-column chunks of a row (d <= 32 NC).  BN: keys per key tile.  T: query tiles per CTA.  ACC: output columns per
// softmax thread.  KS, VS: depth of the K and V rings.  NO: buffers for the product of a key tile.  MAX_FIRST: whether a key tile
// fits the anchor is decided from its maximum before the exponentials, so that the weights replace the scores in registers,
// not from the weights' sum behind them (measured: d = 80 43 -> 36 us; the other shapes lose 2% to 12% by it).  BELOW: head dims up to
// this one take a smaller shape.
template <int NC_, int BN_, int T_, int ACC_, int KS_, int VS_, int NO_, bool MAX_FIRST_, int BELOW_>
struct F32Shape {
    static constexpr int NC = NC_, BN = BN_, T = T_, ACC = ACC_, KS = KS_, VS = VS_, NO = NO_;
    static constexpr bool MAX_FIRST = MAX_FIRST_;
    static constexpr int MAX_D = NC * F3_CHUNK < 2 * ACC ? NC * F3_CHUNK : 2 * ACC;
    static constexpr int MIN_PIECES = BELOW_ / 8 + 1, MAX_PIECES = MAX_D / 8;   // of eight columns
    static constexpr int N_CONV = T == 2 ? 1 : 2;   // warpgroups that convert K; as many for V
    static constexpr int WG_CONVERT = 2 * T, WG_ISSUE = WG_CONVERT + 2 * N_CONV, THREADS = (WG_ISSUE + 1) * 128;
    static constexpr int Q_PART = NC * TILE_M * 64, Q_TILE = 3 * Q_PART, KV_PART = NC * BN * 64, KV_STAGE = 3 * KV_PART;
    static constexpr int SMEM = T * Q_TILE + (KS + VS) * KV_STAGE + 1024;
    // Tensor memory, per query tile: two slots that take the scores of a key tile (BN columns) and then its weights; NO
    // buffers for the product.  A softmax thread's weights go over its own scores (h, m) and behind all scores (l), so the
    // halves of a row need not wait for one another: word `off` of part (h, m) of half x at x BN/2 + (0, BN/4) + off, of
    // part l at BN + x BN/4 + off.
    static constexpr int HALF = BN / 2, SLOT = 3 * BN / 2, O_COLS = 2 * ACC;
    static constexpr bool Q_TMEM = T == 1;             // (two query tiles leave 32 columns: part h, Q_STEPS steps of it)
    static constexpr int Q_COLS = NC * F3_CHUNK / 2;   // of a part
    static constexpr int Q_STEPS = 2;
    static constexpr int TILE_COLS = 2 * SLOT + NO * O_COLS + (Q_TMEM ? 3 * Q_COLS : 8 * Q_STEPS);
    static_assert(T * TILE_COLS <= 512, "tensor memory");
    // registers: the pools of setmaxnreg must not exceed what the CTA was launched with
    static constexpr int LAUNCH_REGS = 65536 / THREADS / 8 * 8;
    // (a few spilled registers in the softmax loop of two query tiles cost 10%: 96 for it, what the others can spare)
    static constexpr int ISSUE_REGS = T == 2 ? 24 : 40, CONVERT_REGS = T == 2 ? 48 : 56, SOFTMAX_REGS = T == 2 ? 96 : 120;
    static constexpr int POOL = 128 * (2 * T * SOFTMAX_REGS + 2 * N_CONV * CONVERT_REGS + ISSUE_REGS);
    static_assert(POOL <= THREADS * LAUNCH_REGS, "setmaxnreg budget");
};
using F32Two = F32Shape<2, 64, 2, 24, 2, 2, 1, false, 0>;                // d <= 48, two query tiles
using F32One = F32Shape<2, 64, 1, 32, 3, 3, 2, false, 0>;                // d <= 64
using F32Mid = F32Shape<3, 64, 1, 48, 2, 2, 1, true, F32One::MAX_D>;     // d <= 96
using F32Wide = F32Shape<5, 32, 1, 80, 2, 1, 1, true, F32Mid::MAX_D>;    // d <= 160
constexpr float F32_TILE_SUM_LIMIT = 1.8446744e19f; // 2^64: no weight above it reaches the products
constexpr float F32_MAX_LIMIT = 58.f;               // log2 of the largest weight where the maximum decides: 64 of them stay below the sum

// Shared-memory matrix descriptor of a 64-byte-swizzled tile (rows of 64 bytes, eight to a 512-byte atom).
__host__ __device__ constexpr uint64_t smem_desc_sw64(uint32_t byte_addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    return (uint64_t)((byte_addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32) | (1ull << 46) | (4ull << 61);
}

// x minus a packed bfloat16 value, the low or the high one: one mixed multiply-add on the FMA pipe, exact here.  (Taking the parts out as
// binary32 values first costs two shifts or masks a pair on the half-rate integer pipe.)
__device__ __forceinline__ float less_low_bf16(float x, uint32_t packed) {
    float d;
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %1;\n\tfma.rn.f32.bf16 %0, l, %2, %3;\n\t}" : "=f"(d) : "r"(packed), "h"((unsigned short)0xBF80), "f"(x));
    return d;
}
__device__ __forceinline__ float less_high_bf16(float x, uint32_t packed) {
    float d;
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %1;\n\tfma.rn.f32.bf16 %0, h, %2, %3;\n\t}" : "=f"(d) : "r"(packed), "h"((unsigned short)0xBF80), "f"(x));
    return d;
}
// The three bf16 parts of a pair of binary32 values, packed (low half = first value), rounded to nearest.
__device__ __forceinline__ void split_pair_rn(float x0, float x1, uint32_t& h, uint32_t& m, uint32_t& l) {
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(x1), "f"(x0));
    const float r0 = less_low_bf16(x0, h), r1 = less_high_bf16(x1, h);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(m) : "f"(r1), "f"(r0));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(l) : "f"(less_high_bf16(r1, m)), "f"(less_low_bf16(r0, m)));
}

// Eight columns, split into their three parts, `part` bytes apart.  PAIRED: what shares their contraction step in each part (see the
// file's comment), of Q or of K.
enum F32Paired { F3_ALONE, F3_PAIR_Q, F3_PAIR_K };
__device__ __forceinline__ void f32_store_at(uint32_t at, uint32_t part, const float4& lo, const float4& hi, F32Paired paired) {
    uint4 h, m, l;
    split_pair_rn(lo.x, lo.y, h.x, m.x, l.x);
    split_pair_rn(lo.z, lo.w, h.y, m.y, l.y);
    split_pair_rn(hi.x, hi.y, h.z, m.z, l.z);
    split_pair_rn(hi.z, hi.w, h.w, m.w, l.w);
    st_shared_v4(at, h);
    st_shared_v4(at + part, m);
    if (paired != F3_PAIR_K) st_shared_v4(at + 2 * part, l);
    if (paired == F3_PAIR_Q) {          // h h | m m | l h
        st_shared_v4(at ^ 16, h);
        st_shared_v4((at + part) ^ 16, m);
        st_shared_v4((at + 2 * part) ^ 16, h);
    } else if (paired == F3_PAIR_K) {   // h l | m h
        st_shared_v4(at ^ 16, l);
        st_shared_v4((at + part) ^ 16, h);
    }
}
// The contraction of Q K^T: steps of 16 columns of one part each, and whether the eight columns behind them share steps with another part's.
// (PIECES eight columns; known at compile time, as steps counted at run time spill in the issuing warps: 2 x 8 x 600 x 600, d = 120
// 63.6 us against 50.2, and 256, d = 160 27.6 against 25.8)
template <int PIECES>
struct F32Steps {
    static constexpr int whole = PIECES / 2;
    static constexpr bool left = PIECES % 2 != 0;
};
template <int LO, int HI, typename F>
__device__ __forceinline__ void f32_with_steps(int pieces, const F& f) {
    if constexpr (LO == HI) {
        f(F32Steps<LO>{});
    } else {
        constexpr int MID = (LO + HI) / 2;
        if (pieces <= MID) f32_with_steps<LO, MID>(pieces, f);
        else f32_with_steps<MID + 1, HI>(pieces, f);
    }
}

// Convert warpgroups: a tile of ROWS rows of d binary32 values as pieces of eight columns; thread i of THREADS takes pieces
// i, i + THREADS, ...  (fetch: into registers; store: split, into the three parts of a shared-memory tile).
template <int NC, int ROWS, int THREADS, int MAX_D>
struct F32Converter {
    static constexpr int MAX_PIECES = (ROWS * MAX_D / 8 + THREADS - 1) / THREADS;
    const float* base;      // row 0 of the head
    long long tile_step;    // elements from one tile to the next
    int rows, d;            // rows of the head
    int at_g[MAX_PIECES], at_s[MAX_PIECES];   // the piece in global memory and in the tile (bit 0: half of it; bit 1: paired); at_s < 0: none
    float4 lo[MAX_PIECES], hi[MAX_PIECES];
    __device__ __forceinline__ void init(const float* head, int ld, int rows_, int d_, int i, const FastDiv& by_pieces, bool is_k) {
        base = head; rows = rows_; d = d_;
        tile_step = (long long)ROWS * ld;
#pragma unroll
        for (int u = 0; u < MAX_PIECES; ++u) {
            const int idx = i + u * THREADS, r = (int)fast_div((uint32_t)idx, by_pieces), p = idx - r * (int)by_pieces.d;
            at_g[u] = r * ld + p * 8;
            at_s[u] = r < ROWS ? (((p >> 2) * ROWS + r) << 6) + (((p & 3) ^ ((r >> 1) & 3)) << 4) : -1;
            if (p * 8 + 8 > d) at_s[u] |= 1;   // half a piece (d is a multiple of 4)
            if (is_k && !(p & 1) && p == (int)by_pieces.d - 1) at_s[u] |= 2;
        }
    }
    __device__ __forceinline__ void fetch(int j) {
        const float* src = base + j * tile_step;
        const bool whole = (j + 1) * ROWS <= rows;
#pragma unroll
        for (int u = 0; u < MAX_PIECES; ++u) {
            lo[u] = hi[u] = make_float4(0.f, 0.f, 0.f, 0.f);   // rows past the head read as zeros
            if (at_s[u] >= 0 && (whole || j * ROWS + ((at_s[u] >> 6) % ROWS) < rows)) {
                lo[u] = __ldg(reinterpret_cast<const float4*>(src + at_g[u]));
                if (!(at_s[u] & 1)) hi[u] = __ldg(reinterpret_cast<const float4*>(src + at_g[u] + 4));
            }
        }
    }
    __device__ __forceinline__ void store(uint32_t tile) const {
#pragma unroll
        for (int u = 0; u < MAX_PIECES; ++u)
            if (at_s[u] >= 0) f32_store_at(tile + (at_s[u] & ~3), NC * ROWS * 64, lo[u], hi[u], at_s[u] & 2 ? F3_PAIR_K : F3_ALONE);
    }
};

// Columns c0 .. c0 + cols - 1 of one output row by one warp, with the operations of simt_kernel.cuh in their order.  For the rows the
// split operands cannot serve (see above), whose loads come straight from global memory: with a NaN in every head, so that all rows of
// 16 x 4096 x 4096, d = 40, are redone, a call takes 21.7 ms (the CUDA-core kernel 3.9); without one 294 us before and after.
template <int ACC>
__device__ __forceinline__ void f32_plain_row(const F32Args& a, int bh, int row, int c0, int cols, int lane) {
    constexpr int CC = (ACC + 31) / 32, GROUP = 8;
    const float* q = head_row(a.q, a.lq, bh, row);
    const float* k = head_row(a.k, a.lk, bh, 0);
    const float* v = head_row(a.v, a.lk, bh, 0) + c0 + lane;
    const long long ld = a.lk.ld;
    float m = -INFINITY, l = 0.f, o[CC];
#pragma unroll
    for (int cc = 0; cc < CC; ++cc) o[cc] = 0.f;
#pragma unroll 1
    for (int j0 = 0; j0 < a.Nk; j0 += 32) {
        float score = -INFINITY;
        if (j0 + lane < a.Nk) {   // lane = key
            const float* kj = k + (j0 + lane) * ld;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
            for (int c = 0; c < a.d; c += 4) {
                const float4 qq = __ldg(reinterpret_cast<const float4*>(q + c)), kk = __ldg(reinterpret_cast<const float4*>(kj + c));
                acc.x = fmaf(qq.x, kk.x, acc.x);
                acc.y = fmaf(qq.y, kk.y, acc.y);
                acc.z = fmaf(qq.z, kk.z, acc.z);
                acc.w = fmaf(qq.w, kk.w, acc.w);
            }
            score = a.scale * ((acc.x + acc.y) + (acc.z + acc.w));
        }
        float mx = score;
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
        const float m_new = fmaxf(m, mx), alpha = expf(m - m_new), p = expf(score - m_new);
        m = m_new;
        l = l * alpha + p;
#pragma unroll
        for (int cc = 0; cc < CC; ++cc) o[cc] *= alpha;
#pragma unroll 1
        for (int g = 0; g < 32; g += GROUP) {   // lane = column
            float x[GROUP][CC];
#pragma unroll
            for (int u = 0; u < GROUP; ++u)
#pragma unroll
                for (int cc = 0; cc < CC; ++cc)
                    x[u][cc] = j0 + g + u < a.Nk && cc * 32 + lane < cols ? __ldg(v + (j0 + g + u) * ld + cc * 32) : 0.f;
#pragma unroll
            for (int u = 0; u < GROUP; ++u) {
                const float pj = __shfl_sync(0xffffffffu, p, g + u);
#pragma unroll
                for (int cc = 0; cc < CC; ++cc) o[cc] = fmaf(pj, x[u][cc], o[cc]);
            }
        }
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) l += __shfl_xor_sync(0xffffffffu, l, s);
    float* out = head_row(a.out, a.lq, bh, row) + c0 + lane;
#pragma unroll
    for (int cc = 0; cc < CC; ++cc)
        if (cc * 32 + lane < cols) out[cc * 32] = o[cc] / l;
}

template <typename SH>
__global__ void __launch_bounds__(SH::THREADS, 1)
f32_attention_kernel(const __grid_constant__ F32Args args) {
    constexpr int NC = SH::NC, BN = SH::BN, KS = SH::KS, VS = SH::VS, NO = SH::NO, ACC = SH::ACC;
    extern __shared__ uint8_t f3_smem_raw[];
    struct Barriers {
        uint64_t q_full[SH::T], s_full[SH::T][2], slot_free[SH::T][2], p_full[SH::T][2], pv_done[SH::T][NO], o_free[SH::T][NO];
        uint64_t k_full[KS], v_full[VS], k_empty[KS], v_empty[VS];
    };
    __shared__ __align__(8) Barriers bars;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;
    __shared__ float half_s[SH::T][2][TILE_M];   // what the halves of a row tell one another: maximum, row sum

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), wg = warp >> 2, wt = tid & 127;   // thread inside its warpgroup
    if (tid == 0) pdl_launch_dependents();
    const int bh = (int)blockIdx.x / args.units_per_head, unit = (int)blockIdx.x - bh * args.units_per_head;
    const int row_base = unit * SH::T * TILE_M;
    int T = (args.Nq - row_base + TILE_M - 1) / TILE_M;   // query tiles of this CTA
    if (T > SH::T) T = SH::T;
    const int n_kv = (args.Nk + BN - 1) / BN, d = args.d;
    const uint32_t smem_base = (smem_u32(f3_smem_raw) + 1023u) & ~1023u;
    const uint32_t q_smem = smem_base, k_smem = q_smem + SH::T * SH::Q_TILE, v_smem = k_smem + KS * SH::KV_STAGE;
    volatile int* abort_p = &abort_flag;

    if (tid == 0) {
        abort_flag = 0;
        for (int t = 0; t < SH::T; ++t) {
            mbar_init(smem_u32(&bars.q_full[t]), 8);
            for (int b = 0; b < 2; ++b) {
                mbar_init(smem_u32(&bars.s_full[t][b]), 1);
                mbar_init(smem_u32(&bars.slot_free[t][b]), 1);
                mbar_init(smem_u32(&bars.p_full[t][b]), 8);
            }
            for (int b = 0; b < NO; ++b) {
                mbar_init(smem_u32(&bars.pv_done[t][b]), 1);
                mbar_init(smem_u32(&bars.o_free[t][b]), 8);
            }
        }
        for (int s = 0; s < KS; ++s) {
            mbar_init(smem_u32(&bars.k_full[s]), 4 * SH::N_CONV);
            mbar_init(smem_u32(&bars.k_empty[s]), T);
        }
        for (int s = 0; s < VS; ++s) {
            mbar_init(smem_u32(&bars.v_full[s]), 4 * SH::N_CONV);
            mbar_init(smem_u32(&bars.v_empty[s]), T);
        }
        mbar_init_fence();
    }
    if (warp == SH::WG_ISSUE * 4) {
        tmem_alloc(smem_u32(&tmem_base_slot), 512);
        tmem_relinquish();
    }
    const int pieces = (d + 7) >> 3;
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    pdl_wait();
    const uint32_t tmem_base = tmem_base_slot;
    auto tmem_slot = [&](int t, int b) { return tmem_base + t * SH::TILE_COLS + b * SH::SLOT; };
    auto tmem_o = [&](int t, int b) { return tmem_base + t * SH::TILE_COLS + 2 * SH::SLOT + b * SH::O_COLS; };
    auto tmem_q = [&](int t) { return tmem_base + t * SH::TILE_COLS + 2 * SH::SLOT + NO * SH::O_COLS; };
    // Q_t, by the 256 threads that will work on its scores: thread i of them
    auto convert_q = [&](int t, int i) {
        constexpr int n = 256, U = SH::T == 1 ? 5 : 4;
        const float* qb = head_row(args.q, args.lq, bh, 0);
        for (int first = i; first < TILE_M * pieces; first += U * n) {
            float4 lo[U], hi[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int idx = first + u * n, r = (int)fast_div((uint32_t)idx, args.by_pieces), c = (idx - r * pieces) * 8;
                const int row = row_base + t * TILE_M + r;
                lo[u] = hi[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (idx < TILE_M * pieces && row < args.Nq) {
                    const float* src = qb + (long long)row * args.lq.ld + c;
                    lo[u] = __ldg(reinterpret_cast<const float4*>(src));
                    if (c + 8 <= d) hi[u] = __ldg(reinterpret_cast<const float4*>(src + 4));
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int idx = first + u * n, r = (int)fast_div((uint32_t)idx, args.by_pieces);
                const int p = idx - r * pieces;
                if (idx < TILE_M * pieces)
                    f32_store_at(q_smem + t * SH::Q_TILE + (p >> 2) * (TILE_M * 64) + r * 64 + (((p & 3) ^ ((r >> 1) & 3)) << 4), SH::Q_PART,
                                 lo[u], hi[u], !(p & 1) && p == pieces - 1 ? F3_PAIR_Q : F3_ALONE);
            }
        }
        if (!SH::Q_TMEM) fence_proxy_async_smem();
        {   // thread = row: its steps of 16 columns, every second one
            named_barrier(1 + t, 256);
            const int row = i & 127, sw = (row >> 1) & 3;
            const uint32_t src = q_smem + t * SH::Q_TILE + row * 64, dst = tmem_q(t) + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll
            for (int part = 0; part < (SH::Q_TMEM ? 3 : 1); ++part)
#pragma unroll
                for (int kk = 0; kk < (SH::Q_TMEM ? 2 * NC : SH::Q_STEPS); ++kk) {
                    if ((kk & 1) != i >> 7 || kk * 16 >= d) continue;
                    const uint32_t at = src + part * SH::Q_PART + (kk >> 1) * (TILE_M * 64);
                    const uint4 a = ld_shared_v4(at + ((((kk & 1) * 2) ^ sw) << 4)), b = ld_shared_v4(at + ((((kk & 1) * 2 + 1) ^ sw) << 4));
                    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
                    tmem_st8(dst + part * SH::Q_COLS + kk * 8, w);
                }
            tmem_wait_st();
            tc_fence_before_sync();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars.q_full[t]));
    };

    if (wg == SH::WG_ISSUE) {
        setmaxnreg_dec<SH::ISSUE_REGS>();
        const int t = (warp & 3) >> 1;
        if (t < T) {
            // the whole warp runs the loops and one thread issues, which keeps descriptors in uniform registers
            const bool leader = elect_one();
            bool ok = true;
            auto wait = [&](uint64_t& bar, int parity, int site, int j) {
                return __all_sync(0xffffffffu, mbar_wait(smem_u32(&bar), parity, abort_p, args.status, site, j)) != 0;
            };
            // parts of the six products, small ones first
            constexpr int PA[6] = {2, 0, 1, 1, 0, 0}, PB[6] = {0, 2, 1, 0, 1, 0};
            if ((warp & 1) == 0) {
                // ------------------------------------------------------------ S_t(j) = Q_t K(j)^T
                const uint32_t idesc = idesc_f16(TILE_M, BN, false, false, args.negate != 0, true);
                const uint64_t q_desc = smem_desc_sw64(q_smem + t * SH::Q_TILE, 16, 512), k_desc = smem_desc_sw64(k_smem, 16, 512);
                auto scores = [&](auto steps) {
                    constexpr int whole = decltype(steps)::whole;
                    constexpr bool left = decltype(steps)::left;
                    ok = wait(bars.q_full[t], 0, SITE_F_Q, t);
                    // The second query tile begins when the first has its first weights: in step, both sweep at once and then both
                    // wait (16 x 4096 x 4096, d = 40 282 -> 280 us).  Tile 0 hands over no further weights through this
                    // barrier before tile 1 has let go of key tile 0, which the ring of K then waits for.
                    if (t == 1) ok = ok && wait(bars.p_full[0][0], 0, SITE_F_P, 0);
                    int s = 0, pk = 0;
                    for (int j = 0; j < n_kv && ok; ++j) {
                        const int b = j & 1;
                        ok = wait(bars.k_full[s], pk, SITE_F_K, j);
                        if (ok && j >= 2) ok = wait(bars.slot_free[t][b], ((j >> 1) - 1) & 1, SITE_F_SLOT, j);
                        if (!ok) break;
                        tc_fence_after_sync();
                        const uint64_t kd = k_desc + (uint64_t)(s * (SH::KV_STAGE >> 4));
                        const uint32_t ts = tmem_slot(t, b);
                        if (leader) {
                            auto step = [&](int pa, int pb, int kk, bool q_tmem, bool acc) {
                                const uint64_t kt = kd + (uint64_t)((pb * SH::KV_PART + (kk >> 1) * (BN * 64) + (kk & 1) * 32) >> 4);
                                if (q_tmem)
                                    mma_f16_ts(ts, tmem_q(t) + pa * SH::Q_COLS + kk * 8, kt, idesc, acc);
                                else
                                    mma_f16_ss(ts, q_desc + (uint64_t)((pa * SH::Q_PART + (kk >> 1) * (TILE_M * 64) + (kk & 1) * 32) >> 4), kt, idesc, acc);
                            };
                            if (left) step(2, 0, whole, SH::Q_TMEM, false);       // l h + h l
#pragma unroll
                            for (int p = 0; p < 6; ++p) {
                                if (left && p == 3) step(1, 1, whole, SH::Q_TMEM, true);   // m m + m h
                                if (left && p == 5) step(0, 1, whole, SH::Q_TMEM, true);   // h m + h h
#pragma unroll
                                for (int kk = 0; kk < 2 * NC; ++kk)   // (offsets are constants)
                                    if (kk < whole) step(PA[p], PB[p], kk, SH::Q_TMEM || (PA[p] == 0 && kk < SH::Q_STEPS), left || p > 0 || kk > 0);
                            }
                            tc_commit(smem_u32(&bars.s_full[t][b]));
                            tc_commit(smem_u32(&bars.k_empty[s]));
                        }
                        if (++s == KS) { s = 0; pk ^= 1; }
                    }
                };
                f32_with_steps<SH::MIN_PIECES, SH::MAX_PIECES>(pieces, scores);
            } else {
                // ------------------------------------------------------------ O_t = P_t(j) V(j)
                auto weights_at = [](int part, int kk) {   // 16 keys of a part (see F32Shape)
                    constexpr int STEPS = SH::HALF / 16;
                    const int x = kk / STEPS, off = kk % STEPS * 8;
                    return part == 2 ? BN + x * (BN / 4) + off : x * SH::HALF + part * (BN / 4) + off;
                };
                const uint32_t idesc = idesc_f16(TILE_M, (d + 15) / 16 * 16, false, true, false, true);
                const uint64_t v_desc = smem_desc_sw64(v_smem, BN * 64, 512);
                int s = 0, pv = 0;
                for (int j = 0; j < n_kv && ok; ++j) {
                    const int b = j & 1, ob = j % NO;
                    const uint32_t tp = tmem_slot(t, b), to = tmem_o(t, ob);
                    ok = wait(bars.v_full[s], pv, SITE_F_V, j);
                    if (ok && j >= NO) ok = wait(bars.o_free[t][ob], (j / NO - 1) & 1, SITE_F_OFREE, j);
                    if (ok) ok = __all_sync(0xffffffffu, mbar_wait_eager(smem_u32(&bars.p_full[t][b]), (j >> 1) & 1, abort_p, args.status, SITE_F_P, j));
                    if (!ok) break;
                    tc_fence_after_sync();
                    const uint64_t vd = v_desc + (uint64_t)(s * (SH::KV_STAGE >> 4));
                    if (leader) {
#pragma unroll
                        for (int p = 0; p < 6; ++p)
#pragma unroll
                            for (int kk = 0; kk < BN / 16; ++kk)
                                mma_f16_ts(to, tp + weights_at(PA[p], kk), vd + (uint64_t)((PB[p] * SH::KV_PART + kk * 1024) >> 4), idesc,
                                           p > 0 || kk > 0);
                        tc_commit(smem_u32(&bars.pv_done[t][ob]));
                        tc_commit(smem_u32(&bars.slot_free[t][b]));
                        tc_commit(smem_u32(&bars.v_empty[s]));
                    }
                    if (++s == VS) { s = 0; pv ^= 1; }
                }
            }
        }
        __syncwarp();
    } else if (wg >= SH::WG_CONVERT) {
        setmaxnreg_dec<SH::CONVERT_REGS>();
        const int which = (wg - SH::WG_CONVERT) / SH::N_CONV;   // 0: K, 1: V
        bool ok = true;
        F32Converter<NC, BN, 128 * SH::N_CONV, SH::MAX_D> cv;
        cv.init(head_row(which == 0 ? args.k : args.v, args.lk, bh, 0), args.lk.ld, args.Nk, d, (wg - SH::WG_CONVERT) % SH::N_CONV * 128 + wt,
                args.by_pieces, which == 0);
        const int depth = which == 0 ? KS : VS;
        const uint32_t ring = which == 0 ? k_smem : v_smem;
        uint64_t* full = which == 0 ? bars.k_full : bars.v_full;
        uint64_t* empty = which == 0 ? bars.k_empty : bars.v_empty;
        cv.fetch(0);
        int s = 0, pe = 1;
        for (int j = 0; j < n_kv; ++j) {
            if (j >= depth) {
                ok = mbar_wait(smem_u32(&empty[s]), pe, abort_p, args.status, which == 0 ? SITE_F_KEMPTY : SITE_F_VEMPTY, j);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
            }
            cv.store(ring + s * SH::KV_STAGE);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&full[s]));
            if (j + 1 < n_kv) cv.fetch(j + 1);
            if (++s == depth) { s = 0; pe ^= 1; }
        }
    } else {
        // ---------------------------------------------------------------- softmax and accumulation
        setmaxnreg_inc<SH::SOFTMAX_REGS>();
        const int t = wg >> 1, half = wg & 1;
        constexpr int HALF = SH::HALF;
        if (t < T) {
            convert_q(t, half * 128 + wt);
            const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
            const float c2 = args.scale_log2e;
            const int c0 = half * ACC, cols = d - c0 < ACC ? d - c0 : ACC;   // this thread's output columns (none where cols <= 0)
            float m_run = 0.f, nm_run = 0.f, l_run = 0.f;   // anchor; -anchor * c2 as rounded; sum of this half's weights
            uint64_t o[ACC / 2];
#pragma unroll
            for (int c = 0; c < ACC / 2; ++c) o[c] = 0ull;
            // maximum of both halves' arguments (every thread of the query tile takes part)
            auto row_max_of_halves = [&](float mx) {
                half_s[t][half][wt] = mx;
                named_barrier(1 + t, 256);
                const float both = fmaxf(half_s[t][0][wt], half_s[t][1][wt]);
                named_barrier(1 + t, 256);
                return both;
            };
            auto add_product = [&](int j) -> bool {   // O += P V of key tile j
                const int ob = j % NO;
                bool good = mbar_wait(smem_u32(&bars.pv_done[t][ob]), (j / NO) & 1, abort_p, args.status, SITE_F_PV, j);
                good = __all_sync(0xffffffffu, good);
                if (!good) return false;
                tc_fence_after_sync();
                const uint32_t src = tmem_o(t, ob) + c0 + lane_off;
                constexpr int TOGETHER = ACC <= 48 ? 16 : 8;   // columns fetched together: a load and its wait are 130 clocks (80 spill)
#pragma unroll
                for (int c = 0; c < ACC; c += TOGETHER) {
                    if (c < cols) {
                        uint32_t x[16];
                        if (TOGETHER == 16 && c + 16 <= ACC) tmem_ld16(src + c, x);
                        else tmem_ld8(src + c, *reinterpret_cast<uint32_t(*)[8]>(x));
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < TOGETHER / 2; ++i)
                            if (c + 2 * i < ACC && (i < 4 || c + 8 < cols))   // (columns behind d are not real)
                                o[c / 2 + i] = add_f32x2(o[c / 2 + i], pack_b64(x[2 * i], x[2 * i + 1]));
                    }
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bars.o_free[t][ob]));
                return true;
            };
            bool ok = true;
            for (int j = 0; j < n_kv; ++j) {
                const int b = j & 1;
                ok = ok && mbar_wait(smem_u32(&bars.s_full[t][b]), (j >> 1) & 1, abort_p, args.status, SITE_F_S, j);
                ok = __all_sync(0xffffffffu, ok);
                const uint32_t slot = tmem_slot(t, b) + lane_off;
                const int valid = args.Nk - j * BN - half * HALF;   // columns past it are zero-filled keys
                uint32_t s[HALF];
                if (ok) {
                    tc_fence_after_sync();
#pragma unroll
                    for (int c = 0; c < HALF; c += 16) tmem_ld16(slot + half * HALF + c, *reinterpret_cast<uint32_t(*)[16]>(&s[c]));
                    tmem_wait_ld();
                } else {
#pragma unroll
                    for (int c = 0; c < HALF; ++c) s[c] = 0u;
                }
                if (j == 0) {
                    m_run = row_max_of_halves(row_max_masked<HALF>(s, valid));
                    nm_run = -m_run * c2;
                }
                auto sweep = [&]() -> float {   // weights of the anchor in use, to tensor memory; their sum
                    const uint64_t c2c2 = pack_b64(__float_as_uint(c2), __float_as_uint(c2));
                    const uint64_t nmnm = pack_b64(__float_as_uint(nm_run), __float_as_uint(nm_run));
                    uint64_t sum[2] = {0ull, 0ull};
#pragma unroll
                    for (int c = 0; c < HALF; c += 8) {
                        uint32_t h[4], m[4], l[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            uint32_t x0, x1;
                            unpack_b64(fma_f32x2(pack_b64(s[c + 2 * i], s[c + 2 * i + 1]), c2c2, nmnm), x0, x1);
                            float p0 = ex2_approx(__uint_as_float(x0)), p1 = ex2_approx(__uint_as_float(x1));
                            if (valid < HALF) {
                                if (c + 2 * i >= valid) p0 = 0.f;
                                if (c + 2 * i + 1 >= valid) p1 = 0.f;
                            }
                            // three parts by truncation: exact, and a pair's high halves are one byte permute
                            const uint32_t q0 = __float_as_uint(p0), q1 = __float_as_uint(p1);
                            const uint64_t pp = pack_b64(q0, q1);
                            sum[i & 1] = add_f32x2(sum[i & 1], pp);
                            h[i] = high_halves(q0, q1);
                            const float r0 = less_low_bf16(p0, h[i]), r1 = less_high_bf16(p1, h[i]);
                            m[i] = high_halves(__float_as_uint(r0), __float_as_uint(r1));
                            l[i] = high_halves(__float_as_uint(less_low_bf16(r0, m[i])), __float_as_uint(less_high_bf16(r1, m[i])));
                        }
                        const uint32_t own = slot + half * HALF + c / 2;   // over scores that sit in registers
                        tmem_st4(own, h);
                        tmem_st4(own + BN / 4, m);
                        tmem_st4(slot + BN + half * (BN / 4) + c / 2, l);
                    }
                    return sum_f32x2(sum[0], sum[1]);
                };
                // Rare: a score far above the anchor.  Everything summed so far is rescaled to the new one.
                auto reanchor = [&]() {
                    const float m_new = fmaxf(m_run, row_max_of_halves(row_max_masked<HALF>(s, valid)));
                    const float nm_new = -m_new * c2, alpha = ex2_approx(nm_new - nm_run);
                    m_run = m_new;
                    nm_run = nm_new;
                    l_run *= alpha;
                    const uint64_t aa = pack_b64(__float_as_uint(alpha), __float_as_uint(alpha));
#pragma unroll
                    for (int c = 0; c < ACC / 2; ++c) o[c] = fma_f32x2(o[c], aa, 0ull);
                };
                // One decision for the query tile's 256 threads: go on, give up (a wait expired), or re-anchor.  The product of the
                // key tile before is added ahead of handing this one's weights over: once their product runs, loads from
                // tensor memory take three times as long.
                float tile_sum;
                if constexpr (SH::MAX_FIRST) {
                    bool added = j == 0;
                    if (j > 0) {
                        float top[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                        for (int c = 0; c < HALF; ++c) top[c & 3] = fmaxf(top[c & 3], __uint_as_float(s[c]));
                        const float mx = fmaxf(fmaxf(top[0], top[1]), fmaxf(top[2], top[3]));
                        if (!named_barrier_and(1 + t, 256, ok && fmaf(mx, c2, nm_run) <= F32_MAX_LIMIT)) {
                            if (!named_barrier_and(1 + t, 256, ok)) { ok = false; break; }
                            ok = add_product(j - 1);
                            added = true;
                            reanchor();
                        }
                    }
                    tile_sum = sweep();
                    if (!added && ok) ok = add_product(j - 1);
                } else {
                    bool live = true;
#pragma unroll 1
                    for (int attempt = 0; attempt < 2; ++attempt) {
                        tile_sum = sweep();
                        if (attempt == 0 && j > 0 && ok) ok = add_product(j - 1);
                        if (attempt == 1 || named_barrier_and(1 + t, 256, ok && tile_sum <= F32_TILE_SUM_LIMIT)) break;
                        live = named_barrier_and(1 + t, 256, ok);
                        if (!live) break;
                        reanchor();
                        tmem_wait_st();
                    }
                    if (!live) { ok = false; break; }
                }
                l_run += tile_sum;
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bars.p_full[t][b]));
            }
            if (ok) ok = add_product(n_kv - 1);
            half_s[t][half][wt] = l_run;
            ok = named_barrier_and(1 + t, 256, ok);
            if (ok) {
                // A thread's columns are 4 ACC bytes of a row of its own: through shared memory (the query tile's, which no product
                // reads any more), so that a warp's stores run along the rows (row by row they took 9000 clocks at d = 160).
                constexpr int PITCH = ACC + 4;   // floats
                static_assert(8 * 32 * PITCH * 4 <= SH::Q_TILE, "staging");
                const float inv = 1.f / (half_s[t][0][wt] + half_s[t][1][wt]);
                const uint32_t stage = q_smem + t * SH::Q_TILE + (uint32_t)((half * 4 + (warp & 3)) * 32 * PITCH * 4);
                float zero = 0.f;   // (until a value is not finite)
#pragma unroll
                for (int c = 0; c < ACC; c += 4) {
                    uint32_t x[4];
                    unpack_b64(o[c / 2], x[0], x[1]);
                    unpack_b64(o[c / 2 + 1], x[2], x[3]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float y = __uint_as_float(x[i]) * inv;
                        zero = fmaf(y, 0.f, zero);
                        x[i] = __float_as_uint(y);
                    }
                    st_shared_v4(stage + (lane * PITCH + c) * 4, make_uint4(x[0], x[1], x[2], x[3]));
                }
                __syncwarp();
                const int row0 = row_base + t * TILE_M + (warp & 3) * 32, rows = args.Nq - row0 < 32 ? args.Nq - row0 : 32;
                // lane = (piece of four columns, row modulo the rows done at once); d and c0 are multiples of 4
                const int per_row = cols > 0 ? cols >> 2 : 1, at_once = 32 / per_row, first = lane / per_row, c = (lane - first * per_row) * 4;
                if (cols > 0 && first < at_once) {
                    float* out = head_row(args.out, args.lq, bh, row0) + c0 + c;
                    for (int r = first; r < rows; r += at_once) {
                        const uint4 v = ld_shared_v4(stage + (r * PITCH + c) * 4);
                        *reinterpret_cast<uint4*>(out + (long long)r * args.lq.ld) = v;
                    }
                }
                uint32_t again = __ballot_sync(0xffffffffu, !(zero == 0.f) && lane < rows);
                for (; again; again &= again - 1) f32_plain_row<ACC>(args, bh, row0 + __ffs(again) - 1, c0, cols, lane);
            }
        }
    }

    // -------------------------------------------------------------------- teardown (every thread arrives)
    tc_fence_before_sync();
    __syncthreads();
    if (warp == SH::WG_ISSUE * 4) {
        __syncwarp();
        tmem_dealloc(tmem_base, 512);
    }
}

}  // namespace sd_attn
