// Direct 3x3 convolution (stride 1, zero padding 1, channels-last fp16) as ONE implicit matrix product on the tensor
// cores: y[pixel][k] = sum over 9 taps and C channels of x[pixel + tap][c] w[k][tap][c], accumulated in binary32.
//
// F(4x4, 3x3) needs a quarter of these products, but its transformed operands are 2.25 times the input, 4 times the
// filter and (binary32) 4.5 times the output, written and read once more each, in three dependent kernels: at 2 x 64 x 64 x
// 320 -> 320 the products of either form take less time than that traffic, and at 1280 channels the transformed filter
// alone is 118 MB.  Here every operand is read where it lies, once per CTA that needs it.
//
// Pixels.  The images of a batch are seen as one stack of rows PW = W + 2 positions wide, with one zero row between
// images: padded row 0 and every (H + 1)-th are zero, the first and last position of a row too.  Output position p of
// that raster (row p / PW, column p % PW) needs positions p + r PW + s for the taps r, s = 0..2 -- a constant offset --
// so a tile of 128 CONSECUTIVE positions is 128 consecutive 128-byte rows of shared memory whatever the tap, and the nine
// taps are nine start addresses into one patch fetched once per 64 channels.  (Positions in the padding are computed and
// not stored: 2 of W + 2 columns and one row per image, 3% to 5% at 64 x 64 against up to half with rectangular tiles of
// odd-sized images.)  Patch rows arrive by TMA, one padded row each, the padding by its zero fill; the 128-byte swizzle is
// a function of the shared-memory address, so rows and tiles may start at any multiple of 128 bytes.
//
// One CTA: 128 positions x n_tile output channels.  B (n_tile filters of one tap, 64 channels) streams through a ring, the
// patch is double-buffered per 64 channels.  The filter is laid out once per layer in the order it is used, swizzle included,
// so that a step's tile is one contiguous bulk copy.  Small images leave too few tiles for the GPU: the (64 channels, tap)
// steps are then split among the CTAs of a cluster, which exchange their accumulators through distributed shared memory.
//   warps 0, 4 filter producers   warps 1, 3 MMA issuers (of the even and the odd steps each)   warp 2 patch producer
// What bounds it is the tensor core only if the threads that feed it keep up: a step is 320 clocks of it at 160 channels, but
// one issuing thread's waits, descriptors, MMAs and commits of a step take 600 and one producing thread's wait and copy 300.  So
// two of either take the steps in turn; the issuers each have an accumulator of their own (products of different threads are
// not ordered), added when they are read out.  With the second producer a step of 80 channels went from 320 to 230 clocks
// (2 x 32 x 32, 640 -> 640: 17.0 -> 14.8 us; 2 x 33 x 43: 24.3 -> 18.2); 160 channels are at the tensor core's rate either way
// (2 x 64 x 64, 320 -> 320: 14.9k of a CTA's 24k clocks are products, 4k the ramp, 2.4k stores at 17 bytes a clock).
// Every wait is bounded and reports to the status block.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "cross_common.cuh"  // TILE_M, CHUNK_COLS, CHUNK_ROW_BYTES
#include "tc_common.cuh"

namespace sd_attn {

constexpr int CD_THREADS = 256;
constexpr int CD_MAX_STAGES = 8;
constexpr int CD_MAX_SPLIT = 8;
constexpr int CD_MAX_N = 256;            // output channels per CTA, at most (one MMA)
constexpr int CD_MAX_W = 126;            // two patch buffers and the filter ring fit shared memory up to here
constexpr int CD_SMEM_BUDGET = 222 * 1024;
enum { SITE_D_AEMPTY = 60, SITE_D_AFULL = 61, SITE_D_BEMPTY = 62, SITE_D_BFULL = 63, SITE_D_DONE = 64, SITE_D_FIRST = 65 };

struct ConvDirectArgs {
    __half* y;
    const __half* bias;     // may be null
    int H, W, K;
    int pw;                 // W + 2
    int padded_rows;        // N * (H + 1): the padded rows that hold images or the zero row before one
    int chunks;             // ceil(C / 64)
    int n_tile, tmem_cols;
    int split;              // CTAs of a cluster that share a tile's steps
    int stages;             // filter ring
    int patch_bytes;        // of one buffer (a multiple of 1024)
    const __half* filter;   // packed: see conv_pack_kernel
    int k_padded;           // K rounded up to 16
    FastDiv by_pw, by_h1;   // division by pw, by H + 1
    int* status;
};

// Padded rows a tile's patch spans, at most: 128 positions and 2 pw + 2 more, from anywhere in a row.
__host__ inline int cd_patch_rows(int pw) { return (TILE_M + 2 * pw + 2 + pw - 1 + pw - 1) / pw; }
__host__ inline int cd_patch_bytes(int pw) { return (cd_patch_rows(pw) * pw * CHUNK_ROW_BYTES + 1023) & ~1023; }
// The accumulator on its way out: binary16 rows of n_tile + 8 (one CTA per tile), or, of every CTA of the cluster, the
// binary32 rows of n_tile + 4 that this CTA finishes.
__host__ __device__ inline int cd_share_rows(int split) { return (TILE_M + split - 1) / split; }
__host__ inline int cd_staging_bytes(int n_tile, int split) {
    return split == 1 ? TILE_M * (n_tile + 8) * 2 : split * cd_share_rows(split) * (n_tile + 4) * 4;
}

__device__ __forceinline__ void cd_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cd_map_to_rank(uint32_t addr, int rank) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(rank));
    return remote;
}
__device__ __forceinline__ void cd_store_remote(uint32_t addr, float a, float b, float c, float d) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// w [K][3][3][C] -> packed [ceil(C / 64)][9][K rounded up to 16][64], zeros in the padding, the eight 16-byte pieces of row k
// in the order of the 128-byte swizzle (piece c at c ^ (k & 7)).  One thread per piece.
__host__ inline size_t conv_packed_elems(int K, int C) {
    return (size_t)((C + CHUNK_COLS - 1) / CHUNK_COLS) * 9 * ((K + 15) / 16 * 16) * CHUNK_COLS;
}
__global__ void __launch_bounds__(256) conv_pack_kernel(const __half* __restrict__ w, __half* __restrict__ packed, int K, int C) {
    const int kp = (K + 15) / 16 * 16;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x, n = (long long)((C + CHUNK_COLS - 1) / CHUNK_COLS) * 9 * kp * 8;
    if (idx >= n) return;
    const int c = (int)(idx & 7);
    const long long row = idx >> 3;
    const int k = (int)(row % kp), tap = (int)(row / kp % 9), chunk = (int)(row / kp / 9);
    const int ch = chunk * CHUNK_COLS + c * 8;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (k < K && ch < C) v = *reinterpret_cast<const uint4*>(w + ((long long)k * 9 + tap) * C + ch);   // (C is a multiple of 8)
    reinterpret_cast<uint4*>(packed)[row * 8 + (c ^ (k & 7))] = v;
}

template <bool CLUSTER>   // the steps of a tile are split among the CTAs of a cluster
__global__ void __launch_bounds__(CD_THREADS, 1)
conv_direct_kernel(const __grid_constant__ CUtensorMap tmap_x, const ConvDirectArgs args) {
    extern __shared__ uint8_t cd_smem_raw[];
    __shared__ __align__(8) uint64_t bar_a_full[2], bar_a_empty[2], bar_b_full[CD_MAX_STAGES], bar_b_empty[CD_MAX_STAGES], bar_done, bar_first;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;
    __shared__ float bias_s[CD_MAX_N];

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    if (tid == 0) pdl_launch_dependents();
    const int split = CLUSTER ? args.split : 1, rank = CLUSTER ? (int)blockIdx.x : 0;   // rank inside the cluster
    const int k0 = blockIdx.y * args.n_tile, p0 = blockIdx.z * TILE_M;
    const int pw = args.pw, n_tile = args.n_tile, stages = args.stages;
    const int row0 = (int)fast_div((uint32_t)p0, args.by_pw), col0 = p0 - row0 * pw;
    const int patch_rows = (int)fast_div((uint32_t)(col0 + TILE_M + 2 * pw + 2 + pw - 1), args.by_pw);
    const int n_steps = 9 * args.chunks;
    const int q_begin = n_steps * rank / split, q_end = n_steps * (rank + 1) / split;   // (64 channels, tap) steps
    const uint32_t smem_base = (smem_u32(cd_smem_raw) + 1023u) & ~1023u;
    const uint32_t patch_smem = smem_base, ring_smem = smem_base + 2 * args.patch_bytes;
    const uint32_t stage_pitch = (uint32_t)(n_tile * CHUNK_ROW_BYTES);   // (n_tile % 16 == 0: a multiple of 1024)

    if (tid == 0) {
        abort_flag = 0;
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&bar_a_full[b]), 1);
            mbar_init(smem_u32(&bar_a_empty[b]), 2);   // both issuers
        }
        for (int s = 0; s < stages; ++s) {
            mbar_init(smem_u32(&bar_b_full[s]), 1);
            mbar_init(smem_u32(&bar_b_empty[s]), 1);
        }
        mbar_init(smem_u32(&bar_done), 2);
        mbar_init(smem_u32(&bar_first), 1);
        mbar_init_fence();
        tma_prefetch_desc(&tmap_x);
    }
    if (warp == 3) {
        tmem_alloc(smem_u32(&tmem_base_slot), (uint32_t)args.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    pdl_wait();   // set-up overlapped the tail of the stream's previous kernel
    const uint32_t tmem_d = tmem_base_slot;
    volatile int* abort_p = &abort_flag;

    if (warp == 0 || warp == 4) {
        if (elect_one()) {
            // ---------------------------------------------------------------- filter producers: every second step each
            // (the last tile of channels may be short: the accumulator columns behind it are not stored).  Behind the first
            // step's filters the first patch goes out, which those products wait for too, and only then the rest of the ring.
            const int mine = warp >> 2;
            const uint32_t bytes = (uint32_t)(min(n_tile, args.k_padded - k0) * CHUNK_ROW_BYTES);
            const __half* src = args.filter + ((size_t)(q_begin + mine) * args.k_padded + k0) * CHUNK_COLS;
            const size_t step = 2 * (size_t)args.k_padded * CHUNK_COLS;
            uint32_t dst = ring_smem + mine * stage_pitch;
            int s = mine, pe = 1;
            bool filled = false;
            for (int q = q_begin + mine; q < q_end; q += 2) {
                if (q == q_begin + mine + 2 && !mbar_wait(smem_u32(&bar_first), 0, abort_p, args.status, SITE_D_FIRST, q)) break;
                if (filled && !mbar_wait(smem_u32(&bar_b_empty[s]), pe, abort_p, args.status, SITE_D_BEMPTY, q)) break;
                const uint32_t bar = smem_u32(&bar_b_full[s]);
                mbar_arrive_expect_tx(bar, bytes);
                bulk_load(dst, src, bytes, bar);
                src += step;
                dst += 2 * stage_pitch;
                if ((s += 2) >= stages) { s = mine; pe ^= 1; dst = ring_smem + mine * stage_pitch; filled = true; }
            }
        }
    } else if (warp == 2) {
        if (elect_one()) {
            // ---------------------------------------------------------------- patch producer
            const int c_begin = q_begin / 9, c_end = (q_end + 8) / 9;
            for (int c = c_begin, i = 0; c < c_end; ++c, ++i) {
                const int b = i & 1;
                if (i >= 2 && !mbar_wait(smem_u32(&bar_a_empty[b]), ((i >> 1) - 1) & 1, abort_p, args.status, SITE_D_AEMPTY, c)) break;
                const uint32_t bar = smem_u32(&bar_a_full[b]);
                mbar_arrive_expect_tx(bar, (uint32_t)(patch_rows * pw * CHUNK_ROW_BYTES));
                for (int r = 0; r < patch_rows; ++r) {
                    const int pr = row0 + r, n = (int)fast_div((uint32_t)pr, args.by_h1);
                    // padded row n (H + 1) is the zero row before image n; rows past the last image read as zeros too
                    const int img_y = pr < args.padded_rows ? pr - n * (args.H + 1) - 1 : -1;
                    tma_load_4d(patch_smem + b * args.patch_bytes + r * pw * CHUNK_ROW_BYTES, &tmap_x, bar, c * CHUNK_COLS, -1, img_y,
                                pr < args.padded_rows ? n : 0);
                }
                if (i == 0) mbar_arrive(smem_u32(&bar_first));
            }
        }
    } else if (warp == 1 || warp == 3) {
        // ------------------------------------------------------------------- MMA issuers: every second step each
        // Descriptors are 32-bit additions to their address field (16-byte units), nothing is divided in the loop; the whole
        // warp runs it and one thread issues, which keeps descriptors in uniform registers.
        const bool leader = elect_one();
        auto wait = [&](uint64_t& bar, int parity, int site, int q) {
            return __all_sync(0xffffffffu, mbar_wait(smem_u32(&bar), parity, abort_p, args.status, site, q)) != 0;
        };
        const int mine = warp >> 1;
        const uint32_t idesc = idesc_f16(TILE_M, n_tile, false, false, false);
        constexpr uint64_t DESC = smem_desc_sw128(0, 16, 1024);
        const uint32_t a0 = (patch_smem + col0 * CHUNK_ROW_BYTES) >> 4, a_buf = (uint32_t)args.patch_bytes >> 4;
        const uint32_t b0 = ring_smem >> 4, b_stage = stage_pitch >> 4, tmem_acc = tmem_d + mine * n_tile;
        int s = mine, pf = 0, chunk_i = 0, tap = q_begin % 9 + mine;
        uint32_t b_at = b0 + mine * b_stage, a_at = a0;
        bool ok = wait(bar_a_full[0], 0, SITE_D_AFULL, q_begin);
        for (int q = q_begin + mine; q < q_end && ok; q += 2) {
            if (tap >= 9) {   // the next 64 channels
                if (leader) tc_commit(smem_u32(&bar_a_empty[chunk_i & 1]));
                tap -= 9;
                ++chunk_i;
                a_at = a0 + (chunk_i & 1) * a_buf;
                ok = wait(bar_a_full[chunk_i & 1], (chunk_i >> 1) & 1, SITE_D_AFULL, q);
            }
            ok = ok && wait(bar_b_full[s], pf, SITE_D_BFULL, q);
            if (!ok) break;
            tc_fence_after_sync();
            const uint32_t a_tap = a_at + (uint32_t)(((tap * 11) >> 5) * (pw - 3) + tap) * 8;   // (tap * 11) >> 5 = tap / 3
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    mma_f16_ss(tmem_acc, DESC | (a_tap + (uint32_t)(kk * 2)), DESC | (b_at + (uint32_t)(kk * 2)), idesc,
                               q > q_begin + mine || kk > 0);
                tc_commit(smem_u32(&bar_b_empty[s]));
            }
            tap += 2;
            s += 2;
            b_at += 2 * b_stage;
            if (s >= stages) { s -= stages; b_at -= stages * b_stage; pf ^= 1; }
        }
        if (ok && leader) tc_commit(smem_u32(&bar_done));
    } else {
        for (int c = tid - 160; c < n_tile; c += 96) bias_s[c] = args.bias && k0 + c < args.K ? __half2float(args.bias[k0 + c]) : 0.f;
    }
    __syncwarp();

    // -------------------------------------------------------------------- out: sum of the two accumulators, thread = row; two
    // warps per quarter of the lanes share its columns.  (The rings are idle: every product has completed.)
    __syncthreads();   // (bias_s; the roles are done)
    bool ok = mbar_wait(smem_u32(&bar_done), 0, abort_p, args.status, SITE_D_DONE, blockIdx.z);
    ok = __all_sync(0xffffffffu, ok);
    if (CLUSTER) cd_cluster_sync();   // every CTA of the cluster is done with its rings
    uint8_t* staging = cd_smem_raw + (smem_base - smem_u32(cd_smem_raw));
    const int pitch = CLUSTER ? n_tile + 4 : n_tile + 8;   // floats, halves
    const int share_rows = cd_share_rows(split);
    if (ok) {
        tc_fence_after_sync();
        const int row = (warp & 3) * 32 + lane, groups = n_tile >> 4, g_begin = warp < 4 ? 0 : groups >> 1, g_end = warp < 4 ? groups >> 1 : groups;
        const uint32_t src = tmem_d + ((uint32_t)((warp & 3) * 32) << 16);
        // CLUSTER: CTA o finishes rows 128 o / split .. 128 (o + 1) / split - 1; every thread stores its row where it is finished
        // (straight from registers: bulk copies of staged rows took 4000 clocks for 42 KB)
        const int owner = CLUSTER ? ((row + 1) * split - 1) >> 7 : 0, in_share = CLUSTER ? row - TILE_M * owner / split : row;
        const uint32_t remote = CLUSTER ? cd_map_to_rank(smem_base + (uint32_t)((rank * share_rows + in_share) * pitch * 4), owner) : 0u;
        for (int g = g_begin; g < g_end; ++g) {
            uint32_t x[16], y[16];
            tmem_ld16(src + g * 16, x);
            tmem_ld16(src + n_tile + g * 16, y);
            tmem_wait_ld();
            float v[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) v[c] = __uint_as_float(x[c]) + __uint_as_float(y[c]);
            if (CLUSTER) {
#pragma unroll
                for (int c = 0; c < 16; c += 4) cd_store_remote(remote + (g * 16 + c) * 4, v[c], v[c + 1], v[c + 2], v[c + 3]);
            } else {
                uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<__half*>(staging) + row * pitch + g * 16);
#pragma unroll
                for (int c = 0; c < 16; ++c) v[c] += bias_s[g * 16 + c];
                dst[0] = make_uint4(pack_half2(v[0], v[1]), pack_half2(v[2], v[3]), pack_half2(v[4], v[5]), pack_half2(v[6], v[7]));
                dst[1] = make_uint4(pack_half2(v[8], v[9]), pack_half2(v[10], v[11]), pack_half2(v[12], v[13]), pack_half2(v[14], v[15]));
            }
        }
    }
    if (abort_flag && tid == 0) {   // gave up: let copies in flight land before shared memory is released
        for (int s = 0; s < stages; ++s) mbar_drain(smem_u32(&bar_b_full[s]), 0);
        for (int b = 0; b < 2; ++b) mbar_drain(smem_u32(&bar_a_full[b]), 0);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (CLUSTER) cd_cluster_sync();   // every row is where it is finished; nobody touches another CTA's memory from here on
    if (ok && !abort_flag) {
        // eight channels (16 bytes) a thread at a time: thread = (piece of a row, row modulo the rows done at once)
        const int r_begin = TILE_M * rank / split, r_end = TILE_M * (rank + 1) / split;
        const int per_row = min(n_tile, args.K - k0) >> 3, at_once = CD_THREADS / per_row, first = tid / per_row, c = (tid - first * per_row) * 8;
        float b8[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) b8[i] = CLUSTER ? bias_s[c + i] : 0.f;
        __half* y = args.y + k0 + c;
        for (int row = r_begin + first; row < r_end && first < at_once; row += at_once) {
            const int p = p0 + row, pr = (int)fast_div((uint32_t)p, args.by_pw), xx = p - pr * pw;
            const int n = (int)fast_div((uint32_t)pr, args.by_h1), yy = pr - n * (args.H + 1);
            if (xx >= args.W || yy >= args.H || pr >= args.padded_rows) continue;
            uint4 o8;
            if (CLUSTER) {
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = b8[i];
                const float* part = reinterpret_cast<const float*>(staging) + (row - r_begin) * pitch + c;
                for (int o = 0; o < split; ++o, part += share_rows * pitch) {   // in rank order, so that the bits repeat
                    const float4 lo = *reinterpret_cast<const float4*>(part), hi = *reinterpret_cast<const float4*>(part + 4);
                    v[0] += lo.x; v[1] += lo.y; v[2] += lo.z; v[3] += lo.w;
                    v[4] += hi.x; v[5] += hi.y; v[6] += hi.z; v[7] += hi.w;
                }
                o8 = make_uint4(pack_half2(v[0], v[1]), pack_half2(v[2], v[3]), pack_half2(v[4], v[5]), pack_half2(v[6], v[7]));
            } else {
                o8 = *reinterpret_cast<const uint4*>(reinterpret_cast<const __half*>(staging) + row * pitch + c);
            }
            *reinterpret_cast<uint4*>(y + (size_t)((uint32_t)(n * args.H + yy) * (uint32_t)args.W + xx) * args.K) = o8;
        }
    }
    if (warp == 3) tmem_dealloc(tmem_d, (uint32_t)args.tmem_cols);
}

}  // namespace sd_attn
