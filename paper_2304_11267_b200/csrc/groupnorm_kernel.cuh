// Fused group normalisation (Sec. 3.1, Eq. 1): mean, variance, normalisation and the per-channel affine of one
// (sample, group) in one kernel, the group read from global memory ONCE.
//
// In the model's NCHW layout a group -- C/G consecutive channels of HW values -- is one contiguous run of memory: 80 KB
// at the 64 x 64 level of the UNet (fp16), less below, up to 0.7 MB (fp32, 96 x 96).  A cluster of one to eight blocks
// takes it into registers, reduces it to mean and variance there and writes the result.  Memory-bound: 4 bytes per
// fp16 element (2 read, 2 written).  A group that does not fit takes the streaming form: three passes over global
// memory (the second and third hit the L2).
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "softmax_math.cuh"  // packed binary32 arithmetic
#include "tc_common.cuh"     // programmatic dependent launch, FastDiv

namespace sd_attn {

constexpr int GN_THREADS = 512;

__device__ __forceinline__ float gn_to_float(__half v) { return __half2float(v); }
__device__ __forceinline__ float gn_to_float(float v) { return v; }
__device__ __forceinline__ void gn_from_float(__half& d, float v) { d = __float2half_rn(v); }
__device__ __forceinline__ void gn_from_float(float& d, float v) { d = v; }

// Sum over the block; every thread gets the result.  `scratch` holds one float per warp (+1).
__device__ __forceinline__ float gn_block_sum(float v, float* scratch) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();   // scratch may still be read from the previous reduction
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    float t = lane < (GN_THREADS >> 5) ? scratch[lane] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

struct GroupNormArgs {
    const void* x;
    const void* gamma;   // may be null
    const void* beta;    // may be null
    void* y;
    int C, G;
    long long HW;
    float eps;
};

__device__ __forceinline__ uint64_t gn_pack(float lo, float hi) { return pack_b64(__float_as_uint(lo), __float_as_uint(hi)); }
__device__ __forceinline__ float gn_sum_pair(uint64_t v) {
    uint32_t lo, hi;
    unpack_b64(v, lo, hi);
    return __uint_as_float(lo) + __uint_as_float(hi);
}
__device__ __forceinline__ void gn_from_pair(float& d0, float& d1, uint64_t v) {   // d0, d1: neighbours in memory
    uint32_t lo, hi;
    unpack_b64(v, lo, hi);
    d0 = __uint_as_float(lo);
    d1 = __uint_as_float(hi);
}
__device__ __forceinline__ void gn_from_pair(__half& d0, __half&, uint64_t v) {
    uint32_t lo, hi;
    unpack_b64(v, lo, hi);
    *reinterpret_cast<__half2*>(&d0) = __floats2half2_rn(__uint_as_float(lo), __uint_as_float(hi));
}
// x * scale + shift for the VEC values of a 16-byte piece
template <typename T, int VEC>
__device__ __forceinline__ void gn_affine_piece(const uint4& x, float scale, float shift, uint4& y) {
    const T* e = reinterpret_cast<const T*>(&x);
    T* o = reinterpret_cast<T*>(&y);
    const uint64_t ss = gn_pack(scale, scale), hh = gn_pack(shift, shift);
#pragma unroll
    for (int i = 0; i < VEC; i += 2)
        gn_from_pair(o[i], o[i + 1], fma_f32x2(gn_pack(gn_to_float(e[i]), gn_to_float(e[i + 1])), ss, hh));
}

// ------------------------------------------------------------------ statistics of a set of values
// (count, mean, sum of squared deviations from that mean).  Two sets merge without cancellation (Chan, Golub and
// LeVeque's pairwise update), so ONE reduction delivers mean and variance: a thread takes its own values' mean and
// deviations from registers, then warps, the block and the cluster merge triples.
struct GnStat {
    float n, mean, m2;
};
__device__ __forceinline__ GnStat gn_merge(const GnStat& a, const GnStat& b) {
    const float n = a.n + b.n, w = n > 0.f ? __fdividef(b.n, n) : 0.f, d = b.mean - a.mean;
    GnStat r;
    r.n = n;
    r.mean = fmaf(d, w, a.mean);
    r.m2 = a.m2 + b.m2 + d * d * (a.n * w);
    return r;
}
// Of LANES neighbouring lanes; every lane gets the result.  `alike` (the same in the whole warp): their counts are equal, as in every
// warp that holds no remainder, and the update needs neither the division nor the count.  (Sums about one lane's mean take fewer
// instructions, but lose up to LANES times the rounding of the variance where that lane lies far from the rest.)
template <int LANES>
__device__ __forceinline__ GnStat gn_merge_lanes(GnStat s, bool alike) {
    if (alike) {
        float half = 0.5f * s.n;
#pragma unroll
        for (int o = LANES / 2; o > 0; o >>= 1) {
            const float mean = __shfl_xor_sync(0xffffffffu, s.mean, o), m2 = __shfl_xor_sync(0xffffffffu, s.m2, o), d = mean - s.mean;
            s.mean = 0.5f * (s.mean + mean);
            s.m2 = fmaf(d * d, half, s.m2 + m2);
            half *= 2.f;
        }
        s.n *= (float)LANES;
        return s;
    }
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) {
        GnStat t;
        t.n = __shfl_xor_sync(0xffffffffu, s.n, o);
        t.mean = __shfl_xor_sync(0xffffffffu, s.mean, o);
        t.m2 = __shfl_xor_sync(0xffffffffu, s.m2, o);
        s = gn_merge(s, t);
    }
    return s;
}
// The means of a warp's lanes, then of a block's warps, are taken about the middle one of three of their values, so that a large common
// mean is rounded once and not in every step of the reduction, also where one lane or warp lies far from the rest (2 x 1280 x 8 x 8 fp32, a mean of
// three deviations: relative error 1.1e-7, with the means themselves 1.5e-7).
__device__ __forceinline__ float gn_middle(float a, float b, float c) { return fmaxf(fminf(a, b), fminf(fmaxf(a, b), c)); }

// Registers form: a group is shared out among the CL blocks of a cluster, a thread holds PPT 16-byte pieces of it in
// registers from the one read to the one write, and the blocks exchange one triple each through distributed shared
// memory.  RAGGED: HW times the element size is no multiple of 16, so groups begin and end inside an aligned 16-byte
// piece and pieces straddle channels.  The pieces are then those that lie whole inside the group, and the values before
// the first and behind the last one (fewer than a piece each) go to the first block's first threads one by one.
// What bounds it is the latency of one pass -- fetch, reduction, exchange, write -- as long as the group is shared out
// finely enough for every SM to take part, and the instructions of a block that holds a large group; see launch_groupnorm in
// sd_attn_api.cu for the split and what it measured.
constexpr int GN_MAX_CLUSTER = 8;
constexpr int GN_MAX_CPG = 1024;   // channels per group whose scale and shift the block keeps in shared memory

struct GroupNormPlan {
    int log2_cluster, pieces_per_block, cpg;   // blocks per group, 16-byte pieces of each, channels per group
    int ahead;                                 // ask for the values in the L2 before the stream's previous kernel has completed
    FastDiv by_hw, by_groups;
};

__device__ __forceinline__ void gn_cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void gn_cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// RESIDENT: blocks whose registers an SM holds.
template <typename T, int THREADS, int PPT, int RESIDENT, bool RAGGED>
__global__ void __launch_bounds__(THREADS, RESIDENT)
groupnorm_cluster_kernel(const GroupNormArgs a, const GroupNormPlan plan) {
    const int cluster = 1 << plan.log2_cluster, pieces_per_block = plan.pieces_per_block;
    constexpr int VEC = 16 / (int)sizeof(T), WARPS = THREADS / 32;
    __shared__ GnStat warp_stat[WARPS];
    __shared__ GnStat block_stat[GN_MAX_CLUSTER];
    __shared__ float2 affine[GN_MAX_CPG];   // y = x * .x + .y
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)blockIdx.x & (cluster - 1), group = (int)blockIdx.x >> plan.log2_cluster;
    const int cpg = plan.cpg, hw = (int)a.HW, n_elems = cpg * hw;
    const int c0 = (group - (int)fast_div((uint32_t)group, plan.by_groups) * a.G) * cpg;
    const long long base = (long long)group * n_elems;   // groups follow one another in memory
    const int head = RAGGED ? (int)((VEC - (base & (VEC - 1))) & (VEC - 1)) : 0;   // values before the first whole piece
    const int n_pieces = (n_elems - head) / VEC;                                    // (n_elems >= hw >= VEC > head)
    const int p0 = rank * pieces_per_block + tid, p_end = min(n_pieces, (rank + 1) * pieces_per_block);
    const T* src = static_cast<const T*>(a.x) + base;
    T* dst = static_cast<T*>(a.y) + base;

    if (tid == 0) pdl_launch_dependents();
    if (cluster > 1) gn_cluster_arrive();   // every block of the cluster has started once the first wait returns
    const uint4* from = reinterpret_cast<const uint4*>(src + head) + p0;
    if (plan.ahead && (tid & 7) == 0) {
#pragma unroll
        for (int k = 0; k < PPT; ++k)
            if (p0 + k * THREADS < p_end) prefetch_l2(from + k * THREADS);
    }
    pdl_wait();

    uint4 v[PPT];
    {
#pragma unroll
        for (int k = 0; k < PPT; ++k)
            if (p0 + k * THREADS < p_end) v[k] = from[k * THREADS];
    }
    // RAGGED: this thread's lone value, if it has one
    const int lone = tid < head ? tid : head + n_pieces * VEC + (tid - head);
    const bool has_lone = RAGGED && rank == 0 && tid < 2 * VEC && lone < n_elems;
    float lone_x = has_lone ? gn_to_float(src[lone]) : 0.f;
#pragma unroll 1
    for (int c = tid; c < cpg; c += THREADS)   // (read back by the thread itself: gamma and beta)
        affine[c] = make_float2(a.gamma ? gn_to_float(static_cast<const T*>(a.gamma)[c0 + c]) : 1.f,
                                a.beta ? gn_to_float(static_cast<const T*>(a.beta)[c0 + c]) : 0.f);

    // ---- statistics: the thread's own values, then warp, block, cluster.  One pass over the registers, about the
    // thread's first value: as that value is one of the set, the sum of squares about it exceeds the one about the mean by
    // at most a factor of the thread's count (and typically two), which is all the subtraction below can lose.
    float pivot = 0.f, count = 0.f;
    uint64_t sum2 = 0ull, sq2 = 0ull;
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
        if (p0 + k * THREADS >= p_end) continue;
        const T* e = reinterpret_cast<const T*>(&v[k]);
        if (k == 0) pivot = gn_to_float(e[0]);
        const uint64_t pp = gn_pack(pivot, pivot);
        count += (float)VEC;
#pragma unroll
        for (int i = 0; i < VEC; i += 2) {
            const uint64_t d = sub_f32x2(gn_pack(gn_to_float(e[i]), gn_to_float(e[i + 1])), pp);
            sum2 = add_f32x2(sum2, d);
            sq2 = fma_f32x2(d, d, sq2);
        }
    }
    if (has_lone) {
        if (count == 0.f) pivot = lone_x;
        const float d = lone_x - pivot;
        count += 1.f;
        sum2 = add_f32x2(sum2, gn_pack(d, 0.f));
        sq2 = add_f32x2(sq2, gn_pack(d * d, 0.f));
    }
    GnStat s;
    {
        const float sum = gn_sum_pair(sum2), sq = gn_sum_pair(sq2), shift = count > 0.f ? __fdividef(sum, count) : 0.f;
        s.n = count;
        s.mean = pivot + shift;
        s.m2 = fmaxf(fmaf(-sum, shift, sq), 0.f);
    }
    // threads below `left` hold a piece more than the others, and the first threads of a ragged group's first block lone values
    const int left = max(p_end - rank * pieces_per_block, 0) % THREADS, warp0 = warp * 32;
    const bool lone_values = RAGGED && rank == 0;
    const float at = gn_middle(__shfl_sync(0xffffffffu, s.mean, 0), __shfl_sync(0xffffffffu, s.mean, 16), __shfl_sync(0xffffffffu, s.mean, 31));
    s.mean = s.n > 0.f ? s.mean - at : 0.f;
    s = gn_merge_lanes<32>(s, (left <= warp0 || left >= warp0 + 32) && !(lone_values && warp == 0));
    s.mean += at;
    if (lane == 0) warp_stat[warp] = s;
    __syncthreads();
    const bool prepares = warp0 < cpg;   // scale and shift of some channels
    if (cluster > 1 ? warp == 0 : prepares) {
        const float about = gn_middle(warp_stat[0].mean, warp_stat[WARPS / 2].mean, warp_stat[WARPS - 1].mean);
        s = warp_stat[lane & (WARPS - 1)];
        s.mean = s.n > 0.f ? s.mean - about : 0.f;
        s = gn_merge_lanes<WARPS>(s, left == 0 && !lone_values);
        s.mean += about;
    }
    if (cluster > 1) {
        gn_cluster_wait();
        if (warp == 0 && lane < cluster) {   // lane r stores the block's triple into block r's slot of this block
            const uint32_t slot = (uint32_t)__cvta_generic_to_shared(&block_stat[rank]);
            uint32_t remote;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(slot), "r"(lane));
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(s.n) : "memory");
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote + 4), "f"(s.mean) : "memory");
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote + 8), "f"(s.m2) : "memory");
        }
        gn_cluster_arrive();
        gn_cluster_wait();
        s = block_stat[0];
        for (int r = 1; r < cluster; ++r) s = gn_merge(s, block_stat[r]);
    }

    // ---- y = x * scale + shift
    if (prepares) {
        const float rstd = 1.0f / sqrtf(s.m2 / (float)n_elems + a.eps);
#pragma unroll 1
        for (int c = tid; c < cpg; c += THREADS) {
            const float scale = rstd * affine[c].x;
            affine[c] = make_float2(scale, fmaf(-s.mean, scale, affine[c].y));
        }
    }
    __syncthreads();
    uint4* to = reinterpret_cast<uint4*>(dst + head) + p0;
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
        if (p0 + k * THREADS >= p_end) continue;
        const int e0 = head + (p0 + k * THREADS) * VEC, c = (int)fast_div((uint32_t)e0, plan.by_hw);
        const float2 f = affine[c];
        uint4 o;
        gn_affine_piece<T, VEC>(v[k], f.x, f.y, o);
        if (RAGGED) {
            const int left = (c + 1) * hw - e0;   // values of the piece before the next channel begins
            if (left < VEC) {
                // a channel boundary inside (one: hw >= VEC), and another channel behind it, as the piece lies inside the group:
                // the words behind the boundary come from a second evaluation
                const float2 f1 = affine[c + 1];
                uint4 o1;
                gn_affine_piece<T, VEC>(v[k], f1.x, f1.y, o1);
                uint32_t* w = reinterpret_cast<uint32_t*>(&o);
                const uint32_t* w1 = reinterpret_cast<const uint32_t*>(&o1);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t m = left * (int)sizeof(T) >= 4 * i + 4 ? 0u : left * (int)sizeof(T) > 4 * i ? 0xffff0000u : 0xffffffffu;
                    w[i] = (w[i] & ~m) | (w1[i] & m);
                }
            }
        }
        to[k * THREADS] = o;
    }
    if (has_lone) {
        const float2 f = affine[fast_div((uint32_t)lone, plan.by_hw)];
        gn_from_float(dst[lone], fmaf(lone_x, f.x, f.y));
    }
}

// Streaming form: any sizes, three passes over global memory.
template <typename T>
__global__ void __launch_bounds__(GN_THREADS)
groupnorm_streaming_kernel(const GroupNormArgs a) {
    __shared__ float scratch[GN_THREADS / 32 + 1];
    const int cpg = a.C / a.G;
    const long long n_elems = (long long)cpg * a.HW;
    const int n = blockIdx.x / a.G, g = blockIdx.x % a.G;
    const long long base = ((long long)n * a.C + (long long)g * cpg) * a.HW;
    const T* x = static_cast<const T*>(a.x) + base;
    T* y = static_cast<T*>(a.y) + base;
    float sum = 0.f;
    for (long long i = threadIdx.x; i < n_elems; i += GN_THREADS) sum += gn_to_float(x[i]);
    const float mu = gn_block_sum(sum, scratch) / (float)n_elems;
    float sq = 0.f;
    for (long long i = threadIdx.x; i < n_elems; i += GN_THREADS) {
        const float d = gn_to_float(x[i]) - mu;
        sq = fmaf(d, d, sq);
    }
    const float var = gn_block_sum(sq, scratch) / (float)n_elems;
    const float rstd = 1.0f / sqrtf(var + a.eps);
    const T* gamma = static_cast<const T*>(a.gamma);
    const T* beta = static_cast<const T*>(a.beta);
    for (long long i = threadIdx.x; i < n_elems; i += GN_THREADS) {
        const int c = g * cpg + (int)(i / a.HW);
        const float ga = gamma ? gn_to_float(gamma[c]) : 1.f, be = beta ? gn_to_float(beta[c]) : 0.f;
        const float scale = rstd * ga, shift = fmaf(-mu, scale, be);
        gn_from_float(y[i], fmaf(gn_to_float(x[i]), scale, shift));
    }
}

}  // namespace sd_attn
