// CaP scoring of f32 pots (Sec. 3.3.1, Eq. 2) with fp32 FMAs, every product computed once.
//
//   f32_tile_kernel    : a block computes the logits of a tile (rows x keys) of one unit in registers, takes each row's
//                        maximum m over the tile's keys, and leaves e = 2^(x - m) in a scratch array and (m, sum e) per
//                        row beside it.  The block that completes a row tile last (a counter, no waiting) folds the
//                        row's pairs over all key tiles into (maximum, 1 / denominator).
//   f32_columns_kernel : u_j = sum_i e_ij 2^(m_tile,i - m_i) / l_i: one weight per row and key tile, no exponential per
//                        element, coalesced reads of the scratch.
//
// Bound: the FMA pipe, 2 M N d flops (recomputing the logits for the column sums, as the generic kernels do, doubles
// that; the scratch, written and read once, costs 8 bytes per logit against 2 d flops, and units are taken in groups whose
// scratch stays in L2).  A thread holds 8 rows x 4 keys as packed pairs over even and odd channels: per four
// channels 12 shared-memory vectors feed 64 packed FMAs.  Where such tiles would leave SMs idle the tiles are smaller
// (32 x 32, 16 x 16).  Measured (64 units x 4096 keys x 128 channels, M = 128): 292 us = 29 TFLOP/s; the
// generic kernels 805.  Four blocks per SM (16 warps) hide the shared-memory latency better than three with more
// registers (324 us), scalar FMAs instead of packed pairs cost 12 %.
#pragma once
#include "common.cuh"
#include "k_select.cuh"  // NucJob
#include "k_score_simt.cuh"  // merge_stats

namespace ipotk {

constexpr int kF32Threads = 128;   // 16 key columns x 8 row groups
constexpr int kF32Chan = 32;       // channels per stage
constexpr int kF32Stride = kF32Chan + 4;

struct F32Params {
    const float *Q, *K;       // [units][M][d], [units][k_unit rows][d]
    float *e;                 // [group units][M][e_stride]
    float2 *part;             // [group units][key tiles][M]
    float2 *row;              // [units][M]: (maximum, 1 / denominator)
    int *counters;            // [group units][row tiles], zero between launches
    const float2 *extra;      // NULL, or [units][M] (max, sum) that join every row's denominator
    float *scores;            // [units][N]
    int unit0, M, N, d, e_stride, key_tiles;
    int fold_here;            // the tile kernel folds the row pairs; else f32_fold_kernel does
    size_t k_unit_stride;
    float scale_log2e;
};

// RT x KT tile; thread (tx, ty) = (t % 16, t / 16) owns rows ty + 8 a and keys tx + 16 b.
// kRank: the blocks of the grid's last layer rank the streams' novelty (up to kF32RankSlots slots): on a stream of its own beside
// a launch of one wave the ranking cost a cycle two events, two waits and a launch, 5 us of 23 (2 units x 512 slots x 64 channels).
constexpr int kF32RankSlots = 16 * kF32Threads;
template <int RT, int KT, bool kRank>
__global__ void __launch_bounds__(kF32Threads, 4)
f32_tile_kernel(const __grid_constant__ F32Params p, const __grid_constant__ NucJob nuc)
{
    if (kRank && blockIdx.z == gridDim.z - 1) {
        __shared__ SelShared sel;
        pdl_wait();
        pdl_release();
        const int b = blockIdx.y * gridDim.x + blockIdx.x;
        if (b < nuc.ctas) nuc_rank_streams<kF32Threads, 16>(nuc.aux, nuc.mask, p.N, nuc.T, nuc.batch, b, nuc.ctas, sel);
        return;
    }
    constexpr int RA = RT / 8, KB = KT / 16;
    __shared__ __align__(16) float qs[2][RT * kF32Stride];
    __shared__ __align__(16) float ks[2][KT * kF32Stride];
    __shared__ int is_last;
    pdl_wait();
    pdl_release();
    const int g = blockIdx.z, unit = p.unit0 + g, i0 = blockIdx.y * RT, j0 = blockIdx.x * KT;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const float *Qu = p.Q + (size_t)unit * p.M * p.d, *Ku = p.K + (size_t)unit * p.k_unit_stride;
    const int stages = (p.d + kF32Chan - 1) / kF32Chan;
    // A thread brings one 16-byte column of a stage for every sixteenth row of the tile.  Rows beyond M or N and channels
    // beyond d become zeros.
    constexpr int kFetch = (RT + KT) / 16;
    const int fr = threadIdx.x >> 3, fc = (threadIdx.x & 7) * 4;
    const float *qp = Qu + (size_t)(i0 + fr) * p.d + fc, *kp = Ku + (size_t)(j0 + fr) * p.d + fc;
    uint32_t in_range = 0;
#pragma unroll
    for (int i = 0; i < kFetch; ++i) in_range |= (i < RT / 16 ? i0 + fr + 16 * i < p.M : j0 + fr + 16 * i - RT < p.N) ? 1u << i : 0u;
    const uint32_t fq = (uint32_t)__cvta_generic_to_shared(&qs[0][fr * kF32Stride + fc]), fk = (uint32_t)__cvta_generic_to_shared(&ks[0][fr * kF32Stride + fc]);
    auto fetch = [&](int s) {
        const int c0 = s * kF32Chan;
        const bool channels = c0 + fc < p.d;
#pragma unroll
        for (int i = 0; i < kFetch; ++i) {
            const bool is_q = i < RT / 16, ok = channels && (in_range >> i & 1u);
            const int r = is_q ? 16 * i : 16 * i - RT;
            const float *src = ok ? (is_q ? qp : kp) + (size_t)r * p.d + c0 : Qu;
            const uint32_t dst = (is_q ? fq : fk) + (uint32_t)((s & 1) * (is_q ? RT : KT) + r) * (kF32Stride * 4);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float2 acc[RA][KB];
#pragma unroll
    for (int a = 0; a < RA; ++a)
#pragma unroll
        for (int b = 0; b < KB; ++b) acc[a][b] = make_float2(0.f, 0.f);
    fetch(0);
    for (int s = 0; s < stages; ++s) {
        if (s + 1 < stages) {
            fetch(s + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const float *q = qs[s & 1] + ty * kF32Stride, *k = ks[s & 1] + tx * kF32Stride;
#pragma unroll 1
        for (int c = 0; c < kF32Chan; c += 4) {
            float4 qv[RA], kv[KB];
#pragma unroll
            for (int a = 0; a < RA; ++a) qv[a] = *reinterpret_cast<const float4 *>(q + 8 * a * kF32Stride + c);
#pragma unroll
            for (int b = 0; b < KB; ++b) kv[b] = *reinterpret_cast<const float4 *>(k + 16 * b * kF32Stride + c);
#pragma unroll
            for (int a = 0; a < RA; ++a)
#pragma unroll
                for (int b = 0; b < KB; ++b) acc[a][b] = __ffma2_rn(make_float2(qv[a].x, qv[a].y), make_float2(kv[b].x, kv[b].y), acc[a][b]);
#pragma unroll
            for (int a = 0; a < RA; ++a)
#pragma unroll
                for (int b = 0; b < KB; ++b) acc[a][b] = __ffma2_rn(make_float2(qv[a].z, qv[a].w), make_float2(kv[b].z, kv[b].w), acc[a][b]);
        }
        __syncthreads();   // the stage may be overwritten
    }
#pragma unroll
    for (int a = 0; a < RA; ++a) {
        const int row = i0 + ty + 8 * a;
        float x[KB], m = -INFINITY, l = 0.f;
#pragma unroll
        for (int b = 0; b < KB; ++b) {
            x[b] = (acc[a][b].x + acc[a][b].y) * p.scale_log2e;
            if (j0 + tx + 16 * b < p.N) m = fmaxf(m, x[b]);
        }
#pragma unroll
        for (int off = 8; off >= 1; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        const float from = m == -INFINITY ? 0.f : m;   // (a tile whose logits all lie below fp32's range: zeros, not NaNs)
#pragma unroll
        for (int b = 0; b < KB; ++b) {
            const int key = j0 + tx + 16 * b;
            const float e = exp2f(x[b] - from);
            if (key < p.N) {
                l += e;
                if (row < p.M) p.e[((size_t)g * p.M + row) * p.e_stride + key] = e;
            }
        }
#pragma unroll
        for (int off = 8; off >= 1; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
        if (tx == 0 && row < p.M) __stcg(&p.part[((size_t)g * p.key_tiles + blockIdx.x) * p.M + row], make_float2(m, l));
    }
    if (!p.fold_here) return;
    __syncthreads();
    if (threadIdx.x == 0) {
        int *counter = p.counters + (size_t)g * gridDim.y + blockIdx.y, done;
        asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(done) : "l"(counter) : "memory");
        is_last = done == p.key_tiles - 1;
        if (is_last) *counter = 0;   // ready for the next launch
    }
    __syncthreads();
    if (!is_last) return;
    // sixteen lanes per row, each over every sixteenth key tile
    for (int r = ty; r < RT && i0 + r < p.M; r += kF32Threads / 16) {
        const int row = i0 + r;
        float m = -INFINITY, l = 0.f;
        for (int t = tx; t < p.key_tiles; t += 16) {
            const float2 s = __ldcg(&p.part[((size_t)g * p.key_tiles + t) * p.M + row]);
            merge_stats(m, l, s.x, s.y);
        }
        const unsigned half = 0xffffu << (threadIdx.x & 16);   // (the two rows of a warp may end apart)
#pragma unroll
        for (int off = 8; off >= 1; off >>= 1) {
            const float m2 = __shfl_xor_sync(half, m, off), l2 = __shfl_xor_sync(half, l, off);
            merge_stats(m, l, m2, l2);
        }
        if (tx == 0) {
            if (p.extra) {
                const float2 s = p.extra[(size_t)unit * p.M + row];
                merge_stats(m, l, s.x, s.y);
            }
            p.row[(size_t)unit * p.M + row] = make_float2(m, 1.f / l);
        }
    }
}

// The fold as a launch of its own, grid (ceil(M / 4), group units): a warp per row.  For rows of many key tiles (more than
// 16 per thread of the block above: its one block's loads would be the longest chain of the cycle).
__global__ void __launch_bounds__(kF32Threads)
f32_fold_kernel(const __grid_constant__ F32Params p)
{
    const int g = blockIdx.y, unit = p.unit0 + g, row = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    pdl_wait();
    pdl_release();
    if (row >= p.M) return;
    float m = -INFINITY, l = 0.f;
    for (int t0 = 0; t0 < p.key_tiles; t0 += 256) {
        float2 s[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int t = t0 + 32 * i + lane;
            s[i] = t < p.key_tiles ? __ldcg(&p.part[((size_t)g * p.key_tiles + t) * p.M + row]) : make_float2(-INFINITY, 0.f);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) merge_stats(m, l, s[i].x, s[i].y);
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, m, off), l2 = __shfl_xor_sync(0xffffffffu, l, off);
        merge_stats(m, l, m2, l2);
    }
    if (lane == 0) {
        if (p.extra) {
            const float2 s = p.extra[(size_t)unit * p.M + row];
            merge_stats(m, l, s.x, s.y);
        }
        p.row[(size_t)unit * p.M + row] = make_float2(m, 1.f / l);
    }
}

// grid (ceil(N / 64), group units), block 256: 64 keys x 4 row quarters.  kt: keys of a tile of the first kernel (16, 32, 64).
constexpr int kF32ColThreads = 256;
__global__ void __launch_bounds__(kF32ColThreads)
f32_columns_kernel(const __grid_constant__ F32Params p, int kt)
{
    __shared__ float w[64 / 16][256];   // weights of up to 256 rows for the block's key tiles
    __shared__ float red[4][64];
    const int g = blockIdx.y, unit = p.unit0 + g, j = threadIdx.x & 63, part = threadIdx.x >> 6, key = blockIdx.x * 64 + j;
    const int tiles = 64 / kt, tile0 = blockIdx.x * tiles;
    pdl_wait();
    pdl_release();
    float u[4] = {0.f, 0.f, 0.f, 0.f};
    for (int i0 = 0; i0 < p.M; i0 += 256) {
        const int n = min(256, p.M - i0);
        __syncthreads();
        for (int v = threadIdx.x; v < tiles * n; v += kF32ColThreads) {
            const int t = v / n, i = v - t * n;
            float f = 0.f;
            if (tile0 + t < p.key_tiles) {
                const float2 s = __ldcg(&p.part[((size_t)g * p.key_tiles + tile0 + t) * p.M + i0 + i]), r = __ldcg(&p.row[(size_t)unit * p.M + i0 + i]);
                f = exp2f(s.x - r.x) * r.y;
            }
            w[t][i] = f;
        }
        __syncthreads();
        if (key < p.N) {
            const float *e = p.e + ((size_t)g * p.M + i0) * p.e_stride + key, *wj = w[j / kt];
            int i = part;
            for (; i + 28 < n; i += 32) {   // eight rows in flight
                float v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = __ldcg(e + (size_t)(i + 4 * k) * p.e_stride);
#pragma unroll
                for (int k = 0; k < 8; ++k) u[k & 3] = fmaf(v[k], wj[i + 4 * k], u[k & 3]);
            }
            for (; i < n; i += 4) u[0] = fmaf(__ldcg(e + (size_t)i * p.e_stride), wj[i], u[0]);
        }
    }
    red[part][j] = (u[0] + u[1]) + (u[2] + u[3]);
    __syncthreads();
    if (threadIdx.x < 64 && key < p.N) p.scores[(size_t)unit * p.N + key] = (red[0][j] + red[1][j]) + (red[2][j] + red[3][j]);
}

// ------------------------------------------------------------------ host side
constexpr size_t kF32Scratch = (size_t)64 << 20;   // half of L2

// Bytes a unit needs: its e values and the row pairs of its key tiles (the smallest tile has 16 keys)
inline size_t f32_unit_bytes(int M, int N) { return (size_t)M * ((N + 3) & ~3) * 4 + (size_t)((N + 15) / 16) * M * 8; }

struct F32Plan {
    char *scratch = nullptr;
    int *counters = nullptr;      // [units][row tiles of 16]
    size_t bytes = 0;
};

inline void f32_plan_init(F32Plan &plan, int units, int max_M, int pot_size, DeviceArena &mem)
{
    const size_t all = (size_t)units * f32_unit_bytes(max_M, pot_size);
    plan.bytes = all < kF32Scratch ? all : kF32Scratch;
    mem.add((void **)&plan.scratch, plan.bytes);
    mem.add((void **)&plan.counters, (size_t)units * ((max_M + 15) / 16) * sizeof(int), true);
}

inline bool f32_applicable(const F32Plan &plan, int M, int N) { return plan.scratch && f32_unit_bytes(M, N) <= plan.bytes; }

// the largest tile that still gives every SM a block
inline int f32_tile(int units, int M, int N, int sm_count)
{
    int t = 64;
    while (t > 16 && (long long)units * ((M + t - 1) / t) * ((N + t - 1) / t) < sm_count) t /= 2;
    return t;
}
// The ranking rides along where the tiles are one wave (four blocks per SM) of one launch: behind more, it runs beside them unnoticed.
inline bool f32_ranks(const F32Plan &plan, int units, int M, int N, int sm_count)
{
    const int t = f32_tile(units, M, N, sm_count);
    return f32_applicable(plan, M, N) && N <= kF32RankSlots && (long long)units * ((M + t - 1) / t) * ((N + t - 1) / t) <= 4LL * sm_count &&
           (size_t)units * f32_unit_bytes(M, N) <= plan.bytes && units < 65535;
}

// nuc.batch > 0: the first launch ranks the streams as well (only where f32_ranks() says so)
inline cudaError_t f32_launch(const F32Plan &plan, const float *Q, const float *K, const float2 *extra, float2 *row_stats, float *scores, int units,
                              int M, int N, int d, size_t k_unit_stride, float scale_log2e, int sm_count, cudaStream_t stream, int *launches, NucJob nuc)
{
    const int t = f32_tile(units, M, N, sm_count);
    F32Params p;
    p.Q = Q; p.K = K; p.extra = extra; p.row = row_stats; p.scores = scores; p.counters = plan.counters;
    p.M = M; p.N = N; p.d = d; p.k_unit_stride = k_unit_stride; p.scale_log2e = scale_log2e;
    p.e_stride = (N + 3) & ~3;
    p.key_tiles = (N + t - 1) / t;
    p.fold_here = t * p.key_tiles <= 16 * kF32Threads;
    int per = (int)(plan.bytes / f32_unit_bytes(M, N));
    if (per > 65535) per = 65535;
    p.e = (float *)plan.scratch;
    for (int u0 = 0; u0 < units; u0 += per) {
        const int n = units - u0 < per ? units - u0 : per;
        p.unit0 = u0;
        p.part = (float2 *)(plan.scratch + (size_t)n * M * p.e_stride * 4);
        const bool rank = nuc.batch > 0 && u0 == 0;
        const dim3 grid(p.key_tiles, (M + t - 1) / t, n + rank);
        if (rank) nuc.ctas = std::min(nuc.batch, (int)(grid.x * grid.y));
        auto tile = t == 64   ? (rank ? f32_tile_kernel<64, 64, true> : f32_tile_kernel<64, 64, false>)
                    : t == 32 ? (rank ? f32_tile_kernel<32, 32, true> : f32_tile_kernel<32, 32, false>)
                              : (rank ? f32_tile_kernel<16, 16, true> : f32_tile_kernel<16, 16, false>);
        cudaError_t err = launch_pdl(tile, grid, dim3(kF32Threads), 0, stream, p, nuc);
        if (!p.fold_here && err == cudaSuccess) {
            err = launch_pdl(f32_fold_kernel, dim3((M + 3) / 4, n), dim3(kF32Threads), 0, stream, p);
            *launches += 1;
        }
        if (err == cudaSuccess) err = launch_pdl(f32_columns_kernel, dim3((N + 63) / 64, n), dim3(kF32ColThreads), 0, stream, p, t);
        if (err != cudaSuccess) return err;
        *launches += 2;
    }
    return cudaGetLastError();
}

}  // namespace ipotk
