// Rankings of the cycle (Sec. 3.3.3, Appendix B "Combine NuC and CaP" and "Final
// Token Selection"):
//   nuc_mask_kernel   : per stream, mark the T slots with the largest novelty;
//   select_kernel     : per unit, give the marked slots the highest possible
//                       key, take the top `keep` keys, emit the survivors'
//                       slot numbers in ascending order.
// Both are an exact radix select on an order-preserving 32-bit image of the
// fp32 value followed by one ordered sweep; among equal keys the lower slot
// wins, so the result is a pure function of the score bits.  The digits (11
// bits) start at the highest bit in which the problem's keys differ - the scores
// of a unit span a few binades, and a digit that all of them share would put
// every count on one address - and the search ends as soon as the boundary
// digit's keys are taken as a whole: two passes nearly always, where digits of 8
// bits from the top took four (one stream's ranking of 4096 slots: 5.7 -> 4.4 us).
//
// One block per problem.  A thread keeps 16 (pot sizes above 16384: 32; 4 or 8 where every unit has an SM) consecutive
// slots' keys in registers from the first load to the last store, and the block has
// only as many threads as that takes (256 for a pot of 4096): the per-thread work of
// a pass (histogram scan, barriers) is then shared by 16 keys, which is what the
// instruction count - the bound of this kernel - is made of.  Slots beyond N carry key
// 0, which no score maps to, and are never taken.
#pragma once
#include "common.cuh"
#include "k_move.cuh"  // GatherPlan

namespace ipotk {

constexpr int kSelMaxWarps = 32;

constexpr int kSelBits = 11, kSelBins = 1 << kSelBits;
struct SelShared {
    __align__(16) uint32_t hist[kSelBins];
    uint32_t wtot[2][kSelMaxWarps];
    uint32_t wmin[kSelMaxWarps], wmax[kSelMaxWarps], wres[kSelMaxWarps];
    uint32_t bin, count;
    int remaining;
};

// The key of a slot that exists: never 0, which the NaN with all bits set would have.
__device__ __forceinline__ uint32_t slot_key(float f) { return max(order_key(f), 1u); }

// Exclusive prefix sum of v over the block in thread order; `total` = block sum.  One barrier; consecutive
// calls alternate `parity` so that a warp that runs ahead does not overwrite totals still being read.
template <int kThreads>
__device__ __forceinline__ uint32_t block_scan_exclusive(uint32_t v, SelShared &sh, int parity, uint32_t &total)
{
    constexpr int kWarps = kThreads / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += t;
    }
    if (lane == 31) sh.wtot[parity][warp] = inc;
    __syncthreads();
    uint32_t w = lane < kWarps ? sh.wtot[parity][lane] : 0u;
#pragma unroll
    for (int off = 1; off < kWarps; off <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, w, off);
        if (lane >= off) w += t;
    }
    total = __shfl_sync(0xffffffffu, w, kWarps - 1);
    const uint32_t before = __shfl_sync(0xffffffffu, w, (warp + 31) & 31);
    return (warp == 0 ? 0u : before) + inc - v;
}

// Key 0 marks no slot, key 0xFFFFFFFF a reserved one, which ranks above all.  The k (>= 1) largest keys of the block are
// those > tau and need_eq of those == tau (need_eq may be 0).  sh.hist must be zero on entry and is zero again on exit.
template <int kThreads, int kKpt>
__device__ __forceinline__ void block_radix_select(const uint32_t (&key)[kKpt], int k, SelShared &sh,
                                                   uint32_t &tau, int &need_eq)
{
    constexpr int kWarps = kThreads / 32, kPer = kSelBins / kThreads;   // bins of a thread
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t mn = 0xFFFFFFFFu, mx = 0u, res = 0u;
#pragma unroll
    for (int i = 0; i < kKpt; ++i) {
        const bool reserved = key[i] == 0xFFFFFFFFu;
        res += reserved ? 1u : 0u;
        mx = max(mx, reserved ? 0u : key[i]);
        mn = min(mn, key[i] ? key[i] : 0xFFFFFFFFu);
    }
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    res = __reduce_add_sync(0xffffffffu, res);
    if (lane == 0) {
        sh.wmin[warp] = mn;
        sh.wmax[warp] = mx;
        sh.wres[warp] = res;
    }
    __syncthreads();
    mn = __reduce_min_sync(0xffffffffu, lane < kWarps ? sh.wmin[lane] : 0xFFFFFFFFu);
    mx = __reduce_max_sync(0xffffffffu, lane < kWarps ? sh.wmax[lane] : 0u);
    res = __reduce_add_sync(0xffffffffu, lane < kWarps ? sh.wres[lane] : 0u);
    int remaining = k - (int)res;
    if (remaining <= 0) {   // only reserved slots, the lowest ones where there are more (a NaN of all ones has their key, too)
        tau = 0xFFFFFFFFu;
        need_eq = k;
        return;
    }
    uint32_t lo = mn, span = mx - mn;   // the boundary lies in [lo, lo + span]
    for (int pass = 0;; ++pass) {
        if (span == 0u) {
            tau = lo;
            need_eq = remaining;
            return;
        }
        const int bits = 32 - __clz(span), shift = bits > kSelBits ? bits - kSelBits : 0;
#pragma unroll
        for (int i = 0; i < kKpt; ++i)
            if (key[i] - lo <= span) atomicAdd(&sh.hist[(key[i] - lo) >> shift], 1u);   // (no slot and reserved ones wrap around or lie above)
        __syncthreads();
        // thread t owns the kPer bins below kSelBins - t * kPer (descending key order) and clears them for the next pass
        uint32_t c[kPer], tot = 0;
        uint2 *h2 = reinterpret_cast<uint2 *>(sh.hist + kSelBins - (threadIdx.x + 1) * kPer);
#pragma unroll
        for (int i = 0; i < kPer / 2; ++i) {
            const uint2 v = h2[i];
            h2[i] = make_uint2(0u, 0u);
            c[kPer - 1 - 2 * i] = v.x;
            c[kPer - 2 - 2 * i] = v.y;
            tot += v.x + v.y;
        }
        uint32_t total;
        uint32_t run = block_scan_exclusive<kThreads>(tot, sh, pass & 1, total);   // keys in the bins above this thread's
        if (run < (uint32_t)remaining && (uint32_t)remaining <= run + tot) {
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                if (run < (uint32_t)remaining && (uint32_t)remaining <= run + c[i]) {
                    sh.bin = kSelBins - 1 - (threadIdx.x * kPer + i);
                    sh.count = c[i];
                    sh.remaining = remaining - (int)run;
                }
                run += c[i];
            }
        }
        __syncthreads();
        remaining = sh.remaining;
        lo += sh.bin << shift;
        if ((uint32_t)remaining == sh.count) {   // the whole digit is taken (the case remaining == count == 1 above all)
            tau = lo - 1u;
            need_eq = 0;
            return;
        }
        span = min((1u << shift) - 1u, mx - lo);
    }
}

// Larger and equal keys in the slots below this thread's, in one block scan (16 bits each: a block has at
// most 32768 slots); `total` = the same counts over the block.
template <int kThreads, int kKpt>
__device__ __forceinline__ uint32_t block_count_before(const uint32_t (&key)[kKpt], uint32_t tau, SelShared &sh, uint32_t &total)
{
    uint32_t mine = 0;
#pragma unroll
    for (int i = 0; i < kKpt; ++i) mine += (key[i] > tau ? 1u : 0u) + (key[i] == tau ? 0x10000u : 0u);
    return block_scan_exclusive<kThreads>(mine, sh, 0, total);
}
// Ordered sweep: slot j is taken iff key > tau, or key == tau and it is among the first need_eq such
// slots.  taken(j, pos) is called for every taken slot with its rank pos among the taken ones;
// every(i, is_taken) for each of the thread's slots i < kKpt.  `before` = block_count_before().
template <int kThreads, int kKpt, typename Taken, typename Every>
__device__ __forceinline__ void block_ordered_sweep(const uint32_t (&key)[kKpt], int slot0, uint32_t tau, int need_eq,
                                                    uint32_t before, Taken taken, Every every)
{
    int gt_before = (int)(before & 0xFFFFu), eq_before = (int)(before >> 16);
#pragma unroll
    for (int i = 0; i < kKpt; ++i) {
        const bool gt = key[i] > tau, eq = key[i] == tau;
        const bool sel = gt || (eq && eq_before < need_eq);
        every(i, sel);
        if (sel) taken(slot0 + i, gt_before + min(eq_before, need_eq));
        gt_before += gt;
        eq_before += eq;
    }
}

struct SelNoTaken { __device__ void operator()(int, int) const {} };
struct SelNoEvery { __device__ void operator()(int, bool) const {} };
constexpr int kSelStage = 4096;   // survivors staged in shared memory per round of the index output
struct SelStageIndex {            // positions [base, base + kSelStage) go to the stage, the rest to another round
    int32_t *stage;
    int base;
    __device__ void operator()(int j, int pos) const
    {
        if ((unsigned)(pos - base) < (unsigned)kSelStage) stage[pos - base] = j;
    }
};
struct SelPackMask {  // byte i of the thread's mask bytes, four to a word
    uint32_t *packed;
    __device__ void operator()(int i, bool s) const { packed[i >> 2] |= (s ? 1u : 0u) << (8 * (i & 3)); }
};

// Slots [slot0, slot0 + kKpt) of a row of N floats that may start on any 4-byte boundary (rows of an odd length): whole
// 16-byte vectors from the boundary below the first slot on, shifted into place (the shift is the same for every
// thread of a block), one by one at the row's ends; slots at or beyond N are left alone.
// (With one 4-byte load per slot, 64 bytes apart across a warp, such a row took 3 us more.)
template <int kKpt, int kShift>
__device__ __forceinline__ void shift_row(const float4 (&q)[kKpt / 4 + 1], float (&s)[kKpt])
{
#pragma unroll
    for (int i = 0; i < kKpt; ++i) {
        const float4 v = q[(i + kShift) / 4];
        s[i] = (i + kShift) % 4 == 0 ? v.x : (i + kShift) % 4 == 1 ? v.y : (i + kShift) % 4 == 2 ? v.z : v.w;
    }
}
template <int kKpt>
__device__ __forceinline__ void load_row(const float *__restrict__ row, int slot0, int N, float (&s)[kKpt])
{
    const int shift = (int)(reinterpret_cast<uintptr_t>(row) >> 2) & 3;
    if (shift == 0 ? slot0 + kKpt <= N : (slot0 > 0 && slot0 + kKpt + 4 <= N)) {
        const float4 *v = reinterpret_cast<const float4 *>(row + slot0 - shift);
        float4 q[kKpt / 4 + 1];
#pragma unroll
        for (int i = 0; i < kKpt / 4; ++i) q[i] = __ldg(v + i);
        q[kKpt / 4] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (shift) q[kKpt / 4] = __ldg(v + kKpt / 4);
        switch (shift) {
        case 0: shift_row<kKpt, 0>(q, s); break;
        case 1: shift_row<kKpt, 1>(q, s); break;
        case 2: shift_row<kKpt, 2>(q, s); break;
        default: shift_row<kKpt, 3>(q, s); break;
        }
    } else {
#pragma unroll
        for (int i = 0; i < kKpt; ++i)
            if (slot0 + i < N) s[i] = row[slot0 + i];
    }
}
__host__ __device__ inline int mask_stride(int N) { return (N + 31) & ~31; }   // bytes of a stream's mask row

// mask[b][j] = 1 iff slot j is one of the T most novel slots of stream b, for the streams first, first + step, ... of batch,
// by kThreads threads of the block.
template <int kThreads, int kKpt>
__device__ __forceinline__ void nuc_rank_streams(const float *__restrict__ aux, uint8_t *__restrict__ mask, int N, int T, int batch, int first,
                                                 int step, SelShared &sh)
{
    const int slot0 = threadIdx.x * kKpt;
    for (int i = threadIdx.x; i < kSelBins; i += kThreads) sh.hist[i] = 0;
    for (int b = first; b < batch; b += step) {
        uint8_t *m = mask + (size_t)b * mask_stride(N);
        uint32_t key[kKpt];
        {
            float s[kKpt];
            load_row<kKpt>(aux + (size_t)b * N, slot0, N, s);
#pragma unroll
            for (int i = 0; i < kKpt; ++i) key[i] = slot0 + i < N ? slot_key(s[i]) : 0u;
        }
        __syncthreads();
        uint32_t tau;
        int need_eq;
        block_radix_select<kThreads, kKpt>(key, T, sh, tau, need_eq);
        uint32_t packed[kKpt / 4];
#pragma unroll
        for (int i = 0; i < kKpt / 4; ++i) packed[i] = 0;
        uint32_t total;
        const uint32_t before = block_count_before<kThreads, kKpt>(key, tau, sh, total);
        block_ordered_sweep<kThreads, kKpt>(key, slot0, tau, need_eq, before, SelNoTaken{}, SelPackMask{packed});
        if (slot0 < N) {   // (a row has room for whole vectors)
#pragma unroll
            for (int i = 0; i < kKpt / 4; i += 4)
                *reinterpret_cast<uint4 *>(m + slot0 + 4 * i) = make_uint4(packed[i], packed[i + 1], packed[i + 2], packed[i + 3]);
        }
        __syncthreads();
    }
}
template <int kThreads, int kKpt>
__global__ void __launch_bounds__(kThreads)
nuc_mask_kernel(const float *__restrict__ aux, uint8_t *__restrict__ mask, int N, int T, int batch)
{
    __shared__ SelShared sh;
    nuc_rank_streams<kThreads, kKpt>(aux, mask, N, T, batch, blockIdx.x, gridDim.x, sh);
}

// The ranking as extra blocks of a scorer's grid, for up to kNucMaxSlots slots: a kernel of its own beside the scorer costs an
// event fork and join, about 5 us of a small cycle.  (Out of line it cost the scorer's own blocks more: 10 % instead of 5.)
struct NucJob {
    const float *aux;   // [batch][N]
    uint8_t *mask;
    int T, batch, ctas;   // ctas == 0: nothing to rank
};
constexpr int kNucThreads = 512, kNucMaxSlots = 16 * kNucThreads;
__device__ __forceinline__ void nuc_rank_extra_block(const NucJob &job, int N, int first, SelShared *sh)
{
    if (threadIdx.x >= kNucThreads) return;   // (the barriers below count the threads that have not exited)
    nuc_rank_streams<kNucThreads, 16>(job.aux, job.mask, N, job.T, job.batch, first, job.ctas, *sh);
}

// grid (units).  scores: `parts` partial score arrays of [units][N] each, `part_stride`
// floats apart, added in index order.  mask may be NULL (T == 0).  The survivors' slot numbers
// are put in order in shared memory and leave in 16-byte stores.
template <int kThreads, int kKpt>
__global__ void __launch_bounds__(kThreads)
select_kernel(const float *__restrict__ scores, int parts, size_t part_stride,
              const uint8_t *__restrict__ mask, int32_t *__restrict__ idx, float *__restrict__ summed,
              int N, int keep, int Hkv, int batch, int *status, GatherPlan plan)
{
    __shared__ SelShared sh;
    __shared__ __align__(16) int32_t stage[kSelStage];
    const int unit = blockIdx.x;
    const int b = (unit / Hkv) % batch;
    const float *u = scores + (size_t)unit * N;
    const uint8_t *m = mask ? mask + (size_t)b * mask_stride(N) : nullptr;
    const int slot0 = threadIdx.x * kKpt;
    for (int i = threadIdx.x; i < kSelBins; i += kThreads) sh.hist[i] = 0;
    int *below = plan.ints + (size_t)unit * plan.per_unit();   // for the gather that follows
    // launched as a programmatic dependent of the scorer: its scores and the ranking's mask are complete after this.  Then
    // the compaction may be made resident; it waits for this grid's end before it reads an index.
    pdl_wait();
    pdl_release();
    uint32_t key[kKpt];
    // a reserved slot outranks every score: finite scores map below 0xFF800000
    constexpr int kPiece = kKpt > 16 ? 8 : kKpt;   // slots loaded at a time (what 64 registers a thread allow)
#pragma unroll
    for (int h = 0; h < kKpt; h += kPiece) {
        const int first = slot0 + h;
        float s[kPiece];
        uint32_t r[kPiece / 4];
        load_row<kPiece>(u, first, N, s);
#pragma unroll
        for (int i = 0; i < kPiece / 4; ++i) r[i] = (m && first < N) ? *reinterpret_cast<const uint32_t *>(m + first + 4 * i) : 0u;
        if (parts > 1) {
#pragma unroll 1
            for (int p = 1; p < parts; ++p) {
                float t[kPiece];
                load_row<kPiece>(u + (size_t)p * part_stride, first, N, t);
#pragma unroll
                for (int i = 0; i < kPiece; ++i) s[i] += t[i];
            }
            float *to = summed + (size_t)unit * N + first;
            if (summed) {
                if ((reinterpret_cast<uintptr_t>(to) & 15u) == 0 && first + kPiece <= N) {
#pragma unroll
                    for (int i = 0; i < kPiece; i += 4) *reinterpret_cast<float4 *>(to + i) = make_float4(s[i], s[i + 1], s[i + 2], s[i + 3]);
                } else {
#pragma unroll
                    for (int i = 0; i < kPiece; ++i)
                        if (first + i < N) to[i] = s[i];
                }
            }
        }
#pragma unroll
        for (int i = 0; i < kPiece; ++i)
            key[h + i] = first + i >= N ? 0u : (r[i >> 2] >> (8 * (i & 3))) & 0xFFu ? 0xFFFFFFFFu : slot_key(s[i]);
    }
    __syncthreads();
    uint32_t tau;
    int need_eq;
    block_radix_select<kThreads, kKpt>(key, keep, sh, tau, need_eq);
    uint32_t total;
    const uint32_t before = block_count_before<kThreads, kKpt>(key, tau, sh, total);
    const int taken = (int)(total & 0xFFFFu) + min((int)(total >> 16), need_eq);
    if (taken != keep && threadIdx.x == 0) set_status(status, kStatusBounds);
    // for the gather: survivors below the first slot of every chunk of slots (at most one or two such slots per thread)
    for (int c = (slot0 + plan.rows - 1) / plan.rows; c <= plan.chunks && c * plan.rows < slot0 + kKpt; ++c) {
        int gt = (int)(before & 0xFFFFu), eq = (int)(before >> 16);
#pragma unroll
        for (int i = 0; i < kKpt; ++i) {
            const bool in = slot0 + i < c * plan.rows;
            gt += in && key[i] > tau;
            eq += in && key[i] == tau;
        }
        below[c] = gt + min(eq, need_eq);
    }
    if (threadIdx.x == 0 && plan.chunks * plan.rows >= kThreads * kKpt) below[plan.chunks] = keep;
    int32_t *out = idx + (size_t)unit * keep;
    for (int base = 0; base < keep; base += kSelStage) {
        block_ordered_sweep<kThreads, kKpt>(key, slot0, tau, need_eq, before, SelStageIndex{stage, base}, SelNoEvery{});
        __syncthreads();
        const int n = min(kSelStage, min(keep, taken) - base);
        if ((keep & 3) == 0) {
            for (int i = 4 * threadIdx.x; i < n; i += 4 * kThreads) {
                if (i + 4 <= n) *reinterpret_cast<int4 *>(out + base + i) = *reinterpret_cast<const int4 *>(stage + i);
                else
                    for (int e = i; e < n; ++e) out[base + e] = stage[e];
            }
        } else {
            for (int i = threadIdx.x; i < n; i += kThreads) out[base + i] = stage[i];
        }
        if (base + kSelStage < keep) __syncthreads();
    }
}

// Launch shapes: the smallest block whose threads hold N slots at 16 a thread (32 above 16384 slots).
inline void launch_nuc_mask(int blocks, cudaStream_t st, const float *aux, uint8_t *mask, int N, int T, int batch)
{
    const int threads = N <= 4096 ? 256 : N <= 8192 ? 512 : 1024;
    auto kern = N <= 4096 ? nuc_mask_kernel<256, 16> : N <= 8192 ? nuc_mask_kernel<512, 16> : N <= 16384 ? nuc_mask_kernel<1024, 16> : nuc_mask_kernel<1024, 32>;
    kern<<<blocks, threads, 0, st>>>(aux, mask, N, T, batch);
}
inline cudaError_t launch_select(int blocks, cudaStream_t st, const float *scores, int parts, size_t part_stride, const uint8_t *mask,
                                 int32_t *idx, float *summed, int N, int keep, int Hkv, int batch, int *status, const GatherPlan &plan, int sm_count)
{
    auto kern = N <= 4096 ? select_kernel<256, 16> : N <= 8192 ? select_kernel<512, 16> : N <= 16384 ? select_kernel<1024, 16> : select_kernel<1024, 32>;
    int threads = N <= 4096 ? 256 : N <= 8192 ? 512 : 1024;
    // A unit per SM: what counts is one block's chain, not the number of instructions, and a thread of 4 (8) keys is through
    // its histogram and its scans earlier (whole passes, us: 8 units x 4096 28.9 -> 26.8, x 2000 25.5 -> 23.0, x 1000 23.4 -> 20.9, x 8192 36.5 -> 36.1;
    // 8 keys below 4096 slots as well: 27.4, 24.6, 21.7).
    if (N <= 8192 && blocks <= sm_count) {
        kern = N <= 512 ? select_kernel<128, 4> : N <= 1024 ? select_kernel<256, 4> : N <= 2048 ? select_kernel<512, 4> : N <= 4096 ? select_kernel<1024, 4> : select_kernel<1024, 8>;
        threads = N <= 512 ? 128 : N <= 1024 ? 256 : N <= 2048 ? 512 : 1024;
    }
    return launch_pdl(kern, dim3(blocks), dim3(threads), 0, st, scores, parts, part_stride, mask, idx, summed, N, keep, Hkv, batch, status, plan);
}

// summed[i] = parts[0][i] + parts[1][i] + ... in index order (the order select_kernel uses).
__global__ void sum_parts_kernel(const float *__restrict__ scores, int parts, size_t part_stride,
                                 float *__restrict__ summed, size_t n)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float s = scores[i];
    for (int p = 1; p < parts; ++p) s += scores[(size_t)p * part_stride + i];
    summed[i] = s;
}

}  // namespace ipotk
