// Row movers of the pot:
//   append_kernel  : Sec. 3.2 - new rows go into the free slots behind the survivors, in order;
//   compact_kernel : Appendix B "KV-cache compression" - K'[r] = K[idx[r]],
//                    V'[r] = V[idx[r]] - done in place.
#pragma once
#include "common.cuh"

namespace ipotk {

constexpr int kMoveThreads = 256;
constexpr int kMoveVecs = 8;  // 16-byte vectors in flight per thread

// One block's share of a copy of n_vecs vectors: pieces blocks of kMoveThreads threads, block `piece`.
__device__ __forceinline__ void append_body(const uint4 *__restrict__ src, uint4 *__restrict__ dst, size_t n_vecs, int piece, int pieces)
{
    const size_t stride = (size_t)pieces * kMoveThreads;
    size_t v = (size_t)piece * kMoveThreads + threadIdx.x;
    for (; v + (kMoveVecs - 1) * stride < n_vecs; v += kMoveVecs * stride) {
        uint4 t[kMoveVecs];
#pragma unroll
        for (int i = 0; i < kMoveVecs; ++i) t[i] = __ldg(src + v + i * stride);
#pragma unroll
        for (int i = 0; i < kMoveVecs; ++i) dst[v + i * stride] = t[i];
    }
    for (; v < n_vecs; v += stride) dst[v] = __ldg(src + v);
}

// grid (pieces, units, 1 or 2): tensor z of unit y (z = 0 alone: the first pair of pointers); src is [units][n_vecs],
// dst is the pot.
// kEarly: set up beside the kernel before it and lets the next one be.  For copies of at most one wave of blocks: there it
// saves most of two launch gaps, while on large ones the wait in every block costs 5 % of the copy.
template <bool kEarly>
__global__ void __launch_bounds__(kMoveThreads)
append_kernel(const uint4 *__restrict__ srcK, const uint4 *__restrict__ srcV, uint4 *__restrict__ potK,
              uint4 *__restrict__ potV, size_t n_vecs, size_t unit_vecs, size_t first_vec)
{
    if (kEarly) {
        pdl_wait();
        pdl_release();
    }
    const uint4 *src = (blockIdx.z ? srcV : srcK) + (size_t)blockIdx.y * n_vecs;
    uint4 *dst = (blockIdx.z ? potV : potK) + (size_t)blockIdx.y * unit_vecs + first_vec;
    append_body(src, dst, n_vecs, blockIdx.x, gridDim.x);
}

// A deferred append's chunk: rows of slot numbers first, first + 1, ... of every unit, still in the caller's buffers
// ([units][rows][row_vecs]); K or V is NULL where the pot already holds those rows.
struct PendingRows {
    const uint4 *K, *V;
    size_t unit_vecs;  // rows * row_vecs
    int first;
};

// ------------------------------------------------------------------ the in-place gather
// row r <- row idx[r] for every tensor (K, V) of every unit.  A tensor's kept rows are cut into chunks of about 16 KiB of
// whole rows; a block takes one chunk, gathers it into shared memory (16-byte cp.async, everything in flight at once), and
// then writes it back as one bulk copy.  idx is ascending, so idx[r] >= r, and a slot of the chunk's own destination
// range can only be the source of a row r' <= r: before a block overwrites slots [r0, r1) it waits until the chunks
// holding those r' (at most two, as at most r1 - r0 survivors come from r1 - r0 slots) have been read.  Chunks are handed out
// by a ticket per tensor in ascending order and a block reads its chunk and raises its flag before it waits for anything, so
// every wait is for a block that is already running and does not itself wait first.  (With the flag raised behind the wait a
// pot that keeps nearly everything, where every chunk waits for the one before, was a chain of flag round trips.)  The flags are relaxed accesses: when one is
// raised the chunk's bytes ARE in shared memory (the copies have been waited for), so there is no access left that a
// fence would have to order, and a release / acquire pair per block costs more than the copy of a chunk
// (256 units x 4096 -> 2048 rows of 256 bytes, all in the pot: 138 us with the pair, 91 without any flag).
//
// Bound: HBM, 2 * keep rows per tensor.  Whole rows per block because a row's 64-byte pieces fetched by different blocks
// at different times cost a DRAM access each (256 units x 4096 -> 2048 rows of 256 bytes: 80 us = 6.7 TB/s instead of 116),
// and because a unit is then not walked by one block (8 units: 11 us instead of 26).  A chunk whose rows all stay where they
// are, as the best rows of a long stream do, is left alone (2048 survivors + 2048 new rows, 256 units, 53 % of the
// survivors in place: 52 us, with every chunk copied 92).
constexpr int kGatherThreads = 128;
constexpr int kGatherBytes = 16384;
// Time limit of a wait for another chunk.  Its own, and not to be set: a chunk that gives up leaves the pot half moved, where a
// scorer that gives up only loses scores.
constexpr unsigned long long kGatherWaitNs = 200ull * 1000 * 1000;

inline int gather_rows(int row_vecs) { return kGatherBytes / 16 / row_vecs; }
inline int gather_chunks(int keep, int row_vecs) { return (keep + gather_rows(row_vecs) - 1) / gather_rows(row_vecs); }

// What the selection leaves for the gather, ints of one unit: [0, chunks] the number of survivors in slots below c * rows
// (which survivors come from a chunk's own slots).  Then per tensor the gather's own: a 64-bit ticket that counts on from launch
// to launch (a launch takes exactly `chunks` of them, so ticket / chunks numbers the launches) and, for every chunk, the
// number of the last launch in which it has been read.  Nothing is put back.
struct GatherPlan {
    int *ints;
    int rows, chunks;
    __host__ __device__ int below_ints() const { return (chunks + 2) & ~1; }
    __host__ __device__ int per_tensor() const { return 2 + ((chunks + 1) & ~1); }
    __host__ __device__ int per_unit() const { return below_ints() + 2 * per_tensor(); }
};

struct GatherParams {
    uint4 *K, *V;
    const int32_t *idx;      // [units][keep]
    GatherPlan plan;
    int *status;
    int keep, N, row_vecs;
    int units, group;        // units in all, and in a group that is walked chunk by chunk
    size_t unit_vecs;
    PendingRows pend;
    int withhold_chunk;      // -1; test hook: this chunk of every tensor is never reported as read
    bool release;            // one wave of blocks: the next kernel may be set up
};

__device__ __forceinline__ void gather_cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// What a rotary pot does with a gathered key chunk in shared memory besides moving it (k_rope.cuh); nothing here.
struct GatherNoRotate {
    static constexpr bool kOn = false;
    __device__ __forceinline__ void operator()(const uint4 *, int, int, int, int) const {}
};

// grid (chunks * 2 * group, groups), block kGatherThreads.  rotate(chunk, unit, r0, rows, row_vecs) is called for key chunks.
template <typename Rotate>
__device__ __forceinline__ void gather_block(const GatherParams &p, const Rotate &rotate)
{
    __shared__ __align__(128) uint4 buf[kGatherBytes / 16];
    __shared__ int src_sm[kGatherBytes / 64];   // (rows have at least 64 bytes)
    __shared__ int chunk_sm, launch_sm, gave_up;
    // Block order: the groups from the last one down, K then V of a unit next to each other.
    const int in_group = (int)(blockIdx.x % (2u * p.group)), unit = p.units - 1 - (int)blockIdx.y * p.group - in_group / 2, tensor = in_group & 1;
    if (unit < 0) return;   // (the last group may be smaller)
    uint4 *base = (tensor ? p.V : p.K) + (size_t)unit * p.unit_vecs;
    const int32_t *ix = p.idx + (size_t)unit * p.keep;
    const int rows = p.plan.rows, chunks = p.plan.chunks;
    const int *below = p.plan.ints + (size_t)unit * p.plan.per_unit();
    int *sync = p.plan.ints + (size_t)unit * p.plan.per_unit() + p.plan.below_ints() + tensor * p.plan.per_tensor();
    const uint4 *alt = tensor ? p.pend.V : p.pend.K;
    const int alt_first = alt ? p.pend.first : 0x7fffffff;
    if (alt) alt += (size_t)unit * p.pend.unit_vecs;
    if (threadIdx.x == 0) {
        gave_up = 0;
        const unsigned long long ticket = atomicAdd(reinterpret_cast<unsigned long long *>(sync), 1ull), launch = ticket / (unsigned)chunks;
        chunk_sm = (int)(ticket - launch * (unsigned)chunks);
        launch_sm = (int)(uint32_t)(launch + 1);
    }
    __syncthreads();
    // launched as a programmatic dependent of the selection: the blocks may be resident before it has ended and
    // wait here for its index lists (returns at once after an ordinary launch)
    pdl_wait();
    if (p.release) pdl_release();
    const int launch = launch_sm, chunk = chunk_sm, r0 = chunk * rows, n = min(rows, p.keep - r0);
    const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(buf);
    const int nvec = n * p.row_vecs;
    int q0 = 0, q1 = 0;   // the survivors whose sources lie in this chunk's slots
    if (threadIdx.x == kGatherThreads - 32) {
        q0 = __ldg(below + chunk);
        q1 = __ldg(below + chunk + 1);
    }
    for (int i = threadIdx.x; i < n; i += kGatherThreads) {
        int src = __ldg(ix + r0 + i);
        if (src < r0 + i || src >= p.N) {
            set_status(p.status, kStatusBounds);
            src = r0 + i;
        }
        src_sm[i] = src;
    }
    __syncthreads();
    // the survivors up to here have not moved (src ascends and is no less than its row): so are the bytes, in the rotated copy too
    if (src_sm[n - 1] == r0 + n - 1 && r0 + n <= alt_first) {
        if (threadIdx.x == 0 && chunk != p.withhold_chunk) asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(sync + 2 + chunk), "r"(launch) : "memory");
        return;
    }
    {
        int r = (int)threadIdx.x / p.row_vecs, c = (int)threadIdx.x - r * p.row_vecs;
        const int dr = kGatherThreads / p.row_vecs, dc = kGatherThreads - dr * p.row_vecs;
        for (int v = threadIdx.x; v < nvec; v += kGatherThreads) {
            const int src = src_sm[r];
            gather_cp_async16(sbuf + 16 * v, src >= alt_first ? alt + (size_t)(src - alt_first) * p.row_vecs + c : base + (size_t)src * p.row_vecs + c);
            r += dr;
            c += dc;
            if (c >= p.row_vecs) {
                c -= p.row_vecs;
                r += 1;
            }
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    // The lane that has the flags.  Which chunks' sources lie in this chunk's slots (none in slots whose rows are outside the pot),
    // and a first look at their flags while the rows are on their way.
    const bool lead = threadIdx.x == kGatherThreads - 32;
    int wait_c = 0, wait_end = -1;
    auto read_up = [&]() {
        int seen;
        asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(seen) : "l"(sync + 2 + wait_c) : "memory");
        return seen == launch;
    };
    if (lead && r0 < alt_first && q1 > q0) {
        wait_c = q0 / rows;
        wait_end = min(chunk - 1, (q1 - 1) / rows);
        while (wait_c <= wait_end && read_up()) ++wait_c;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the bulk copy below reads what the threads have brought in
    __syncthreads();
    if (lead) {
        if (chunk != p.withhold_chunk) asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(sync + 2 + chunk), "r"(launch) : "memory");
        const unsigned long long t0 = wait_c <= wait_end ? global_timer_ns() : 0;
        for (uint32_t tries = 1; wait_c <= wait_end; ++tries) {
            if (read_up()) {
                ++wait_c;
            } else if ((tries & 255u) == 0 && global_timer_ns() - t0 > kGatherWaitNs) {
                set_status(p.status, kStatusTimeout);
                gave_up = 1;
                break;
            }
        }
        if (!gave_up) {   // (a wait that ran out: the rows stay as they are)
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                         ::"l"(base + (size_t)r0 * p.row_vecs), "r"(sbuf), "r"((uint32_t)nvec * 16u) : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
    }
    if (Rotate::kOn && tensor == 0) {
        if (r0 < alt_first) __syncthreads();   // (else nothing was waited for)
        if (!gave_up) rotate(buf, unit, r0, n, p.row_vecs);   // (nor does the rotated copy change)
    }
    if (lead) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the block's memory is free again
}

__global__ void __launch_bounds__(kGatherThreads) compact_kernel(const __grid_constant__ GatherParams p)
{
    gather_block(p, GatherNoRotate{});
}

}  // namespace ipotk
