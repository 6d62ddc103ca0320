// CaP scoring on the 5th-generation tensor cores (Sec. 3.3.1, Eq. 2), bf16, any d up to 256.
//
// Item  = (unit, block of 128 folded query rows): one row-softmax problem over the
//         unit's N pot keys.
// Task  = (item, slab of 256 keys).  Tasks are numbered item-major and dealt round
//         robin to a persistent grid of one CTA per SM, so the slabs of an item are
//         in flight on neighbouring SMs at the same time.
//
// Per task, inside one CTA (warp-specialised, two tasks in flight):
//   TMA      Q tile (128 x 128 bf16) and the slab's keys (256 x 128 bf16) land in
//            shared memory in the 128-byte-swizzled K-major layout (2 stages);
//   tcgen05  S = Q K^T (128 x 256 fp32) accumulates in one of two 256-column tensor
//            memory buffers, one 128-column half at a time: the logits never leave
//            the SM;
//   epilogue (16 warps in four groups, a group per 128 columns of tensor memory; groups 0, 1 have the CTA's even
//            tasks, 2, 3 the odd ones, so that one pair computes while the other waits for the exchange)
//     pass 1   a thread owns one query row: e = 2^x is written back over the logits and summed, against the reference
//              0 - no maximum is taken as long as a row's first logits add up to 1 and none is 2^100 above the reference; other rows get one of
//              their own (+3 %) -; a quarter of the exponentials run on the FMA pipe.  The warps of a scheduler take pass 1 in turns, pair after pair: both
//              pairs at once finish later than one of them could, and every reader of their sums waits;
//     exchange the two groups of a pair add their row sums through shared memory and publish them with one 4-byte store
//              that carries the launch's sign as a "fresh" mark; a thread reads half of its row's sums of the whole item
//              (the other group of the pair the other half), re-reading until every one is fresh, and the pair turns
//              them into the row's denominator l (plus, when given, the share of the CaP's own keys);
//     pass 2   u_j = sum_i e_ij / l_i as a weighted column sum: the 16x256b tensor-memory load shape hands every
//              thread four rows of a column pair, so the sum over a warp's 32 rows is four packed FMAs plus a
//              three-step exchange between lanes; the four row quarters meet in shared memory and are added and
//              stored behind the next task's barrier: 256 floats per task.
// A row block of fewer rows keeps the warps of its empty quarters out of all of this.
//
// Bound: a task's way through tensor memory, and tensor memory holds two tasks: product 700 cycles, pass 1 4100 beside the other
// pair's work, exchange 2000, pass 2 1800, hand-overs 500.  (Pass 1 and pass 2 alone would take an SM 2500 cycles per task, without the
// exchange a launch of 256 units takes 66 us.)  The polls are what the exchange costs: with an entry per 128 keys instead of one per
// 256 the last of these figures were 85.2, 173, 18.5 and 384.  Keys far beyond a row's others cost it more: 256 units x 4096 keys of Student t
// (3 degrees) 88 us, with one far key in every unit 101.  Measured against the form in which all 16 warps
// shared a task, took maxima, and four more warps combined and polled (us, alone): 256 units x 4096 keys, M = 128 90.1 -> 82; 128 x
// 8192, M = 256 197 -> 157; 60 x 2999, M = 57 20.8 -> 18.5; 64 x 16384, M = 512 537 -> 333; items -> this: 64 x 4096 x 256 channels, M = 64 51 -> 33.  Error of the scores against
// 64 bits 4.5e-7 -> 1.6e-7 (fewer roundings, a polynomial of degree 5, the tensor core's cut sums made good).
//
// Blocks of one grid wait on each other (pass 2 needs the other slabs' statistics),
// so the grid is launched cooperatively with at most one CTA per SM: all of it is
// resident.  A pair publishes its task before it waits for others, and takes its tasks in
// order, so the waits cannot form a cycle.  Every wait (mbarrier or statistics) is bounded by a time
// limit (a launch parameter); one that runs out records IPOT_E_TIMEOUT in the status
// word and raises a block-wide flag.  From then on every wait of the block returns at
// once: the producer and the MMA issuer stop putting work in flight and wait for what
// they have issued (loads into this CTA's shared memory, MMAs into its tensor memory)
// before the block releases tensor memory and ends; the epilogue warps run through
// their remaining iterations without waiting (their results are void).
#pragma once
#include <algorithm>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "../../include/ipot.h"
#include "common.cuh"
#include "k_select.cuh"  // NucJob

namespace ipotk {

constexpr int kTcThreads = 576;      // warp 0: TMA, 1: MMA + TMEM owner, 2-17: epilogue, four groups of four warps
constexpr int kTcRows = 128;         // query rows per item (TMEM lanes)
constexpr int kTcHalf = 128;         // keys per epilogue group and entry of the statistics
// The first look at a task's statistics comes this much after its own have left: the others' are never there at once, and what is not
// polled leaves L2 to the keys.  Measured (256 units x 4096 keys, M = 128 / 128 x 8192, M = 256, us): 0 ns 88.6 / 175.1, 300 85.2 / 172.7,
// 600 85.8 / 180.5 (before the pair's sums were joined; since then 0 to 300 are equal); a CTA's first task (all there is in a small launch) does not wait (8 units x 4096: 8.3, 8.4, 10.1).
constexpr unsigned kTcPollDelayNs = 300;
constexpr int kTcSlab = 256;         // keys per task (TMEM columns per buffer)
constexpr int kTcFmaEighths = 2;     // share of pass 1's exponentials evaluated on the FMA pipe
constexpr int kTcD = 128;            // channels of a stage; up to 64 use the first half of every tile.  Wider rows are another variant (kWide)
constexpr uint32_t kTcQBytes = kTcRows * kTcD * 2;           // 32 KiB: two halves of 128 rows x 64 channels
constexpr uint32_t kTcKBytes = kTcSlab * kTcD * 2;           // 64 KiB: two halves of 256 rows x 64 channels
constexpr uint32_t kTcStageBytes = kTcQBytes + kTcKBytes;    // 96 KiB
// More than 128 channels: one or two query tiles and two or three half slabs of keys share the space of the two stages, each a slot
// of its own - a whole stage of 256 channels would be all there is room for.  (Slots like these for every width: 4 % slower at 128 channels.)
constexpr uint32_t kTcKBlk = kTcHalf * 128;                  // 64 channels of a half slab's keys
constexpr int kTcMaxK = 4;

// shared-memory carve-up (bytes from the 1024-aligned base)
constexpr uint32_t kTcOffStage = 0;                                        // [2] { Q, K }
constexpr uint32_t kTcOffColpart = 2 * kTcStageBytes;                      // [4 groups][2 parities][4 row quarters][128] float
constexpr uint32_t kTcOffLpart = kTcOffColpart + 4 * 2 * 4 * kTcHalf * 4;      // [2 pairs][2 parities][2 halves][128] float
constexpr uint32_t kTcOffLfar = kTcOffLpart + 2 * 2 * 2 * kTcRows * 4;         // [2 pairs][2 parities][2 halves][128] float2: (reference, sum) of those that are infinite
constexpr uint32_t kTcOffSpart = kTcOffLfar + 2 * 2 * 2 * kTcRows * 8;        // [2 pairs][2 parities][128] float2
constexpr uint32_t kTcOffBar = kTcOffSpart + 2 * 2 * kTcRows * 8;
constexpr uint32_t kTcOffTmemSlot = kTcOffBar + 208;                       // the allocated TMEM base address
constexpr uint32_t kTcOffAbort = kTcOffBar + 212;                          // set once a wait of the CTA has run out; + 4: the block's deadline (8 bytes)
constexpr uint32_t kTcSmemBytes = kTcOffBar + 256;                         // no static shared memory: the base is 1024-aligned

// barriers: per stage Full, Empty; per group (= buffer half 2 * buffer + half) SFull, TEmpty; wide rows: per query and key slot Full, Empty
enum {
    kBarFull = 0, kBarEmpty = 2, kBarSFull = 4, kBarTEmpty = 8, kBarDrain = 12, kBarQFull = 13, kBarQEmpty = 15, kBarKFull = 17,
    kBarKEmpty = kBarKFull + kTcMaxK, kBarCount = kBarKEmpty + kTcMaxK
};

struct TcParams {
    float *scores;        // partial array p (query rows 128p ...) at scores + p * part_stride, unit stride N
    size_t part_stride;
    float *stats;         // [items][slabs][128] a row's sum over a slab's keys, times the launch's sign (infinite: beyond the plain range, see
                          // refs); all of the other sign or 0 at launch
    float2 *refs;         // [items][slabs][128] (reference, sum) of those
    const float2 *cap_stats;  // NULL, or [units][M] (max, sum) over the CaP's own keys that join every row's denominator
    float sign;           // +1 or -1: this launch's "fresh" mark
    unsigned long long wait_ns;  // limit of every wait
    int withhold_cta;     // -1; test hook: this CTA never publishes its slab statistics
    int *status;
    int N, M, mtiles, slabs, tasks;
    int dhalves;          // 64-channel blocks of a row; what the last one lacks is filled with zeros
    // wide rows: 16-channel steps; bytes of 64 channels of a query tile, of the tile, of a half slab's keys; slots.  M <= 64: the tile has 64
    // rows; a product still has 128, of which the lower half multiplies whatever lies behind the tile and is never read
    int ksteps;
    uint32_t q_blk, q_bytes, k_bytes;
    int qslots, kslots;
    int new_slab0;        // slabs from this one on are read through the second key map (the chunk of a deferred
                          // append, row 0 = key 256 * new_slab0); INT_MAX if all keys are in the pot
    float scale_log2e;
    int ctas;             // blocks that score; those behind them rank the streams' novelty
    NucJob nuc;
};

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait.  Every block notes a deadline (its start + the launch's wait limit) next to its give-up flag; a
// wait that is still unsatisfied then records IPOT_E_TIMEOUT and raises the flag.  Once the flag is up, later waits
// of the block return at once (false) - unless heed_flag is off, which is how a role waits for work it has itself
// put in flight before the block may end.  (Clock and flag are looked at every 1024 rounds only: the kernel's
// speed depends on this loop staying small.)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status, bool heed_flag = true)
{
    for (uint32_t i = 0;; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 1023u) == 1023u) {
            if (heed_flag && *abort_flag) return false;
            if (global_timer_ns() > *reinterpret_cast<volatile unsigned long long *>(abort_flag + 1)) {
                *abort_flag = 1;
                set_status(status, kStatusTimeout);
                return false;
            }
        }
    }
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

// 32 consecutive fp32 columns of this thread's TMEM lane (asynchronous: see tmem_wait_ld).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr) : "memory");
}
// 16 TMEM lanes x 32 fp32 columns in the 16x256b shape: for each block j of 8 columns, thread t of the warp
// receives v[4j], v[4j+1] = lane t/4, columns 8j + 2(t%4), +1 and v[4j+2], v[4j+3] = lane t/4 + 8, same columns.
__device__ __forceinline__ void tmem_ld_16x256b_x4(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld16(uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.wait::ld.sync.aligned;"
        : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
          "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
        :: "memory");
}
// Waits for this thread's outstanding TMEM loads.  The loaded registers are passed
// through so that no use of them can be scheduled ahead of the wait.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.wait::ld.sync.aligned;"
        : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
          "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
          "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
          "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
        :: "memory");
}
// 16 consecutive fp32 columns of this thread's TMEM lane (asynchronous: see tmem_wait_ld16).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};"
        ::"r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
          "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Named barriers: of the four warps of an epilogue group, and of the two groups that share a buffer.
// (With those of the turns below, fifteen of the SM's sixteen: one block has the SM to itself.)
__device__ __forceinline__ void group_sync(int g)
{
    switch (g) {
    case 0: asm volatile("bar.sync 1, 128;" ::: "memory"); break;
    case 1: asm volatile("bar.sync 2, 128;" ::: "memory"); break;
    case 2: asm volatile("bar.sync 3, 128;" ::: "memory"); break;
    default: asm volatile("bar.sync 4, 128;" ::: "memory"); break;
    }
}
__device__ __forceinline__ void pair_sync(int pair)
{
    if (pair == 0) asm volatile("bar.sync 5, 256;" ::: "memory");
    else asm volatile("bar.sync 6, 256;" ::: "memory");
}
// Turns: the warps of a TMEM lane quarter (= scheduler) of one pair take pass 1 after those of the other pair have done theirs.
__device__ __forceinline__ void turn_wait(int pair, int q) { asm volatile("bar.sync %0, 128;" ::"r"(7 + pair * 4 + q) : "memory"); }
__device__ __forceinline__ void turn_pass(int pair, int q) { asm volatile("bar.arrive %0, 128;" ::"r"(11 - pair * 4 + q) : "memory"); }
// The statistics are exchanged between CTAs with relaxed accesses at gpu scope: a reader sees the old or the new value of each entry.
__device__ __forceinline__ float ld_gpu_f32(const float *p)
{
    float v;
    asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_gpu_f32(float *p, float v)
{
    asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float y;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}

// The reference of a row over a half slab: 0 if the largest of its first logits (in binary orders) lies between 0 and kTcNear, else that logit
// rounded down to a whole number (moving a sum to another reference is then exact, and no exponential is below its
// probability).  Where no logit is within fp32's range it is 0 and pass1_slow looks at the others.
constexpr float kTcNear = 32.f;
__device__ __forceinline__ float row_reference(float mx, float c)
{
    const float r = floorf(mx * c);
    return (r >= 0.f && r <= kTcNear) || !(fabsf(r) < INFINITY) ? 0.f : r;
}
// 16 columns against the reference r: v <- 2^(v c - r), added into two packed running sums; pm: the largest logit among those that went
// to the FMA pipe, whose exponent arithmetic wraps around where the special-function unit returns +inf.
struct PieceSum {
    float2 s[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    float pm = -INFINITY;
    __device__ __forceinline__ float total() const
    {
        const float2 t = __fadd2_rn(s[0], s[1]);
        return t.x + t.y;
    }
};
template <int kFma = kTcFmaEighths>
__device__ __forceinline__ void piece_exp(uint32_t (&v)[16], float c, float r, PieceSum &p)
{
    const float2 c2 = make_float2(c, c), nr2 = make_float2(-r, -r);
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
        const float2 x = make_float2(__uint_as_float(v[i]), __uint_as_float(v[i + 1])), t = __ffma2_rn(x, c2, nr2);
        float2 e2;
        if (pair_on_fma<kFma>(i >> 1)) {
            p.pm = max3(p.pm, x.x, x.y);
            e2 = exp2_fma_pair5(t);
        } else {
            e2 = make_float2(ex2(t.x), ex2(t.y));
        }
        p.s[(i >> 1) & 1] = __fadd2_rn(p.s[(i >> 1) & 1], e2);
        v[i] = __float_as_uint(e2.x);
        v[i + 1] = __float_as_uint(e2.y);
    }
}
// A row's exponentials are taken against its reference and kept where they are up to 2^100 above it; what is 2^126 below it is lost, and its
// probability is smaller than that.  A weight then is as small as 2^-226 before nothing of its row counts: see kTcLift.
constexpr float kTcSumMax = 1.2676506e30f;    // 2^100
constexpr float kTcSumMin = 0.99f;            // of a row's first logits; with a reference its own term is 1 (less: they are all beyond fp32's range)
constexpr float kTcReach = 100.f;
constexpr float kTcRefLow = -90.f, kTcPlainMax = 3.3230700e35f;   // a sum is published as it is, times 2^reference, up to 2^118 (128 of them are still finite)
constexpr float kTcTiny = 1.1754944e-38f;     // an entry that adds nothing is still not 0
// Where a row's weight is below 2^-100 its warp's weights are multiplied by 2^110 and the column sums divided by it: 2^-226 times
// exponentials of up to 2^100 is a probability that fp32 holds.
constexpr float kTcLift = 110.f, kTcLifted = 1.2980742e33f, kTcUnlift = 7.7037198e-34f;

// (reference, sum) with the sum in [1, 2): sums that are far apart can then be brought to one reference without a factor that underflows
// while what it multiplies still counts.  An empty sum has no reference.
__device__ __forceinline__ float2 normalised(float2 a)
{
    const int b = __float_as_int(a.y);
    if (!(a.y < INFINITY)) return a;
    if (b < 0x00800000) return make_float2(-INFINITY, 0.f);
    return make_float2(a.x + (float)((b >> 23) - 127), __int_as_float((b & 0x007FFFFF) | 0x3F800000));
}
__device__ __noinline__ float2 add_sums(float2 a, float2 b)
{
    a = normalised(a);
    b = normalised(b);
    const float m = fmaxf(a.x, b.x);
    if (m == -INFINITY) return make_float2(0.f, kTcTiny);
    return make_float2(m, fmaf(a.y, ex2(a.x - m), b.y * ex2(b.x - m)));
}

__device__ __forceinline__ float piece_max(const uint32_t (&v)[16])
{
    float mx[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) mx[j] = fmaxf(__uint_as_float(v[j]), __uint_as_float(v[j + 4]));
#pragma unroll
    for (int j = 0; j < 4; ++j) mx[j] = max3(mx[j], __uint_as_float(v[j + 8]), __uint_as_float(v[j + 12]));
    return fmaxf(max3(mx[0], mx[1], mx[2]), mx[3]);
}
// Pass 1 for a warp some of whose rows left the range: the first `done` pieces of 16 columns have been stored against the reference r;
// everything is brought to the reference that the rest needs.  (reference, sum)
// (The other CTAs of the item wait for this: summed column by column it took twice as long, 256 units x 4096 keys with one far key each 120 us
// against 100.  A second register set would make it shorter still, but the kernel's own values then no longer survive the call in registers, 85 us
// against 79 without any far key.)
__device__ __noinline__ float2 pass1_slow(uint32_t taddr, int done, int nvalid, float c, float r)
{
    const int n = (nvalid + 15) >> 4;
    uint32_t A[16];
    auto keys_only = [&](uint32_t (&v)[16], int i) {
        if (16 * i + 16 <= nvalid) return;
#pragma unroll
        for (int e = 0; e < 16; ++e)
            if (16 * i + e >= nvalid) v[e] = __float_as_uint(-INFINITY);
    };
    float mx = -INFINITY;
    tmem_wait_st();
#pragma unroll 1
    for (int i = done; i < n; ++i) {
        tmem_ld16(taddr + 16 * i, A);
        tmem_wait_ld16(A);
        keys_only(A, i);
        mx = fmaxf(mx, piece_max(A));
    }
    float m = floorf(mx * c);
    if (done) m = fmaxf(m, r);
    if (m == -INFINITY) m = 0.f;   // every logit beyond fp32's range
    const float d = m - r, d1 = fminf(d, 113.f), down1 = ex2(-d1), down2 = ex2(d1 - d);   // (one factor would underflow beside 2^100)
    PieceSum p;
#pragma unroll 1
    for (int i = done; i < n; ++i) {
        tmem_ld16(taddr + 16 * i, A);
        tmem_wait_ld16(A);
        keys_only(A, i);
        piece_exp<0>(A, c, m, p);   // (the FMA pipe has no 0 for a logit beyond fp32's range)
        tmem_st16(taddr + 16 * i, A);
    }
#pragma unroll 1
    for (int i = 0; i < done; ++i) {
        tmem_ld16(taddr + 16 * i, A);
        tmem_wait_ld16(A);
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
            float2 y = __fmul2_rn(make_float2(__uint_as_float(A[e]), __uint_as_float(A[e + 1])), make_float2(down1, down1));
            y = __fmul2_rn(y, make_float2(down2, down2));
            p.s[(e >> 1) & 1] = __fadd2_rn(p.s[(e >> 1) & 1], y);
            A[e] = __float_as_uint(y.x);
            A[e + 1] = __float_as_uint(y.y);
        }
        tmem_st16(taddr + 16 * i, A);
    }
    return make_float2(m, p.total());
}
// Pass 1 for 128 keys: (reference, sum).  kSeek: with references, else against 0; false if that does not do for the first logits.
// Pieces of 16 columns in two register sets.  A piece is looked at and stored behind the exponentials of the next one: with the look straight
// after its own, every piece waited out its own chain of sums.
template <bool kSeek>
__device__ __forceinline__ bool pass1_full(uint32_t tb, float c, float2 &s)
{
    uint32_t A[16], B[16];
    PieceSum pa, pb;
    float r = 0.f;
    auto fits = [&](const PieceSum &p) {   // (false for NaN; what the second set adds need not be large)
        const float t = p.total();
        return __all_sync(0xffffffffu, t <= kTcSumMax && (&p == &pb || t >= kTcSumMin) && fmaf(p.pm, c, -r) <= kTcReach) != 0;
    };
    int done = 0;
    tmem_ld16(tb, A);
    tmem_wait_ld16(A);
    if (kSeek) r = row_reference(piece_max(A), c);
    tmem_ld16(tb + 16, B);
    piece_exp(A, c, r, pa);
#pragma unroll 1
    for (;;) {
        tmem_wait_ld16(B);
        piece_exp(B, c, r, pb);
        if (!fits(pa)) {
            if (!kSeek && !done) return false;
            break;
        }
        tmem_st16(tb + 16 * done, A);
        if (++done < 7) {
            tmem_ld16(tb + 16 * done + 16, A);
            tmem_wait_ld16(A);
            piece_exp(A, c, r, pa);
        }
        if (!fits(pb)) break;
        tmem_st16(tb + 16 * done, B);
        if (++done == 8) break;
        tmem_ld16(tb + 16 * done + 16, B);
    }
    if (done == 8) s = make_float2(r, pa.total() + pb.total());
    else s = pass1_slow(tb, done, kTcHalf, c, r);
    return true;
}
__device__ __noinline__ float2 pass1_seek(uint32_t tb, float c)
{
    float2 s;
    pass1_full<true>(tb, c, s);
    return s;
}
// Pass 1 where only the first nvalid (1 .. 127) of the 128 columns hold keys
__device__ __noinline__ float2 pass1_ragged(uint32_t taddr, int nvalid, float c)
{
    float s = 0.f, r = 0.f;
#pragma unroll 1
    for (int i = 0; 16 * i < nvalid; ++i) {
        uint32_t v[16];
        tmem_ld16(taddr + 16 * i, v);
        tmem_wait_ld16(v);
        if (i == 0) {
            float mx = -INFINITY;
#pragma unroll
            for (int e = 0; e < 16; ++e) mx = fmaxf(mx, e < nvalid ? __uint_as_float(v[e]) : -INFINITY);
            r = row_reference(mx, c);
        }
        float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const float y = 16 * i + e < nvalid ? ex2(fmaf(__uint_as_float(v[e]), c, -r)) : 0.f;
            a[e & 3] += y;
            v[e] = __float_as_uint(y);
        }
        s += (a[0] + a[1]) + (a[2] + a[3]);
        if (!__all_sync(0xffffffffu, s >= kTcSumMin && s <= kTcSumMax)) return pass1_slow(taddr, i, nvalid, c, r);
        tmem_st16(taddr + 16 * i, v);
    }
    return make_float2(r, s);
}
// Sum of n (up to kMost) of a row's entries, re-read until each carries the launch's mark.  Only what is still stale is read again: the polls
// of all CTAs together are a large part of what L2 delivers (all of it again, in 16-byte loads of a transposed array: 109 us against 90).
template <int kMost>
__device__ __forceinline__ float poll_entries(const float *st, int n, float sgn, volatile int *ab, int *status)
{
    float v[kMost];
#pragma unroll
    for (int e = 0; e < kMost; ++e) v[e] = e < n ? 0.f : kTcTiny * sgn;
    for (uint32_t tries = 1;; ++tries) {
        bool fresh = true;
#pragma unroll
        for (int e = 0; e < kMost; ++e)
            if (!(v[e] * sgn > 0.f)) v[e] = ld_gpu_f32(st + (size_t)e * kTcRows);
#pragma unroll
        for (int e = 0; e < kMost; ++e) fresh = fresh && v[e] * sgn > 0.f;
        if (fresh) break;
        if ((tries & 63u) == 0 && (*ab || global_timer_ns() > *reinterpret_cast<volatile unsigned long long *>(ab + 1))) {
            if (!*ab) {
                *ab = 1;
                set_status(status, kStatusTimeout);
            }
            break;
        }
    }
#pragma unroll
    for (int e = 0; e < kMost; ++e) v[e] = fabsf(v[e]);
#pragma unroll
    for (int step = 1; step < kMost; step <<= 1) {
#pragma unroll
        for (int e = 0; e < kMost; e += 2 * step) v[e] += v[e + step];
    }
    return v[0];
}
// A slab's entry of a row whose halves have references, or whose sum is no number.  (This and weight_apart are functions of their own to be out of
// the way: in line they cost a launch of one round 0.3 us, one layer's cycle 29.4 against 29.0.)
__device__ __noinline__ void publish_apart(const TcParams &prm, size_t at, float2 s, float2 o)
{
    float m = fmaxf(s.y == 0.f ? -INFINITY : s.x, o.y == 0.f ? -INFINITY : o.x);
    if (m == -INFINITY) m = 0.f;
    const float sum = (s.y == 0.f ? 0.f : s.y * ex2(s.x - m)) + (o.y == 0.f ? 0.f : o.y * ex2(o.x - m));
    const float plain = m >= kTcRefLow && m <= 118.f ? sum * ex2(m) : INFINITY;
    if (plain <= kTcPlainMax) {   // (a NaN takes the other way, or it would never count as fresh)
        st_gpu_f32(prm.stats + at, plain * prm.sign);
        return;
    }
    float *r = reinterpret_cast<float *>(prm.refs + at);
    st_gpu_f32(r, m);
    st_gpu_f32(r + 1, sum);
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    st_gpu_f32(prm.stats + at, INFINITY * prm.sign);
}
// Sum of n of a row's entries of which some are given as (reference, sum), by the thread that has seen their marks: all loads
// in flight, relative to the largest.  (Every block that has a slab of the item comes here for one far logit in one of them.)
__device__ __noinline__ void fold_entries(const TcParams &prm, int item, int row, int half, float2 *to)
{
    asm volatile("fence.acq_rel.gpu;" ::: "memory");   // what was written before the marks that this thread has read
    const int mid = (prm.slabs + 1) >> 1, n = half ? prm.slabs - mid : mid;
    const size_t first = ((size_t)item * prm.slabs + (half ? mid : 0)) * kTcRows + row;
    const float *st = prm.stats + first;
    const float2 *refs = prm.refs + first;
    float m = -INFINITY, l = 0.f;
#pragma unroll 1
    for (int e0 = 0; e0 < n; e0 += 8) {
        float s[8], x[8], y[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const size_t at = (size_t)(e0 + e < n ? e0 + e : n - 1) * kTcRows;
            s[e] = fabsf(ld_gpu_f32(st + at));
            const float *r = reinterpret_cast<const float *>(refs + at);
            x[e] = ld_gpu_f32(r);
            y[e] = ld_gpu_f32(r + 1);
        }
        float mb = m;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            float2 t = s[e] == INFINITY ? make_float2(x[e], y[e]) : make_float2(0.f, s[e]);
            t = e0 + e >= n || t.y <= kTcTiny ? make_float2(-INFINITY, 0.f) : normalised(t);   // (an empty entry has no reference)
            x[e] = t.x;
            s[e] = t.y;
            mb = fmaxf(mb, t.x);
        }
        if (mb == -INFINITY) continue;
        l *= m == -INFINITY ? 0.f : ex2(m - mb);
#pragma unroll
        for (int e = 0; e < 8; ++e) l = fmaf(s[e], ex2(x[e] - mb), l);
        m = mb;
    }
    *to = m == -INFINITY ? make_float2(0.f, kTcTiny) : make_float2(m, l);
}

// A row's weight where a sum is not plain or the slab has a reference, and whether it is given 2^kTcLift times as large
__device__ __noinline__ float2 weight_apart(float l0, float l1, const float2 *lfar, float2 own, float ref)
{
    float2 t = make_float2(0.f, l0 + l1);
    if (t.y == INFINITY) t = add_sums(l0 == INFINITY ? lfar[0] : make_float2(0.f, l0), l1 == INFINITY ? lfar[kTcRows] : make_float2(0.f, l1));
    if (own.x > -INFINITY) t = add_sums(t, own);
    t = normalised(t);
    const float d = fminf(ref - t.x, 8.f);   // (above 2 only where there is nothing to weigh)
    const bool far = d < -kTcReach;
    float w;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(w) : "f"(t.y));
    return make_float2(w * ex2(far ? d + kTcLift : d), far ? 1.f : 0.f);
}

// Pass 2 for one warp over 32 rows x 32 columns: a[] and b[] are the 16x256b loads of the warp's TMEM lanes
// 0..15 and 16..31, fr2[i] the weight of row lane/4 + 8i duplicated into both halves.  On exit
// x[2j + h] = sum over this thread's four rows of f_r e[r][8j + 2(lane%4) + h].
__device__ __forceinline__ void pass2_rows(const uint32_t (&a)[16], const uint32_t (&b)[16], const float2 (&fr2)[4], float (&x)[8])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float2 s = __ffma2_rn(fr2[0], make_float2(__uint_as_float(a[4 * j]), __uint_as_float(a[4 * j + 1])), make_float2(0.f, 0.f));
        s = __ffma2_rn(fr2[1], make_float2(__uint_as_float(a[4 * j + 2]), __uint_as_float(a[4 * j + 3])), s);
        s = __ffma2_rn(fr2[2], make_float2(__uint_as_float(b[4 * j]), __uint_as_float(b[4 * j + 1])), s);
        s = __ffma2_rn(fr2[3], make_float2(__uint_as_float(b[4 * j + 2]), __uint_as_float(b[4 * j + 3])), s);
        x[2 * j] = s.x;
        x[2 * j + 1] = s.y;
    }
}

// Adds the partial sums of the eight lanes that share lane % 4: on entry lane (g, p) = (lane / 4, lane % 4) holds
// x[2c + h] = its partial of column 8c + 2p + h (c < 4, h < 2); on exit it holds the complete sum of column
// 8 (g / 2) + 2p + (g % 2).  Three exchange steps, each halving the values a lane carries.
__device__ __forceinline__ float pass2_reduce(float (&x)[8], int lane)
{
    const bool up4 = lane & 16, up2 = lane & 8, up1 = lane & 4;
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // g bit 2 picks x[4..7] or x[0..3]
        const float keep = up4 ? x[i + 4] : x[i], give = up4 ? x[i] : x[i + 4];
        x[i] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {  // g bit 1 picks x[2..3] or x[0..1]
        const float keep = up2 ? x[i + 2] : x[i], give = up2 ? x[i] : x[i + 2];
        x[i] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
    }
    const float keep = up1 ? x[1] : x[0], give = up1 ? x[0] : x[1];
    return keep + __shfl_xor_sync(0xffffffffu, give, 4);
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows of 128
// bytes, 8-row groups 1024 bytes apart (the layout TMA writes with SWIZZLE_128B).
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// Instruction descriptor: D = fp32, A = B = bf16, both K-major, M = 128, N = 128 (one column half).
constexpr uint32_t kTcIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

// ------------------------------------------------------------------ the kernel
// kRank: blocks from prm.ctas on rank the streams' novelty.  (Their code costs the others about 5 % through the register
// allocation, so launches of more than a dozen rounds use the variant without it and a ranking kernel on the side.)
// kWide: rows of more than 128 channels.
template <bool kRank, bool kWide>
__global__ void __launch_bounds__(kTcThreads, 1)
cap_score_tc_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                    const __grid_constant__ CUtensorMap mapKnew, const __grid_constant__ TcParams prm)
{
    extern __shared__ __align__(1024) uint8_t tc_smem_raw[];
    const uint32_t base = smem_u32(tc_smem_raw);
    if (base & 1023u) {  // the swizzled tiles need this alignment; nothing has been started yet
        if (threadIdx.x == 0) set_status(prm.status, kStatusBounds);
        return;
    }
    if (kRank && (int)blockIdx.x >= prm.ctas) {
        nuc_rank_extra_block(prm.nuc, prm.N, (int)blockIdx.x - prm.ctas, reinterpret_cast<SelShared *>(tc_smem_raw));
        return;
    }
    uint8_t *gbase = tc_smem_raw;
    uint32_t &tmem_base_slot = *reinterpret_cast<uint32_t *>(gbase + kTcOffTmemSlot);
    int &abort_flag = *reinterpret_cast<int *>(gbase + kTcOffAbort);
    const uint32_t bar0 = base + kTcOffBar;
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (uniform: what follows from it lives in uniform registers)

    if (threadIdx.x == 0) {
        abort_flag = 0;
        *reinterpret_cast<unsigned long long *>(gbase + kTcOffAbort + 4) = global_timer_ns() + prm.wait_ns;
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar(kBarFull + b), 1);
            mbar_init(bar(kBarEmpty + b), 1);
        }
        for (int i = kBarQFull; i < kBarCount; ++i) mbar_init(bar(i), 1);
        for (int g = 0; g < 4; ++g) {
            mbar_init(bar(kBarSFull + g), 1);
            mbar_init(bar(kBarTEmpty + g), 4);
        }
        mbar_init(bar(kBarDrain), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {  // tensor memory: two buffers of 256 columns
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_slot;
    volatile int *ab = &abort_flag;
    const int tasks_per_item = prm.slabs;

    if (warp == 0) {
        // ---------------------------------------------------------------- TMA producer
        if (lane == 0) {
            if (kWide) {
                const uint32_t q_blk = prm.q_blk, q_bytes = prm.q_bytes, k_bytes = prm.k_bytes, q_base = base + kTcOffStage, k_base = q_base + prm.qslots * q_bytes;
                uint32_t qn = 0, kn = 0, qs = 0, qph = 1, ks = 0, kph = 1;   // (slots and phases are counted on: divisions would delay every load)
                bool ok = true;
                for (int task = blockIdx.x; task < prm.tasks && ok; task += prm.ctas) {
                    const int item = task / tasks_per_item, slab = task - item * tasks_per_item;
                    const int unit = item / prm.mtiles, mt = item - unit * prm.mtiles;
                    if (!mbar_wait(bar(kBarQEmpty + qs), qph, ab, prm.status)) break;   // nothing more is put in flight
                    ++qn;
                    mbar_expect_tx(bar(kBarQFull + qs), q_bytes);
                    for (int blk = 0; blk < prm.dhalves; ++blk)
                        tma_load_3d(q_base + qs * q_bytes + blk * q_blk, &mapQ, 64 * blk, mt * kTcRows, unit, bar(kBarQFull + qs));
                    if (++qs == (uint32_t)prm.qslots) {
                        qs = 0;
                        qph ^= 1;
                    }
                    const bool fresh_rows = slab >= prm.new_slab0;
                    const CUtensorMap *mk = fresh_rows ? &mapKnew : &mapK;
                    const int krow = (fresh_rows ? slab - prm.new_slab0 : slab) * kTcSlab;
                    for (int h = 0; h < 2; ++h) {
                        ok = mbar_wait(bar(kBarKEmpty + ks), kph, ab, prm.status);
                        if (!ok) break;
                        ++kn;
                        mbar_expect_tx(bar(kBarKFull + ks), k_bytes);
                        for (int blk = 0; blk < prm.dhalves; ++blk)
                            tma_load_3d(k_base + ks * k_bytes + blk * kTcKBlk, mk, 64 * blk, krow + h * kTcHalf, unit, bar(kBarKFull + ks));
                        if (++ks == (uint32_t)prm.kslots) {
                            ks = 0;
                            kph ^= 1;
                        }
                    }
                }
                // loads that were issued land in this CTA's shared memory: see the last one into every slot complete before
                // the CTA may end (load j went to slot j % slots as its (j / slots)-th fill)
                for (uint32_t j = qn > (uint32_t)prm.qslots ? qn - prm.qslots : 0; j < qn; ++j)
                    mbar_wait(bar(kBarQFull + j % prm.qslots), (j / prm.qslots) & 1, ab, prm.status, false);
                for (uint32_t j = kn > (uint32_t)prm.kslots ? kn - prm.kslots : 0; j < kn; ++j)
                    mbar_wait(bar(kBarKFull + j % prm.kslots), (j / prm.kslots) & 1, ab, prm.status, false);
            } else {
                uint32_t k = 0;
                for (int task = blockIdx.x; task < prm.tasks; task += prm.ctas, ++k) {
                    const int item = task / tasks_per_item, slab = task - item * tasks_per_item;
                    const int unit = item / prm.mtiles, mt = item - unit * prm.mtiles;
                    const uint32_t b = k & 1, ph = (k >> 1) & 1;
                    if (!mbar_wait(bar(kBarEmpty + b), ph ^ 1, ab, prm.status)) break;   // nothing more is put in flight
                    mbar_expect_tx(bar(kBarFull + b), (uint32_t)prm.dhalves * (kTcStageBytes / 2));
                    const uint32_t q = base + kTcOffStage + b * kTcStageBytes, kk = q + kTcQBytes;
                    const bool fresh_rows = slab >= prm.new_slab0;
                    const CUtensorMap *mk = fresh_rows ? &mapKnew : &mapK;
                    const int krow = (fresh_rows ? slab - prm.new_slab0 : slab) * kTcSlab;
                    tma_load_3d(q, &mapQ, 0, mt * kTcRows, unit, bar(kBarFull + b));
                    tma_load_3d(kk, mk, 0, krow, unit, bar(kBarFull + b));
                    if (prm.dhalves == 2) {
                        tma_load_3d(q + kTcQBytes / 2, &mapQ, 64, mt * kTcRows, unit, bar(kBarFull + b));
                        tma_load_3d(kk + kTcKBytes / 2, mk, 64, krow, unit, bar(kBarFull + b));
                    }
                }
                // loads that were issued land in this CTA's shared memory: see the last one of either stage complete before
                // the CTA may end (k loads were issued; load j went to stage j & 1 as its (j >> 1)-th fill)
                for (uint32_t j = (k > 2 ? k - 2 : 0); j < k; ++j)
                    mbar_wait(bar(kBarFull + (j & 1)), (j >> 1) & 1, ab, prm.status, false);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issuer
        // The whole warp walks the schedule and one lane issues: descriptors and counters then live in uniform registers, where the MMA
        // instruction wants them (a lone thread gets eight MMAs of 128 columns accepted in about 900 cycles, an elected lane in 530;
        // alone: 256 units x 4096 keys, M = 128 91.4 -> 90.2 us, 60 x 2999 22.5 -> 21.4, 8 x 4096 9.2 -> 8.6).
        const bool leader = elect_one();
        bool any = false;
        if (kWide) {
            const uint32_t q_blk = prm.q_blk, q_bytes = prm.q_bytes, k_bytes = prm.k_bytes, q_base = base + kTcOffStage;
            const uint64_t q_desc = smem_desc_sw128(q_base), k_desc = smem_desc_sw128(q_base + prm.qslots * q_bytes);
            uint32_t k = 0, qs = 0, qph = 0, ks = 0, kph = 0;
            bool ok = true;
            for (int task = blockIdx.x; task < prm.tasks && ok; task += prm.ctas, ++k) {
                const uint32_t b = k & 1, ph = (k >> 1) & 1;
                ok = __all_sync(0xffffffffu, mbar_wait(bar(kBarQFull + qs), qph, ab, prm.status));
                for (uint32_t h = 0; h < 2 && ok; ++h) {
                    ok = __all_sync(0xffffffffu, mbar_wait(bar(kBarKFull + ks), kph, ab, prm.status) && mbar_wait(bar(kBarTEmpty + 2 * b + h), ph ^ 1, ab, prm.status));
                    if (!ok) break;
                    any = true;
                    tc_fence_after();
                    uint64_t da = q_desc + qs * (q_bytes >> 4), db = k_desc + ks * (k_bytes >> 4);
                    const uint32_t d = tmem + b * kTcSlab + h * kTcHalf;
                    if (leader) {
                        for (int c = 0; c < prm.ksteps; c += 4, da += q_blk >> 4, db += kTcKBlk >> 4) {
                            tc_mma_bf16(d, da, db, kTcIdesc, c ? 1u : 0u);
#pragma unroll
                            for (int i = 1; i < 4; ++i)
                                if (c + i < prm.ksteps) tc_mma_bf16(d, da + 2 * i, db + 2 * i, kTcIdesc, 1u);
                        }
                        tc_commit(bar(kBarSFull + 2 * b + h));   // this half's logits are complete
                        tc_commit(bar(kBarKEmpty + ks));         // the slots may be refilled once the MMAs have read them
                        if (h) tc_commit(bar(kBarQEmpty + qs));
                    }
                    __syncwarp();
                    if (++ks == (uint32_t)prm.kslots) {
                        ks = 0;
                        kph ^= 1;
                    }
                }
                if (++qs == (uint32_t)prm.qslots) {
                    qs = 0;
                    qph ^= 1;
                }
            }
        } else {
            const uint64_t q_desc = smem_desc_sw128(base + kTcOffStage), k_desc = smem_desc_sw128(base + kTcOffStage + kTcQBytes);
            uint32_t k = 0;
            for (int task = blockIdx.x; task < prm.tasks; task += prm.ctas, ++k) {
                const uint32_t b = k & 1, ph = (k >> 1) & 1;
                if (!__all_sync(0xffffffffu, mbar_wait(bar(kBarFull + b), ph, ab, prm.status))) break;
                bool ok = true;
                for (uint32_t h = 0; h < 2; ++h) {
                    ok = __all_sync(0xffffffffu, mbar_wait(bar(kBarTEmpty + 2 * b + h), ph ^ 1, ab, prm.status));
                    if (!ok) break;
                    any = true;
                    tc_fence_after();
                    const uint64_t da = q_desc + b * (kTcStageBytes >> 4), db = k_desc + b * (kTcStageBytes >> 4) + h * (128 * 128 >> 4);
                    const uint32_t d = tmem + b * kTcSlab + h * 128;
                    if (leader) {
#pragma unroll
                        for (uint32_t k4 = 0; k4 < 4; ++k4) tc_mma_bf16(d, da + 2 * k4, db + 2 * k4, kTcIdesc, k4 ? 1u : 0u);
                        if (prm.dhalves == 2) {
#pragma unroll
                            for (uint32_t k4 = 0; k4 < 4; ++k4)
                                tc_mma_bf16(d, da + (kTcQBytes / 2 >> 4) + 2 * k4, db + (kTcKBytes / 2 >> 4) + 2 * k4, kTcIdesc, 1u);
                        }
                        tc_commit(bar(kBarSFull + 2 * b + h));   // this half's logits are complete
                        if (h) tc_commit(bar(kBarEmpty + b));    // the stage may be refilled once the MMAs have read it
                    }
                    __syncwarp();
                }
                if (!ok) break;
            }
        }
        if (any) {  // every MMA has finished (and read its operands) before tensor memory is released
            if (leader) tc_commit(bar(kBarDrain));
            mbar_wait(bar(kBarDrain), 0, ab, prm.status, false);
        }
        __syncwarp();
    } else {
        // ---------------------------------------------------------------- epilogue: groups 0, 1 have the even tasks, 2, 3 the odd ones
        const int q = warp & 3;                 // TMEM lane quarter this warp may touch
        const int g = (warp - 2) >> 2;          // group: buffer g >> 1, columns 128 (g & 1) ... of it
        const int pair = g >> 1, half = g & 1;
        const int row = q * 32 + lane;
        const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + g * kTcHalf;
        float *lpart = reinterpret_cast<float *>(gbase + kTcOffLpart) + pair * (4 * kTcRows);
        float2 *lfar = reinterpret_cast<float2 *>(gbase + kTcOffLfar) + pair * (4 * kTcRows);
        float2 *spart = reinterpret_cast<float2 *>(gbase + kTcOffSpart) + pair * (2 * kTcRows);
        float *colpart = reinterpret_cast<float *>(gbase + kTcOffColpart) + g * (8 * kTcHalf);
        const float c = prm.scale_log2e, sgn = prm.sign;
        const int S = prm.slabs, mid = (S + 1) >> 1;
        // task -> (unit, row block, slab) is counted on from task to task: three divisions at the head of each were 250 ns of a pair's cycle
        const int step = 2 * prm.ctas, dslab = step % tasks_per_item, ditem = step / tasks_per_item, dmt = ditem % prm.mtiles, dunit = ditem / prm.mtiles;
        const int task0 = blockIdx.x + pair * prm.ctas;
        int slab = task0 % tasks_per_item, item = task0 / tasks_per_item, mt = item % prm.mtiles, unit = item / prm.mtiles;
        float *out = nullptr;                   // where this thread's score of the task before goes
        int out_rows = 0;
        auto store = [&](uint32_t par) {        // adds the row quarters
            if (!out) return;
            const float *cp = colpart + par * 4 * kTcHalf + row;
            *out = out_rows > 96 ? (cp[0] + cp[kTcHalf]) + (cp[2 * kTcHalf] + cp[3 * kTcHalf])
                   : out_rows > 64 ? (cp[0] + cp[kTcHalf]) + cp[2 * kTcHalf]
                   : out_rows > 32 ? cp[0] + cp[kTcHalf] : cp[0];
        };
        uint32_t j = 0;                         // tasks of this pair so far
        bool seek = false;                      // this warp's rows have needed references
        for (int task = task0; task < prm.tasks; task += step, ++j) {
            const int rows = min(kTcRows, prm.M - mt * kTcRows), nvalid = min(kTcHalf, prm.N - slab * kTcSlab - half * kTcHalf);
            const bool works = q * 32 < rows && nvalid > 0;   // (uniform over the warp)
            const uint32_t par = j & 1;
            float2 own = make_float2(-INFINITY, 0.f);  // the CaP keys' share of this row's denominator (Appendix B listing)
            auto load_own = [&]() {
                if (prm.cap_stats && row < rows) own = __ldg(&prm.cap_stats[(size_t)unit * prm.M + mt * kTcRows + row]);
            };
            if (!kWide) load_own();
            float2 s = make_float2(0.f, nvalid > 0 ? 1.f : 0.f);
            mbar_wait(bar(kBarSFull + g), par, ab, prm.status);
            if (pair | j) turn_wait(pair, q);
            // ---- pass 1: exponentials against the row's reference, written back over the logits, and their sum
            if (works) {
                tc_fence_after();
                if (nvalid == kTcHalf) {
                    // Rows whose first logits are all below 0 need references: looking for them costs 3 %, and most warps never do.  The first time
                    // a warp does it starts again, from then on it looks first.
                    if (seek || !pass1_full<false>(tb, c, s)) {
                        s = pass1_seek(tb, c);
                        seek = true;
                    }
                } else {
                    s = pass1_ragged(tb, nvalid, c);
                }
            }
            if (task + prm.ctas < prm.tasks) turn_pass(pair, q);
            if (kWide) load_own();   // (two registers that pass 1 of this variant does not have)
            // ---- the pair's two sums together are the slab's entry
            if (half) spart[par * kTcRows + row] = s;
            pair_sync(pair);
            if (!half && (int)blockIdx.x != prm.withhold_cta) {
                const float2 o = spart[par * kTcRows + row];
                const size_t at = ((size_t)item * S + slab) * kTcRows + row;
                if (s.x == 0.f && o.x == 0.f && s.y + o.y <= kTcPlainMax) st_gpu_f32(prm.stats + at, s.y + o.y == 0.f ? kTcTiny * sgn : (s.y + o.y) * sgn);
                else publish_apart(prm, at, s, o);
            }
            // ---- the row's entries of the whole item, each half of the pair one half of them
            float l = 0.f;
            const float *st = prm.stats + (size_t)item * S * kTcRows + row;
            if (row < rows) {
                if (j) __nanosleep(kTcPollDelayNs);
                const int end = half ? S : mid;
                int i = half ? mid : 0;
                for (; i + 8 < end; i += 16) l += poll_entries<16>(st + (size_t)i * kTcRows, end - i, sgn, ab, prm.status);
                if (i < end) l += poll_entries<8>(st + (size_t)i * kTcRows, end - i, sgn, ab, prm.status);
            }
            lpart[(par * 2 + half) * kTcRows + row] = l;
            if (l == INFINITY) fold_entries(prm, item, row, half, lfar + (par * 2 + half) * kTcRows + row);
            if (works) {
                tmem_wait_st();
                tc_fence_before();
            }
            pair_sync(pair);
            // ---- the row's weight
            float weight = 0.f;
            bool far = false;
            if (row < rows) {
                const float l0 = lpart[(par * 2) * kTcRows + row], l1 = lpart[(par * 2 + 1) * kTcRows + row];
                float l = l0 + l1;
                const bool plain_own = own.x > -INFINITY && own.x <= 110.f;
                if (plain_own) l = fmaf(own.y, ex2(own.x), l);
                if (s.x == 0.f && l < INFINITY && (plain_own || own.x == -INFINITY)) {
                    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(weight) : "f"(l));
                } else {
                    const float2 t = weight_apart(l0, l1, lfar + (par * 2) * kTcRows + row, own, s.x);
                    weight = t.x;
                    far = t.y != 0.f;
                }
            }
            const bool lift = __any_sync(0xffffffffu, far);
            if (lift && !far) weight *= kTcLifted;
            // ---- pass 2: weighted column sums
            if (works) {
                tc_fence_after();
                float2 fr2[4];  // the weights of rows lane/4 + 8i, duplicated for the packed FMAs
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float f = __shfl_sync(0xffffffffu, weight, (lane >> 2) + 8 * i);
                    fr2[i] = make_float2(f, f);
                }
                const int at = 8 * (lane >> 3) + 2 * (lane & 3) + ((lane >> 2) & 1);
                float *cp = colpart + (par * 4 + q) * kTcHalf + at;
                uint32_t va[2][16], vb[2][16];
                tmem_ld_16x256b_x4(tb, va[0]);
                tmem_ld_16x256b_x4(tb + (16u << 16), vb[0]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    tmem_wait_ld16(va[i & 1]);
                    tmem_wait_ld16(vb[i & 1]);
                    if (i < 3) {
                        tmem_ld_16x256b_x4(tb + 32 * i + 32, va[(i + 1) & 1]);
                        tmem_ld_16x256b_x4(tb + 32 * i + 32 + (16u << 16), vb[(i + 1) & 1]);
                    } else {   // the buffer half may be overwritten by the next task of this group
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar(kBarTEmpty + g));
                    }
                    float x[8];
                    pass2_rows(va[i & 1], vb[i & 1], fr2, x);
                    cp[32 * i] = pass2_reduce(x, lane) * (lift ? kTcUnlift : 1.f);
                }
            } else if (lane == 0) {
                mbar_arrive(bar(kBarTEmpty + g));
            }
            store(par ^ 1);   // the task before: its column sums have been complete since the barrier
            out = nullptr;
            if (row < nvalid) {   // (here a key)
                out = prm.scores + (size_t)mt * prm.part_stride + (size_t)unit * prm.N + slab * kTcSlab + half * kTcHalf + row;
                out_rows = rows;
            }
            slab += dslab;
            int carry = 0;
            if (slab >= tasks_per_item) {
                slab -= tasks_per_item;
                carry = 1;
            }
            item += ditem + carry;
            mt += dmt + carry;
            unit += dunit;
            if (mt >= prm.mtiles) {
                mt -= prm.mtiles;
                ++unit;
            }
        }
        group_sync(g);
        store((j & 1) ^ 1);
    }

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// ------------------------------------------------------------------ host side
// log2(e) / sqrt(d) for products of the tensor core, which cuts its running sums instead of rounding them: a logit comes out short by about
// 1.2e-8 of itself per 16-channel step, which is made good here.  (Right on average: products that happen to be exact become as much too large.
// Error of the item scorer's scores against 64 bits, 2-norm, without / with: 4096 keys of 256 channels 7.7e-7 / 4.5e-7, 3000 of 192
// 5.5e-7 / 3.1e-7, 8192 of 128 4.2e-7 / 2.5e-7; warp-level tensor cores 6.3e-7, 4.5e-7, 2.9e-7.)
inline float tensor_scale_log2e(int d) { return (float)(1.4426950408889634 / sqrt((double)d) * (1.0 + 1.2e-8 * ((d + 15) / 16))); }

typedef CUresult (*TcEncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                               const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                               CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Device memory of a pot: every buffer is registered first and all of them come out of one allocation (a cudaMalloc
// each cost a pot of 20 buffers several milliseconds).  Those that have to start as zeros lie together at the front.
struct DeviceArena {
    struct Want { void **ptr; size_t bytes; bool zero; };
    static constexpr int kMost = 32;
    Want wants[kMost];
    int n = 0;
    void add(void **ptr, size_t bytes, bool zero = false)
    {
        if (n < kMost) wants[n] = {ptr, (bytes + 255) / 256 * 256 + (bytes ? 0 : 256), zero};
        ++n;
    }
    // false: out of memory.  The zeros are queued on `stream`: kernels rely on their counters from the first launch on, so every stream
    // of the pot waits for them.
    bool allocate(void **base, cudaStream_t stream)
    {
        if (n > kMost) return false;
        size_t total = 0, zeros = 0;
        for (int i = 0; i < n; ++i) {
            total += wants[i].bytes;
            if (wants[i].zero) zeros += wants[i].bytes;
        }
        if (cudaMalloc(base, total) != cudaSuccess) return false;
        if (cudaMemsetAsync(*base, 0, zeros, stream) != cudaSuccess) return false;
        char *at = (char *)*base, *at_zero = at;
        at += zeros;
        for (int i = 0; i < n; ++i) {
            char *&from = wants[i].zero ? at_zero : at;
            *wants[i].ptr = from;
            from += wants[i].bytes;
        }
        return true;
    }
};

// A tensor map and what it was made from.  A pot's buffers and the caller's few query and chunk buffers come back every
// cycle; making a map is about a microsecond of host work, three times a cycle.
struct TcMapSlot {
    CUtensorMap map;
    const void *ptr = nullptr;
    int d = 0, rows = 0, units = 0, box_rows = 0;
    size_t unit_rows = 0;
};
constexpr int kTcMapSlots = 16;

struct TcPlan {
    TcMapSlot maps[kTcMapSlots];
    int next_map = 0;                 // the slot that is overwritten next
    bool usable = false;
    TcEncodeFn encode = nullptr;
    int sm_count = 0;
    int max_items = 0, max_slabs = 0;
    float *stats = nullptr;           // [max_items][max_slabs][128]
    float2 *refs = nullptr;           // the same
    // "fresh" marking of the statistics: every launch writes all entries of its (items x slabs) layout
    // with the sign opposite to the previous launch's; a layout change, or a launch that gave up or failed, clears the array first.
    // A captured launch runs again and again with the one sign it was captured with, between launches that nobody counts: it
    // clears the array itself, and so does every launch after it.
    float sign = 1.f;
    int last_items = 0, last_slabs = 0;
    bool captured = false;
};

inline void tc_plan_init(TcPlan &plan, const ipot_config_t &cfg, int sm_count, DeviceArena &mem)
{
    plan.usable = false;
    plan.sm_count = sm_count;
    if (cfg.dtype != IPOT_BF16) return;
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess || !fn) {
        cudaGetLastError();
        return;
    }
    plan.encode = reinterpret_cast<TcEncodeFn>(fn);   // (the two-sweep scorers need it too)
    // Rows of other sizes than 64 and 128 are AUTO's alone (ipot_api.cu), and a row block fetches its unit's keys anew: beyond four of them
    // such a pot keeps to the item kernel, whose sweeps fetch the keys once for all, and to the scratch that it has always had.
    const int G = cfg.Hq / cfg.Hkv;
    if (cfg.d != 64 && cfg.d != 128 && G * cfg.max_cap_rows > 4 * kTcRows) return;
    int coop = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
        cudaGetLastError();
        return;
    }
    for (auto kern : {cap_score_tc_kernel<false, false>, cap_score_tc_kernel<true, false>, cap_score_tc_kernel<false, true>, cap_score_tc_kernel<true, true>})
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmemBytes) != cudaSuccess) {
            cudaGetLastError();
            return;
        }
    const int units = cfg.layers * cfg.batch * cfg.Hkv;
    plan.max_items = units * ((G * cfg.max_cap_rows + kTcRows - 1) / kTcRows);
    plan.max_slabs = (cfg.pot_size + kTcSlab - 1) / kTcSlab;
    mem.add((void **)&plan.stats, (size_t)plan.max_items * plan.max_slabs * kTcRows * sizeof(float));
    mem.add((void **)&plan.refs, (size_t)plan.max_items * plan.max_slabs * kTcRows * sizeof(float2));
    plan.usable = true;
}

inline bool tc_applicable(TcPlan &plan, const ipot_config_t &cfg, int N, int M)
{
    if (!plan.usable || cfg.dtype != IPOT_BF16 || N < 1 || M < 1) return false;
    const int units = cfg.layers * cfg.batch * cfg.Hkv;
    return units * ((M + kTcRows - 1) / kTcRows) <= plan.max_items && (N + kTcSlab - 1) / kTcSlab <= plan.max_slabs;
}

// [units][unit_rows][d] bf16, of which `rows` per unit are addressable; box = 64 x box_rows x 1, 128-byte swizzle.
inline int tc_encode_rows(TcPlan &plan, CUtensorMap *map, const void *ptr, int d, int rows, int units, size_t unit_rows, int box_rows)
{
    for (const TcMapSlot &s : plan.maps)
        if (s.ptr == ptr && s.d == d && s.rows == rows && s.units == units && s.box_rows == box_rows && s.unit_rows == unit_rows) {
            *map = s.map;
            return IPOT_OK;
        }
    cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)rows, (cuuint64_t)units};
    cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)unit_rows * d * 2};
    cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = plan.encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), dims, strides, box, estr,
                             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return IPOT_E_CUDA;
    TcMapSlot &s = plan.maps[plan.next_map];
    plan.next_map = (plan.next_map + 1) % kTcMapSlots;
    s.map = *map;
    s.ptr = ptr; s.d = d; s.rows = rows; s.units = units; s.box_rows = box_rows; s.unit_rows = unit_rows;
    return IPOT_OK;
}

// scores: partial array p (query rows 128 p ...) is written at scores + p * part_stride, unit stride N.
// Knew (may be NULL): the keys from slot new_first on are not in the pot yet but in this [units][N - new_first][d]
// array (the chunk of a deferred append); new_first must be a multiple of the slab size.
inline int tc_launch(TcPlan &plan, const ipot_config_t &cfg, const void *Q, const void *K, const float2 *cap_stats, float *scores,
                     size_t part_stride, int N, int M, int units, int *status, cudaStream_t stream, int *parts, int *n_launch,
                     const void *Knew = nullptr, int new_first = 0, unsigned long long wait_ns = 200ull * 1000 * 1000,
                     int withhold_cta = -1, int spare_sms = 0, NucJob nuc = NucJob{})
{
    if (!tc_applicable(plan, cfg, N, M)) return IPOT_E_INVALID;
    if (Knew && (new_first % kTcSlab != 0 || new_first >= N)) return IPOT_E_INVALID;
    const int mtiles = (M + kTcRows - 1) / kTcRows;
    const bool wide = cfg.d > kTcD;
    const int qrows = wide && M <= kTcRows / 2 ? kTcRows / 2 : kTcRows, krows = wide ? kTcHalf : kTcSlab;   // of a TMA box
    CUtensorMap mapQ, mapK, mapKnew;
    if (tc_encode_rows(plan, &mapQ, Q, cfg.d, M, units, (size_t)M, qrows) != IPOT_OK) return IPOT_E_CUDA;
    if (Knew && new_first == 0) {  // every key is in the chunk
        if (tc_encode_rows(plan, &mapK, Knew, cfg.d, N, units, (size_t)N, krows) != IPOT_OK) return IPOT_E_CUDA;
        Knew = nullptr;
    } else if (tc_encode_rows(plan, &mapK, K, cfg.d, Knew ? new_first : N, units, (size_t)cfg.pot_size, krows) != IPOT_OK) {
        return IPOT_E_CUDA;
    }
    if (!Knew) mapKnew = mapK;
    else if (tc_encode_rows(plan, &mapKnew, Knew, cfg.d, N - new_first, units, (size_t)(N - new_first), krows) != IPOT_OK) return IPOT_E_CUDA;
    TcParams prm;
    prm.scores = scores; prm.part_stride = part_stride; prm.stats = plan.stats; prm.refs = plan.refs; prm.cap_stats = cap_stats; prm.status = status;
    prm.N = N; prm.M = M; prm.mtiles = mtiles; prm.slabs = (N + kTcSlab - 1) / kTcSlab;
    const int items = units * mtiles;
    prm.tasks = items * prm.slabs;
    prm.dhalves = (cfg.d + 63) / 64;
    prm.ksteps = (cfg.d + 15) / 16;
    prm.q_blk = (uint32_t)qrows * 128u;
    prm.q_bytes = (uint32_t)prm.dhalves * prm.q_blk;
    prm.k_bytes = (uint32_t)prm.dhalves * kTcKBlk;
    prm.qslots = 2 * prm.q_bytes + 2 * prm.k_bytes <= 2 * kTcStageBytes ? 2 : 1;   // 256 channels: 2 + 2 slots up to 64 query rows, else 1 + 2; 192: 2 + 3, 2 + 2
    prm.kslots = std::min<int>(kTcMaxK, (2 * kTcStageBytes - prm.qslots * prm.q_bytes) / prm.k_bytes);
    prm.new_slab0 = Knew ? new_first / kTcSlab : 0x7fffffff;
    prm.scale_log2e = tensor_scale_log2e(cfg.d);
    prm.wait_ns = wait_ns;
    prm.withhold_cta = withhold_cta;
    if (!plan.captured) {
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(stream, &capture) != cudaSuccess) {
            cudaGetLastError();
            return IPOT_E_CUDA;
        }
        plan.captured = capture != cudaStreamCaptureStatusNone;
    }
    if (plan.captured || items != plan.last_items || prm.slabs != plan.last_slabs) {
        if (cudaMemsetAsync(plan.stats, 0, (size_t)items * prm.slabs * kTcRows * sizeof(float), stream) != cudaSuccess) {
            cudaGetLastError();
            return IPOT_E_CUDA;
        }
        plan.last_items = items;
        plan.last_slabs = prm.slabs;
    }
    plan.sign = -plan.sign;
    prm.sign = plan.sign;
    cudaLaunchConfig_t lc = {};
    // spare_sms: SMs left to a small kernel of the same cycle that runs beside this one on another stream, or, with nuc, to
    // the ranking's blocks of this launch (at least; SMs without a task are theirs too)
    const int ctas = plan.sm_count - spare_sms > 0 ? plan.sm_count - spare_sms : 1;
    prm.ctas = prm.tasks < ctas ? prm.tasks : ctas;
    if (nuc.batch > 0) nuc.ctas = nuc.batch < plan.sm_count - prm.ctas ? nuc.batch : plan.sm_count - prm.ctas;
    prm.nuc = nuc;
    lc.gridDim = dim3(prm.ctas + nuc.ctas, 1, 1);
    lc.blockDim = dim3(kTcThreads, 1, 1);
    lc.dynamicSmemBytes = kTcSmemBytes;
    lc.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;  // all CTAs resident: they wait on each other's statistics
    at[0].val.cooperative = 1;
    lc.attrs = at; lc.numAttrs = 1;
    auto kern = wide ? (nuc.ctas > 0 ? cap_score_tc_kernel<true, true> : cap_score_tc_kernel<false, true>)
                     : (nuc.ctas > 0 ? cap_score_tc_kernel<true, false> : cap_score_tc_kernel<false, false>);
    if (cudaLaunchKernelEx(&lc, kern, mapQ, mapK, mapKnew, prm) != cudaSuccess) {
        cudaGetLastError();
        plan.last_items = 0;   // the array still holds what the last launch that ran has left
        return IPOT_E_CUDA;
    }
    *parts = mtiles;
    *n_launch = 1;
    return IPOT_OK;
}

}  // namespace ipotk
