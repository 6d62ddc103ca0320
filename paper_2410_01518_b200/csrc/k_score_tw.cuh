// CaP scoring in two sweeps over the keys with work dealt item by item (Sec. 3.3.1, Eq. 2): bf16, any d up to 256, up to
// 1024 folded query rows per unit.
//
// u_j = sum_i softmax_j(q_i . k_j / sqrt d) needs every row's denominator over ALL keys before rows may be added.
// The unit's keys are cut into jobs of a few 128-key tiles, and every job is visited twice by whichever CTA draws it:
//
//   S1 item  row statistics of the job: S = Q K^T (128 rows x 128 keys per task) on tcgen05 into one of four
//            tensor-memory buffers; an epilogue thread owns one query row and keeps sum_j 2^(x_ij c - ref) in a
//            register against a reference that is 0 unless the sum then leaves the range fp32 holds well, so no maximum is
//            taken.  The job's (ref, sum) pairs go to memory; the CTA that completes a row block of a unit last
//            folds the jobs' pairs into -log2 of the denominators.
//   S2 item  the same tiles with the operands swapped, S^T = K Q^T: a KEY per tensor-memory lane, so that u_j is a sum
//            over the thread's own registers of 2^(x_ij c - L_i) - no exchange between lanes, one coalesced store.
//
// A CTA draws items one by one from two counters: its next S2 item as soon as the unit's denominators are known, else its
// next S1 item, so that it does not wait for another CTA while it has anything else to do, and a job's keys are still in L2
// when they are read again.  It waits only once the S1 items are all drawn; each of them is then with a running CTA that
// waits for nothing before it has done it, so the kernel needs no co-residency and is launched like any other.  The
// CTA that leaves last puts the counters back to zero.
//
// Bound: the exponentials, two per logit (special-function unit 16 a clock and SM, a quarter of them on the FMA pipe).
// Four warps per scheduler work on four different buffers, each at its own place of the load - exponential - sum
// sequence, so that the two pipes stay busy (16 warps that share a buffer idle together at its ends).  A unit's keys
// are fetched once per sweep for all of its row blocks.  Measured alone: 64 units x 4096 keys x 256 channels, M = 64:
// 51 us (warp-level tensor cores: 221); 64 x 16384 x 128, M = 512: 313 us (clusters: 377, one sweep: 541).
//
// Warp roles (640 threads): 0 issues TMA loads, 1 issues MMAs and owns tensor memory, 2 merges and publishes row
// statistics, 3 draws items and fetches the denominators of S2 items, 4-19 epilogue: four groups of four warps (one per
// tensor-memory lane quarter), tasks dealt round robin.  All hand-overs are mbarriers with a time limit; one that runs
// out sets IPOT_E_TIMEOUT and a block-wide flag, every role leaves its loop, loads and MMAs in flight are waited for.
#pragma once
#include "k_score_ts.cuh"

namespace ipotk {

constexpr int kTwGroups = 4;             // epilogue groups of four warps, one per buffer
constexpr int kTwThreads = 128 + 128 * kTwGroups;
constexpr int kTwTile = 128;             // keys per tile = query rows per row block
constexpr int kTwMaxBlocks = 8;          // row blocks per unit
constexpr int kTwPoly = 2;               // eighths of the exponentials on the FMA pipe
constexpr int kTwRing = 8;               // items on their way through the warps of a CTA (the statistics warp is the last to see one)
constexpr int kTwAhead = 2;              // of which the MMA warp has not seen: no more, so that an S1 item is not held back by the CTA that drew it
constexpr uint32_t kTwBlkBytes = kTwTile * 128;   // 64 channels of a tile
constexpr int kTwMaxK = 8;

// barrier slots
enum {
    kTwIFull = 0, kTwIEmpty = kTwIFull + kTwRing, kTwPace = kTwIEmpty + kTwRing, kTwQFull = kTwPace + kTwAhead,
    kTwQEmpty = kTwQFull + 2, kTwKFull = kTwQEmpty + 2, kTwKEmpty = kTwKFull + kTwMaxK, kTwSFull = kTwKEmpty + kTwMaxK,
    kTwTEmpty = kTwSFull + 4, kTwRFull = kTwTEmpty + 4, kTwREmpty = kTwRFull + 2, kTwLFull = kTwREmpty + 2,
    kTwLEmpty = kTwLFull + 2, kTwDrain = kTwLEmpty + 2, kTwBarCount
};

// shared-memory carve-up (bytes); the tiles follow at the next multiple of 1024
constexpr uint32_t kTwOffRow = 0;                                             // [2][groups][128] float2
constexpr uint32_t kTwOffLtab = kTwOffRow + 2 * kTwGroups * 128 * 8;          // [2][kTwMaxBlocks * 128] float
constexpr uint32_t kTwOffBar = kTwOffLtab + 2 * kTwMaxBlocks * 128 * 4;
constexpr uint32_t kTwOffItem = kTwOffBar + 8 * kTwBarCount;
constexpr uint32_t kTwOffSlot = kTwOffItem + 4 * kTwRing;                     // tensor-memory base, abort flag, last-CTA flag
constexpr uint32_t kTwOffTiles = (kTwOffSlot + 16 + 1023) / 1024 * 1024;
constexpr uint32_t kTwSmemMax = 227 * 1024;

struct TwParams {
    float *scores;            // [units][N]
    const float2 *cap_stats;  // NULL, or [units][M] (max, sum) over the CaP's own keys that join every row's denominator
    float *sums, *refs;       // [units][J][mt * 128]: the jobs' (ref, sum) pairs
    float *nl;                // [units][mt * 128]: -log2 of the denominators
    int *sync;                // next S1 job, next S2 job, CTAs that have left, then [units] row blocks whose denominators are known,
                              // [units * mt] jobs that have reported (65536 added for one with a reference other than 0); zero between launches
    int *status;
    int N, M, mt, units, tiles;   // tiles: 128-key tiles of a unit
    int nt, J, jobs;              // tiles per job, jobs per unit, jobs in all
    int ksteps, dblk;             // 16-channel steps and 64-channel blocks of a row
    int qrows;                    // rows of a query tile in shared memory and columns of an S2 product: 64 if M <= 64, else 128
    int qslots, kslots;
    int new_tile0;            // tiles from this one on are read through the second key map; INT_MAX if all keys are in the pot
    float scale_log2e;
    unsigned long long wait_ns;
    int withhold_job;         // -1; test hook: this job's statistics are never published
    int ctas;                 // blocks that score; those behind them rank the streams' novelty
    NucJob nuc;
};

// An item as it is handed out: the job's number, kTwSecond added for its S2 visit; negative: no more.
constexpr int kTwSecond = 1 << 30;
constexpr int kTwSyncHead = 3;
struct TwItem { int sweep, unit, r, t0, n, w; };

__device__ __forceinline__ TwItem tw_item(const TwParams &p, int code)
{
    TwItem it;
    const int job = code & (kTwSecond - 1);
    it.sweep = code >= kTwSecond ? 1 : 0;
    it.unit = job / p.J;
    it.r = job - it.unit * p.J;
    it.t0 = it.r * p.nt;
    it.n = min(p.nt, p.tiles - it.t0);
    // Task i of a CTA uses buffer i % 4 and belongs to group i % 4: every wait on a buffer's barrier then sees each of its
    // phases (a group that skipped tasks could run so far ahead that a phase parity repeats).  With several row blocks the
    // tiles of one key must also meet in one group: a row block then takes four tasks, those beyond the item's tiles
    // being handed over empty.
    it.w = p.mt > 1 ? kTwGroups : it.n;
    return it;
}

constexpr float kTwSumMax = 1.2676506e30f;    // 2^100
constexpr float kTwSumMin = 8.0779357e-28f;   // 2^-90
constexpr float kTwReach = 100.f;             // the polynomial's exponent field is safe up to 2^127: stay well inside

// General path of S1 for the 128 logits of a thread's row: the tile's maximum becomes the reference (first nvalid
// columns only).  Taken when the reference did not fit.
__device__ __noinline__ float2 tw_row_slow(uint32_t taddr, int nvalid, float c, float ref, float l)
{
    float mx = -INFINITY;
#pragma unroll 1
    for (int i = 0; i < 8; ++i) {
        uint32_t v[16];
        tmem_ld16(taddr + 16 * i, v);
        tmem_wait_ld16(v);
#pragma unroll
        for (int e = 0; e < 16; ++e)
            if (16 * i + e < nvalid) mx = fmaxf(mx, __uint_as_float(v[e]));
    }
    if (mx == -INFINITY) return make_float2(ref, l);   // no key, or logits beyond fp32's range: nothing to add
    const float m = mx * c;
    float s = 0.f;
#pragma unroll 1
    for (int i = 0; i < 8; ++i) {
        uint32_t v[16];
        tmem_ld16(taddr + 16 * i, v);
        tmem_wait_ld16(v);
        float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int e = 0; e < 16; ++e)
            if (16 * i + e < nvalid) a[e & 3] += ex2(fmaf(__uint_as_float(v[e]), c, -m));
        s += (a[0] + a[1]) + (a[2] + a[3]);
    }
    const float mn = l > 0.f ? fmaxf(ref, m) : m;
    return make_float2(mn, (l > 0.f ? l * ex2(ref - mn) : 0.f) + s * ex2(m - mn));
}

// A tile of which only the first nvalid columns hold keys: their sum against the reference there is (the caller looks at whether
// it fits; taking the tile's maximum instead would give the job a reference of its own and its unit the general fold).
__device__ __noinline__ float tw_row_ragged(uint32_t taddr, int nvalid, float c, float ref)
{
    float s = 0.f;
#pragma unroll 1
    for (int i = 0; 16 * i < nvalid; ++i) {
        uint32_t v[16];
        tmem_ld16(taddr + 16 * i, v);
        tmem_wait_ld16(v);
        float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int e = 0; e < 16; ++e)
            if (16 * i + e < nvalid) a[e & 3] += ex2(fmaf(__uint_as_float(v[e]), c, -ref));
        s += (a[0] + a[1]) + (a[2] + a[3]);
    }
    return s;
}

// S1, 16 of the row's logits: adds 2^(x c + nm) (nm = minus the row's reference).  All arithmetic is on pairs; pm: the largest
// logit among those that went to the FMA pipe, whose exponent arithmetic wraps around where the special-function unit returns +inf.
template <int kPoly>
__device__ __forceinline__ void tw_sweep1(const uint32_t (&v)[16], float c, float nm, float2 (&sa)[2], float2 (&pa)[2], float (&pm)[2])
{
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float2 x = make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])), t = __ffma2_rn(x, make_float2(c, c), make_float2(nm, nm));
        if (pair_on_fma<kPoly>(i)) {
            pm[i & 1] = max3(pm[i & 1], x.x, x.y);
            pa[i & 1] = __fadd2_rn(pa[i & 1], exp2_fma_pair5(t));
        } else {
            sa[i & 1] = __fadd2_rn(sa[i & 1], make_float2(ex2(t.x), ex2(t.y)));
        }
    }
}
// S2, a key's logits against 16 query rows: adds 2^(x c + nl) (nl: shared memory, the same for every lane).  The rounding of nl, some
// 20 to 40, is 4e-7 of a row's probabilities; kept apart as a whole exponent and a factor it would be gone, but over a unit's
// rows it evens out (error of the scores 5 to 15 % less), and the second table in shared memory costs what the MMAs need of it (64 units
// x 16384 keys, M = 512, whole pass: 411 us against 402).
template <int kPoly>
__device__ __forceinline__ void tw_sweep2(const uint32_t (&v)[16], float c, const float *nl, float2 (&sa)[2], float2 (&pa)[2])
{
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const float4 n4 = *reinterpret_cast<const float4 *>(nl + 4 * g);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = 2 * g + h;
            const float2 x = make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
            const float2 t = __ffma2_rn(x, make_float2(c, c), h ? make_float2(n4.z, n4.w) : make_float2(n4.x, n4.y));
            if (pair_on_fma<kPoly>(i)) pa[i & 1] = fadd2_ftz(pa[i & 1], exp2_fma_pair5(t));
            else sa[i & 1] = fadd2_ftz(sa[i & 1], make_float2(ex2(t.x), ex2(t.y)));
        }
    }
}

// (ref, sum) pairs of disjoint key sets -> one pair; a sum of 0 is an empty set whatever its reference is
__device__ __forceinline__ void tw_merge(float &m, float &l, float m2, float l2)
{
    if (l2 > 0.f) {
        const float mn = l > 0.f ? fmaxf(m, m2) : m2;
        l = (l > 0.f ? l * ex2(m - mn) : 0.f) + l2 * ex2(m2 - mn);
        m = mn;
    }
}
// keeps the sum of a pair near 1 so that later merges cannot underflow (the reference moves by a whole number)
__device__ __forceinline__ void tw_normalise(float &m, float &l)
{
    if (l > 0.f && (l < 8.6736174e-19f || l > 1.1529215e18f)) {   // 2^-60, 2^60
        const int e = (int)((__float_as_uint(l) >> 23) & 255u) - 127;
        l = __uint_as_float((__float_as_uint(l) & 0x7FFFFFu) | 0x3F800000u);
        m += (float)e;
    }
}
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap *map, int c0, int c1, int c2)
{
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ int ld_acquire_gpu(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int atom_add_acq_rel_gpu(int *p, int v)
{
    int old;
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// ------------------------------------------------------------------ the kernel
__global__ void __launch_bounds__(kTwThreads, 1)
cap_score_tw_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                    const __grid_constant__ CUtensorMap mapKnew, const __grid_constant__ TwParams prm)
{
    constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);   // 128 rows, bf16 -> fp32; columns: << 17, in eights
    extern __shared__ __align__(1024) uint8_t tw_smem[];
    const uint32_t base = smem_u32(tw_smem);
    if ((int)blockIdx.x >= prm.ctas) {
        pdl_wait();
        nuc_rank_extra_block(prm.nuc, prm.N, (int)blockIdx.x - prm.ctas, reinterpret_cast<SelShared *>(tw_smem));
        return;
    }
    uint32_t &tmem_slot = *reinterpret_cast<uint32_t *>(tw_smem + kTwOffSlot);
    int &abort_flag = *reinterpret_cast<int *>(tw_smem + kTwOffSlot + 4);
    int &last_cta = *reinterpret_cast<int *>(tw_smem + kTwOffSlot + 8);
    volatile int *items = reinterpret_cast<volatile int *>(tw_smem + kTwOffItem);
    auto bar = [&](int i) { return base + kTwOffBar + 8u * (uint32_t)i; };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mt = prm.mt;
    const bool smem_ok = (base & 1023u) == 0;   // the swizzled tiles need this alignment

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int i = 0; i < kTwRing; ++i) {
            mbar_init(bar(kTwIFull + i), 1);
            mbar_init(bar(kTwIEmpty + i), 3 + 4 * kTwGroups);   // the TMA, MMA and statistics warps and the epilogue warps
        }
        for (int i = 0; i < kTwAhead; ++i) mbar_init(bar(kTwPace + i), 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(kTwQFull + i), 1);
            mbar_init(bar(kTwQEmpty + i), 1);
            mbar_init(bar(kTwRFull + i), 4 * kTwGroups);
            mbar_init(bar(kTwREmpty + i), 1);
            mbar_init(bar(kTwLFull + i), 1);
            mbar_init(bar(kTwLEmpty + i), 4 * kTwGroups);
        }
        for (int i = 0; i < kTwMaxK; ++i) {
            mbar_init(bar(kTwKFull + i), 1);
            mbar_init(bar(kTwKEmpty + i), 1);
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(bar(kTwSFull + i), 1);
            mbar_init(bar(kTwTEmpty + i), 4);
        }
        mbar_init(bar(kTwDrain), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (!smem_ok) set_status(prm.status, kStatusBounds);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_wait();   // the keys and queries are complete; everything above ran beside the kernel that brings them
    pdl_release();
    const TsWait wait{&abort_flag, prm.status, prm.wait_ns, warp == 0 || warp == 3 ? 20u : 0u};
    const uint32_t tile_bytes = (uint32_t)prm.dblk * kTwBlkBytes;
    // M <= 64: an S1 product still has 128 rows, of which the lower half multiplies whatever lies behind the tile and is never read
    const uint32_t q_blk = (uint32_t)prm.qrows * 128u, q_bytes = (uint32_t)prm.dblk * q_blk;
    const uint32_t q_base = base + kTwOffTiles, k_base = q_base + (uint32_t)prm.qslots * q_bytes;

    // the item list as a consumer warp sees it: item n of this CTA, negative at the end
    auto take_item = [&](uint32_t n, bool &ok) {
        ok = wait(bar(kTwIFull + (n & (kTwRing - 1))), (n / kTwRing) & 1);
        return ok ? items[n & (kTwRing - 1)] : -1;
    };
    auto take_item_warp = [&](uint32_t n, bool &ok) {
        int v = take_item(n, ok);
        ok = __all_sync(0xffffffffu, ok);
        if (lane == 0 && ok) mbar_arrive(bar(kTwIEmpty + (n & (kTwRing - 1))));
        return ok ? v : -1;
    };

    if (!smem_ok) {
        // nothing was started
    } else if (warp == 0) {
        // ---------------------------------------------------------------- TMA producer
        if (lane == 0) {
            uint32_t kn = 0, qn = 0;
            bool ok = true;
            for (uint32_t n = 0; ok; ++n) {
                const int pos = take_item(n, ok);
                if (!ok || pos < 0) break;
                mbar_arrive(bar(kTwIEmpty + (n & (kTwRing - 1))));
                const TwItem it = tw_item(prm, pos);
                auto key_map = [&](int t, int &row) {
                    const int tile = it.t0 + t;
                    const bool fresh_rows = tile >= prm.new_tile0;
                    row = (fresh_rows ? tile - prm.new_tile0 : tile) * kTwTile;
                    return fresh_rows ? &mapKnew : &mapK;
                };
                auto load_k = [&](int t) {
                    int row;
                    if (!it.sweep && t >= 2 && t + 1 < it.n) {   // keys seen for the first time: on their way to L2 while the tile before them waits for its slot
                        const CUtensorMap *mk = key_map(t + 1, row);
                        for (int blk = 0; blk < prm.dblk; ++blk) tma_prefetch_3d(mk, 64 * blk, row, it.unit);
                    }
                    const uint32_t s = kn % (uint32_t)prm.kslots, use = kn / (uint32_t)prm.kslots;
                    ok = wait(bar(kTwKEmpty + s), (use & 1) ^ 1);
                    if (!ok) return;
                    ++kn;
                    mbar_expect_tx(bar(kTwKFull + s), tile_bytes);
                    const CUtensorMap *mk = key_map(t, row);
                    for (int blk = 0; blk < prm.dblk; ++blk)
                        tma_load_3d(k_base + s * tile_bytes + blk * kTwBlkBytes, mk, 64 * blk, row, it.unit, bar(kTwKFull + s));
                };
                auto load_q = [&](int b) {
                    const uint32_t s = qn % (uint32_t)prm.qslots, use = qn / (uint32_t)prm.qslots;
                    ok = wait(bar(kTwQEmpty + s), (use & 1) ^ 1);
                    if (!ok) return;
                    ++qn;
                    mbar_expect_tx(bar(kTwQFull + s), q_bytes);
                    for (int blk = 0; blk < prm.dblk; ++blk)
                        tma_load_3d(q_base + s * q_bytes + blk * q_blk, &mapQ, 64 * blk, b * kTwTile, it.unit, bar(kTwQFull + s));
                };
                // with two query slots the query tile first (its slot is free); with one it waits for the previous item's
                // last MMA, and the key slots that are free by then are filled meanwhile
                const int ahead = prm.qslots > 1 ? 0 : min(it.n, prm.kslots);
                for (int t = 0; t < ahead && ok; ++t) load_k(t);
                if (ok) load_q(0);
                for (int t = ahead; t < it.n && ok; ++t) load_k(t);
                for (int b = 1; b < mt && ok; ++b) load_q(b);
            }
            // loads that were issued land in this CTA's shared memory: see the last one into each slot complete
            for (uint32_t j = kn > (uint32_t)prm.kslots ? kn - prm.kslots : 0; j < kn; ++j)
                wait(bar(kTwKFull + j % prm.kslots), (j / prm.kslots) & 1);
            for (uint32_t j = qn > (uint32_t)prm.qslots ? qn - prm.qslots : 0; j < qn; ++j)
                wait(bar(kTwQFull + j % prm.qslots), (j / prm.qslots) & 1);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issuer
        // The whole warp walks the schedule and one lane issues: descriptors and counters then live in uniform registers,
        // where the MMA instruction wants them.  The warp shares its scheduler with four epilogue warps, so slots and
        // phases are counted on, not divided out.
        const bool leader = elect_one();
        uint32_t qs = 0, qph = 0, ks = 0, kph = 0, buf = 0, bph = 1;
        bool ok = true, any = false;
        const uint64_t q_desc = smem_desc_sw128(q_base), k_desc = smem_desc_sw128(k_base);
        const uint32_t tile16 = tile_bytes >> 4, q_tile16 = q_bytes >> 4;
        for (uint32_t n = 0; ok; ++n) {
            int pos = take_item(n, ok);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            pos = __shfl_sync(0xffffffffu, pos, 0);
            if (pos < 0) break;
            if (leader) {
                mbar_arrive(bar(kTwIEmpty + (n & (kTwRing - 1))));
                mbar_arrive(bar(kTwPace + n % kTwAhead));
            }
            const TwItem it = tw_item(prm, pos);
            uint32_t ks1 = ks, kph1 = kph;
            for (int b = 0; b < mt; ++b) {
                wait(bar(kTwQFull + qs), qph);   // (a wait that gives up is seen at the next item: what is issued until then only fills buffers)
                ks1 = ks;
                kph1 = kph;
                for (int t = 0; t < it.w; ++t) {
                    if (b == 0 && t < it.n) wait(bar(kTwKFull + ks1), kph1);
                    wait(bar(kTwTEmpty + buf), bph);
                    if (t >= it.n) {   // an empty task
                        if (leader) mbar_arrive(bar(kTwSFull + buf));
                    } else {
                        tc_fence_after();
                        const uint64_t dq = q_desc + qs * q_tile16, dk = k_desc + ks1 * tile16;
                        uint64_t da = it.sweep ? dk : dq, db = it.sweep ? dq : dk;
                        const uint32_t step_a = it.sweep ? kTwBlkBytes >> 4 : q_blk >> 4, step_b = it.sweep ? q_blk >> 4 : kTwBlkBytes >> 4;
                        const uint32_t idesc = kIdesc | (it.sweep ? (uint32_t)prm.qrows : 128u) >> 3 << 17;
                        const uint32_t d = tmem + buf * 128;
                        if (leader) {
                            for (int k = 0; k < prm.ksteps; k += 4, da += step_a, db += step_b) {
                                tc_mma_bf16(d, da, db, idesc, k ? 1u : 0u);
#pragma unroll
                                for (int i = 1; i < 4; ++i)
                                    if (k + i < prm.ksteps) tc_mma_bf16(d, da + 2 * i, db + 2 * i, idesc, 1u);
                            }
                            tc_commit(bar(kTwSFull + buf));
                            if (b == mt - 1) tc_commit(bar(kTwKEmpty + ks1));   // the slot may be refilled once these MMAs have read it
                        }
                        __syncwarp();
                        if (++ks1 == (uint32_t)prm.kslots) {
                            ks1 = 0;
                            kph1 ^= 1;
                        }
                    }
                    buf = (buf + 1) & 3;
                    if (buf == 0) bph ^= 1;
                }
                if (leader) tc_commit(bar(kTwQEmpty + qs));
                if (++qs == (uint32_t)prm.qslots) {
                    qs = 0;
                    qph ^= 1;
                }
            }
            ks = ks1;
            kph = kph1;
            any = true;
        }
        if (any) {  // every MMA has finished (and read its operands) before tensor memory is released
            if (leader) tc_commit(bar(kTwDrain));
            wait(bar(kTwDrain), 0);
        }
        __syncwarp();
    } else if (warp == 2) {
        // ---------------------------------------------------------------- row statistics of S1 items: merge, publish, fold
        const float2 *rows = reinterpret_cast<const float2 *>(tw_smem + kTwOffRow);
        const int R = mt * kTwTile;
        uint32_t nb = 0;
        bool ok = true;
        for (uint32_t n = 0; ok; ++n) {
            const int pos = take_item_warp(n, ok);
            if (pos < 0) break;
            const TwItem it = tw_item(prm, pos);
            if (it.sweep) continue;
            for (int b = 0; b < mt && ok; ++b, ++nb) {
                const uint32_t par = nb & 1;
                ok = __all_sync(0xffffffffu, wait(bar(kTwRFull + par), (nb >> 1) & 1));
                if (!ok) break;
                // A lane has rows 4 * lane ... + 3.  As long as every reference is 0 the sums add up as they are: this warp gets
                // few issue slots beside the epilogue, and a unit whose denominators are late holds up everybody's S2 items.
                const float4 *in = reinterpret_cast<const float4 *>(rows + par * kTwGroups * kTwTile) + 2 * lane;
                float m[4] = {0.f, 0.f, 0.f, 0.f}, l[4] = {0.f, 0.f, 0.f, 0.f};
                bool plain = true;
#pragma unroll
                for (int g = 0; g < kTwGroups; ++g) {
                    const float4 x = in[g * (kTwTile / 2)], y = in[g * (kTwTile / 2) + 1];
                    plain = plain && x.x == 0.f && x.z == 0.f && y.x == 0.f && y.z == 0.f;
                    l[0] += x.y;
                    l[1] += x.w;
                    l[2] += y.y;
                    l[3] += y.w;
                }
                if (!__all_sync(0xffffffffu, plain)) {
#pragma unroll 1
                    for (int g = 0; g < kTwGroups; ++g) {
                        const float4 x = in[g * (kTwTile / 2)], y = in[g * (kTwTile / 2) + 1];
                        if (g == 0) l[0] = l[1] = l[2] = l[3] = 0.f;
                        tw_merge(m[0], l[0], x.x, x.y);
                        tw_merge(m[1], l[1], x.z, x.w);
                        tw_merge(m[2], l[2], y.x, y.y);
                        tw_merge(m[3], l[3], y.z, y.w);
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) tw_normalise(m[i], l[i]);
                plain = __all_sync(0xffffffffu, m[0] == 0.f && m[1] == 0.f && m[2] == 0.f && m[3] == 0.f);
                if (lane == 0) mbar_arrive(bar(kTwREmpty + par));
                if (it.unit * prm.J + it.r == prm.withhold_job) continue;
                if (prm.J > 1) {
                    const size_t first = (size_t)it.unit * prm.J * R + b * kTwTile + 4 * lane, mine = first + (size_t)it.r * R;
                    __stcg(reinterpret_cast<float4 *>(prm.sums + mine), make_float4(l[0], l[1], l[2], l[3]));
                    __stcg(reinterpret_cast<float4 *>(prm.refs + mine), make_float4(m[0], m[1], m[2], m[3]));
                    __syncwarp();
                    int done = 0;
                    if (lane == 0) done = atom_add_acq_rel_gpu(prm.sync + kTwSyncHead + prm.units + it.unit * mt + b, plain ? 1 : 65537);
                    done = __shfl_sync(0xffffffffu, done, 0);
                    if ((done & 65535) != prm.J - 1) continue;   // another CTA completes the row block
                    __syncwarp();   // what lane 0 has acquired is ordered before the other lanes' reads too (a shuffle alone orders no memory)
                    // in job order, so that the result does not depend on who folds
#pragma unroll
                    for (int i = 0; i < 4; ++i) m[i] = l[i] = 0.f;
                    if (plain && done == prm.J - 1) {
#pragma unroll 1
                        for (int e0 = 0; e0 < prm.J; e0 += 8) {   // eight loads in flight
                            const float *src = prm.sums + first + (size_t)e0 * R;
                            float4 v[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e, src += R) v[e] = e0 + e < prm.J ? __ldcg(reinterpret_cast<const float4 *>(src)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                l[0] += v[e].x;
                                l[1] += v[e].y;
                                l[2] += v[e].z;
                                l[3] += v[e].w;
                            }
                        }
                    } else {
                        // the largest reference, then the sums moved to it (an empty pair's reference does not count)
                        auto pairs = [&](int e0, float4 (&a)[4], float4 (&v)[4]) {
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const size_t at = first + (size_t)min(e0 + e, prm.J - 1) * R;
                                a[e] = __ldcg(reinterpret_cast<const float4 *>(prm.refs + at));
                                v[e] = __ldcg(reinterpret_cast<const float4 *>(prm.sums + at));
                                if (e0 + e >= prm.J) v[e] = make_float4(0.f, 0.f, 0.f, 0.f);
                            }
                        };
                        float4 a[4], v[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) m[i] = -INFINITY;
#pragma unroll 1
                        for (int e0 = 0; e0 < prm.J; e0 += 4) {
                            pairs(e0, a, v);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                m[0] = fmaxf(m[0], v[e].x > 0.f ? a[e].x : -INFINITY);
                                m[1] = fmaxf(m[1], v[e].y > 0.f ? a[e].y : -INFINITY);
                                m[2] = fmaxf(m[2], v[e].z > 0.f ? a[e].z : -INFINITY);
                                m[3] = fmaxf(m[3], v[e].w > 0.f ? a[e].w : -INFINITY);
                            }
                        }
#pragma unroll 1
                        for (int e0 = 0; e0 < prm.J; e0 += 4) {
                            pairs(e0, a, v);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                l[0] += v[e].x > 0.f ? v[e].x * ex2(a[e].x - m[0]) : 0.f;
                                l[1] += v[e].y > 0.f ? v[e].y * ex2(a[e].y - m[1]) : 0.f;
                                l[2] += v[e].z > 0.f ? v[e].z * ex2(a[e].z - m[2]) : 0.f;
                                l[3] += v[e].w > 0.f ? v[e].w * ex2(a[e].w - m[3]) : 0.f;
                            }
                        }
                    }
                }
                float nl[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int row = b * kTwTile + 4 * lane + i;
                    nl[i] = -INFINITY;   // rows beyond M: probability 0
                    if (row < prm.M) {
                        if (prm.cap_stats) {   // the CaP keys' share of this row's denominator (Appendix B listing)
                            const float2 own = __ldg(&prm.cap_stats[(size_t)it.unit * prm.M + row]);
                            tw_merge(m[i], l[i], own.x, own.y);
                        }
                        nl[i] = -(m[i] + log2f(l[i]));
                    }
                }
                __stcg(reinterpret_cast<float4 *>(prm.nl + (size_t)it.unit * R + b * kTwTile + 4 * lane), make_float4(nl[0], nl[1], nl[2], nl[3]));
                __syncwarp();
                if (lane == 0) atom_add_acq_rel_gpu(prm.sync + kTwSyncHead + it.unit, 1);
            }
        }
    } else if (warp == 3) {
        // ---------------------------------------------------------------- draws items, fetches the denominators of S2 items
        // Every look at a counter is a trip to L2, so one S2 job is always held in advance, and whether it is ready is asked while
        // the ring is full.  An S1 job is drawn when it is handed out: one held back behind S2 items (which go first) kept its
        // unit's denominators, and at the end every CTA, waiting.
        if (lane == 0) {
            uint32_t ns = 0;
            bool ok = true;
            int known = -1;   // the last unit found ready
            bool first_left = true;   // S1 jobs may be left
            int s2 = atomicAdd(prm.sync + 1, 1);
            for (uint32_t n = 0; ok; ++n) {
                if (first_left && s2 < prm.jobs && s2 / prm.J != known && ld_acquire_gpu(prm.sync + kTwSyncHead + s2 / prm.J) == mt)
                    known = s2 / prm.J;
                ok = wait(bar(kTwPace + n % kTwAhead), ((n / kTwAhead) & 1) ^ 1) && wait(bar(kTwIEmpty + (n & (kTwRing - 1))), ((n / kTwRing) & 1) ^ 1);
                if (!ok) break;
                int pos = -1;
                if (first_left && !(s2 < prm.jobs && s2 / prm.J == known)) {
                    const int s1 = atomicAdd(prm.sync, 1);
                    first_left = s1 < prm.jobs;
                    if (first_left) pos = s1;
                }
                if (pos < 0 && s2 < prm.jobs) {
                    pos = s2 | kTwSecond;
                    s2 = atomicAdd(prm.sync + 1, 1);
                }
                items[n & (kTwRing - 1)] = pos;
                mbar_arrive(bar(kTwIFull + (n & (kTwRing - 1))));
                if (pos < 0) break;
                if (pos < kTwSecond) continue;
                const int unit = (pos - kTwSecond) / prm.J;
                const uint32_t par = ns & 1;
                ok = wait(bar(kTwLEmpty + par), ((ns >> 1) & 1) ^ 1);
                if (!ok) break;
                if (unit != known) {   // drawn when no S1 item was left: its denominators may still be on their way
                    const unsigned long long t0 = global_timer_ns();
                    while (ld_acquire_gpu(prm.sync + kTwSyncHead + unit) != mt) {
                        if (*(volatile int *)&abort_flag) ok = false;
                        else if (global_timer_ns() - t0 > prm.wait_ns) {
                            abort_flag = 1;
                            set_status(prm.status, kStatusTimeout);
                            ok = false;
                        }
                        if (!ok) break;
                        __nanosleep(100);
                    }
                    if (!ok) break;
                    known = unit;
                }
                // the copy engine reads what other SMs wrote with ordinary stores
                asm volatile("fence.proxy.async;" ::: "memory");
                const uint32_t bytes = (uint32_t)mt * kTwTile * 4;
                mbar_expect_tx(bar(kTwLFull + par), bytes);
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(base + kTwOffLtab + par * kTwMaxBlocks * kTwTile * 4), "l"(prm.nl + (size_t)unit * mt * kTwTile), "r"(bytes),
                               "r"(bar(kTwLFull + par)) : "memory");
                ++ns;
            }
            for (uint32_t j = ns > 2 ? ns - 2 : 0; j < ns; ++j) wait(bar(kTwLFull + (j & 1)), (j >> 1) & 1);   // copies in flight land in this CTA
        }
        __syncwarp();
    } else {
        // ---------------------------------------------------------------- epilogue: task i belongs to group and buffer i % 4
        const int q = warp & 3;                 // TMEM lane quarter this warp may touch
        const uint32_t g = (uint32_t)(warp - 4) >> 2;
        const int row = q * 32 + lane;          // S1: query row of the block; S2: key of the tile
        const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + g * 128;
        float2 *rows = reinterpret_cast<float2 *>(tw_smem + kTwOffRow);
        const float *ltab = reinterpret_cast<const float *>(tw_smem + kTwOffLtab);
        const float c = prm.scale_log2e;
        uint32_t task0 = 0, nb = 0, ns = 0;     // task0: number of the row block's first task
        bool ok = true;
        auto wwait = [&](uint32_t b, uint32_t parity) { return __all_sync(0xffffffffu, wait(b, parity)) != 0; };
        auto release = [&]() {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kTwTEmpty + g));
        };
        for (uint32_t n = 0; ok; ++n) {
            const int pos = take_item_warp(n, ok);
            if (pos < 0) break;
            const TwItem it = tw_item(prm, pos);
            const int first = (int)((g - task0) & 3u);   // this group's tiles of the item: first, first + 4, ... (task0 moves by fours within an item of several row blocks)
            if (it.sweep == 0) {
                for (int b = 0; b < mt && ok; ++b, ++nb, task0 += (uint32_t)it.w) {
                    float ref = 0.f, l = 0.f;
                    for (int t = first; t < it.w; t += kTwGroups) {
                        ok = wwait(bar(kTwSFull + g), ((task0 + (uint32_t)t) >> 2) & 1);
                        if (!ok) break;
                        if (t >= it.n || q * 32 >= prm.qrows) {   // (an empty task; rows that no query has)
                            release();
                            continue;
                        }
                        tc_fence_after();
                        const int nvalid = prm.N - (it.t0 + t) * kTwTile;
                        bool redo = nvalid < kTwTile;
                        if (!redo) {
                            float pm[2] = {-INFINITY, -INFINITY};
                            float2 sa[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, pa[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                            // sum in range and no logit beyond the reach of the polynomial's exponent arithmetic (false for NaN)
                            auto fits = [&](float sum) { return sum <= kTwSumMax && fmaxf(pm[0], pm[1]) * c <= ref + kTwReach; };
                            auto total = [&]() { return ((sa[0].x + sa[0].y) + (sa[1].x + sa[1].y)) + ((pa[0].x + pa[0].y) + (pa[1].x + pa[1].y)); };
                            uint32_t r0[16], r1[16];
                            tmem_ld16(tb, r0);
                            tmem_wait_ld16(r0);
                            // a piece's load flies behind the previous piece's arithmetic; rolled: the warps of a
                            // scheduler are at different places of this code, and it has to stay in the instruction cache
#pragma unroll 1
                            for (int i = 0; i < 6; i += 2) {
                                tmem_ld16(tb + 16 * (i + 1), r1);
                                tw_sweep1<kTwPoly>(r0, c, -ref, sa, pa, pm);
                                tmem_wait_ld16(r1);
                                tmem_ld16(tb + 16 * (i + 2), r0);
                                tw_sweep1<kTwPoly>(r1, c, -ref, sa, pa, pm);
                                tmem_wait_ld16(r0);
                            }
                            tmem_ld16(tb + 112, r1);
                            const float most = l + total();
                            redo = !__all_sync(0xffffffffu, fits(most) && most >= kTwSumMin);
                            tmem_wait_ld16(r1);
                            if (!redo) {
                                // the last quarter is in registers: the buffer goes back, its next product runs behind the rest
                                release();
                                tw_sweep1<kTwPoly>(r0, c, -ref, sa, pa, pm);
                                tw_sweep1<kTwPoly>(r1, c, -ref, sa, pa, pm);
                                const float sum = l + total();
                                if (__all_sync(0xffffffffu, fits(sum))) {
                                    l = sum;
                                } else {
                                    l = most;
                                    sweep1_slow<16>(r0, 0, 16, c, ref, l);
                                    sweep1_slow<16>(r1, 0, 16, c, ref, l);
                                }
                            }
                        }
                        if (nvalid < kTwTile) {
                            const float sum = l + tw_row_ragged(tb, nvalid, c, ref);
                            redo = !__all_sync(0xffffffffu, sum <= kTwSumMax && sum >= kTwSumMin);
                            if (!redo) {
                                l = sum;
                                release();
                            }
                        }
                        if (redo) {
                            const float2 s = tw_row_slow(tb, nvalid, c, ref, l);
                            ref = s.x;
                            l = s.y;
                            release();
                        }
                    }
                    if (!ok) break;
                    const uint32_t par = nb & 1;
                    ok = wwait(bar(kTwREmpty + par), ((nb >> 1) & 1) ^ 1);
                    if (!ok) break;
                    rows[(par * kTwGroups + first) * kTwTile + row] = make_float2(ref, l);   // by place in the item: the merge must not depend on who had it
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kTwRFull + par));
                }
            } else {
                const uint32_t par = ns & 1;
                ok = wwait(bar(kTwLFull + par), (ns >> 1) & 1);
                const int cols = prm.qrows;
                float u = 0.f;   // with several row blocks a group has at most one tile of an item, and u adds over them
                for (int b = 0; b < mt && ok; ++b, task0 += (uint32_t)it.w) {
                    const float *nl = ltab + (par * kTwMaxBlocks + b) * kTwTile;
                    for (int t = first; t < it.w; t += kTwGroups) {
                        ok = wwait(bar(kTwSFull + g), ((task0 + (uint32_t)t) >> 2) & 1);
                        if (!ok) break;
                        if (t >= it.n) {
                            release();
                            continue;
                        }
                        tc_fence_after();
                        float2 sa[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, pa[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                        uint32_t r0[16], r1[16];
                        tmem_ld16(tb, r0);
                        tmem_wait_ld16(r0);
#pragma unroll 1
                        for (int i = 0; i < cols / 16 - 2; i += 2) {
                            tmem_ld16(tb + 16 * (i + 1), r1);
                            tw_sweep2<kTwPoly>(r0, c, nl + 16 * i, sa, pa);
                            tmem_wait_ld16(r1);
                            tmem_ld16(tb + 16 * (i + 2), r0);
                            tw_sweep2<kTwPoly>(r1, c, nl + 16 * i + 16, sa, pa);
                            tmem_wait_ld16(r0);
                        }
                        tmem_ld16(tb + cols - 16, r1);
                        tmem_wait_ld16(r1);
                        release();
                        tw_sweep2<kTwPoly>(r0, c, nl + cols - 32, sa, pa);
                        tw_sweep2<kTwPoly>(r1, c, nl + cols - 16, sa, pa);
                        const float2 s2 = fadd2_ftz(fadd2_ftz(sa[0], sa[1]), fadd2_ftz(pa[0], pa[1]));
                        float sum = s2.x + s2.y;
                        if (mt > 1) sum = u += sum;
                        if (b == mt - 1) {
                            const int key = (it.t0 + t) * kTwTile + row;
                            if (key < prm.N) prm.scores[(size_t)it.unit * prm.N + key] = sum;
                        }
                    }
                }
                __syncwarp();
                if (lane == 0 && ok) mbar_arrive(bar(kTwLEmpty + par));
                ++ns;
            }
        }
    }

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
    if (threadIdx.x == 0) {
        __threadfence();
        last_cta = atomicAdd(prm.sync + 2, 1) == prm.ctas - 1;
    }
    __syncthreads();
    if (last_cta)   // every other CTA has left: the counters are put back for the next launch
        for (int i = threadIdx.x; i < kTwSyncHead + prm.units * (1 + mt); i += kTwThreads) prm.sync[i] = 0;
}

// ------------------------------------------------------------------ host side
constexpr int kTwMaxJobs = 128;   // jobs a unit is cut into at most (the fold reads one pair per job and row)

struct TwPlan {
    bool usable = false;
    int sm_count = 0, max_mt = 0, max_jobs = 0;
    float *part = nullptr;
    float *nl = nullptr;
    int *sync = nullptr;
};

inline void tw_plan_init(TwPlan &plan, const TcPlan &enc, const ipot_config_t &cfg, int sm_count, DeviceArena &mem)
{
    plan.sm_count = sm_count;
    if (cfg.dtype != IPOT_BF16 || !enc.encode) return;
    if (cudaFuncSetAttribute(cap_score_tw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTwSmemMax) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    const int units = cfg.layers * cfg.batch * cfg.Hkv, G = cfg.Hq / cfg.Hkv;
    plan.max_mt = (G * cfg.max_cap_rows + kTwTile - 1) / kTwTile;
    if (plan.max_mt > kTwMaxBlocks) plan.max_mt = kTwMaxBlocks;
    const int tiles = (cfg.pot_size + kTwTile - 1) / kTwTile;
    plan.max_jobs = tiles < kTwMaxJobs ? tiles : kTwMaxJobs;
    const size_t rows = (size_t)units * plan.max_mt * kTwTile, sync_ints = kTwSyncHead + (size_t)units * (1 + plan.max_mt);
    mem.add((void **)&plan.part, 2 * rows * plan.max_jobs * sizeof(float));
    mem.add((void **)&plan.nl, rows * sizeof(float));
    mem.add((void **)&plan.sync, sync_ints * sizeof(int), true);
    plan.usable = true;
}

inline bool tw_applicable(const TwPlan &plan, int N, int M) { return plan.usable && N >= 1 && M >= 1 && (M + kTwTile - 1) / kTwTile <= plan.max_mt; }

// scores [units][N].  Knew (may be NULL): the keys from slot new_first on (a multiple of the tile) are not in the pot yet
// but in this [units][N - new_first][d] array.
inline int tw_launch(TwPlan &plan, TcPlan &enc, const ipot_config_t &cfg, const void *Q, const void *K, const float2 *cap_stats, float *scores,
                     int N, int M, int units, int *status, cudaStream_t stream, unsigned long long wait_ns, int withhold_job,
                     const void *Knew, int new_first, int spare_sms, NucJob nuc = NucJob{})
{
    if (!tw_applicable(plan, N, M) || (Knew && (new_first % kTwTile != 0 || new_first >= N))) return IPOT_E_INVALID;
    CUtensorMap mapQ, mapK, mapKnew;
    const int qrows = M <= kTwTile / 2 ? kTwTile / 2 : kTwTile;
    if (tc_encode_rows(enc, &mapQ, Q, cfg.d, M, units, (size_t)M, qrows) != IPOT_OK) return IPOT_E_CUDA;
    if (Knew && new_first == 0) {  // every key is in the chunk
        if (tc_encode_rows(enc, &mapK, Knew, cfg.d, N, units, (size_t)N, kTwTile) != IPOT_OK) return IPOT_E_CUDA;
        Knew = nullptr;
    } else if (tc_encode_rows(enc, &mapK, K, cfg.d, Knew ? new_first : N, units, (size_t)cfg.pot_size, kTwTile) != IPOT_OK) {
        return IPOT_E_CUDA;
    }
    if (!Knew) mapKnew = mapK;
    else if (tc_encode_rows(enc, &mapKnew, Knew, cfg.d, N - new_first, units, (size_t)(N - new_first), kTwTile) != IPOT_OK) return IPOT_E_CUDA;
    TwParams prm;
    prm.scores = scores; prm.cap_stats = cap_stats; prm.nl = plan.nl; prm.sync = plan.sync; prm.status = status;
    prm.N = N; prm.M = M; prm.mt = (M + kTwTile - 1) / kTwTile; prm.units = units; prm.tiles = (N + kTwTile - 1) / kTwTile;
    prm.dblk = (cfg.d + 63) / 64;
    prm.ksteps = (cfg.d + 15) / 16;
    const uint32_t tile_bytes = (uint32_t)prm.dblk * kTwBlkBytes;
    prm.qrows = qrows;
    const uint32_t q_bytes = tile_bytes * (uint32_t)qrows / kTwTile, room = kTwSmemMax - kTwOffTiles;
    // Up to 64 query rows take half a tile: rows of 256 channels then have room for a second one, so that an item's queries no
    // longer wait for the item before it, and half of the exponentials are not computed (64 units x 4096 keys x 256 channels,
    // M = 64: 55.3 -> 51.4 us; 256 x 2048 x 96, M = 64: 48.3 -> 45.9).
    prm.qslots = (room - 2 * q_bytes) / tile_bytes >= (qrows < kTwTile ? 2 : 3) ? 2 : 1;
    const int slots = (int)((room - (uint32_t)prm.qslots * q_bytes) / tile_bytes);
    prm.kslots = slots < kTwMaxK ? slots : kTwMaxK;
    const int ctas = plan.sm_count - spare_sms > 0 ? plan.sm_count - spare_sms : 1;   // spare_sms: left to the ranking, as in tc_launch
    // Tiles per job: few, so that the items spread evenly over the CTAs, but not so few that the start of an item (query
    // tile, hand-over of the statistics: about half a tile's time) weighs.  With several row blocks a job's key tiles stay
    // in shared memory for all of them and a group keeps one key's running sum, hence at most kslots and kTwGroups.
    const int most = prm.mt > 1 ? (prm.kslots < kTwGroups ? prm.kslots : kTwGroups) : 2 * kTwGroups;
    double best = 1e300;
    prm.nt = 0;
    for (int nt = 1; nt <= most; nt = nt < kTwGroups ? nt + 1 : nt + kTwGroups) {
        const int J = (prm.tiles + nt - 1) / nt;
        if (J > plan.max_jobs) continue;
        const double items = 2.0 * J * units, rounds = items <= ctas ? 1.0 : items / ctas + 0.5;
        // with several row blocks the groups without a tile idle: an item of one tile takes about as long as one of three
        const double cost = rounds * ((prm.mt > 1 && nt < 3 ? 3 : nt) * prm.mt + 0.5);
        if (cost < best) {
            best = cost;
            prm.nt = nt;
        }
    }
    if (!prm.nt) return IPOT_E_INVALID;
    prm.J = (prm.tiles + prm.nt - 1) / prm.nt;
    prm.jobs = prm.J * units;
    prm.sums = plan.part;
    prm.refs = plan.part + (size_t)prm.jobs * prm.mt * kTwTile;
    prm.new_tile0 = Knew ? new_first / kTwTile : 0x7fffffff;
    prm.scale_log2e = tensor_scale_log2e(cfg.d);
    prm.wait_ns = wait_ns;
    prm.withhold_job = withhold_job;
    prm.ctas = 2 * prm.jobs < ctas ? 2 * prm.jobs : ctas;
    if (nuc.batch > 0) nuc.ctas = nuc.batch < plan.sm_count - prm.ctas ? nuc.batch : plan.sm_count - prm.ctas;
    prm.nuc = nuc;
    const size_t smem = kTwOffTiles + (size_t)prm.qslots * q_bytes + (size_t)prm.kslots * tile_bytes;
    return launch_pdl(cap_score_tw_kernel, dim3(prm.ctas + nuc.ctas), dim3(kTwThreads), smem, stream, mapQ, mapK, mapKnew, prm) == cudaSuccess ? IPOT_OK : IPOT_E_CUDA;
}

}  // namespace ipotk
