// Host side of the memory-pot library: pot state, argument checks, launches.
// The C ABI is declared and documented in include/ipot.h.
#include "../../include/ipot.h"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>

#include "common.cuh"
#include "k_cap_self.cuh"
#include "k_decode.cuh"
#include "k_move.cuh"
#include "k_novelty.cuh"
#include "k_rope.cuh"
#include "k_score_mma.cuh"
#include "k_score_simt.cuh"
#include "k_score_tc.cuh"
#include "k_score_f32.cuh"
#include "k_score_ts.cuh"
#include "k_score_tw.cuh"
#include "k_select.cuh"

using namespace ipotk;

struct ipot {
    ipot_config_t cfg;
    int len;
    int device;
    int sm_count;
    int scorer;
    int G, units, elem_bytes, row_bytes;
    cudaStream_t stream;
    // Deferred append (ipot_set_deferred_append): the newest chunk's rows (slots pend_first .. len - 1) still lie in
    // the caller's buffers; the tensor-core scorer reads its keys there and the compaction fetches the survivors
    // from there, so rows that the cycle drops are never copied.  NULL = those rows are in the pot.  In rotary mode
    // pend_K are the unrotated keys; their rotated copy is complete.
    int deferred;
    const void *pend_K, *pend_V;
    int pend_n, pend_first;
    // device memory (library-owned; all but Krot and nov_scratch in one allocation)
    void *arena;
    void *K, *V;
    // CR-RoPE (ipot_enable_rope): K then holds the keys without rotary embedding, Krot the copy rotated at the slot
    // numbers, which is what the scorers read; the tables are the caller's
    void *Krot;
    const void *rope_cos, *rope_sin;
    int rope;            // 0 off, IPOT_ROPE_HALF, IPOT_ROPE_INTERLEAVED
    float *scores;       // [max_parts][units * pot_size]; array q holds [units][N] partial scores of the
                         // q-th block of 128 query rows (the SIMT scorer writes array 0 only)
    float *summed;       // [units][N]: sum of the partial arrays when there are several
    int max_parts;
    float2 *row_stats;   // [units][max M]
    float2 *mma_part;    // [kMmaSplits][units][max M]: partial row statistics of the warp-level tensor-core scorer
    float2 *cap_stats;   // [units][max M]: (max, sum) over the CaP's own keys, CaP-inclusive scoring only
    uint8_t *nuc_mask;   // [batch][mask_stride(N)]
    int32_t *idx;        // [units][keep]
    GatherPlan gather;   // what the selection leaves for the gather
    int withhold_chunk;  // IPOT_TUNE_TEST_WITHHOLD_CHUNK
    int *status;         // sticky device status word
    void *stage_q;       // device staging for the *_host calls
    void *stage_kc;
    float *dec_partial;  // [units][dec_splits][G][d + 2]: ipot_decode_attention's split results
    int *dec_counters;   // [units], zero between calls
    int dec_splits;
    bool dec_ready[2];   // the fp32-FMA and the tensor-core kernel's shared memory limit is set (once per pot)
    char *nov_scratch;   // scratch of ipot_nuc_scores, grown on demand: 65536 row counters (always zero between
                         // calls), then [tokens][segments] float2
    size_t nov_capacity;  // float2 entries behind the counters
    float *stage_aux;
    // results of the last cycle
    int last_len_before;
    const float *last_scores;
    int last_scorer;
    // timing
    int profiling;
    cudaEvent_t (*ev)[5];  // kProfSlots event quintuples, one per recorded cycle
    int ev_used;
    long long launches;
    TcPlan tc;           // tensor-core scorer state
    TwPlan tw;
    F32Plan f32;         // scorer of f32 pots
    TsTuning ts;         // launch parameters of the two-sweep tensor-core scorer
    TsOccupancy ts_occ;
    // the novelty ranking does not depend on the scores: it runs beside the scorer on a stream of its own
    cudaStream_t side;
    cudaEvent_t ev_fork, ev_join;
    cudaEvent_t ev_zero;   // the counters are zero (queued on the side stream by ipot_create)
};

namespace {

constexpr int kProfSlots = 2048;
constexpr int kMmaSplits = 8;
constexpr size_t kNovCounterBytes = (size_t)(kNovMaxRows + 1) * sizeof(int);

#define IPOT_CUDA(call)                                                             \
    do {                                                                            \
        cudaError_t e_ = (call);                                                    \
        if (e_ != cudaSuccess) {                                                    \
            if (getenv("IPOT_DEBUG"))                                               \
                fprintf(stderr, "ipot: %s -> %s\n", #call, cudaGetErrorString(e_)); \
            return IPOT_E_CUDA;                                                     \
        }                                                                           \
    } while (0)

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// the keys the CaP queries attend to
const void *score_keys(const ipot *p) { return p->rope ? p->Krot : p->K; }

int check_config(const ipot_config_t &c)
{
    if (c.pot_size <= 0 || c.pot_size > 32768) return IPOT_E_INVALID;
    if (c.keep <= 0 || c.keep >= c.pot_size) return IPOT_E_INVALID;
    if (c.layers <= 0 || c.batch <= 0 || c.Hq <= 0 || c.Hkv <= 0 || c.Hq % c.Hkv) return IPOT_E_INVALID;
    if (c.d < 32 || c.d > 256 || c.d % 8) return IPOT_E_INVALID;
    if (c.dtype != IPOT_BF16 && c.dtype != IPOT_F32) return IPOT_E_INVALID;
    if (c.nuc_slots < -1 || c.nuc_slots > c.keep) return IPOT_E_INVALID;
    if (c.max_cap_rows <= 0 || c.max_cap_rows > 4096) return IPOT_E_INVALID;
    return IPOT_OK;
}

void free_all(ipot *p)
{
    cudaFree(p->arena); cudaFree(p->Krot); cudaFree(p->nov_scratch);
    if (p->ev_fork) cudaEventDestroy(p->ev_fork);
    if (p->ev_join) cudaEventDestroy(p->ev_join);
    if (p->ev_zero) cudaEventDestroy(p->ev_zero);
    if (p->side) cudaStreamDestroy(p->side);
    if (p->ev) {
        for (int i = 0; i < kProfSlots; ++i)
            for (auto &e : p->ev[i]) if (e) cudaEventDestroy(e);
        delete[] p->ev;
    }
}

// Nothing on stream s runs before the counters are zero.  A stream whose work is being captured cannot wait for what is outside its
// graph; there the host waits.
int wait_for_zeros(ipot *p, cudaStream_t s)
{
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone) {
        IPOT_CUDA(cudaStreamWaitEvent(s, p->ev_zero, 0));
        return IPOT_OK;
    }
    cudaGetLastError();
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    IPOT_CUDA(cudaThreadExchangeStreamCaptureMode(&mode));
    const cudaError_t waited = cudaEventSynchronize(p->ev_zero);
    IPOT_CUDA(cudaThreadExchangeStreamCaptureMode(&mode));
    IPOT_CUDA(waited);
    return IPOT_OK;
}

// Blocks that fit the device at once (the row movers keep eight per SM).
bool one_wave(const ipot *p, dim3 grid) { return (long long)grid.x * grid.y * grid.z <= 8LL * p->sm_count; }

cudaError_t launch_append(ipot *p, dim3 grid, const uint4 *srcK, const uint4 *srcV, uint4 *potK, uint4 *potV, size_t n_vecs, size_t unit_vecs,
                          size_t first_vec)
{
    if (one_wave(p, grid))
        return launch_pdl(append_kernel<true>, grid, dim3(kMoveThreads), 0, p->stream, srcK, srcV, potK, potV, n_vecs, unit_vecs, first_vec);
    append_kernel<false><<<grid, kMoveThreads, 0, p->stream>>>(srcK, srcV, potK, potV, n_vecs, unit_vecs, first_vec);
    return cudaGetLastError();
}

// Copies the rows of a deferred append that are still in the caller's buffers into the pot (keys, values or both).
int materialise(ipot *p, bool keys, bool values)
{
    const void *k = keys ? p->pend_K : nullptr, *v = values ? p->pend_V : nullptr;
    if (!k && !v) return IPOT_OK;
    const size_t row_vecs = p->row_bytes / 16, n_vecs = (size_t)p->pend_n * row_vecs;
    int pieces = (int)((n_vecs + (size_t)kMoveThreads * kMoveVecs - 1) / ((size_t)kMoveThreads * kMoveVecs));
    if (pieces < 1) pieces = 1;
    dim3 grid(pieces, p->units, (k && v) ? 2 : 1);
    if (k && v)
        IPOT_CUDA(launch_append(p, grid, (const uint4 *)k, (const uint4 *)v, (uint4 *)p->K, (uint4 *)p->V, n_vecs,
                                                           (size_t)p->cfg.pot_size * row_vecs, (size_t)p->pend_first * row_vecs));
    else
        IPOT_CUDA(launch_append(p, grid, (const uint4 *)(k ? k : v), nullptr, (uint4 *)(k ? p->K : p->V), nullptr, n_vecs,
                                                           (size_t)p->cfg.pot_size * row_vecs, (size_t)p->pend_first * row_vecs));
    p->launches += 1;
    IPOT_CUDA(cudaGetLastError());
    if (k) p->pend_K = nullptr;
    if (v) p->pend_V = nullptr;
    return IPOT_OK;
}

PendingRows pending_rows(const ipot *p)
{
    PendingRows r;
    r.K = (const uint4 *)p->pend_K;
    r.V = (const uint4 *)p->pend_V;
    r.unit_vecs = (size_t)p->pend_n * (p->row_bytes / 16);
    r.first = p->pend_first;
    return r;
}

// Row statistics over the CaP's own keys (causal): what Appendix B's listing adds to every row's denominator.
int launch_cap_self(ipot *p, const void *Q, const void *Kc, int M, int P)
{
    const int d = p->cfg.d;
    const float scale_log2e = (float)(1.4426950408889634 / std::sqrt((double)d));
    if (p->cfg.dtype == IPOT_BF16 && d % 16 == 0) {
        dim3 g((M + kSelfRows - 1) / kSelfRows, p->units);
        cap_self_stats_bf16<<<g, kSelfWarps * 32, self_smem_bytes(d), p->stream>>>((const __nv_bfloat16 *)Q, (const __nv_bfloat16 *)Kc, p->cap_stats,
                                                                 M, P, d, scale_log2e);
    } else {
        dim3 g((M + kSimtRows - 1) / kSimtRows, p->units);
        if (p->cfg.dtype == IPOT_F32)
            cap_row_stats<float><<<g, kSimtThreads, simt_smem_bytes(d), p->stream>>>(
                (const float *)Q, (const float *)Kc, p->cap_stats, M, P, d, (size_t)P * d, scale_log2e, nullptr, P, 0);
        else
            cap_row_stats<__nv_bfloat16><<<g, kSimtThreads, simt_smem_bytes(d), p->stream>>>(
                (const __nv_bfloat16 *)Q, (const __nv_bfloat16 *)Kc, p->cap_stats, M, P, d, (size_t)P * d, scale_log2e, nullptr, P, 0);
    }
    p->launches += 1;
    IPOT_CUDA(cudaGetLastError());
    return IPOT_OK;
}

template <typename T>
int launch_simt(ipot *p, const void *Q, const float2 *cap_stats, int M, int N)
{
    const int d = p->cfg.d;
    const size_t smem = simt_smem_bytes(d);
    const float scale_log2e = (float)(1.4426950408889634 / std::sqrt((double)d));
    const size_t kstride = (size_t)p->cfg.pot_size * d;
    dim3 g1((M + kSimtRows - 1) / kSimtRows, p->units), g2((N + kSimtKeys - 1) / kSimtKeys, p->units);
    cap_row_stats<T><<<g1, kSimtThreads, smem, p->stream>>>((const T *)Q, (const T *)score_keys(p), p->row_stats, M, N, d, kstride, scale_log2e,
                                                            cap_stats, 0, 1);
    cap_column_sums<T><<<g2, kSimtThreads, smem, p->stream>>>((const T *)Q, (const T *)score_keys(p), p->row_stats, p->scores, M, N, d, kstride, scale_log2e);
    p->launches += 2;
    IPOT_CUDA(cudaGetLastError());
    return IPOT_OK;
}

// f32 pots: every logit computed once, unless one unit's logits exceed the scratch (M * N above 14.9 million: 4.5 bytes each) or it
// did not fit into the device's memory
int launch_f32(ipot *p, const void *Q, const float2 *cap_stats, int M, int N, NucJob nuc)
{
    if (!f32_applicable(p->f32, M, N)) return launch_simt<float>(p, Q, cap_stats, M, N);
    const int d = p->cfg.d;
    int n = 0;
    IPOT_CUDA(f32_launch(p->f32, (const float *)Q, (const float *)score_keys(p), cap_stats, p->row_stats, p->scores, p->units, M, N, d,
                         (size_t)p->cfg.pot_size * d, (float)(1.4426950408889634 / std::sqrt((double)d)), p->sm_count, p->stream, &n, nuc));
    p->launches += n;
    return IPOT_OK;
}

// bf16 pots with d a multiple of 16 that the tcgen05 kernel does not take: the same two launches on warp-level tensor cores
int launch_warp_mma(ipot *p, const void *Q, const float2 *cap_stats, int M, int N)
{
    const int d = p->cfg.d;
    const size_t smem = mma_scorer_smem_bytes(d);
    const float scale_log2e = (float)(1.4426950408889634 / std::sqrt((double)d));
    const size_t kstride = (size_t)p->cfg.pot_size * d;
    const int row_tiles = (M + kMsRows - 1) / kMsRows;
    // the row pass splits the keys so that it launches about four blocks per SM (at most kMmaSplits splits of whole tiles)
    int nsplit = (4 * p->sm_count + row_tiles * p->units - 1) / (row_tiles * p->units);
    const int key_tiles = (N + kMsKeys - 1) / kMsKeys;
    if (nsplit > kMmaSplits) nsplit = kMmaSplits;
    if (nsplit > key_tiles) nsplit = key_tiles;
    if (nsplit < 1) nsplit = 1;
    const int per = ((key_tiles + nsplit - 1) / nsplit) * kMsKeys;
    dim3 g1(row_tiles, p->units, nsplit), g2(key_tiles, p->units);
    const __nv_bfloat16 *Qb = (const __nv_bfloat16 *)Q, *Kb = (const __nv_bfloat16 *)score_keys(p);
    cap_row_stats_mma<<<g1, kMsWarps * 32, smem, p->stream>>>(Qb, Kb, p->mma_part, M, N, d, kstride, scale_log2e, per);
    cap_column_sums_mma<<<g2, kMsWarps * 32, smem, p->stream>>>(Qb, Kb, p->mma_part, cap_stats, nsplit, p->scores, M, N, d, kstride,
                                                               scale_log2e);
    p->launches += 2;
    IPOT_CUDA(cudaGetLastError());
    return IPOT_OK;
}

// The fastest scorer the shape allows.  The one-sweep kernel computes every exponential once; only where an item is spread over most of the
// blocks (beyond 64 slabs of 256 keys) do they wait for each other's statistics long enough for the two-sweep kernel, whose work is dealt item
// by item, to be faster - if there are items enough to deal.  How long they wait depends on the keys: one logit beyond 2^118 takes every block
// of the item through the general fold.  So each line is drawn where neither ordinary nor heavy-tailed keys (Student t, 3 degrees) lose
// much by it.  Rows of 64 channels cost the one-sweep kernel as much as wider ones: there the other is from fewer keys on.  Up to 40 slabs the
// lines are those that the one-sweep kernel had with its former, slower exchange, and test_automatic_choice holds them: between them and 40 slabs
// it would be 8 to 15 % faster on ordinary keys.  A chunk that starts between two slabs is read in place by the item kernel (tiles of 128 keys) and
// copied first for the other: there the lines are the former ones for every length (64 units x 12800, M = 256: 182 us against 228).
// Measured as steps of a stream with deferred appends (us, one sweep / items; ordinary keys, heavy-tailed ones), d = 128:
//   units x keys      M = 64              M = 128             M = 256             M = 512
//   64 x 12288    112/121, 128/126    114/120, 130/129    165/176, 210/205    277/280, 299/306
//   64 x 14336            -                   -           198/204, 240/231            -
//   64 x 15360            -                   -           211/212, 282/242            -
//   64 x 16384    147/150, 157/162    149/151, 168/164    228/227, 298/261    408/371, 450/408
//   32 x 16384     86/94,  108/104     88/95,  114/104    127/138, 154/199    208/193, 258/288
//   64 x 20480    205/200, 253/211    207/206, 268/213    321/294, 437/331    567/461, 778/510
//   32 x 20480    124/126, 159/136    124/126, 156/141    182/174, 242/256    298/245, 392/369
//   24 x 20480    103/107, 126/116    105/107, 131/120    150/154, 195/218    240/211, 286/308
//   16 x 24576     92/94,   98/105     92/97,  108/110    129/142, 155/225    198/237, 255/397
//   16 x 32768    116/119, 159/136    118/121, 172/138    176/179, 243/290    284/254, 432/429
// and d = 64:
//   64 x 12288     91/90,  130/90      92/95,  124/97     145/154, 208/186    250/248, 334/280
//   32 x 16384     73/73,   95/80      74/77,  102/85     115/115, 169/167    193/175, 282/256
//   32 x 12288     59/62,   78/70      59/64,   74/72      87/94,  120/128    141/151, 198/235
//   16 x 16384     51/56,   59/71      51/58,   61/81      72/76,   86/108    111/113, 133/177
// Other head dimensions up to 128 are as 128 beyond 64 slabs (96: 64 x 20480, M = 64 191/175, 237/188; 16 x 32768, M = 128 108/105, 135/122), wider ones
// keep the one-sweep kernel with up to 128 rows (256: 32 x 20480, M = 64 161/195, 183/195; 16 x 32768 149/172, 172/183).  Below 64 slabs it is faster for
// all of them (256: 64 x 4096, M = 64, 256: 58/84, 82/137; 192: 64 x 4096, M = 256 71/104; 96: 64 x 4096, M = 64 41/54; 64 x 8192, M = 256 105/112,
// 123/137; 8 x 2048, M = 64 19/26).  A handful of slabs is left to the item kernel (fewer than 16 have not been measured).
int auto_scorer(int units, int N, int M, int d, bool tile_chunk, bool tc_ok, bool items_ok, bool mma_ok)
{
    const long long keys = (long long)units * N;
    bool many, long_items;
    if (N <= 40 * kTcSlab || (tile_chunk && (d == 64 || d == 128))) {
        many = d == 64 && N >= 6144 && keys >= 64 * 6144;
        long_items = (N > 8192 || (N == 8192 && M > 512)) && keys >= 32 * 8192 && (M > kTcRows || N >= 16384 || keys >= 32 * 10240);
    } else {
        many = d == 64 && keys >= 32 * 16384;
        const bool rows = M > kTcRows || d <= kTcD;
        long_items = keys >= 32 * 8192 && ((N > 96 * kTcSlab && rows) || (N > 64 * kTcSlab && rows && units >= 32) || (M > 2 * kTcRows && N > 48 * kTcSlab) ||
                                           (M > kTcRows && keys >= 60 * 16384));
    }
    if (d != 64 && d != 128) {
        const long long tasks = (long long)units * ((M + kTcRows - 1) / kTcRows) * ((N + kTcSlab - 1) / kTcSlab);
        many = tasks < 16 || tile_chunk;
        long_items = long_items && N > 64 * kTcSlab;
    }
    if (items_ok && (!tc_ok || many || long_items)) return IPOT_SCORER_TENSOR_ITEMS;
    if (tc_ok) return IPOT_SCORER_TENSOR;
    return mma_ok ? IPOT_SCORER_WARP_MMA : IPOT_SCORER_SIMT;
}

// Steps 1-2 (and the timing events around them).  On success *parts tells how many
// partial score arrays the scorer wrote.
int run_scoring(ipot *p, const void *Q, const void *Kc, int cap_rows, const float *aux, int *parts)
{
    const int N = p->len, T = p->cfg.nuc_slots, M = p->G * cap_rows;
    int scorer = p->scorer;
    const bool tc_ok = tc_applicable(p->tc, p->cfg, N, M);
    const bool ts_ok = ts_applicable(p->tc, p->cfg, N, M);
    const bool mma_ok = p->cfg.dtype == IPOT_BF16 && p->cfg.d % 16 == 0;
    // on request only for the row sizes it has always been offered for; AUTO takes it for others too
    if (scorer == IPOT_SCORER_TENSOR && !(tc_ok && (p->cfg.d == 64 || p->cfg.d == 128))) return IPOT_E_INVALID;
    if (scorer == IPOT_SCORER_TENSOR_SWEEPS && !ts_ok) return IPOT_E_INVALID;
    if (scorer == IPOT_SCORER_WARP_MMA && !mma_ok) return IPOT_E_INVALID;
    const bool items_ok = tw_applicable(p->tw, N, M);
    if (scorer == IPOT_SCORER_TENSOR_ITEMS && !items_ok) return IPOT_E_INVALID;
    if (scorer == IPOT_SCORER_AUTO) {
        // a chunk that starts between two slabs is read in place by the item kernel (tiles of 128 keys), copied first for the other
        const bool tile_chunk = p->pend_K && !p->rope && p->pend_first % kTcSlab != 0 && p->pend_first % kTwTile == 0;
        scorer = auto_scorer(p->units, N, M, p->cfg.d, tile_chunk, tc_ok, items_ok, mma_ok);
    }
    // keys of a deferred append: the tensor-core scorers read whole slabs of them where they are, anything else
    // wants them in the pot
    const int slab_keys = scorer == IPOT_SCORER_TENSOR         ? kTcSlab
                          : scorer == IPOT_SCORER_TENSOR_SWEEPS ? kTsSlab
                          : scorer == IPOT_SCORER_TENSOR_ITEMS  ? kTwTile
                                                                : 0;
    const bool keys_in_chunk = p->pend_K && !p->rope && slab_keys && p->pend_first % slab_keys == 0;
    if (p->pend_K && !p->rope && !keys_in_chunk) {
        int mrc = materialise(p, true, false);
        if (mrc != IPOT_OK) return mrc;
    }

    cudaEvent_t *ev = (p->profiling && p->ev_used < kProfSlots) ? p->ev[p->ev_used] : nullptr;
    if (ev) IPOT_CUDA(cudaEventRecord(ev[0], p->stream));
    // Sec. 3.3.3: the T most novel slots per stream.  Independent of the scores, so it is queued on the side stream (after
    // everything the caller has queued so far) and the tensor-core scorers leave it SMs of their own (a scorer block
    // holds an SM's registers); the selection waits for both.  Other scorers' blocks are small and need no such
    // care.  A block ranks several streams, one after the other, when that ends before the scorer does: about 8 us
    // a stream against 3 us per round of (128 rows x 256 keys).
    const long long rounds = ((long long)p->units * ((M + kTcRows - 1) / kTcRows) * ((N + kTcSlab - 1) / kTcSlab) + p->sm_count - 1) / p->sm_count;
    // ... or rides along in the scorer's own launch: the fork and join by events cost a small cycle 5 us
    const bool in_scorer = T > 0 && aux && (p->cfg.dtype == IPOT_F32 ? f32_ranks(p->f32, p->units, M, N, p->sm_count)
                                            : N > kTcSlab && N <= kNucMaxSlots && rounds <= 12 && p->sm_count > 1 && (scorer == IPOT_SCORER_TENSOR || scorer == IPOT_SCORER_TENSOR_ITEMS));
    const bool side_nuc = T > 0 && aux && p->side && !in_scorer;
    const int nuc_blocks = slab_keys ? (int)std::min<long long>(std::min(p->cfg.batch, std::max(1, p->sm_count / 4)), 1 + (8LL * p->cfg.batch - 1) / (3 * rounds)) : p->cfg.batch;
    NucJob nuc{};
    if (in_scorer) nuc = NucJob{aux, p->nuc_mask, T, p->cfg.batch, 0};
    else if (T > 0 && aux) {
        cudaStream_t ns = side_nuc ? p->side : p->stream;
        if (side_nuc) {
            IPOT_CUDA(cudaEventRecord(p->ev_fork, p->stream));
            IPOT_CUDA(cudaStreamWaitEvent(p->side, p->ev_fork, 0));
        }
        launch_nuc_mask(side_nuc ? nuc_blocks : p->cfg.batch, ns, aux, p->nuc_mask, N, T, p->cfg.batch);
        p->launches += 1;
        IPOT_CUDA(cudaGetLastError());
        if (side_nuc) IPOT_CUDA(cudaEventRecord(p->ev_join, p->side));
    }
    if (ev) IPOT_CUDA(cudaEventRecord(ev[1], p->stream));
    *parts = 1;
    int rc;
    if (Kc) {
        rc = launch_cap_self(p, Q, Kc, M, cap_rows);
        if (rc != IPOT_OK) return rc;
    }
    const float2 *cap_stats = Kc ? p->cap_stats : nullptr;
    if (scorer == IPOT_SCORER_TENSOR) {
        int n_launch = 0;
        rc = tc_launch(p->tc, p->cfg, Q, score_keys(p), cap_stats, p->scores, (size_t)p->units * p->cfg.pot_size, N, M, p->units, p->status,
                       p->stream, parts, &n_launch, keys_in_chunk ? p->pend_K : nullptr, keys_in_chunk ? p->pend_first : 0, p->ts.wait_ns,
                       p->ts.withhold_rank, side_nuc || in_scorer ? nuc_blocks : 0, nuc);
        p->launches += n_launch;
    } else if (scorer == IPOT_SCORER_TENSOR_ITEMS) {
        rc = tw_launch(p->tw, p->tc, p->cfg, Q, score_keys(p), cap_stats, p->scores, N, M, p->units, p->status, p->stream, p->ts.wait_ns,
                       p->ts.withhold_rank, keys_in_chunk ? p->pend_K : nullptr, keys_in_chunk ? p->pend_first : 0, side_nuc || in_scorer ? nuc_blocks : 0, nuc);
        p->launches += 1;
    } else if (scorer == IPOT_SCORER_TENSOR_SWEEPS) {
        rc = ts_launch(p->tc, p->ts_occ, p->ts, p->cfg, Q, score_keys(p), cap_stats, p->scores, N, M, p->units, p->status, p->stream,
                       keys_in_chunk ? p->pend_K : nullptr, keys_in_chunk ? p->pend_first : 0, side_nuc ? nuc_blocks : 0);
        p->launches += 1;
    } else if (scorer == IPOT_SCORER_WARP_MMA) {
        rc = launch_warp_mma(p, Q, cap_stats, M, N);
    } else {
        rc = p->cfg.dtype == IPOT_F32 ? launch_f32(p, Q, cap_stats, M, N, nuc) : launch_simt<__nv_bfloat16>(p, Q, cap_stats, M, N);
    }
    if (ev && rc == IPOT_OK) IPOT_CUDA(cudaEventRecord(ev[2], p->stream));   // the scorer's end, before the join below
    if (side_nuc) IPOT_CUDA(cudaStreamWaitEvent(p->stream, p->ev_join, 0));   // (also when the scorer refused: nothing is left behind on the side stream)
    if (rc != IPOT_OK) return rc;
    p->last_scorer = scorer;
    p->last_len_before = N;
    p->last_scores = (*parts > 1) ? p->summed : p->scores;
    return IPOT_OK;
}

int check_cycle_args(ipot *p, const void *Q, int cap_rows, const float *aux, bool compress)
{
    if (!p || !Q) return IPOT_E_INVALID;
    if (cap_rows < 1 || cap_rows > p->cfg.max_cap_rows) return IPOT_E_INVALID;
    if (compress && p->cfg.nuc_slots > 0 && !aux) return IPOT_E_INVALID;
    if (compress ? (p->len <= p->cfg.keep) : (p->len < 1)) return IPOT_E_STATE;
    return IPOT_OK;
}

// The gather of the survivors (and, in rotary mode, the rotated copy of the keys).
template <typename Kernel, typename... Rot>
cudaError_t launch_gather(ipot *p, Kernel kern, const GatherParams &g, const Rot &...rot)
{
    return launch_pdl(kern, dim3(p->gather.chunks * 2 * g.group, (g.units + g.group - 1) / g.group), dim3(kGatherThreads), 0, p->stream, g, rot...);
}

template <typename T>
cudaError_t launch_gather_rope(ipot *p, const GatherParams &g)
{
    if (p->rope == IPOT_ROPE_INTERLEAVED)
        return launch_gather(p, compact_rope_kernel<T, true>, g,
                             GatherRotate<T, true>{(uint4 *)p->Krot, (const T *)p->rope_cos, (const T *)p->rope_sin, g.unit_vecs});
    return launch_gather(p, compact_rope_kernel<T, false>, g,
                         GatherRotate<T, false>{(uint4 *)p->Krot, (const T *)p->rope_cos, (const T *)p->rope_sin, g.unit_vecs});
}

// New key rows (src, unit stride src_unit_vecs) -> pot rows [len, len + n) rotated and, with keys_too, unrotated; if srcV
// is not NULL the same launch copies the value rows ([units][n rows]) into the pot.
template <typename T>
cudaError_t launch_append_rope_t(ipot *p, const void *src, size_t src_unit_vecs, const void *srcV, int n, bool keys_too)
{
    const int row_vecs = p->row_bytes / 16;
    const size_t items = (size_t)n * (row_vecs / 2), unit_vecs = (size_t)p->cfg.pot_size * row_vecs;
    int pieces = (int)((items + (size_t)kMoveThreads * 4 - 1) / ((size_t)kMoveThreads * 4));
    if (pieces < 1) pieces = 1;
    dim3 grid(pieces, p->units, srcV ? 2 : 1);
    auto kern = p->rope == IPOT_ROPE_INTERLEAVED ? append_rope_kernel<T, true> : append_rope_kernel<T, false>;
    kern<<<grid, kMoveThreads, 0, p->stream>>>((const uint4 *)src, src_unit_vecs, (uint4 *)(keys_too ? p->K : nullptr), (uint4 *)p->Krot, (const T *)p->rope_cos,
                                               (const T *)p->rope_sin, n, row_vecs, unit_vecs, p->len, (const uint4 *)srcV, (uint4 *)p->V);
    return cudaGetLastError();
}

cudaError_t launch_append_rope(ipot *p, const void *src, size_t src_unit_vecs, const void *srcV, int n, bool keys_too = true)
{
    if (p->cfg.dtype == IPOT_F32) return launch_append_rope_t<float>(p, src, src_unit_vecs, srcV, n, keys_too);
    return launch_append_rope_t<__nv_bfloat16>(p, src, src_unit_vecs, srcV, n, keys_too);
}

int run_cycle(ipot *p, const void *Q, const void *Kc, int cap_rows, const float *aux)
{
    const int N = p->len, keep = p->cfg.keep, T = p->cfg.nuc_slots, row_vecs = p->row_bytes / 16;
    int parts = 1;
    cudaEvent_t *ev = (p->profiling && p->ev_used < kProfSlots) ? p->ev[p->ev_used] : nullptr;
    int rc = run_scoring(p, Q, Kc, cap_rows, aux, &parts);
    if (rc != IPOT_OK) return rc;
    const size_t part_stride = (size_t)p->units * p->cfg.pot_size;
    IPOT_CUDA(launch_select(p->units, p->stream, p->scores, parts, part_stride, T > 0 ? p->nuc_mask : nullptr, p->idx,
                  parts > 1 ? p->summed : nullptr, N, keep, p->cfg.Hkv, p->cfg.batch, p->status, p->gather, p->sm_count));
    p->launches += 1;
    IPOT_CUDA(cudaGetLastError());
    if (ev) IPOT_CUDA(cudaEventRecord(ev[3], p->stream));

    // Where nothing is read from the pot no block waits for another, and unit after unit finds the last units' keys still in
    // L2 from the scorer (256 units, 4096 -> 2048 rows: cycle 186 us, chunk after chunk over all units 188).  Otherwise
    // chunk after chunk: the chunks a block waits for have then been read long ago (all rows in the pot: 92 us instead of
    // 104; groups of 64 units 94, of 16 units 100).
    const PendingRows pend = pending_rows(p);
    const bool outside = pend.K && pend.V && pend.first == 0;
    const int group = outside ? 1 : (int)std::min<long long>(p->units, (1LL << 30) / p->gather.chunks);
    const GatherParams g{(uint4 *)p->K, (uint4 *)p->V, p->idx, p->gather, p->status, keep, N, row_vecs, p->units, group,
                         (size_t)p->cfg.pot_size * row_vecs, pend, p->withhold_chunk, one_wave(p, dim3(p->gather.chunks, 2, p->units))};
    if (!p->rope) IPOT_CUDA(launch_gather(p, compact_kernel, g));
    else IPOT_CUDA(p->cfg.dtype == IPOT_F32 ? launch_gather_rope<float>(p, g) : launch_gather_rope<__nv_bfloat16>(p, g));
    p->launches += 1;
    p->pend_K = p->pend_V = nullptr;  // the survivors are in the pot, the rest of the chunk is dropped
    if (ev) {
        IPOT_CUDA(cudaEventRecord(ev[4], p->stream));
        p->ev_used += 1;
    }
    p->len = keep;
    return IPOT_OK;
}

}  // namespace

namespace {
template <typename T>
int launch_novelty(ipot *p, const void *logits, size_t row_stride, const int32_t *labels, int n_tokens, int vocab,
                   float *out, size_t out_stride, int slot0)
{
    const size_t rows = (size_t)p->cfg.batch * n_tokens;
    // whole segments where every row starts on a 16-byte boundary (measured: 128256 words 1 % faster than even ones), even
    // ones otherwise
    const bool aligned = aligned16(logits) && row_stride * sizeof(T) % 16 == 0;
    const int segs = (vocab + kNovSegElems - 1) / kNovSegElems;
    const int seg_elems = aligned ? kNovSegElems : ((vocab + segs - 1) / segs + 63) / 64 * 64;   // at most kNovSegElems, itself a multiple of 64
    int *counters = reinterpret_cast<int *>(p->nov_scratch);
    float2 *partial = reinterpret_cast<float2 *>(p->nov_scratch + kNovCounterBytes);
    dim3 grid(segs, (unsigned)rows);
    IPOT_CUDA(launch_pdl(aligned ? novelty_kernel<T, true> : novelty_kernel<T, false>, grid, dim3(kNovThreads), 0, p->stream, 
        (const T *)logits, row_stride, vocab, segs, seg_elems, partial, counters, labels, n_tokens, out, out_stride, slot0, p->status));
    p->launches += 1;
    IPOT_CUDA(cudaGetLastError());
    return IPOT_OK;
}
}  // namespace

// Blocks of one decode launch are equally long, so they run in waves over the resident slots, and every block
// pays a start-up and a merge.  Measured on 64 to 256 units: the fewest splits per unit whose last wave is at
// least 85 % full win (256 blocks on 296 slots beat 384, 768 or 2048); if no count up to 32 gets there, the fullest.
int decode_splits(int units, int slots)
{
    int best = 1;
    double best_eff = 0.0;
    for (int s = 1; s <= 32; ++s) {
        const double waves = (double)units * s / slots;
        const double eff = waves / std::ceil(waves);
        if (eff >= 0.85) return s;
        if (eff > best_eff + 1e-9) {
            best_eff = eff;
            best = s;
        }
    }
    return best;
}

template <typename T, int G>
int launch_decode_g(ipot *p, const void *q, float *out, float *lse)
{
    const int d = p->cfg.d, N = p->len;
    int splits = p->dec_splits;
    const int tile_keys = kDecStageVecs / (p->row_bytes / 16);
    if (splits > (N + tile_keys - 1) / tile_keys) splits = (N + tile_keys - 1) / tile_keys;  // at least one stage of rows per block
    const size_t smem = decode_smem_bytes(G, d);
    auto kern = decode_attn_kernel<T, G>;
    if (smem > 48 * 1024 && !p->dec_ready[0]) IPOT_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    p->dec_ready[0] = true;
    dim3 grid(splits, p->units);
    IPOT_CUDA(launch_pdl(kern, grid, dim3(kDecThreads), smem, p->stream, (const T *)score_keys(p), (const T *)p->V, (const T *)q, out, lse, p->dec_partial,
                                                 p->dec_counters, N, d, p->row_bytes / 16, (size_t)p->cfg.pot_size * d,
                                                 (float)(1.4426950408889634 / std::sqrt((double)d))));
    p->launches += 1;
    IPOT_CUDA(cudaGetLastError());
    return IPOT_OK;
}

// bf16 rows of 64 or 128 channels: the tensor-core stream
template <int D>
int launch_decode_mma(ipot *p, const void *q, float *out, float *lse)
{
    const int N = p->len;
    int splits = p->dec_splits;
    if (splits > (N + 63) / 64) splits = (N + 63) / 64;  // at least one 16-key tile per warp
    const size_t smem = decode_mma_smem_bytes(p->G, D);
    auto kern = decode_attn_mma_kernel<D>;
    if (!p->dec_ready[1]) IPOT_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    p->dec_ready[1] = true;
    dim3 grid(splits, p->units);
    IPOT_CUDA(launch_pdl(kern, grid, dim3(kMmaWarps * 32), smem, p->stream, (const __nv_bfloat16 *)score_keys(p), (const __nv_bfloat16 *)p->V,
                                                    (const __nv_bfloat16 *)q, out, lse, p->dec_partial, p->dec_counters, N, p->G,
                                                    (size_t)p->cfg.pot_size * D, (float)(1.4426950408889634 / std::sqrt((double)D))));
    p->launches += 1;
    IPOT_CUDA(cudaGetLastError());
    return IPOT_OK;
}

template <typename T>
int launch_decode(ipot *p, const void *q, float *out, float *lse)
{
    switch (p->G) {
    case 1: return launch_decode_g<T, 1>(p, q, out, lse);
    case 2: return launch_decode_g<T, 2>(p, q, out, lse);
    case 4: return launch_decode_g<T, 4>(p, q, out, lse);
    case 8: return launch_decode_g<T, 8>(p, q, out, lse);
    default: return IPOT_E_INVALID;
    }
}

extern "C" {

int ipot_create(int pot_size, int keep, int layers, int Hq, int Hkv, int d, ipot_t **out)
{
    ipot_config_t c;
    memset(&c, 0, sizeof(c));
    c.pot_size = pot_size; c.keep = keep; c.layers = layers; c.Hq = Hq; c.Hkv = Hkv; c.d = d;
    c.batch = 1; c.dtype = IPOT_BF16; c.nuc_slots = -1; c.max_cap_rows = 64; c.stream = nullptr;
    return ipot_create_ex(&c, out);
}

int ipot_create_ex(const ipot_config_t *cfg, ipot_t **out)
{
    if (!cfg || !out) return IPOT_E_INVALID;
    int rc = check_config(*cfg);
    if (rc != IPOT_OK) return rc;
    ipot *p = new (std::nothrow) ipot();
    if (!p) return IPOT_E_NOMEM;
    p->cfg = *cfg;
    if (p->cfg.nuc_slots < 0) p->cfg.nuc_slots = p->cfg.keep / 2;
    p->G = cfg->Hq / cfg->Hkv;
    p->units = cfg->layers * cfg->batch * cfg->Hkv;
    p->elem_bytes = cfg->dtype == IPOT_F32 ? 4 : 2;
    p->row_bytes = cfg->d * p->elem_bytes;
    p->stream = (cudaStream_t)cfg->stream;
    p->scorer = IPOT_SCORER_AUTO;
    p->withhold_chunk = -1;
    if (cudaGetDevice(&p->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&p->sm_count, cudaDevAttrMultiProcessorCount, p->device) != cudaSuccess) {
        cudaGetLastError();
        delete p;
        return IPOT_E_CUDA;
    }
    if (cudaStreamCreateWithFlags(&p->side, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&p->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&p->ev_join, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&p->ev_zero, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        free_all(p);
        delete p;
        return IPOT_E_CUDA;
    }
    const size_t pot_bytes = (size_t)p->units * cfg->pot_size * p->row_bytes;
    const int maxM = p->G * cfg->max_cap_rows;
    p->max_parts = (maxM + 127) / 128;
    const size_t score_elems = (size_t)p->units * cfg->pot_size;
    DeviceArena mem;
    auto alloc = [&](void **ptr, size_t bytes, bool zero = false) { mem.add(ptr, bytes, zero); };
    alloc(&p->K, pot_bytes);
    alloc(&p->V, pot_bytes);
    alloc((void **)&p->scores, score_elems * 4 * p->max_parts);
    alloc((void **)&p->summed, score_elems * 4);
    alloc((void **)&p->row_stats, (size_t)p->units * maxM * sizeof(float2));
    alloc((void **)&p->cap_stats, (size_t)p->units * maxM * sizeof(float2));
    alloc((void **)&p->mma_part, (size_t)kMmaSplits * p->units * maxM * sizeof(float2));
    alloc((void **)&p->nuc_mask, (size_t)cfg->batch * mask_stride(cfg->pot_size));
    alloc((void **)&p->idx, (size_t)p->units * cfg->keep * 4);
    p->gather.rows = gather_rows(p->row_bytes / 16);
    p->gather.chunks = gather_chunks(cfg->keep, p->row_bytes / 16);
    alloc((void **)&p->gather.ints, (size_t)p->units * p->gather.per_unit() * 4, true);
    alloc((void **)&p->status, 16, true);
    p->dec_splits = decode_splits(p->units, 2 * p->sm_count);  // both decode kernels keep two blocks per SM
    alloc((void **)&p->dec_partial, (size_t)p->units * p->dec_splits * p->G * (cfg->d + 2) * sizeof(float));
    alloc((void **)&p->dec_counters, (size_t)p->units * sizeof(int), true);
    alloc(&p->stage_q, (size_t)p->units * maxM * p->row_bytes);
    alloc(&p->stage_kc, (size_t)p->units * cfg->max_cap_rows * p->row_bytes);
    alloc((void **)&p->stage_aux, (size_t)cfg->batch * cfg->pot_size * 4);
    // The scratch of the faster scorers comes last: where it does not fit any more a pot does without, the item and f32 scorers'
    // first (6 to 25 % of a bf16 pot of many query rows), then the one-sweep scorer's.
    const int without_tc = mem.n;
    tc_plan_init(p->tc, p->cfg, p->sm_count, mem);
    const int without_tw = mem.n;
    tw_plan_init(p->tw, p->tc, p->cfg, p->sm_count, mem);
    if (cfg->dtype == IPOT_F32) f32_plan_init(p->f32, p->units, maxM, cfg->pot_size, mem);
    bool ok = mem.allocate(&p->arena, p->side);
    if (!ok && !p->arena && mem.n > without_tw) {
        cudaGetLastError();
        mem.n = without_tw;
        p->tw.usable = false;
        p->f32 = F32Plan();
        ok = mem.allocate(&p->arena, p->side);
    }
    if (!ok && !p->arena && mem.n > without_tc) {
        cudaGetLastError();
        mem.n = without_tc;
        p->tc.usable = false;
        ok = mem.allocate(&p->arena, p->side);
    }
    if (!ok) {
        cudaGetLastError();
        free_all(p);
        delete p;
        return IPOT_E_NOMEM;
    }
    // kernels whose dynamic shared memory can exceed the default limit
    ok = cudaFuncSetAttribute(cap_row_stats<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)simt_smem_bytes(256)) == cudaSuccess &&
         cudaFuncSetAttribute(cap_column_sums<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)simt_smem_bytes(256)) == cudaSuccess &&
         cudaFuncSetAttribute(cap_row_stats<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)simt_smem_bytes(256)) == cudaSuccess &&
         cudaFuncSetAttribute(cap_column_sums<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)simt_smem_bytes(256)) == cudaSuccess &&
         cudaFuncSetAttribute(cap_self_stats_bf16, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)self_smem_bytes(256)) == cudaSuccess &&
         cudaFuncSetAttribute(cap_row_stats_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mma_scorer_smem_bytes(256)) == cudaSuccess &&
         cudaFuncSetAttribute(cap_column_sums_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mma_scorer_smem_bytes(256)) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        free_all(p);
        delete p;
        return IPOT_E_CUDA;
    }
    if (cudaEventRecord(p->ev_zero, p->side) != cudaSuccess || wait_for_zeros(p, p->stream) != IPOT_OK) {
        cudaGetLastError();
        free_all(p);
        delete p;
        return IPOT_E_CUDA;
    }
    *out = p;
    return IPOT_OK;
}

int ipot_destroy(ipot_t *p)
{
    if (!p) return IPOT_OK;
    cudaStreamSynchronize(p->stream);
    free_all(p);
    delete p;
    return IPOT_OK;
}

int ipot_set_stream(ipot_t *p, void *s)
{
    if (!p) return IPOT_E_INVALID;
    int rc = materialise(p, true, true);  // queued on the stream that is being left
    if (rc == IPOT_OK) rc = wait_for_zeros(p, (cudaStream_t)s);
    if (rc != IPOT_OK) return rc;
    p->stream = (cudaStream_t)s;
    return IPOT_OK;
}

int ipot_set_nuc_slots(ipot_t *p, int T)
{
    if (!p || T < 0 || T > p->cfg.keep) return IPOT_E_INVALID;
    p->cfg.nuc_slots = T;
    return IPOT_OK;
}

int ipot_set_scorer(ipot_t *p, int scorer)
{
    if (!p || scorer < IPOT_SCORER_AUTO || scorer > IPOT_SCORER_TENSOR_ITEMS) return IPOT_E_INVALID;
    p->scorer = scorer;
    return IPOT_OK;
}

int ipot_set_tuning(ipot_t *p, int what, long long value)
{
    if (!p) return IPOT_E_INVALID;
    switch (what) {
    case IPOT_TUNE_SWEEPS_CLUSTER:
        if (value != 0 && value != 1 && value != 2 && value != 4 && value != 8) return IPOT_E_INVALID;
        p->ts.cluster = (int)value;
        return IPOT_OK;
    case IPOT_TUNE_SWEEPS_FMA_EIGHTHS:
        if (value != -1 && value != 2 && value != 3) return IPOT_E_INVALID;
        p->ts.poly = (int)value;
        return IPOT_OK;
    case IPOT_TUNE_WAIT_LIMIT_NS:
        if (value < 1000) return IPOT_E_INVALID;
        p->ts.wait_ns = (unsigned long long)value;
        return IPOT_OK;
    case IPOT_TUNE_TEST_WITHHOLD_RANK:
        if (value < -1 || value > 7) return IPOT_E_INVALID;
        p->ts.withhold_rank = (int)value;
        return IPOT_OK;
    case IPOT_TUNE_TEST_WITHHOLD_CHUNK:
        if (value < -1 || value > 7) return IPOT_E_INVALID;
        p->withhold_chunk = (int)value;
        return IPOT_OK;
    default:
        return IPOT_E_INVALID;
    }
}

int ipot_set_deferred_append(ipot_t *p, int on)
{
    if (!p) return IPOT_E_INVALID;
    if (!on) {
        int rc = materialise(p, true, true);
        if (rc != IPOT_OK) return rc;
    }
    p->deferred = on ? 1 : 0;
    return IPOT_OK;
}

int ipot_reset(ipot_t *p)
{
    if (!p) return IPOT_E_INVALID;
    p->len = 0;
    p->pend_K = p->pend_V = nullptr;
    return IPOT_OK;
}

int ipot_append_chunk(ipot_t *p, const void *K, const void *V, int n)
{
    if (!p || !K || !V || n <= 0 || !aligned16(K) || !aligned16(V)) return IPOT_E_INVALID;
    if (p->len + n > p->cfg.pot_size) return IPOT_E_STATE;
    const size_t row_vecs = p->row_bytes / 16;
    const size_t n_vecs = (size_t)n * row_vecs;
    int pieces = (int)((n_vecs + (size_t)kMoveThreads * kMoveVecs - 1) / ((size_t)kMoveThreads * kMoveVecs));
    if (pieces < 1) pieces = 1;
    int rc = materialise(p, true, true);  // at most one chunk is kept outside the pot
    if (rc != IPOT_OK) return rc;
    if (p->deferred) {
        p->pend_first = p->len;
        p->pend_n = n;
        p->pend_V = V;
        p->pend_K = K;
        if (p->rope) {  // the rotated copy is what the scorers read: it is made now
            IPOT_CUDA(launch_append_rope(p, K, n_vecs, nullptr, n, false));
            p->launches += 1;
            IPOT_CUDA(cudaGetLastError());
        }
        p->len += n;
        return IPOT_OK;
    }
    if (!p->rope) {
        dim3 grid(pieces, p->units, 2);
        IPOT_CUDA(launch_append(p, grid, (const uint4 *)K, (const uint4 *)V, (uint4 *)p->K, (uint4 *)p->V,
                                                           n_vecs, (size_t)p->cfg.pot_size * row_vecs, (size_t)p->len * row_vecs));
    } else {
        IPOT_CUDA(launch_append_rope(p, K, n_vecs, V, n));
    }
    p->launches += 1;
    IPOT_CUDA(cudaGetLastError());
    p->len += n;
    return IPOT_OK;
}

int ipot_append_chunk_host(ipot_t *p, const void *K, const void *V, int n)
{
    if (!p || !K || !V || n <= 0) return IPOT_E_INVALID;
    if (p->len + n > p->cfg.pot_size) return IPOT_E_STATE;
    int rc = materialise(p, true, true);
    if (rc != IPOT_OK) return rc;
    const size_t width = (size_t)n * p->row_bytes, dpitch = (size_t)p->cfg.pot_size * p->row_bytes;
    char *dK = (char *)p->K + (size_t)p->len * p->row_bytes, *dV = (char *)p->V + (size_t)p->len * p->row_bytes;
    IPOT_CUDA(cudaMemcpy2DAsync(dK, dpitch, K, width, width, p->units, cudaMemcpyHostToDevice, p->stream));
    IPOT_CUDA(cudaMemcpy2DAsync(dV, dpitch, V, width, width, p->units, cudaMemcpyHostToDevice, p->stream));
    if (p->rope) {  // the key rows are in place: rotate them into the copy
        IPOT_CUDA(launch_append_rope(p, dK, (size_t)p->cfg.pot_size * (p->row_bytes / 16), nullptr, n));
        p->launches += 1;
        IPOT_CUDA(cudaGetLastError());
    }
    p->len += n;
    return IPOT_OK;
}

int ipot_score_and_compress(ipot_t *p, const void *Q, int cap_rows, const float *aux)
{
    int rc = check_cycle_args(p, Q, cap_rows, aux, true);
    if (rc != IPOT_OK) return rc;
    if (!aligned16(Q) || (aux && (reinterpret_cast<uintptr_t>(aux) & 3u))) return IPOT_E_INVALID;
    return run_cycle(p, Q, nullptr, cap_rows, aux);
}

int ipot_score_and_compress_host(ipot_t *p, const void *Q, int cap_rows, const float *aux, int32_t *idx_host)
{
    int rc = check_cycle_args(p, Q, cap_rows, aux, true);
    if (rc != IPOT_OK) return rc;
    const size_t qbytes = (size_t)p->units * p->G * cap_rows * p->row_bytes;
    IPOT_CUDA(cudaMemcpyAsync(p->stage_q, Q, qbytes, cudaMemcpyHostToDevice, p->stream));
    if (aux) IPOT_CUDA(cudaMemcpyAsync(p->stage_aux, aux, (size_t)p->cfg.batch * p->len * 4, cudaMemcpyHostToDevice, p->stream));
    rc = run_cycle(p, p->stage_q, nullptr, cap_rows, aux ? p->stage_aux : nullptr);
    if (rc != IPOT_OK) return rc;
    if (idx_host)
        IPOT_CUDA(cudaMemcpyAsync(idx_host, p->idx, (size_t)p->units * p->cfg.keep * 4, cudaMemcpyDeviceToHost, p->stream));
    return IPOT_OK;
}

namespace {
int score_only(ipot *p, const void *Q, const void *Kc, int cap_rows, const float *aux)
{
    int parts = 1;
    int rc = run_scoring(p, Q, Kc, cap_rows, aux, &parts);
    if (rc != IPOT_OK) return rc;
    if (parts > 1) {
        const size_t n = (size_t)p->units * p->len;
        sum_parts_kernel<<<(unsigned)((n + 255) / 256), 256, 0, p->stream>>>(
            p->scores, parts, (size_t)p->units * p->cfg.pot_size, p->summed, n);
        p->launches += 1;
        IPOT_CUDA(cudaGetLastError());
    }
    return IPOT_OK;
}
}  // namespace

int ipot_score_only(ipot_t *p, const void *Q, int cap_rows, const float *aux)
{
    int rc = check_cycle_args(p, Q, cap_rows, aux, false);
    if (rc != IPOT_OK) return rc;
    if (!aligned16(Q)) return IPOT_E_INVALID;
    return score_only(p, Q, nullptr, cap_rows, aux);
}

int ipot_score_and_compress_cap(ipot_t *p, const void *Q, const void *K_cap, int cap_rows, const float *aux)
{
    int rc = check_cycle_args(p, Q, cap_rows, aux, true);
    if (rc != IPOT_OK) return rc;
    if (!K_cap || !aligned16(Q) || !aligned16(K_cap) || (aux && (reinterpret_cast<uintptr_t>(aux) & 3u))) return IPOT_E_INVALID;
    return run_cycle(p, Q, K_cap, cap_rows, aux);
}

int ipot_score_and_compress_cap_host(ipot_t *p, const void *Q, const void *K_cap, int cap_rows, const float *aux, int32_t *idx_host)
{
    int rc = check_cycle_args(p, Q, cap_rows, aux, true);
    if (rc != IPOT_OK) return rc;
    if (!K_cap) return IPOT_E_INVALID;
    const size_t qbytes = (size_t)p->units * p->G * cap_rows * p->row_bytes, kcbytes = (size_t)p->units * cap_rows * p->row_bytes;
    IPOT_CUDA(cudaMemcpyAsync(p->stage_q, Q, qbytes, cudaMemcpyHostToDevice, p->stream));
    IPOT_CUDA(cudaMemcpyAsync(p->stage_kc, K_cap, kcbytes, cudaMemcpyHostToDevice, p->stream));
    if (aux) IPOT_CUDA(cudaMemcpyAsync(p->stage_aux, aux, (size_t)p->cfg.batch * p->len * 4, cudaMemcpyHostToDevice, p->stream));
    rc = run_cycle(p, p->stage_q, p->stage_kc, cap_rows, aux ? p->stage_aux : nullptr);
    if (rc != IPOT_OK) return rc;
    if (idx_host)
        IPOT_CUDA(cudaMemcpyAsync(idx_host, p->idx, (size_t)p->units * p->cfg.keep * 4, cudaMemcpyDeviceToHost, p->stream));
    return IPOT_OK;
}

int ipot_score_only_cap(ipot_t *p, const void *Q, const void *K_cap, int cap_rows, const float *aux)
{
    int rc = check_cycle_args(p, Q, cap_rows, aux, false);
    if (rc != IPOT_OK) return rc;
    if (!K_cap || !aligned16(Q) || !aligned16(K_cap)) return IPOT_E_INVALID;
    return score_only(p, Q, K_cap, cap_rows, aux);
}

int ipot_nuc_scores(ipot_t *p, const void *logits, int logits_dtype, long long row_stride, const int32_t *labels,
                    int n_tokens, int vocab, float *aux_out, long long aux_stride, int slot0)
{
    if (!p || !logits || !labels || !aux_out) return IPOT_E_INVALID;
    if (logits_dtype != IPOT_BF16 && logits_dtype != IPOT_F32) return IPOT_E_INVALID;
    if (n_tokens < 1 || n_tokens > kNovMaxRows / p->cfg.batch || vocab < 1 || row_stride < vocab) return IPOT_E_INVALID;
    if (slot0 < 0 || aux_stride < (long long)slot0 + n_tokens) return IPOT_E_INVALID;
    const size_t elem = logits_dtype == IPOT_F32 ? 4 : 2;
    if ((reinterpret_cast<uintptr_t>(logits) % elem) || (reinterpret_cast<uintptr_t>(labels) & 3u) ||
        (reinterpret_cast<uintptr_t>(aux_out) & 3u))
        return IPOT_E_INVALID;
    const size_t rows = (size_t)p->cfg.batch * n_tokens;
    const size_t need = rows * ((vocab + kNovSegElems - 1) / kNovSegElems);
    if (!p->nov_scratch || need > p->nov_capacity) {  // first use or a larger shape: the only allocation outside ipot_create
        IPOT_CUDA(cudaStreamSynchronize(p->stream));
        cudaFree(p->nov_scratch);  // only this call's own scratch: every other buffer keeps its owner
        p->nov_scratch = nullptr;
        p->nov_capacity = 0;
        if (cudaMalloc((void **)&p->nov_scratch, kNovCounterBytes + need * sizeof(float2)) != cudaSuccess) {
            cudaGetLastError();
            return IPOT_E_NOMEM;
        }
        IPOT_CUDA(cudaMemsetAsync(p->nov_scratch, 0, kNovCounterBytes, p->stream));
        p->nov_capacity = need;
    }
    return logits_dtype == IPOT_F32
               ? launch_novelty<float>(p, logits, (size_t)row_stride, labels, n_tokens, vocab, aux_out, (size_t)aux_stride, slot0)
               : launch_novelty<__nv_bfloat16>(p, logits, (size_t)row_stride, labels, n_tokens, vocab, aux_out, (size_t)aux_stride, slot0);
}

int ipot_decode_attention(ipot_t *p, const void *q, float *out, float *lse)
{
    if (!p || !q || !out || !aligned16(q) || (reinterpret_cast<uintptr_t>(out) & 3u) || (reinterpret_cast<uintptr_t>(lse) & 3u))
        return IPOT_E_INVALID;
    const int lpk = p->row_bytes / 16;
    if (p->row_bytes % 16 || (lpk != 4 && lpk != 8 && lpk != 16 && lpk != 32)) return IPOT_E_INVALID;
    if (p->G > 8) return IPOT_E_INVALID;
    if (p->len < 1) return IPOT_E_STATE;
    int rc = materialise(p, true, true);
    if (rc != IPOT_OK) return rc;
    if (p->cfg.dtype == IPOT_BF16 && p->scorer != IPOT_SCORER_SIMT && (p->cfg.d == 64 || p->cfg.d == 128))
        return p->cfg.d == 64 ? launch_decode_mma<64>(p, q, out, lse) : launch_decode_mma<128>(p, q, out, lse);
    if (p->G != 1 && p->G != 2 && p->G != 4 && p->G != 8) return IPOT_E_INVALID;
    return p->cfg.dtype == IPOT_F32 ? launch_decode<float>(p, q, out, lse) : launch_decode<__nv_bfloat16>(p, q, out, lse);
}

int ipot_enable_rope(ipot_t *p, const void *cos_table, const void *sin_table, int pairing)
{
    if (!p || !cos_table || !sin_table || !aligned16(cos_table) || !aligned16(sin_table)) return IPOT_E_INVALID;
    if (pairing != IPOT_ROPE_HALF && pairing != IPOT_ROPE_INTERLEAVED) return IPOT_E_INVALID;
    if (p->row_bytes % 32) return IPOT_E_INVALID;  // a row must split into two halves of whole 16-byte vectors
    if (p->len != 0) return IPOT_E_STATE;
    if (!p->Krot) {
        IPOT_CUDA(cudaStreamSynchronize(p->stream));
        if (cudaMalloc(&p->Krot, (size_t)p->units * p->cfg.pot_size * p->row_bytes) != cudaSuccess) {
            cudaGetLastError();
            p->Krot = nullptr;
            return IPOT_E_NOMEM;
        }
    }
    p->rope_cos = cos_table;
    p->rope_sin = sin_table;
    p->rope = pairing;
    return IPOT_OK;
}

int ipot_view_rope(ipot_t *p, void **K_rot)
{
    if (!p || !K_rot) return IPOT_E_INVALID;
    if (!p->rope) return IPOT_E_STATE;
    *K_rot = p->Krot;
    return IPOT_OK;
}

int ipot_view(ipot_t *p, void **K, void **V, int *len)
{
    if (!p) return IPOT_E_INVALID;
    int rc = materialise(p, true, true);
    if (rc != IPOT_OK) return rc;
    if (K) *K = p->K;
    if (V) *V = p->V;
    if (len) *len = p->len;
    return IPOT_OK;
}

int ipot_last_indices(ipot_t *p, const int32_t **idx)
{
    if (!p || !idx) return IPOT_E_INVALID;
    *idx = p->idx;
    return IPOT_OK;
}

int ipot_last_scores(ipot_t *p, const float **u, int *len_before)
{
    if (!p || !u) return IPOT_E_INVALID;
    *u = p->last_scores ? p->last_scores : p->scores;
    if (len_before) *len_before = p->last_len_before;
    return IPOT_OK;
}

int ipot_sync_status(ipot_t *p)
{
    if (!p) return IPOT_E_INVALID;
    int rc = materialise(p, true, true);  // after this call the caller's chunk buffers are free again
    if (rc != IPOT_OK) return rc;
    IPOT_CUDA(cudaStreamSynchronize(p->stream));
    int st = 0;
    IPOT_CUDA(cudaMemcpy(&st, p->status, sizeof(int), cudaMemcpyDeviceToHost));
    if (st) p->tc.last_items = 0;  // a launch that gave up half way: the tensor scorer clears its statistics before its next launch
    return st;
}

int ipot_set_profiling(ipot_t *p, int on)
{
    if (!p) return IPOT_E_INVALID;
    if (on && !p->ev) {  // the event pool is created on first use
        p->ev = new (std::nothrow) cudaEvent_t[kProfSlots][5]();
        if (!p->ev) return IPOT_E_NOMEM;
        for (int i = 0; i < kProfSlots; ++i)
            for (auto &e : p->ev[i]) IPOT_CUDA(cudaEventCreate(&e));
    }
    p->profiling = on != 0;
    p->ev_used = 0;
    return IPOT_OK;
}

int ipot_kernel_ms(ipot_t *p, float ms[4], int *cycles, int *scorer_used)
{
    if (!p || !ms) return IPOT_E_INVALID;
    if (!p->profiling || p->ev_used == 0) return IPOT_E_STATE;
    IPOT_CUDA(cudaEventSynchronize(p->ev[p->ev_used - 1][4]));
    double sum[4] = {0, 0, 0, 0};
    for (int c = 0; c < p->ev_used; ++c)
        for (int i = 0; i < 4; ++i) {
            float t = 0.f;
            IPOT_CUDA(cudaEventElapsedTime(&t, p->ev[c][i], p->ev[c][i + 1]));
            sum[i] += t;
        }
    for (int i = 0; i < 4; ++i) ms[i] = (float)(sum[i] / p->ev_used);
    if (cycles) *cycles = p->ev_used;
    if (scorer_used) *scorer_used = p->last_scorer;
    p->ev_used = 0;
    return IPOT_OK;
}

int ipot_launch_count(ipot_t *p, long long *launches)
{
    if (!p || !launches) return IPOT_E_INVALID;
    *launches = p->launches;
    return IPOT_OK;
}

const char *ipot_strerror(int code)
{
    switch (code) {
    case IPOT_OK: return "ok";
    case IPOT_E_INVALID: return "invalid argument";
    case IPOT_E_STATE: return "call not allowed in the pot's current state";
    case IPOT_E_NOMEM: return "out of memory";
    case IPOT_E_CUDA: return "CUDA call failed or no usable device";
    case IPOT_E_TIMEOUT: return "a bounded device-side wait gave up";
    case IPOT_E_BOUNDS: return "a device-side self-check found an index out of range";
    case IPOT_E_LIMIT: return "size exceeds the fixed scratch capacity of the allocation-free entry point";
    default: return "unknown error code";
    }
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Allocation-free CaP scoring.  The two SIMT launches hand the per-row softmax
// statistics to each other through global memory; here that scratch is a fixed
// array inside the library image instead of a cudaMalloc'ed buffer.
// ---------------------------------------------------------------------------
static __device__ __align__(256) float2 g_noalloc_row_stats[IPOT_NOALLOC_MAX_ROWS];

namespace {
std::mutex g_noalloc_mutex;
float2 *g_noalloc_ptr[64];  // device address of the array, per device ordinal

// The array's name is only a host-side handle; kernels need the address the
// runtime reports for the device that is current.
int noalloc_scratch(float2 **out)
{
    int dev = 0;
    IPOT_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return IPOT_E_INVALID;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void *ptr = nullptr;
        IPOT_CUDA(cudaGetSymbolAddress(&ptr, g_noalloc_row_stats));
        g_noalloc_ptr[dev] = static_cast<float2 *>(ptr);
    }
    *out = g_noalloc_ptr[dev];
    return IPOT_OK;
}

template <typename T>
int noalloc_launch(const void *Q, const void *K, float *scores, float2 *stats, int units, int M, int N, int d,
                   size_t k_unit_rows, cudaStream_t stream)
{
    const size_t smem = simt_smem_bytes(d);
    IPOT_CUDA(cudaFuncSetAttribute(cap_row_stats<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)simt_smem_bytes(256)));
    IPOT_CUDA(cudaFuncSetAttribute(cap_column_sums<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)simt_smem_bytes(256)));
    const float scale_log2e = (float)(1.4426950408889634 / std::sqrt((double)d));
    dim3 g1((M + kSimtRows - 1) / kSimtRows, units), g2((N + kSimtKeys - 1) / kSimtKeys, units);
    cap_row_stats<T><<<g1, kSimtThreads, smem, stream>>>((const T *)Q, (const T *)K, stats, M, N, d, k_unit_rows * d, scale_log2e, nullptr, 0, 1);
    cap_column_sums<T><<<g2, kSimtThreads, smem, stream>>>((const T *)Q, (const T *)K, stats, scores, M, N, d, k_unit_rows * d, scale_log2e);
    IPOT_CUDA(cudaGetLastError());
    return IPOT_OK;
}
}  // namespace

extern "C" int ipot_cap_scores_noalloc(const void *Q, const void *K, float *scores, int units, int rows, int N, int d,
                                       int k_unit_rows, int dtype, void *cuda_stream)
{
    if (!Q || !K || !scores || !aligned16(Q) || !aligned16(K) || (reinterpret_cast<uintptr_t>(scores) & 3u))
        return IPOT_E_INVALID;
    if (units < 1 || rows < 1 || N < 1 || k_unit_rows < N || d < 32 || d > 256 || d % 8) return IPOT_E_INVALID;
    if (dtype != IPOT_BF16 && dtype != IPOT_F32) return IPOT_E_INVALID;
    if ((long long)units * rows > IPOT_NOALLOC_MAX_ROWS) return IPOT_E_LIMIT;
    float2 *stats = nullptr;
    int rc = noalloc_scratch(&stats);
    if (rc != IPOT_OK) return rc;
    // every statistics entry that the second launch reads is written by the first one,
    // so nothing left behind by an earlier call needs clearing
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    return dtype == IPOT_F32
               ? noalloc_launch<float>(Q, K, scores, stats, units, rows, N, d, (size_t)k_unit_rows, stream)
               : noalloc_launch<__nv_bfloat16>(Q, K, scores, stats, units, rows, N, d, (size_t)k_unit_rows, stream);
}
