// rpd_internal.h - shared between the host entry points and the kernels' translation
// units: scratch layout, launch parameters and launcher declarations.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/rpd.h"

namespace rpd {

// Head-statistics tiles (tcgen05 cta_group::2: a cluster of two CTAs, one per SM, M = 256).
// Pair tiles: 256 rows x 256 vocabulary columns per pair; each CTA stages its own 128 rows of
// u and 128 rows of W per K-step of 64 (32 KB), 7 stages deep.
constexpr int kTileM = 128;   // rows of u per CTA (TMEM lanes) and the row padding unit of scratch
constexpr int kTileN = 256;   // vocabulary entries per tile
constexpr int kTileK = 64;
constexpr int kPairTileM = 256;
constexpr int kPairStages = 7;
constexpr int kPairHalfRows = 128;
constexpr int kPairStageBytesA = kPairHalfRows * kTileK * 2;
constexpr int kPairStageBytesB = kPairHalfRows * kTileK * 2;
// "Rows on N" tiles: a pair multiplies 256 vocabulary entries (128 per CTA, the MMA's M side)
// by a group of up to 512 projected rows (the N side, in steps of 32), so rows are padded to a
// multiple of 32 instead of a multiple of 256.  Each CTA stages its 128 head rows (16 KB) and
// half of the group's rows per K-step.  Tiles alternate between two places in TMEM: its two halves
// for groups of at most 256 rows, its two ends, overlapping in the middle, for larger ones.
constexpr int kSwapMaxRows = 512;
constexpr int kSwapRowStep = 32;  // N of the M = 256 MMA: a multiple of 32, at least 32
// At most 8 operand stages per CTA: small groups would fit 12, but with 12 the HBM-bound
// head streamed 2 % slower (20 rows: 0.158 against 0.153 ms) - the extra copies in flight
// bought nothing; 6 was slower again.  The barrier arrays are sized by this, so it must also
// cover the pair tiling's stages.
constexpr int kSwapMaxStages = 8;
constexpr int kSwapStageBytesA = kPairHalfRows * kTileK * 2;

constexpr int kSwapEpiWarps = 8;   // two per TMEM sub-partition, alternating its chunks
constexpr int kSwapXposeStride = 33;                             // floats per padded row
constexpr int kSwapXposeBytes = kSwapEpiWarps * 32 * kSwapXposeStride * 4;  // 32 x 32 fp32 per warp
// rows on N, per row of the group: running statistics of the four sub-partitions, RMS factor
constexpr int kSwapRowBytes = 4 * 16 + 4;
constexpr int kUBoxRows = 16;  // granularity of a half group's rows (the TMA box heights)
// Roles: warp 0 TMA, warp 1 MMA + TMEM owner, warps 2-9 epilogue (pair tiles use warps 2-5).
constexpr int kHeadKernelThreads = 64 + 32 * kSwapEpiWarps;
constexpr int kPairEpiWarps = 4;
constexpr int kHeadBarrierBytes = 448;
// Canvas positions (B * N) whose masks the head kernel compacts itself, as a bitmap in its shared
// memory: any single canvas, and batches of up to this many positions together.
constexpr int kFusedMaxPositions = 8192;
constexpr int kMaskWords = kFusedMaxPositions / 32;
constexpr int kHeadMaskBytes = kMaskWords * 4 + (kMaskWords + 8) * 2 + 32;  // bitmap, prefixes, plan
// The pair tiles' operand ring, or the rows-on-N ring, transpose blocks and statistics (the
// ring takes what the other two leave): the 7-stage pair ring, 224 KB.
constexpr int kHeadRegionBytes = 224 * 1024;
static_assert(kPairStages <= kSwapMaxStages, "the stage barriers are shared by both tilings");
static_assert(kPairStages * (kPairStageBytesA + kPairStageBytesB) <= kHeadRegionBytes,
              "the pair tiles' operand ring fits the region");
static_assert(kHeadRegionBytes - kSwapXposeBytes - kSwapMaxRows * kSwapRowBytes >=
                  3 * (kSwapStageBytesA + (kSwapMaxRows / 2) * kTileK * 2),
              "a 512-row group still gets three stages");
// 1024-byte alignment slack + that region + barriers + the compaction's bitmap
constexpr int kHeadKernelSmemBytes = 1024 + kHeadRegionBytes + kHeadBarrierBytes + kHeadMaskBytes;
static_assert(kHeadKernelSmemBytes <= 232448, "dynamic shared memory per CTA");
// Values of meta[kMetaHeadMode].
constexpr int kHeadModePair = 2;
constexpr int kHeadModeRowsN = 3;
constexpr int kMaxBatch = 128;
constexpr int kMaxCanvas = 8192;
static_assert(kMaxCanvas <= kFusedMaxPositions, "a single canvas never needs k_compact");
constexpr int kScoreThreads = 1024;
// Longest canvas that the head kernel scores itself.  Its 320 threads take 3.2 times as many turns, each
// a trip to L2 for the rows' statistics, as k_score_commit's 1024, which cost a launch of 1.5 to 2 us:
// half masked, d = 256, V = 4096, K = 2: 1024 positions 27.8 us here, 27.6 there; 2048: 36.9, 35.2;
// 4096: 49.9, 46.4; 8192: 91.0, 78.5.  With 5 masked: 1024 20.5, 22.6; 2048 22.4, 22.6; 8192 30.8, 29.0.
constexpr int kFuseScoreMaxN = 2048;
constexpr uint64_t kWaitLimitNs = 2000000000ull;  // bounded mbarrier waits: 2 s
constexpr long long kBandBytes = 32ll << 20;       // u tiles a band of head work units re-reads

// Indices into the per-step device metadata words.
enum MetaIndex : int {
    kMetaMasked = 0,   // total masked positions over all canvases (NMT)
    kMetaRows = 1,     // projected rows R = K * NMT
    kMetaStatus = 2,   // RPD_OK or RPD_ERR_TIMEOUT, latched by kernels
    kMetaSplits = 3,   // vocabulary splits G chosen for the head kernel
    kMetaHeadMode = 4, // kHeadModePair or kHeadModeRowsN: the pass's head tiling
    kMetaSel = 5,      // positions projected by the current pass
    kMetaLayer0 = 6,   // first window layer of the current pass (rows are layer-major)
    kMetaRowsTotal = 7,// rows projected by all passes of this step
    kMetaLazy = 8,     // 1 when this step projects lazily (two passes)
    kMetaUnitNext = 9, // next head work unit to claim
    kMetaMergeDone = 10, // merged blocks of rows
    kMetaSwapRows = 11,  // rows per row group of the "rows on N" tiling (mode 3)
    kMetaRowNext = 12,   // next rows of the pass to gather (claimed by the head kernel's warps)
    kMetaMergeNext = 13, // next block of rows to merge (claimed by the head kernel's CTAs)
    kMetaExit = 14,      // CTAs of the head kernel that are done; the last one zeroes the counters
    kMetaStepStatus = 15,// the step's status, published when its last head kernel ends
    kMetaClearLater = 16,// the canvas was scored before every CTA had read its mask: the last CTA to
                         // leave clears the committed bits
    kMetaScored = 17,    // the first of two passes scored the canvas: nothing is left for the second
    // counts that the head kernel's CTAs wait for, on a line of their own
    kMetaRowsDone = 32,  // gathered rows of the pass
    kMetaUnitsDone = 33, // head work units whose partials are written, counted by each epilogue warp
    kMetaMaskRead = 48,  // CTAs of the head kernel that have read the mask
    kMetaWords = 64
};

// A projection pass as the head kernel sees it (from its own compaction, or from the meta words).
struct PassInfo {
    int rows, sel, layer0, masked, lazy;
    int mode, splits, swap_rows;
};

// Tiling plan of a projection pass (head_plan.h): which tiling the head kernel runs, with how
// many vocabulary splits.
struct HeadPlan {
    int mode;       // kHeadModePair or kHeadModeRowsN
    int splits;     // partials per row the merge reads (vocabulary splits; twice that for rows on N)
    int swap_rows;  // rows per group of the rows-on-N tiling; pair tiles: 0, or kSplitTail
    float est;      // estimated time, in 128 x 256-tile units
};
struct HeadPlanInputs {
    int num_n;        // vocabulary tiles of 256
    int max_splits;   // partials per row the scratch holds
    int pair_slots;   // CTA pairs of the head kernel
    float hbm_tiles;  // time to stream the head once, in tile units
    int force;        // RPD_TILING_*
    int regroup;      // also weigh more, smaller row groups (regroup_plan)
    int d;            // hidden size
};
// Pair tiles whose last, partly filled wave is issued as half tiles (split_tail).
constexpr int kSplitTail = 1;
// Rows up to which a context tabulates the plan row by row (a multiple of kPairTileM).
constexpr int kPlanRows = 16384;

// The plans of passes of up to kStepPlanRows rows as a kernel argument: a plan depends on the row
// count only through its multiple of 32 (groups are padded to 32 rows, pair tiles to 256).  Reading
// a table in global memory, or evaluating the plan on the device (9 us), lay between a step's
// compaction and its first copies.
constexpr int kStepPlanRows = 1024;
struct StepPlan {
    int32_t splits[kStepPlanRows / 32];  // negative: rows on N
    uint16_t swap_rows[kStepPlanRows / 32];
    float est[kStepPlanRows / 32];
};

struct CompactParams {
    const uint8_t *mask;  // [B*N]
    int32_t *q_of_pos;    // [B*N] compact index or -1
    int32_t *pos_of_q;    // [B*N] flat position b*N+i of compact index q
    int32_t *meta;        // [kMetaWords]
    int B, N, K;
    const HeadPlan *plan; // the context's tables (table_plan)
    int plan_rows;
    int block;            // 0: every masked position; > 0: only each canvas's active block
    int lazy;             // 0: all window layers; 1: lazy; 2: lazy when it is estimated cheaper
};

// Band fraction assumed when the device weighs lazy against full projection before the
// first pass (the real band is known only after it).
constexpr float kLazyBandGuess = 0.25f;

// Where merged per-row statistics go: split partials (log2 units) in, argmax / max
// probability / entropy per (layer, compact position) out, at layer * NMT + q.
struct MergeArgs {
    const float4 *partials;  // [rows][max_splits]
    int max_splits;
    int32_t *row_arg;
    float *row_pmax;
    float *row_H;
    // Vocabulary-sharded steps: when shard_out is set, each row's merged statistics themselves
    // (max, sum, tsum, argmax + v_offset) go to shard_out[layer * shard_stride + position]
    // instead of the derived outputs above.
    float4 *shard_out;
    int shard_stride;
    int v_offset;
};

// Merge of the statistics of P vocabulary shards (rpd_step_shard_finish): per (layer k, masked
// position) the P records gathered[(p * K + k) * N + position], p = 0..P-1 in order, give the
// row's argmax, probability and entropy at k * NMT + q.
struct ShardMergeParams {
    const float4 *gathered;   // [P][K][B*N]
    int P, K, BN;
    const int32_t *pos_of_q;  // [NMT]
    const int32_t *meta;
    int32_t *row_arg;
    float *row_pmax;
    float *row_H;
};

// Second pass of lazy projection, of batches that the head kernel does not compact itself: selects the
// positions whose final confidence lies in the stability band theta_c <= c < tau of their canvas and
// sets up the pass over their earlier window layers (tiling, split count, row mapping).
struct BandParams {
    int32_t *meta;
    MergeArgs mg;              // merged first-pass statistics (final-layer confidences)
    const int32_t *pos_of_q;   // [NMT] flat position b*N+i of compact index q
    int32_t *sel_q;            // out: compact indices of the band positions
    int B, N, K;
    float theta_c;
    const HeadPlan *plan;
    int plan_rows;
    float tau[kMaxBatch];
};

// Costs of the tiling choice are in units of one 128-row x 256-entry tile's MMA work on one SM
// at the nominal rate below (24.4 us).  The per-tile costs are measured ones (LLaDA head,
// d = 4096, GB300, head time / tiles per pair, both tilings forced at 20 to 1024 rows):
//   pair tile (256 rows x 256 entries per pair): 22.3 us, 0.914 units;
//   rows-on-N tile (256 entries x a group of ng rows): 20.5 + 0.025 ng us (0.840 + 0.00102 ng
//   units) for ng <= 256, whose accumulators are double-buffered, and 4.9 + 0.0888 ng us
//   (0.201 + 0.00364 ng units) for larger groups (288 rows: 30.5 us, 416: 42.8 us, 512: 50.4 us).
// When streaming the head bounds a pass, pair tiles - half of whose staged bytes are rows of u -
// stream it about 4 % slower than rows-on-N tiles (20 rows: 0.159 against 0.153 ms).
constexpr float kPairTileCost = 0.914f;
constexpr float kSwapTileBase = 0.840f;
constexpr float kSwapTilePerRow = 0.00102f;
constexpr float kSwapWideTileBase = 0.201f;
constexpr float kSwapWideTilePerRow = 0.00364f;
constexpr float kPairStreamFactor = 1.04f;
// Per-SM MMA rate of the unit tile and the sustained HBM read rate used by the tiling choice
// (GB300 measurements; only their ratio matters).
constexpr double kSingleTileFlopsPerSm = 1.1e13;
constexpr double kHeadStreamBytesPerSec = 6.5e12;

// Row r of a projection pass: layer k = meta[kMetaLayer0] + r / S and position
// q = sel[r % S] (sel = the pass's list of compact indices, or the identity when null),
// S = meta[kMetaSel]; its merged statistics land at k * NMT + q.
struct NormParams {
    const __nv_bfloat16 *hidden;  // [K][B*N][d]
    const __nv_bfloat16 *gain;    // [d]
    const int32_t *pos_of_q;
    const int32_t *sel_list;      // null: every compact position
    const int32_t *meta;
    __nv_bfloat16 *u;             // [rows][d] compact head operand bf16(g*h)
    float *inv_rms;               // [rows]
    int BN, d;
    float eps;
};

// Time to stream the head once, in units of one 128 x 256 tile's MMA time on one SM.
inline float head_stream_in_tiles(int V, int d, int num_sms) {
    (void)num_sms;
    const double t_hbm = 2.0 * V * static_cast<double>(d) / kHeadStreamBytesPerSec;
    const double t_tile = 2.0 * kTileM * kTileN * static_cast<double>(d) / kSingleTileFlopsPerSm;
    return static_cast<float>(t_hbm / t_tile);
}

struct ScoreParams {
    uint8_t *mask;              // [B][N] in/out
    const int32_t *q_of_pos;    // [B*N]
    const int32_t *meta;
    const int32_t *row_arg;
    const float *row_pmax;
    const float *row_H;
    uint8_t *out_commit;        // [B][N]
    int32_t *out_token;         // [B][N]
    rpd_stats *out_stats;       // [B]
    rpd_debug dbg;
    int B, N, K;
    float theta_c, theta_s, w;
    int k_max, window;
    int block;                  // 0: full RPD; > 0: RPD-block (no budget, in-block fallback)
    float tau, budget;          // of a single canvas
};

// Several canvases, each with thresholds of its own.
struct BatchScoreParams {
    ScoreParams canvas;
    float tau[kMaxBatch];
    float budget[kMaxBatch];
};

struct HeadParams {
    CompactParams compact; // the mask and what its compaction writes
    StepPlan plan;         // of the passes that the kernel compacts itself
    NormParams norm;       // the rows gathered before the contraction
    float4 *partials;      // [rows][max_splits]: (max, sum, tsum, argmax bits), log2 units
    int32_t *meta;
    int from_mask;         // the kernel compacts the mask itself (B * N <= kFusedMaxPositions);
                           // otherwise the pass is described by the meta words
    int last_pass;         // the step's last projection pass: publish its status
    int score_canvas;      // score the (single) canvas once nothing is left to project
    int select_band;       // the first of two passes: select the second's positions after the merge
    int32_t *sel_q;        // out: their compact indices
    float tau[kMaxBatch];  // upper end of each canvas's band (the lower one is score.theta_c)
    MergeArgs merge;
    ScoreParams score;
    int V, d, max_splits;
    uint64_t wait_limit_ns;  // bound on every mbarrier wait
    int stall;               // diagnostics: issue no loads (the waits run out)
    int w_tiled;             // W is the context's tiled copy (rpd_set_head_layout), else row-major
};

// Launch with programmatic stream serialisation, so that the kernel's prologue overlaps the
// tail of its predecessor in the stream (the kernel itself waits with griddepcontrol.wait
// before it reads what the predecessor wrote).
// Set on a host thread while it records launches that may not carry programmatic dependencies
// (a graph body that refuses them): the launches are then plainly stream-ordered, and the
// kernels' griddepcontrol instructions have nothing to wait for.
inline thread_local bool t_no_pdl = false;

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t s, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = t_no_pdl ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Args &&>(args)...);
}

// Bounds checks of the checked build (compiled with -DRPD_CHECKS): a failed check latches
// RPD_ERR_CHECK in the step's status word (`status`, device memory) and the guarded access is
// skipped; without RPD_CHECKS every check is `true` and compiles away.
#ifdef RPD_CHECKS
__device__ __forceinline__ bool rpd_check(bool ok, const int32_t *status) {
    if (!ok) atomicCAS(const_cast<int32_t *>(status), RPD_OK, RPD_ERR_CHECK);
    return ok;
}
#else
__device__ __forceinline__ bool rpd_check(bool, const int32_t *) { return true; }
#endif

// Record the message returned by rpd_last_error() on this host thread.
void set_last_error(const char *msg);

// ------------------------------------------------------------------ argument checks
// Shared by every entry point, so that they accept and refuse the same arguments.  Each
// returns nullptr when the argument is acceptable, else the message to report.

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Rule parameters (Table 4): theta_c, w finite and >= 0, theta_s not NaN, k_max, window >= 1,
// block >= 0.
inline const char *rule_error(const rpd_rule &r) {
    if (!(r.theta_c >= 0.f) || !(r.theta_c <= 3.402823466e38f)) return "theta_c must be finite and >= 0";
    if (r.theta_s != r.theta_s) return "theta_s is NaN";
    if (!(r.w >= 0.f) || !(r.w <= 3.402823466e38f)) return "w must be finite and >= 0";
    if (r.k_max < 1) return "k_max must be >= 1";
    if (r.window < 1) return "window must be >= 1";
    if (r.block < 0) return "block must be >= 0";
    return nullptr;
}

// Per-call thresholds: 0 < tau <= 1, theta_c < tau (Eq. 5 needs theta_c < theta_h), budget >= 0.
inline const char *call_error(const rpd_rule &r, float tau, float budget) {
    if (!(tau > 0.f && tau <= 1.f)) return "tau must be in (0, 1]";
    if (!(r.theta_c < tau)) return "theta_c must be below tau";
    if (!(budget >= 0.f)) return "budget must be >= 0";
    return nullptr;
}

// Memory the kernels read with TMA (the head, the gain) must be device or managed memory of
// `device`; memory the head kernel gathers with plain loads (hidden states) may also be
// page-locked host memory mapped into the device's address space.  Any other pointer - pageable
// host memory, another device's memory - would make the kernels fault, so it is refused.
inline bool pointer_usable(const void *p, int device, bool host_mapped_ok) {
    cudaPointerAttributes a{};
    const bool ok = cudaPointerGetAttributes(&a, p) == cudaSuccess &&
                    (((a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) &&
                      a.device == device) ||
                     (host_mapped_ok && a.type == cudaMemoryTypeHost && a.devicePointer == p));
    cudaGetLastError();  // clear the (non-sticky) error the query may have recorded
    return ok;
}

cudaError_t launch_compact(const CompactParams &p, cudaStream_t s);
// Tensor maps of the head kernel's operands (128-byte swizzling, K boxes of 64): u in boxes of
// 128 rows (pair tiles) and, for the rows-on-N tiles, in boxes of 16, 32, ..., 256 rows (one
// per half-group height, so that a stage copies a CTA's half of the group with one instruction:
// the TMA unit's time per copy, not its bytes, bounded a stage built from 16-row boxes); W in
// boxes of 128 rows, and of 64 for half tiles.
constexpr int kUMaps = (kSwapMaxRows / 2) / kUBoxRows;  // box heights kUBoxRows * (1 .. kUMaps)
struct HeadMaps {
    CUtensorMap u;                // box 64 x 128 rows
    CUtensorMap w128, w64;        // boxes 64 x 128 and 64 x 64 rows of W
    CUtensorMap u_rows[kUMaps];   // u_rows[j]: box 64 x kUBoxRows*(j+1) rows
};
// The head kernel (every tiling; the pass's is looked up by its row count, or read from the meta words
// where another kernel set the pass up), launched as `grid` CTAs in clusters of two, one per SM.
cudaError_t launch_head(const HeadMaps &maps, const HeadParams &p, int grid, cudaStream_t s);
// Copy W [V][d] (d % 64 == 0) into blocks of 128 rows x 64 columns, block (t, k) at element
// ((t * (d / 64) + k) * 128) * 64, rows past V zero; Wt holds ceil(V/128)*128*d elements.
cudaError_t launch_tile_head(const void *W, void *Wt, int V, int d, cudaStream_t s);
// Largest number of clusters of the head kernel that can be resident at once.
int head_max_clusters();
cudaError_t launch_band(const BandParams &p, cudaStream_t s);
cudaError_t launch_score_commit(const BatchScoreParams &p, cudaStream_t s);
// Stop test of the decoding loop: counts the step and sets the loop's condition (one thread).
cudaError_t launch_loop_test(cudaGraphConditionalHandle handle, const rpd_stats *stats, int B, int N,
                             float stop_frac, int max_steps, int32_t *steps, cudaStream_t s);
cudaError_t launch_merge_shards(const ShardMergeParams &p, int grid, cudaStream_t s);
}  // namespace rpd
