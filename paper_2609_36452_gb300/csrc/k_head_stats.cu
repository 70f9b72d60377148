// k_head_stats.cu - the layerwise projection's contraction with online softmax statistics
// (logit lens of §2.2 / App. A.2 through the LM head; Eq. 1 needs only the final layer's
// entropy, Eq. 2-3 only each layer's argmax and its probability).
//
//   z[r][v] = inv_rms[r] * sum_d u[r][d] * W[v][d]
//
// is computed tile by tile on the 5th-generation tensor cores (tcgen05.mma kind::f16,
// bf16 operands staged in shared memory by TMA with 128-byte swizzling, fp32 accumulators
// in TMEM) and reduced in the epilogue straight out of TMEM into per-row running
// statistics in base-2 units (x = z * log2 e):
//   m = max x,  s = sum 2^(x-m),  t = sum 2^(x-m) (x-m),  a = argmax (lowest index).
// Logits never reach global memory.  Each work unit is (row tile, contiguous range of
// 256-wide vocabulary tiles); its statistics are written once per row as one partial
// (float4); the rows' partials are merged after the last unit (step_epilogue.cuh).
//
// One persistent kernel, launched as clusters of two CTAs (one per SM), serves two tilings.  Each
// CTA counts the mask's set bits and looks the pass's plan up by its row count (or, for large
// batches and second passes, reads both from the step's meta words).  Both tilings run on CTA
// pairs (tcgen05 cta_group::2, M = 256):
//   pair tiles:  256 rows (M, 128 per CTA) x 256 vocabulary entries (N);
//   rows on N:   256 vocabulary entries (M, 128 per CTA) x a group of up to 512 rows (N,
//                padded to a multiple of 32), so that a pass whose row count is not a multiple
//                of 256 pads by at most 31 rows per group.
// Roles: warp 0 TMA producer (one thread), warp 1 TMEM owner (512 columns) and MMA issuer
// (the whole warp in the even CTA, one elected lane issuing), warps 2-9 epilogue (pair tiles
// use warps 2-5); before the contraction they gather the rows of u (step_prologue.cuh).  Every wait is
// bounded; a timeout latches RPD_ERR_TIMEOUT in the step's status word and the CTA drains and
// exits.
#include <atomic>

#include "ptx.cuh"
#include "rpd_internal.h"
#include "step_counters.h"
#include "step_epilogue.cuh"
#include "step_prologue.cuh"

namespace rpd {
namespace {

constexpr uint32_t kTmemCols = 2 * kTileN;
constexpr float kLog2e = 1.4426950408889634f;

// Work units are claimed at run time from a per-pass counter (meta[kMetaUnitNext]) by the
// TMA producer, in the walk's order, so the units in flight are always a window of
// consecutive indices however the CTAs' speeds differ.  The producer passes each claimed
// index to the MMA issuer and the epilogue warps through a small ring in shared memory
// (-1: no unit left).
constexpr int kUnitRing = 4;

struct UnitCursor {
    int slot = 0;
    uint32_t phase = 0;
    __device__ __forceinline__ void advance() {
        if (++slot == kUnitRing) {
            slot = 0;
            phase ^= 1u;
        }
    }
};

// Fold one 32-entry chunk of a row's logits, column col0 + i in v[i], into the row's running
// statistics: top = the largest logit so far (unscaled), and in log2 units, x = logit * scale,
// s = sum 2^(x - x_top), t = sum 2^(x - x_top) (x - x_top), a = its lowest index.
//
// Bound by instruction issue (two warps per scheduler, beside the MMA issuer): the maximum is
// taken of the unscaled logits, three at a time, its index is looked for only in a chunk that
// raises it, and the rest runs on pairs.  5 instructions per logit where scaling, comparing and
// exponentiating one logit at a time took 11.  (v - top) * scale is also closer to x - x_top than
// the difference of two rounded products.
template <bool kFull>
__device__ __forceinline__ void fold_chunk(float (&v)[32], float scale, int col0, int V, float &top,
                                           float &s, float &t, int &a) {
    if (!kFull) {
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (col0 + i >= V) v[i] = -INFINITY;
    }
    float c = v[0];
#pragma unroll
    for (int i = 1; i < 32; ++i) c = fmaxf(c, v[i]);
    if (c > top) {
        if (s > 0.f) {
            const float d = (top - c) * scale;
            const float alpha = ex2(d);
            t = alpha * fmaf(d, s, t);
            s = alpha * s;
        }
        top = c;
        int first = 31;
#pragma unroll
        for (int i = 30; i >= 0; --i) first = v[i] == c ? i : first;
        a = col0 + first;
    }
    if (kFull) {
        const f32x2 minus = pack2(-top, -top), scale2 = pack2(scale, scale);
        f32x2 s2 = pack2(s, 0.f), t2 = pack2(t, 0.f);
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
            const f32x2 d = mul2(add2(pack2(v[i], v[i + 1]), minus), scale2);
            float lo, hi;
            unpack2(d, lo, hi);
            const f32x2 e = pack2(ex2(lo), ex2(hi));
            s2 = add2(s2, e);
            t2 = fma2(e, d, t2);
        }
        float lo, hi;
        unpack2(s2, lo, hi);
        s = lo + hi;
        unpack2(t2, lo, hi);
        t = lo + hi;
    } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            if (col0 + i < V) {
                const float d = (v[i] - top) * scale;
                const float e = ex2(d);
                s += e;
                t = fmaf(e, d, t);
            }
        }
    }
}

// Shared memory of the head kernel: the operand ring (and for rows on N the transpose blocks
// and running statistics), then the barriers.
struct HeadSmem {
    uint8_t *ring;            // 1024-byte aligned

    uint64_t *full;           // [kSwapMaxStages] TMA -> MMA (in the even CTA for pair tilings)
    uint64_t *empty;          // [kSwapMaxStages] MMA -> TMA
    uint64_t *acc_full;       // [2] MMA -> epilogue
    uint64_t *acc_empty;      // [2] epilogue -> MMA (in the even CTA for pair tilings)
    uint64_t *drain;          // [1] MMA completion at exit
    uint64_t *unit_full;      // [kUnitRing] producer -> MMA, epilogue
    uint64_t *unit_empty;     // [kUnitRing] MMA, epilogue -> producer
    uint64_t *epi;            // [1] rows-on-N tiling: barrier of the epilogue warps
    uint64_t *chunk_free;     // [16] rows-on-N tiling: TMEM chunk read (in the even CTA)
    uint32_t *tmem_slot;
    volatile int *abort_flag;
    volatile int *unit_ring;  // [kUnitRing] claimed unit indices
    MaskMap map;              // the compaction (and the pass) of this CTA
};

__device__ __forceinline__ HeadSmem carve_smem(uint8_t *raw) {
    HeadSmem s;
    uint8_t *base = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(raw) + 1023) & ~static_cast<uintptr_t>(1023));
    s.ring = base;  // the rows-on-N tiles place their transpose blocks and statistics after their ring
    uint64_t *bars = reinterpret_cast<uint64_t *>(base + kHeadRegionBytes);
    s.full = bars;
    s.empty = bars + kSwapMaxStages;
    s.acc_full = bars + 2 * kSwapMaxStages;
    s.acc_empty = s.acc_full + 2;
    s.drain = s.acc_empty + 2;
    s.unit_full = s.drain + 1;
    s.unit_empty = s.unit_full + kUnitRing;
    s.epi = s.unit_empty + kUnitRing;
    s.chunk_free = s.epi + 1;
    s.tmem_slot = reinterpret_cast<uint32_t *>(s.chunk_free + kTmemCols / 32);
    s.abort_flag = reinterpret_cast<volatile int *>(s.tmem_slot + 1);
    s.unit_ring = s.abort_flag + 1;
    s.map.words = reinterpret_cast<uint32_t *>(base + kHeadRegionBytes + kHeadBarrierBytes);
    s.map.before = reinterpret_cast<uint16_t *>(s.map.words + kMaskWords);
    s.map.pass = reinterpret_cast<PassInfo *>(s.map.before + kMaskWords + 8);
    return s;
}

static_assert((2 * kSwapMaxStages + 6 + 2 * kUnitRing + kTmemCols / 32) * 8 + 8 + 4 * kUnitRing <=
                  kHeadBarrierBytes,
              "barrier region");

// Barriers and tensor memory of a CTA, the same for both tilings so that neither depends on the
// pass.  full[s] lives in the even CTA and receives both CTAs' TMA completions; empty[s],
// acc_full[a] and drain receive multicast commits from the MMA issuer in both CTAs; acc_empty[a]
// lives in the even CTA and counts the 8 epilogue warps of both CTAs (with pair tiles half of
// the warps work and each arrives twice); unit_empty[i] also counts the even CTA's MMA issuer and
// the odd CTA's producer.
__device__ __forceinline__ void init_barriers(const HeadSmem &sm) {
    for (int i = 0; i < kSwapMaxStages; ++i) {
        mbar_init(&sm.full[i], 1);
        mbar_init(&sm.empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
        mbar_init(&sm.acc_full[i], 1);
        mbar_init(&sm.acc_empty[i], 2 * kSwapEpiWarps);
    }
    for (int i = 0; i < kUnitRing; ++i) {
        mbar_init(&sm.unit_full[i], 1);
        mbar_init(&sm.unit_empty[i], 2 + 2 * kSwapEpiWarps);
    }
    // a chunk is read by one warp per TMEM sub-partition in each CTA
    for (uint32_t i = 0; i < kTmemCols / 32; ++i) mbar_init(&sm.chunk_free[i], 8);
    mbar_init(sm.epi, 32 * kSwapEpiWarps);
    mbar_init(sm.drain, 1);
    *sm.abort_flag = 0;
    fence_mbar_init();
}

// Wait for every CTA's gathered rows (the bound grows with what the grid has to gather).
__device__ __forceinline__ bool wait_for_rows(const HeadParams &p, const HeadSmem &sm, int rows,
                                              unsigned sleep_ns) {
    return counter_wait(&p.meta[kMetaRowsDone], rows, sm.abort_flag,
                        p.wait_limit_ns * (1 + static_cast<unsigned>(rows) / 4096), sleep_ns);
}

// The TMA producer's claim of the next work unit (-1: none left): the even CTA takes it from the
// pass's counter - its first claim was made before the pass was known - and hands it to both
// CTAs' rings.  Returns false if a wait gave up.
__device__ __forceinline__ bool claim_unit(const HeadParams &p, const HeadSmem &sm, uint32_t rank,
                                           int units, UnitCursor &uc, int &first, int &u) {
    volatile int *unit_ring = sm.unit_ring;
    if (rank == 0) {
        const uint32_t unit_full1 = mapa_shared(smem_u32(&sm.unit_full[0]), 1);
        const uint32_t unit_ring1 = mapa_shared(smem_u32(const_cast<int *>(&unit_ring[0])), 1);
        if (!mbar_wait_bounded_cluster(&sm.unit_empty[uc.slot], uc.phase ^ 1u, sm.abort_flag, p.wait_limit_ns))
            return false;
        const int claimed = first >= 0 ? first : atomicAdd(&p.meta[kMetaUnitNext], 1);
        first = -1;
        u = claimed < units ? claimed : -1;
        unit_ring[uc.slot] = u;
        st_shared_cluster(unit_ring1 + static_cast<uint32_t>(uc.slot * sizeof(int)), u);
        mbar_arrive(&sm.unit_full[uc.slot]);
        mbar_arrive_cluster(unit_full1 + static_cast<uint32_t>(uc.slot * sizeof(uint64_t)));
    } else {
        const uint32_t unit_empty0 = mapa_shared(smem_u32(&sm.unit_empty[0]), 0);
        if (!mbar_wait_bounded_cluster(&sm.unit_full[uc.slot], uc.phase, sm.abort_flag, p.wait_limit_ns))
            return false;
        u = unit_ring[uc.slot];
        mbar_arrive_cluster(unit_empty0 + static_cast<uint32_t>(uc.slot * sizeof(uint64_t)));
    }
    uc.advance();
    return true;
}

// Rows on N: a stage of 128 head rows and half a group's rows, and how many there are in the region
// beside the transpose blocks and the rows' statistics and RMS factors.
__device__ __forceinline__ int swap_stage_bytes(int ng) { return kSwapStageBytesA + (ng / 2) * kTileK * 2; }
__device__ __forceinline__ int swap_stages(int ng) {
    return min((kHeadRegionBytes - kSwapXposeBytes - ng * kSwapRowBytes) / swap_stage_bytes(ng), kSwapMaxStages);
}

// What one CTA's TMA producer copies: per stage 128 head rows x 64 columns (w_off bytes into the
// stage) and this CTA's rows of u x 64 columns (u_off), u_rows * m + u_row0 on for row tile m.
struct Copies {
    const CUtensorMap *w, *w_half, *u;
    int stages, stage_bytes, w_off, u_off, u_rows, u_row0;
};

// Bytes of a stage that the pair expects: a half tile brings 64 head rows to each CTA, not 128.
__device__ __forceinline__ uint32_t stage_bytes(const Copies &c, bool half) {
    return 2u * (c.stage_bytes - (half ? 64 * kTileK * 2 : 0));
}

// First row of the head that this CTA copies for the tile at half tile v, in rows of W (of the tiled
// copy: block (v + rank, kb = 0), 128 contiguous rows of 64 columns).
__device__ __forceinline__ int head_row(const HeadParams &p, int v, bool half, uint32_t rank, int num_kb) {
    const int block = half ? v : v + static_cast<int>(rank);
    return (p.w_tiled ? block * num_kb : block) * kPairHalfRows + (half ? static_cast<int>(rank) * 64 : 0);
}

// One tile's K-steps kb0 .. num_kb - 1; returns how many were issued (fewer if a wait gave up).
// The loop is kept as tight as it gets: the same copies issued
// from a loop with a few more branches and address computations in it made whole first-step and
// mid-decode passes 1.5 to 3 % slower.  kOnce: drop the head tile from L2 first (see produce).
template <bool kOnce>
__device__ __forceinline__ int copy_tile(const HeadParams &p, const HeadSmem &sm, const Copies &c,
                                          uint32_t rank, uint32_t full0, uint64_t evict_first, int v,
                                          bool half, int u_row, int kb0, int num_kb, int &stage,
                                          uint32_t &phase) {
    const int dx = p.w_tiled ? 0 : kTileK, dy = p.w_tiled ? kPairHalfRows : 0;
    int x = kb0 * dx;
    int y = head_row(p, v, half, rank, num_kb) + kb0 * dy;
    const CUtensorMap *w = half ? c.w_half : c.w;
    const uint32_t bytes = stage_bytes(c, half);
    int kb = kb0;
    for (; kb < num_kb; ++kb, x += dx, y += dy) {
        if (!mbar_wait_bounded(&sm.empty[stage], phase ^ 1u, sm.abort_flag, p.wait_limit_ns)) break;
        if (rank == 0) mbar_arrive_expect_tx(&sm.full[stage], bytes);
        const uint32_t bar = full0 + static_cast<uint32_t>(stage * sizeof(uint64_t));
        uint8_t *st = sm.ring + stage * c.stage_bytes;
        tma_load_2d_pair(st + c.u_off, c.u, bar, kb * kTileK, u_row);
        if (kOnce)
            tma_load_2d_pair_hint(st + c.w_off, w, bar, x, y, evict_first);
        else
            tma_load_2d_pair(st + c.w_off, w, bar, x, y);
        if (++stage == c.stages) {
            stage = 0;
            phase ^= 1u;
        }
    }
    return kb - kb0;
}

// The first stages of a CTA's first tile, while the ring is empty and the rows of u are still
// being gathered: the head tiles at once, the rows once all of them are counted.  Returns the
// K-steps issued, or -1 if the wait gave up.
__device__ __forceinline__ int copy_ahead(const HeadParams &p, const HeadSmem &sm, const Copies &c,
                                          uint32_t rank, uint32_t full0, bool once, uint64_t evict_first,
                                          int v, bool half, int u_row, int rows, int num_kb) {
    const int ahead = min(c.stages, num_kb);
    const int y0 = head_row(p, v, half, rank, num_kb);
    const CUtensorMap *w = half ? c.w_half : c.w;
    for (int s = 0; s < ahead; ++s) {
        if (rank == 0) mbar_arrive_expect_tx(&sm.full[s], stage_bytes(c, half));
        const uint32_t bar = full0 + static_cast<uint32_t>(s * sizeof(uint64_t));
        uint8_t *dst = sm.ring + s * c.stage_bytes + c.w_off;
        const int x = p.w_tiled ? 0 : s * kTileK;
        const int y = y0 + (p.w_tiled ? s * kPairHalfRows : 0);
        if (once)
            tma_load_2d_pair_hint(dst, w, bar, x, y, evict_first);
        else
            tma_load_2d_pair(dst, w, bar, x, y);
    }
    if (!wait_for_rows(p, sm, rows, 0)) return -1;
    proxy_fence_global();
    for (int s = 0; s < ahead; ++s)
        tma_load_2d_pair(sm.ring + s * c.stage_bytes + c.u_off, c.u,
                         full0 + static_cast<uint32_t>(s * sizeof(uint64_t)), s * kTileK, u_row);
    return ahead;
}

// The TMA producer of one CTA (one thread).
//
// With a single row tile every head tile is read once and is dropped from L2 first, which leaves the
// hidden rows, the partials and the code of the step's later phases there: at 20 rows (LLaDA head)
// 181.8 -> 178.6 us where 1 GB of other traffic lies between two steps, as a forward pass would, and
// 164.2 -> 163.4 where step follows step.  Several row tiles re-read a head tile at slightly different
// times: with that policy, and with an explicit normal one instead of none, first-step and serving
// passes were 1.5 % slower.
__device__ __forceinline__ void produce(const HeadParams &p, const HeadSmem &sm, const Copies &c,
                                        uint32_t rank, const TileWalk &tw, int rows, int num_kb, int first) {
    const uint32_t full0 = mapa_shared(smem_u32(&sm.full[0]), 0);
    const uint64_t evict_first = l2_evict_first();
    const bool once = tw.num_m == 1;
    bool started = false;
    int stage = 0;
    uint32_t phase = 0;
    long long fills = 0;
    bool ok = true;
    UnitCursor uc;
    proxy_fence();  // the compaction's scratch lay in the ring
    while (ok) {
        int u;
        if (!claim_unit(p, sm, rank, tw.units, uc, first, u) || u < 0) break;
        int m, g, v0, v1;
        tw.unit(u, m, g, v0, v1);
        const int u_row = m * c.u_rows + c.u_row0;
        int kb0 = 0;
        if (!started) {
            started = true;
            kb0 = copy_ahead(p, sm, c, rank, full0, once, evict_first, v0, v0 + 1 == v1, u_row, rows, num_kb);
            fills = kb0 < 0 ? min(c.stages, num_kb) : kb0;
            if (kb0 < 0) break;
            if (kb0 == c.stages)
                phase = 1u;
            else
                stage = kb0;
        }
        for (int v = v0; ok && v < v1; v += 2, kb0 = 0) {
            const bool half = v + 1 == v1;
            const int issued =
                once ? copy_tile<true>(p, sm, c, rank, full0, evict_first, v, half, u_row, kb0, num_kb, stage, phase)
                     : copy_tile<false>(p, sm, c, rank, full0, evict_first, v, half, u_row, kb0, num_kb, stage, phase);
            fills += issued;
            ok = issued == num_kb - kb0;
        }
    }
    // Drain: a stage's copies have landed once the MMAs that read it have completed, which the
    // multicast commit on empty[s] reports in this CTA.
    for (int s = 0; s < c.stages; ++s) {
        const long long n_s = fills / c.stages + (s < fills % c.stages ? 1 : 0);
        if (n_s > 0)
            mbar_wait_drain(&sm.empty[s], static_cast<uint32_t>((n_s - 1) & 1), p.wait_limit_ns / 8);
    }
}

// ------------------------------------------------------------------------------------------
// Tiling 1: CTA pairs, rows on M (tcgen05 cta_group::2).  A pair (cluster of 2 CTAs) computes a tile of
// 256 rows x 256 vocabulary columns: CTA r of the pair stages rows [128r, 128r+128) of the row
// tile and W rows [128r, 128r+128) of the vocabulary tile; the even CTA issues
// tcgen05.mma.cta_group::2 with M=256, N=256, which reads both CTAs' shared memory and
// accumulates rows [128r, 128r+128) x all 256 columns into CTA r's TMEM.  Per SM and K-step
// that is 32 KB of operands for the MMA work a single CTA's 128 x 256 tile would need 48 KB for.
//
// Barriers: full[s] lives in the even CTA and receives both CTAs' TMA completions (tx bytes
// 64 KB per stage); empty[s], acc_full[a] and drain receive multicast commits from the MMA
// thread in both CTAs; acc_empty[a] lives in the even CTA and counts two arrivals
// from each of the 4 epilogue warps of both CTAs (16, as many as with rows on N).
__device__ __forceinline__ void head_pair(const HeadParams &p, const HeadSmem &sm, const TileWalk &tw,
                                          int rows, int splits, bool tail, int num_kb, uint32_t tmem_base) {
    constexpr int kStageBytes = kPairStageBytesA + kPairStageBytesB;
    uint64_t *full = sm.full, *empty = sm.empty, *acc_full = sm.acc_full,
             *acc_empty = sm.acc_empty, *unit_full = sm.unit_full, *unit_empty = sm.unit_empty;
    volatile int *abort_flag = sm.abort_flag;
    volatile int *unit_ring = sm.unit_ring;
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();  // 0 = even CTA (issues the MMAs), 1 = odd

    if (warp == 1) {
        if (rank == 0) {
            // -------------------------------------------- MMA issuer (even CTA only): the whole
            // warp runs the loop, one elected lane issues (every branch below is warp-uniform)
            int stage = 0;
            uint32_t phase = 0;
            uint32_t tile_iter = 0;
            bool ok = true;
            UnitCursor uc;
            while (ok) {
                if (!mbar_wait_bounded_warp(&unit_full[uc.slot], uc.phase, abort_flag, p.wait_limit_ns))
                    break;
                const int u = unit_ring[uc.slot];
                __syncwarp();
                if (lane == 0) mbar_arrive(&unit_empty[uc.slot]);
                uc.advance();
                if (u < 0) break;
                int m, g, v0, v1;
                tw.unit(u, m, g, v0, v1);
                const uint32_t idesc = idesc_bf16_f32(kPairTileM, v0 + 1 == v1 ? kTileN / 2 : kTileN);
                for (int v = v0; ok && v < v1; v += 2, ++tile_iter) {
                    const uint32_t acc = tile_iter & 1u;
                    const uint32_t acc_phase = (tile_iter >> 1) & 1u;
                    if (!mbar_wait_bounded_warp(&acc_empty[acc], acc_phase ^ 1u, abort_flag,
                                                p.wait_limit_ns)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after_sync();
                    const uint32_t d_tmem = tmem_base + acc * kTileN;
                    for (int kb = 0; kb < num_kb; ++kb) {
                        if (!mbar_wait_bounded_warp(&full[stage], phase, abort_flag, p.wait_limit_ns)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after_sync();
                        const uint32_t a0 = smem_u32(sm.ring + stage * kStageBytes);
                        const uint32_t b0 = a0 + kPairStageBytesA;
#pragma unroll
                        for (int kk = 0; kk < kTileK / 16; ++kk) {
                            umma_bf16_pair_warp(d_tmem, smem_desc_sw128(a0 + kk * 32),
                                                smem_desc_sw128(b0 + kk * 32), idesc,
                                                (kb > 0 || kk > 0) ? 1u : 0u);
                        }
                        umma_commit_pair_multicast_warp(&empty[stage], 0x3);
                        if (++stage == kPairStages) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                    if (!ok) break;
                    umma_commit_pair_multicast_warp(&acc_full[acc], 0x3);
                }
            }
            umma_commit_pair_multicast_warp(sm.drain, 0x3);
        }
        // Both CTAs: every MMA writing this CTA's TMEM has completed before it is freed.
        if (lane == 0) mbar_wait_drain(sm.drain, 0, p.wait_limit_ns);
        __syncwarp();
    } else if (warp < 6) {
        // ---------------------------------------------------------- epilogue (both CTAs)
        const int sub = warp & 3;
        const int row_in_tile = static_cast<int>(rank) * kPairHalfRows + sub * 32 + lane;
        const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(sub * 32) << 16);
        const uint32_t acc_empty0 = mapa_shared(smem_u32(&acc_empty[0]), 0);
        const uint32_t unit_empty0 = mapa_shared(smem_u32(&unit_empty[0]), 0);
        uint32_t tile_iter = 0;
        // the other CTAs' inv_rms, long before this warp's first tile is done
        bool ok = wait_for_rows(p, sm, rows, 500);
        UnitCursor uc;
        while (ok) {
            if (!mbar_wait_bounded_cluster(&unit_full[uc.slot], uc.phase, abort_flag, p.wait_limit_ns))
                break;
            const int u = unit_ring[uc.slot];
            __syncwarp();
            if (lane < 2)  // half of the warps work: each arrives twice
                mbar_arrive_cluster(unit_empty0 + static_cast<uint32_t>(uc.slot * sizeof(uint64_t)));
            uc.advance();
            if (u < 0) break;
            int m, g, v0, v1;
            tw.unit(u, m, g, v0, v1);
            const int chunks = (v0 + 1 == v1 ? kTileN / 2 : kTileN) / 32;
            const int r = m * kPairTileM + row_in_tile;
            const bool valid = r < rows;
            const float scale = valid ? p.norm.inv_rms[r] * kLog2e : 0.f;
            float run_m = -INFINITY, run_s = 0.f, run_t = 0.f;
            int run_a = 0;
            for (int tile = v0; tile < v1; tile += 2, ++tile_iter) {
                const uint32_t acc = tile_iter & 1u;
                const uint32_t acc_phase = (tile_iter >> 1) & 1u;
                if (!mbar_wait_bounded(&acc_full[acc], acc_phase, abort_flag, p.wait_limit_ns)) {
                    ok = false;
                    break;
                }
                tc_fence_after_sync();
                const int col_base = tile * (kTileN / 2);
                const bool full_tile = col_base + chunks * 32 <= p.V;
#pragma unroll 1
                for (int c = 0; c < chunks; ++c) {
                    float v[32];
                    tmem_ld_32x32b_x32(lane_base + acc * kTileN + c * 32, v);
                    if (full_tile)
                        fold_chunk<true>(v, scale, col_base + c * 32, p.V, run_m, run_s, run_t, run_a);
                    else
                        fold_chunk<false>(v, scale, col_base + c * 32, p.V, run_m, run_s, run_t, run_a);
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane < 2) mbar_arrive_cluster(acc_empty0 + acc * static_cast<uint32_t>(sizeof(uint64_t)));
            }
            if (!ok) break;
            // with a split tail a row has a partial per half tile: a whole tile's second one is empty
            const int slot = tail ? v0 : g;
            if (valid && rpd_check(slot + (tail && v0 + 1 < v1) < p.max_splits, p.meta + kMetaStatus)) {
                float4 *part = p.partials + static_cast<size_t>(r) * p.max_splits + slot;
                part[0] = make_float4(run_m * scale, run_s, run_t, __int_as_float(run_a));
                if (tail && v0 + 1 < v1) part[1] = make_float4(-INFINITY, 0.f, 0.f, __int_as_float(0));
            }
            __syncwarp();
            if (lane == 0) counter_add_release(&p.meta[kMetaUnitsDone], 1);
        }
    }
}

// Barrier of the rows-on-N epilogue's threads: every thread arrives (release) and waits
// for the phase (acquire), bounded like every other wait.  Returns false if it gave up.
__device__ __forceinline__ bool epi_sync(uint64_t *bar, uint32_t &phase, volatile int *abort,
                                         uint64_t limit_ns) {
    mbar_arrive(bar);
    const bool ok = mbar_wait_bounded(bar, phase, abort, limit_ns);
    phase ^= 1u;
    return ok;
}

// ------------------------------------------------------------------------------------------
// Tiling 2: "rows on N" CTA pairs.  The pair's MMA (cta_group::2, M = 256) takes the head as
// its A operand - CTA r stages vocabulary rows [256n + 128r, +128) of tile n, 16 KB per
// K-step - and a group of G rows of u as its B operand (N = G, a multiple of 32 up to 512).
// So CTA r's TMEM holds logits for 128 vocabulary entries (lanes) x the group's rows
// (columns): per row the softmax statistics reduce across lanes.
//
// Operands: each CTA stages its half of the group (rows [r G/2, +G/2)) as one TMA copy per
// stage, from the tensor map whose box has that height (16 to 256 rows; a stage with a second,
// small copy measured far slower).
//
// TMEM: 16 chunks of 32 columns, in which tiles alternate between two places (swap_place); the
// MMAs of a tile wait for the chunks that it shares with its predecessor - two with 288 rows,
// all of them with 512 -, which the epilogue reads and releases first.  A segment's MMA takes the
// first half of its columns' rows from the even CTA's half of the group and the rest from the odd
// CTA's; the epilogue maps each column back to its row.
//
// Epilogue: 8 warps, two per TMEM sub-partition, alternating its chunks.  A warp loads a
// 32 x 32 block, releases a shared chunk, transposes the block through shared memory
// so that each thread holds one row's 32 vocabulary entries, and folds them into that row's
// running statistics (per sub-partition, in shared memory).  At the end of a work unit the
// four sub-partitions' statistics of each row are combined and each CTA writes one partial
// per row (the merge sees 2 partials per split).
// The K-steps of one rows-on-N tile issued as kSegs MMAs per 16-wide step (one per column
// segment), run by the whole issuing warp.  A separate loop per segment count keeps the loop
// free of branches: with the segment tests inside it a tile measured 60 % slower.
template <int kSegs>
__device__ __forceinline__ bool swap_tile_mmas(const HeadSmem &sm, int num_kb, int stages,
                                               int stage_bytes, int &stage, uint32_t &phase,
                                               uint32_t d0, uint32_t d1, uint32_t id0, uint32_t id1,
                                               uint32_t bo1, volatile int *abort_flag, uint64_t limit) {
    for (int kb = 0; kb < num_kb; ++kb) {
        if (!mbar_wait_bounded_warp(&sm.full[stage], phase, abort_flag, limit)) return false;
        tc_fence_after_sync();
        const uint32_t a0 = smem_u32(sm.ring + stage * stage_bytes);
        const uint32_t b0 = a0 + kSwapStageBytesA;
#pragma unroll
        for (int kk = 0; kk < kTileK / 16; ++kk) {
            const uint32_t accum = (kb > 0 || kk > 0) ? 1u : 0u;
            umma_bf16_pair_warp(d0, smem_desc_sw128(a0 + kk * 32), smem_desc_sw128(b0 + kk * 32), id0, accum);
            if (kSegs > 1)
                umma_bf16_pair_warp(d1, smem_desc_sw128(a0 + kk * 32), smem_desc_sw128(b0 + bo1 + kk * 32),
                                    id1, accum);
        }
        umma_commit_pair_multicast_warp(&sm.empty[stage], 0x3);
        if (++stage == stages) {
            stage = 0;
            phase ^= 1u;
        }
    }
    return true;
}

// Where a rows-on-N tile of ng columns lies in TMEM, and its column segments (the MMA's N is at
// most 256).  Tiles alternate between two placements.  Up to 256 columns: the two halves, one
// segment.  More: the two ends of TMEM, overlapping in the middle, and two segments as equal as
// whole 32-column steps allow: an MMA of few columns costs nearly as much as one of 128 (the
// head's half of the operands has to be read all the same; 44 cycles for 32 columns, 64 for 128),
// so 288 columns take 144 cycles a step as 160 + 128 and 173 as 256 + 32.
struct SwapPlace {
    uint32_t chunk0;      // first TMEM chunk (of 32 columns)
    uint32_t shared0, shared1;  // chunks that both placements use: [shared0, shared1)
    int n0, n1;           // segment widths (n1 = 0: one segment)
};
__device__ __forceinline__ SwapPlace swap_place(int ng, uint32_t odd_tile) {
    constexpr uint32_t kChunks = kTmemCols / 32;
    const uint32_t nch = static_cast<uint32_t>(ng) / 32;
    SwapPlace s;
    const uint32_t odd0 = nch > kChunks / 2 ? kChunks - nch : kChunks / 2;
    s.chunk0 = odd_tile ? odd0 : 0u;
    s.shared0 = odd0;
    s.shared1 = nch > odd0 ? nch : odd0;
    s.n0 = ng <= kPairTileM ? ng : static_cast<int>((nch + 1) / 2) * 32;
    s.n1 = ng - s.n0;
    return s;
}

__device__ __forceinline__ void head_swap(const HeadParams &p, const HeadSmem &sm, const TileWalk &tw,
                                          int rows, int splits, int num_kb, int ng, uint32_t tmem_base) {
    uint64_t *acc_full = sm.acc_full, *acc_empty = sm.acc_empty, *unit_full = sm.unit_full, *unit_empty = sm.unit_empty,
             *chunk_free = sm.chunk_free;
    volatile int *abort_flag = sm.abort_flag;
    volatile int *unit_ring = sm.unit_ring;
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const uint32_t nch = static_cast<uint32_t>(ng / 32);
    const int stage_bytes = swap_stage_bytes(ng);
    const int stages = swap_stages(ng);
    float *xpose = reinterpret_cast<float *>(sm.ring + stages * stage_bytes);
    float4 *stats = reinterpret_cast<float4 *>(sm.ring + stages * stage_bytes + kSwapXposeBytes);
    float *scales = reinterpret_cast<float *>(stats + 4 * ng);
    constexpr int kEpiThreads = 32 * kSwapEpiWarps;

    if (warp == 1) {
        if (rank == 0) {
            // -------------------------------------------- MMA issuer (even CTA only): the whole
            // warp runs the loop, one elected lane issues (every branch below is warp-uniform)
            int stage = 0;
            uint32_t phase = 0;
            uint32_t tile_iter = 0;
            bool ok = true;
            UnitCursor uc;
            while (ok) {
                if (!mbar_wait_bounded_warp(&unit_full[uc.slot], uc.phase, abort_flag, p.wait_limit_ns))
                    break;
                const int u = unit_ring[uc.slot];
                __syncwarp();
                if (lane == 0) mbar_arrive(&unit_empty[uc.slot]);
                uc.advance();
                if (u < 0) break;
                int m, g, v0, v1;
                tw.unit(u, m, g, v0, v1);
                for (int v = v0; ok && v < v1; v += 2, ++tile_iter) {
                    // tile t-2, which had the same place, has been read ...
                    const uint32_t acc = tile_iter & 1u;
                    if (!mbar_wait_bounded_warp(&acc_empty[acc], ((tile_iter >> 1) & 1u) ^ 1u, abort_flag,
                                                p.wait_limit_ns)) {
                        ok = false;
                        break;
                    }
                    // ... and so have the chunks that this tile shares with tile t-1
                    const SwapPlace place = swap_place(ng, acc);
                    for (uint32_t c = place.shared0; ok && tile_iter > 0 && c < place.shared1; ++c)
                        ok = mbar_wait_bounded_warp(&chunk_free[c], (tile_iter - 1) & 1u, abort_flag,
                                                    p.wait_limit_ns);
                    if (!ok) break;
                    tc_fence_after_sync();
                    const uint32_t d0 = tmem_base + place.chunk0 * 32, d1 = d0 + place.n0;
                    const uint32_t id0 = idesc_bf16_f32(kPairTileM, place.n0);
                    const uint32_t id1 = idesc_bf16_f32(kPairTileM, place.n1 > 0 ? place.n1 : 32);
                    // the second segment's rows of u start at row n0 / 2 of each CTA's half
                    const uint32_t bo1 = static_cast<uint32_t>((place.n0 / 2) * kTileK * 2);
                    ok = place.n1 > 0 ? swap_tile_mmas<2>(sm, num_kb, stages, stage_bytes, stage, phase, d0,
                                                          d1, id0, id1, bo1, abort_flag, p.wait_limit_ns)
                                      : swap_tile_mmas<1>(sm, num_kb, stages, stage_bytes, stage, phase, d0,
                                                          d1, id0, id1, bo1, abort_flag, p.wait_limit_ns);
                    if (!ok) break;
                    umma_commit_pair_multicast_warp(&acc_full[acc], 0x3);
                }
            }
            umma_commit_pair_multicast_warp(sm.drain, 0x3);
        }
        if (lane == 0) mbar_wait_drain(sm.drain, 0, p.wait_limit_ns);
        __syncwarp();
    } else {
        // ---------------------------------------------------------- epilogue (both CTAs)
        const int sub = warp & 3;                 // TMEM sub-partition (lanes 32*sub..+31)
        const int etid = (warp - 2) * 32 + lane;  // 0 .. kEpiThreads-1
        const int chunk0 = (warp - 2) / 4;        // the two warps of a sub-partition alternate chunks
        constexpr int kChunkStep = kSwapEpiWarps / 4;
        static_assert(kChunkStep == 2, "chunks are shared out by parity");
        const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(sub * 32) << 16);
        const uint32_t acc_empty0 = mapa_shared(smem_u32(&acc_empty[0]), 0);
        const uint32_t chunk_free0 = mapa_shared(smem_u32(&chunk_free[0]), 0);
        const uint32_t unit_empty0 = mapa_shared(smem_u32(&unit_empty[0]), 0);
        float *xp = xpose + (warp - 2) * 32 * kSwapXposeStride;
        const float4 kEmpty = make_float4(-INFINITY, 0.f, 0.f, __int_as_float(0));
        for (int i = etid; i < 4 * ng; i += kEpiThreads) stats[i] = kEmpty;
        uint32_t epi_phase = 0;
        uint32_t tile_iter = 0;
        bool ok = epi_sync(sm.epi, epi_phase, abort_flag, p.wait_limit_ns) &&
                  // the other CTAs' inv_rms, long before this warp's first tile is done
                  wait_for_rows(p, sm, rows, 500);
        UnitCursor uc;
        while (ok) {
            if (!mbar_wait_bounded_cluster(&unit_full[uc.slot], uc.phase, abort_flag, p.wait_limit_ns))
                break;
            const int u = unit_ring[uc.slot];
            __syncwarp();
            if (lane == 0)
                mbar_arrive_cluster(unit_empty0 + static_cast<uint32_t>(uc.slot * sizeof(uint64_t)));
            uc.advance();
            if (u < 0) break;
            int m, g, v0, v1;
            tw.unit(u, m, g, v0, v1);
            // the group's RMS factors, once per unit (read from global memory for every chunk of
            // every tile, steps of two 320-row groups were 0.6 % slower)
            for (int rl = etid; rl < ng; rl += kEpiThreads)
                scales[rl] = m * ng + rl < rows ? p.norm.inv_rms[m * ng + rl] * kLog2e : 0.f;
            if (!epi_sync(sm.epi, epi_phase, abort_flag, p.wait_limit_ns)) break;
            for (int tile = v0; tile < v1; tile += 2, ++tile_iter) {
                const uint32_t acc = tile_iter & 1u;
                if (!mbar_wait_bounded(&acc_full[acc], (tile_iter >> 1) & 1u, abort_flag, p.wait_limit_ns)) {
                    ok = false;
                    break;
                }
                tc_fence_after_sync();
                const SwapPlace place = swap_place(ng, acc);
                // the 32 vocabulary entries of this warp's sub-partition
                const int vbase = tile * (kTileN / 2) + static_cast<int>(rank) * kPairHalfRows + sub * 32;
                const bool full_tile = vbase + 32 <= p.V;
                // This warp's chunks are always the same ones (their statistics are its own); the
                // next tile waits for the shared chunks, so those come first.
                const int chunks = (static_cast<int>(nch) - chunk0 + kChunkStep - 1) / kChunkStep;
                int c = chunk0;
                if (place.shared1 > place.shared0) {
                    const int first = static_cast<int>(place.shared0 - place.chunk0);
                    c = first + ((first ^ chunk0) & 1);
                    if (c >= static_cast<int>(nch)) c = chunk0;
                }
#pragma unroll 1
                for (int i = 0; i < chunks; ++i) {
                    float v[32];
                    const uint32_t slot = place.chunk0 + static_cast<uint32_t>(c);
                    tmem_ld_32x32b_x32(lane_base + slot * 32, v);
                    if (slot >= place.shared0 && slot < place.shared1) {  // the next tile may overwrite it
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(chunk_free0 + slot * static_cast<uint32_t>(sizeof(uint64_t)));
                    }
                    // thread `lane` holds vocabulary entry vbase + lane for rows c*32 + i; write
                    // it as row `lane` of a block padded to 33 floats a row (bank lane + i: no
                    // conflict) and read back column `lane` (bank i + lane: no conflict)
#pragma unroll
                    for (int i = 0; i < 32; ++i) xp[lane * kSwapXposeStride + i] = v[i];
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = xp[i * kSwapXposeStride + lane];
                    __syncwarp();
                    // now v[i] = logit of vocabulary entry vbase + i for column c*32 + lane, i.e. for
                    // row rl of the group: a segment's MMA takes its first half of columns from the
                    // even CTA's rows [o, o + n/2) and the rest from the odd CTA's, and CTA r holds
                    // the group's rows [r * ng/2, +ng/2) (o = 0, then n0/2)
                    const int col = c * 32 + lane;
                    const int x0 = col < place.n0 ? 0 : place.n0;
                    const int half_n = (col < place.n0 ? place.n0 : place.n1) / 2;
                    const int x = col - x0;
                    const int rl = x0 / 2 + (x < half_n ? x : ng / 2 + (x - half_n));
                    const float scale = scales[rl];
                    float4 st = stats[sub * ng + rl];
                    int a = __float_as_int(st.w);
                    if (full_tile)
                        fold_chunk<true>(v, scale, vbase, p.V, st.x, st.y, st.z, a);
                    else
                        fold_chunk<false>(v, scale, vbase, p.V, st.x, st.y, st.z, a);
                    st.w = __int_as_float(a);
                    stats[sub * ng + rl] = st;
                    c += kChunkStep;
                    if (c >= static_cast<int>(nch)) c = chunk0;
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(acc_empty0 + acc * static_cast<uint32_t>(sizeof(uint64_t)));
            }
            if (!ok) break;
            // Combine the four sub-partitions' statistics of each row of the group, write this
            // CTA's partial and reset the entries for the next unit.  The epilogue warps meet at
            // an mbarrier rather than a named barrier, so that a wait that runs out (or another
            // role's abort) can never leave a warp blocked.
            if (!epi_sync(sm.epi, epi_phase, abort_flag, p.wait_limit_ns)) break;
            for (int rl = etid; rl < ng; rl += kEpiThreads) {
                const int r = m * ng + rl;
                const float scale = scales[rl];
                Stat all{-INFINITY, 0.f, 0.f, 0};
#pragma unroll 1
                for (int s4 = 0; s4 < 4; ++s4) {
                    const float4 st = stats[s4 * ng + rl];
                    stats[s4 * ng + rl] = kEmpty;
                    all = merge2(all, Stat{st.x * scale /* log2 units */, st.y, st.z, __float_as_int(st.w)});
                }
                if (r < rows && rpd_check(2 * g + static_cast<int>(rank) < p.max_splits, p.meta + kMetaStatus))
                    p.partials[static_cast<size_t>(r) * p.max_splits + 2 * g + static_cast<int>(rank)] =
                        make_float4(all.m, all.s, all.t, __int_as_float(all.a));
            }
            __syncwarp();
            if (lane == 0) counter_add_release(&p.meta[kMetaUnitsDone], 1);
            if (!epi_sync(sm.epi, epi_phase, abort_flag, p.wait_limit_ns)) break;
        }
    }
}

// After the contraction: CTAs claim blocks of rows and merge them once every work unit of the
// pass is done, and the CTA that completes the merge scores the canvas, or selects what the second
// of two passes projects.

// The kernel is compiled twice: for the plain step - one canvas, one pass over every window layer,
// scored in the kernel (kPlain) - and for everything else.  What the plain step does not run is
// not in its code, which it has to fetch anew in every step.
template <bool kPlain>
struct StepKind {
    const HeadParams &p;
    __device__ __forceinline__ bool from_mask() const { return kPlain || p.from_mask; }
    __device__ __forceinline__ bool scores() const { return kPlain || p.score_canvas; }
    __device__ __forceinline__ bool selects() const { return !kPlain && p.select_band; }
    __device__ __forceinline__ bool lazy() const { return !kPlain && p.compact.lazy; }
    // whether kernels after this one read of its compaction
    __device__ __forceinline__ bool publishes() const { return !kPlain && p.from_mask && (!p.score_canvas || p.select_band); }
};

// A CTA's first claim of a block of rows and the wait for the units (the producer's thread, which
// is done before the epilogue is); `blocks` if there is nothing to merge.  Only running CTAs hold
// units, so the wait ends whatever part of the grid is resident.  It also ends when a CTA has
// given up (the step's outputs are then meaningless), and after the time in which a unit's own
// waits would have run out.
template <bool kPlain>
__device__ __forceinline__ int claim_merge(const HeadParams &p, const HeadSmem &sm, const PassInfo &pass,
                                           int blocks) {
    int32_t *meta = p.meta;
    if (blocks == 0) return blocks;
    const int block = atomicAdd(&meta[kMetaMergeNext], 1);
    if (block >= blocks) return blocks;
    const bool pair = pass.mode == kHeadModePair;
    const int splits = pair ? pass.splits : pass.splits / 2;
    const int tile_rows = pair ? kPairTileM : pass.swap_rows;
    int units = (pass.rows + tile_rows - 1) / tile_rows * splits;
    if (pair && pass.swap_rows == kSplitTail)
        units = tail_split((pass.rows + tile_rows - 1) / tile_rows * (splits / 2), gridDim.x / 2).units;
    // and the warp that publishes the pass
    const int target = 2 * units * (pair ? kPairEpiWarps : kSwapEpiWarps) + (StepKind<kPlain>{p}.publishes() ? 1 : 0);
    const uint64_t limit = p.wait_limit_ns * (p.V / kTileN / splits + 2);
    uint64_t t0 = globaltimer_ns();
    int seen = 0;
    while (true) {
        const int done = ld_acquire(&meta[kMetaUnitsDone]);
        if (done >= target || *sm.abort_flag || ld_acquire(&meta[kMetaStatus]) != RPD_OK) break;
        const uint64_t now = globaltimer_ns();
        if (done != seen) t0 = now;
        seen = done;
        if (now - t0 > limit) {
            *sm.abort_flag = 1;
            break;
        }
    }
    return block;
}

template <bool kPlain>
__device__ __forceinline__ void finish_pass(const HeadParams &p, const HeadSmem &sm,
                                            const PassInfo &pass) {
    const StepKind<kPlain> kind{p};
    int32_t *meta = p.meta;
    volatile int *share = reinterpret_cast<volatile int *>(sm.ring + kHeadRegionBytes - 16);
    const int gs = merge_lanes(pass.splits);
    const int per_block = kHeadKernelThreads / gs;
    const int blocks = (pass.rows + per_block - 1) / per_block;
    const int first = threadIdx.x == 0 ? claim_merge<kPlain>(p, sm, pass, blocks) : 0;
    __syncthreads();  // the ring is free: every role of this CTA is done
    if (threadIdx.x == 0) {
        if (*sm.abort_flag) atomicExch(&meta[kMetaStatus], RPD_ERR_TIMEOUT);
        share[0] = first;
        // nothing to merge: the first CTA goes on
        share[1] = blocks == 0 && blockIdx.x == 0 && (kPlain || !meta[kMetaScored]);
    }
    __syncthreads();
    const int num_words = kind.from_mask() ? (p.compact.B * p.compact.N + 31) >> 5 : 0;
    for (int block = share[0]; block < blocks; block = share[0]) {
        int next = 0;
        if (threadIdx.x == 0) next = atomicAdd(&meta[kMetaMergeNext], 1);  // while this block is merged
        merge_block<kPlain>(p.merge, pass, p.norm.sel_list, block, gs, meta + kMetaStatus,
                    [&](int q) { return sm.map.position(q, num_words); });
        __syncthreads();
        if (threadIdx.x == 0) {
            share[1] = counter_add_acq_rel(&meta[kMetaMergeDone], 1) == blocks - 1;
            share[0] = next;
        }
        __syncthreads();
    }
    if (!share[1]) return;
    if (kind.selects()) {
        // The positions whose earlier window layers a second pass projects (none if this one had
        // every layer); without any the canvas can be scored now.
        const int per_canvas = p.compact.N;
        const int band = pass.lazy
                             ? select_band(p.merge.row_pmax + static_cast<size_t>(p.compact.K - 1) * pass.masked,
                                           pass.masked, p.score.theta_c, p.tau, p.sel_q,
                                           reinterpret_cast<int *>(sm.ring), [&](int q) {
                                               return p.compact.B == 1 ? 0 : sm.map.position(q, num_words) / per_canvas;
                                           })
                             : 0;
        const int rows = (p.compact.K - 1) * band;
        if (threadIdx.x < 32) {
            const HeadPlan hp = pass_plan(p.compact, p.plan, rows);
            if (threadIdx.x == 0) {
                meta[kMetaRows] = rows;
                meta[kMetaRowsTotal] = pass.rows + rows;
                meta[kMetaSel] = band;
                meta[kMetaLayer0] = 0;
                meta[kMetaSwapRows] = hp.swap_rows;
                meta[kMetaSplits] = hp.splits;
                meta[kMetaHeadMode] = hp.mode;
                meta[kMetaScored] = band == 0 && p.score_canvas;
            }
        }
        if (band > 0) return;
    }
    if (!kind.scores()) return;
    int status = RPD_OK, rows_total = pass.rows;
    if (threadIdx.x == kHeadKernelThreads - 1) {  // a thread with nothing to score on short canvases
        // The scoring's barriers lie between this and the first mask byte that changes.
        const bool all = !kind.from_mask() || ld_acquire(&meta[kMetaMaskRead]) == static_cast<int>(gridDim.x);
        share[2] = all;
        if (!all) meta[kMetaClearLater] = 1;
    }
    if (threadIdx.x == 0) {
        status = *reinterpret_cast<volatile int32_t *>(&meta[kMetaStatus]);
        if (!kind.from_mask()) rows_total = meta[kMetaRowsTotal];
    }
    score_canvas(p.score, 0, p.score.tau, p.score.budget, pass, status, rows_total,
                 carve_score(sm.ring, p.score.N), [&](int i, bool masked) {
                     if (kind.from_mask()) return sm.map.scored(i) ? sm.map.rank(i) : -1;
                     const int q = p.score.q_of_pos[i];
                     return masked ? q : -1;
                 },
                 [&] { return share[2] != 0; });
}

// The counters in global memory.
struct DeviceWords {
    int32_t *meta;
    __device__ unsigned inc_wrap(int i, unsigned top) { return atomicInc(reinterpret_cast<unsigned *>(&meta[i]), top); }
    __device__ void zero(int i) { meta[i] = 0; }
};

// The head kernel: one launch per projection pass, clusters of two CTAs, one CTA per SM.  It
// compacts the mask (or reads the pass from the meta words), gathers and normalises the pass's
// rows, contracts them with the head, merges the splits' statistics and scores a single canvas of at
// most kFuseScoreMaxN positions.
template <bool kPlain>
__global__ void __launch_bounds__(kHeadKernelThreads, 1)
    k_head(const __grid_constant__ HeadMaps maps, const __grid_constant__ HeadParams p) {
    extern __shared__ uint8_t smem_raw[];
    const HeadSmem sm = carve_smem(smem_raw);
    const StepKind<kPlain> kind{p};
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    pdl_trigger();  // successors may launch now; they wait for this grid before reading
    for (int i = threadIdx.x * 64; i < p.d; i += blockDim.x * 64)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(p.norm.gain + i));
    if (threadIdx.x == 0) {
        init_barriers(sm);
        tma_prefetch_desc(&maps.w128);
        tma_prefetch_desc(&maps.u);
    }
    if (warp == 1) tmem_alloc_pair(sm.tmem_slot, kTmemCols);
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync();  // both CTAs' barriers initialised before any cross-CTA signal
    tc_fence_after_sync();
    const uint32_t tmem_base = *sm.tmem_slot;
    pdl_wait();  // mask, hidden states and meta words come from preceding work of the stream

    // The first claims need nothing of the pass, and return while it is worked out.  (Claiming and
    // loading the mask before the set-up above is slower: its fences wait for both.)
    int first_unit = -1, first_row = 0;
    if (threadIdx.x == 0 && rank == 0) first_unit = atomicAdd(&p.meta[kMetaUnitNext], 1);
    if (warp >= 2 && lane == 0) first_row = atomicAdd(&p.meta[kMetaRowNext], 1);

    PassInfo pass;
    int num_words = 0;
    if (kind.from_mask()) {
        const int masked = compact_mask(p.compact, sm.map, reinterpret_cast<int *>(sm.ring));
        num_words = (p.compact.B * p.compact.N + 31) >> 5;
        // Every CTA of the grid works its pass out of the same mask, also one that starts when the
        // others are done (kernels of other streams may hold some of the SMs): the canvas is scored
        // without waiting for it, but no bit is cleared before all have been counted here.
        if (threadIdx.x == 32) counter_add_release(&p.meta[kMetaMaskRead], 1);
        int lazy = 0;
        if (kind.lazy()) {  // which rows there are may depend on the plan
            if (warp == 0) {
                lazy = choose_lazy(p.compact, p.plan, masked);
                if (lane == 0) sm.map.pass->lazy = lazy;
            }
            __syncthreads();
            lazy = sm.map.pass->lazy;
        }
        pass.masked = masked;
        pass.lazy = lazy;
        pass.sel = masked;
        pass.layer0 = lazy ? p.compact.K - 1 : 0;
        pass.rows = lazy ? masked : p.compact.K * masked;
        if (warp == 0) {
            const HeadPlan hp = pass_plan(p.compact, p.plan, pass.rows);
            pass.mode = hp.mode;
            pass.splits = hp.splits;
            pass.swap_rows = hp.swap_rows;
            if (lane == 0) *sm.map.pass = pass;
        }
    } else {
        pass.rows = p.meta[kMetaRows];
        pass.masked = p.meta[kMetaMasked];
        pass.lazy = p.meta[kMetaLazy];
        pass.sel = p.meta[kMetaSel];
        pass.layer0 = p.meta[kMetaLayer0];
        pass.mode = p.meta[kMetaHeadMode];
        pass.splits = p.meta[kMetaSplits];
        pass.swap_rows = p.meta[kMetaSwapRows];
    }

    if (warp >= 2) {
        first_row = __shfl_sync(0xffffffffu, first_row, 0);
        gather_rows<kPlain>(p.norm, sm.map, num_words, pass.rows, pass.sel, pass.layer0, first_row,
                    rows_per_claim(pass.rows, gridDim.x * kSwapEpiWarps), p.meta, lane);
    }
    if (kind.from_mask()) {  // the plan, from warp 0, which does not wait for the others
        if (warp == 0) {
            __syncwarp();
            asm volatile("bar.arrive 1, %0;" ::"n"(kHeadKernelThreads) : "memory");
        } else {
            asm volatile("bar.sync 1, %0;" ::"n"(kHeadKernelThreads) : "memory");
            pass = *sm.map.pass;
            if (kind.publishes() && warp >= 2) {
                publish_maps(p.compact, sm.map, (blockIdx.x * kSwapEpiWarps + warp - 2) * 32 + lane,
                             gridDim.x * kSwapEpiWarps * 32);
                // the pass: by the warp that gathered row 0 (or, without rows, one of the first CTA)
                if (lane == 0 && (pass.rows > 0 ? first_row == 0 : blockIdx.x == 0 && warp == 2)) {
                    publish_pass(p.compact, pass);
                    counter_add_release(&p.meta[kMetaUnitsDone], 1);
                }
            }
        }
    }

    if (pass.rows > 0) {
        const bool pair = pass.mode == kHeadModePair;
        const int ng = pair ? kPairTileM : pass.swap_rows;
        const int splits = pair ? pass.splits : pass.splits / 2;
        const int num_kb = (p.d + kTileK - 1) / kTileK;
        TileWalk tw;
        const bool tail = pair && pass.swap_rows == kSplitTail;
        tw.init(pass.rows, ng, p.V, p.d, splits, tail, gridDim.x / 2);
        if (warp == 0) {
            if (lane == 0 && !p.stall) {
                // this CTA's half of the tile's rows, one copy (rows on N: the map whose box is half
                // a group high)
                const int half = ng / 2;
                const CUtensorMap *u = pair ? &maps.u : &maps.u_rows[half / kUBoxRows - 1];
                if (!pair) tma_prefetch_desc(u);
                const Copies copies{&maps.w128, &maps.w64, u,
                                    pair ? kPairStages : swap_stages(ng),
                                    pair ? kPairStageBytesA + kPairStageBytesB : swap_stage_bytes(ng),
                                    pair ? kPairStageBytesA : 0,
                                    pair ? 0 : kSwapStageBytesA,
                                    ng, static_cast<int>(rank) * half};
                produce(p, sm, copies, rank, tw, pass.rows, num_kb, first_unit);
            }
        } else if (pair) {
            head_pair(p, sm, tw, pass.rows, splits, tail, num_kb, tmem_base);
        } else {
            head_swap(p, sm, tw, pass.rows, splits, num_kb, ng, tmem_base);
        }
    }
    __syncwarp();
    tc_fence_before_sync();
    finish_pass<kPlain>(p, sm, pass);  // begins with a barrier of the CTA
    cluster_sync();  // no signal may still be in flight to a CTA that is about to exit
    tc_fence_after_sync();
    if (warp == 1) {
        __syncwarp();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
    // The last CTA of the grid leaves the counters at zero for the next pass.
    int clear_later = 0;
    if (threadIdx.x == 0) {
        __threadfence();
        DeviceWords words{p.meta};
        if (last_to_leave(words, gridDim.x)) {
            __threadfence();
            if (kind.from_mask() && kind.scores())
                clear_later = *reinterpret_cast<volatile int32_t *>(&p.meta[kMetaClearLater]);
            zero_counters(words);
            if (!kPlain && p.last_pass) p.meta[kMetaScored] = 0;
            if (kPlain || p.last_pass) p.meta[kMetaStepStatus] = atomicExch(&p.meta[kMetaStatus], RPD_OK);
        }
    }
    if (kind.from_mask() && kind.scores() && warp == 0 && __shfl_sync(0xffffffffu, clear_later, 0))
        clear_committed(p.score, lane);
}

// The tiled copy of the head: thread i writes 16-byte vector i of Wt, which is vector k8 of
// row r of block blk = t * (d / 64) + k, i.e. W[128 t + r][64 k + 8 k8 ...].
__global__ void k_tile_head(const uint4 *__restrict__ W, uint4 *__restrict__ Wt, int V, int d) {
    const int nkb = d / 64;
    const long long total = static_cast<long long>((V + 127) / 128) * nkb * 128 * 8;
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int k8 = static_cast<int>(i & 7);
        const long long rest = i >> 3;
        const int r = static_cast<int>(rest & 127);
        const long long blk = rest >> 7;
        const int k = static_cast<int>(blk % nkb);
        const int row = static_cast<int>(blk / nkb) * 128 + r;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (row < V) v = W[(static_cast<long long>(row) * d + k * 64) / 8 + k8];
        Wt[i] = v;
    }
}

// Per-device one-time settings (the dynamic shared-memory opt-in is a property of the
// kernel on each device).
constexpr int kMaxDevices = 64;
std::atomic<int> g_head_ready[kMaxDevices];
std::atomic<int> g_head_clusters[kMaxDevices];  // resident pairs + 1 (0: not queried yet)

int current_device() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -1;
    return dev;
}

cudaError_t opt_in_smem() {
    const int dev = current_device();
    if (dev < 0) return cudaErrorInvalidDevice;
    if (g_head_ready[dev].load(std::memory_order_acquire)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_head<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kHeadKernelSmemBytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_head<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kHeadKernelSmemBytes);
    if (e == cudaSuccess) g_head_ready[dev].store(1, std::memory_order_release);
    return e;
}

}  // namespace

int head_max_clusters() {
    const int dev = current_device();
    if (dev < 0) return 0;
    const int cached = g_head_clusters[dev].load(std::memory_order_acquire);
    if (cached > 0) return cached - 1;
    if (opt_in_smem() != cudaSuccess) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(kHeadKernelThreads);
    cfg.dynamicSmemBytes = kHeadKernelSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_head<false>, &cfg) != cudaSuccess) n = 0;
    g_head_clusters[dev].store(n + 1, std::memory_order_release);
    return n;
}

cudaError_t launch_tile_head(const void *W, void *Wt, int V, int d, cudaStream_t s) {
    k_tile_head<<<1024, 256, 0, s>>>(static_cast<const uint4 *>(W), static_cast<uint4 *>(Wt), V, d);
    return cudaGetLastError();
}

cudaError_t launch_head(const HeadMaps &maps, const HeadParams &p, int grid, cudaStream_t s) {
    cudaError_t e = opt_in_smem();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kHeadKernelThreads);
    cfg.dynamicSmemBytes = kHeadKernelSmemBytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = t_no_pdl ? 1 : 2;
    const bool plain = p.from_mask && p.score_canvas && !p.select_band && p.last_pass && p.compact.lazy == 0 &&
                       !p.norm.sel_list && !p.merge.shard_out;
    return cudaLaunchKernelEx(&cfg, plain ? k_head<true> : k_head<false>, maps, p);
}

}  // namespace rpd
