// step_prologue.cuh - the part of the head kernel that runs before the contraction: compaction
// of the mask (App. A.6: only masked positions are projected) and the RMSNorm prologue of the
// layerwise projection (App. A.2: the model's final normalisation is applied to every window
// layer).
//
// Every CTA builds the compaction for itself: the mask as a bitmap in shared memory and the
// number of set bits before each word, so that position -> compact index is a popcount and
// compact index -> position a search.  A canvas is a few hundred bytes; reading it in every CTA
// costs less than passing the result from one CTA to the others.
//
// The rows are gathered by warps that claim them from a counter: row r of the pass (layer k,
// compact position q) reads hidden[k][pos(q)], writes the head operand u[r] = bf16_rne(g * h)
// (exact product, one rounding) and inv_rms[r] = (mean(h^2) + eps)^(-1/2); the RMS factor is
// applied after the contraction.  Finished rows are counted, and a CTA's first copy of u waits for
// the count.  Only running warps claim rows and no warp waits before its row is done, so the wait
// ends whatever part of the grid is resident (other streams' kernels may hold some of the SMs).
//
// Bound: latency.  As two kernels of their own before the head kernel (one CTA for the
// compaction, a warp per row for the gather) this took 16 us of every step, in which the memory
// system idled; here the head's first tiles stream into shared memory meanwhile.
#pragma once

#include "head_plan.h"
#include "ptx.cuh"
#include "rpd_internal.h"
#include "step_common.cuh"

namespace rpd {
namespace {

static_assert(sizeof(PassInfo) == 32, "kHeadMaskBytes");

struct MaskMap {
    uint32_t *words;   // [kMaskWords] scored positions, flat index b * N + i
    uint16_t *before;  // [kMaskWords + 1] set bits before each word; the total after the last
    PassInfo *pass;

    // Compact index of flat position i (also the count before any i <= B * N).
    __device__ __forceinline__ int rank(int i) const {
        const uint32_t below = (i & 31) ? words[i >> 5] & ((1u << (i & 31)) - 1u) : 0u;
        return before[i >> 5] + __popc(below);
    }
    __device__ __forceinline__ bool scored(int i) const { return (words[i >> 5] >> (i & 31)) & 1u; }
    // Flat position of compact index q < total.
    __device__ __forceinline__ int position(int q, int num_words) const {
        int lo = 0, hi = num_words;  // before[lo] <= q < before[hi]
#pragma unroll 1
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (before[mid] <= q) lo = mid; else hi = mid;
        }
        uint32_t w = words[lo];
#pragma unroll 1
        for (int n = q - before[lo]; n > 0; --n) w &= w - 1;  // drop the set bits before it
        return lo * 32 + __ffs(w) - 1;
    }
};

// The bits of 4 mask bytes (nonzero = masked), byte i at bit i.
__device__ __forceinline__ uint32_t mask_bits4(uint32_t v) {
    return ((__vcmpne4(v, 0u) & 0x01010101u) * 0x10204080u) >> 28;
}

// The bitmap of the scored positions (every masked one, or with RPD-block each canvas's active
// block) and its prefix counts; the whole CTA, `scratch`: kMaxBatch ints of shared memory.
// Returns the number of scored positions.
__device__ __forceinline__ int compact_mask(const CompactParams &p, const MaskMap &map, int *scratch) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int total = p.B * p.N;
    const int num_words = (total + 31) >> 5;
    // 16 positions per thread and step: one 16-byte load where the mask allows it
    const bool aligned = (reinterpret_cast<uintptr_t>(p.mask) & 15u) == 0;
    uint16_t *halves = reinterpret_cast<uint16_t *>(map.words);
    for (int h = tid; h < 2 * num_words; h += blockDim.x) {
        const int i0 = h * 16;
        uint32_t bits = 0;
        if (aligned && i0 + 16 <= total) {
            const uint4 v = *reinterpret_cast<const uint4 *>(p.mask + i0);
            bits = mask_bits4(v.x) | mask_bits4(v.y) << 4 | mask_bits4(v.z) << 8 | mask_bits4(v.w) << 12;
        } else {
            uint8_t v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = i0 + j < total ? p.mask[i0 + j] : 0;
#pragma unroll
            for (int j = 0; j < 16; ++j) bits |= (v[j] != 0 ? 1u : 0u) << j;
        }
        halves[h] = static_cast<uint16_t>(bits);
    }
    __syncthreads();
    if (p.block > 0) {
        // first masked position of each canvas, rounded down to its block
        for (int b = tid; b < p.B; b += blockDim.x) {
            const int first = b * p.N, end = first + p.N;
            int lo = p.N;
            for (int w = first >> 5; w <= (end - 1) >> 5 && lo == p.N; ++w) {
                uint32_t v = map.words[w];
                if (w == first >> 5) v &= 0xffffffffu << (first & 31);
                if (v) lo = min(p.N, w * 32 + __ffs(v) - 1 - first);
            }
            scratch[b] = lo < p.N ? lo / p.block * p.block : p.N;
        }
        __syncthreads();
        for (int w = tid; w < num_words; w += blockDim.x) {
            uint32_t keep = 0;
            const int i1 = min(total, w * 32 + 32);
            for (int i = w * 32; i < i1;) {  // the canvases that this word touches
                const int b = i / p.N, end = min(i1, (b + 1) * p.N);
                const int from = max(i, b * p.N + scratch[b]);
                const int to = static_cast<int>(min(static_cast<long long>(end),
                                                    static_cast<long long>(b) * p.N + scratch[b] + p.block));
                if (from < to) keep |= (0xffffffffu >> (32 - (to - from))) << (from & 31);
                i = end;
            }
            map.words[w] &= keep;
        }
        __syncthreads();
    }
    if (warp == 0) {
        constexpr int kPerLane = kMaskWords / 32;
        int n[kPerLane], sum = 0;
#pragma unroll
        for (int j = 0; j < kPerLane; ++j) {
            const int w = lane * kPerLane + j;
            n[j] = w < num_words ? __popc(map.words[w]) : 0;
            sum += n[j];
        }
        int at = warp_inclusive_scan(sum, lane) - sum;
#pragma unroll
        for (int j = 0; j < kPerLane; ++j) {
            map.before[lane * kPerLane + j] = static_cast<uint16_t>(at);
            at += n[j];
        }
        if (lane == 31) map.before[kMaskWords] = static_cast<uint16_t>(at);
    }
    __syncthreads();
    return map.before[kMaskWords];
}

// The plan of a pass that the kernel compacts itself; one warp.
__device__ __forceinline__ HeadPlan pass_plan(const CompactParams &p, const StepPlan &plan, long long rows) {
    return rows <= kStepPlanRows ? step_plan(plan, rows) : table_plan(rows, p.plan, p.plan_rows);
}

// Which window layers the step's first pass projects; one warp.  Automatic choice: lazy when its
// two passes (the final layer of every position, then the earlier layers of an assumed band
// fraction) are estimated cheaper than one pass over all layers.
__device__ __forceinline__ bool choose_lazy(const CompactParams &p, const StepPlan &plan, int masked) {
    if (p.lazy != 2 || p.K <= 1) return p.lazy == 1 && p.K > 1;
    const float e_all = pass_plan(p, plan, static_cast<long long>(p.K) * masked).est;
    const float e_fin = pass_plan(p, plan, masked).est;
    const float e_band = pass_plan(p, plan, static_cast<long long>(kLazyBandGuess * (p.K - 1) * masked)).est;
    return e_fin + e_band < e_all;
}

// What the kernels after this one read of the compaction.  The maps: every warp of the grid writes
// its share (positions first, first + step, ...), and the grid's end is all that their readers wait
// for.  By one warp, which the merge waited for, the maps of 8192 positions took some 25 us of a step.
__device__ __forceinline__ void publish_maps(const CompactParams &p, const MaskMap &map, int first, int step) {
    const int total = p.B * p.N;
    for (int i = first; i < total; i += step) {
        const int q = map.rank(i);
        const bool on = map.scored(i);
        p.q_of_pos[i] = on ? q : -1;
        if (on) p.pos_of_q[q] = i;
    }
}

// The pass, by one thread of the grid; the second pass's takes its place after the merge.
__device__ __forceinline__ void publish_pass(const CompactParams &p, const PassInfo &pass) {
    p.meta[kMetaMasked] = pass.masked;
    p.meta[kMetaRows] = pass.rows;
    p.meta[kMetaRowsTotal] = pass.rows;
    p.meta[kMetaSel] = pass.sel;
    p.meta[kMetaLayer0] = pass.layer0;
    p.meta[kMetaLazy] = pass.lazy;
    p.meta[kMetaHeadMode] = pass.mode;
    p.meta[kMetaSplits] = pass.splits;
    p.meta[kMetaSwapRows] = pass.swap_rows;
}

// bf16(a * b) of both halves, one rounding (the product of two bf16 is exact in fp32).
__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

__device__ __forceinline__ float add_squares(uint32_t h, float ss) {
    const float lo = __uint_as_float(h << 16), hi = __uint_as_float(h & 0xffff0000u);
    return fmaf(hi, hi, fmaf(lo, lo, ss));
}

constexpr int kVecPerLane = 4;  // 16-byte vectors of a row a lane has in registers at a time

// Rows r .. r + kRows - 1 of the pass from `src` (null: left out, the first is there); one warp.  The
// rows were prefetched into L2 and are walked in short steps: this code runs a few times per launch on
// instructions that the previous step's stream through L2 has evicted, and as one unrolled block (16 KB
// of them) it took 10 us a row, nearly all of it instruction fetches.
template <int kRows>
__device__ __forceinline__ void gather_row(const NormParams &p, int r, const uint4 *const (&src)[kRows],
                                           int lane) {
    const int nvec = p.d >> 3;  // 8 bf16 per 16-byte vector
    const uint4 *__restrict__ gvec = reinterpret_cast<const uint4 *>(p.gain);
    uint4 *__restrict__ dst = reinterpret_cast<uint4 *>(p.u + static_cast<size_t>(r) * p.d);
    float ss[kRows];
#pragma unroll
    for (int i = 0; i < kRows; ++i) ss[i] = 0.f;
#pragma unroll 1
    for (int v0 = lane; v0 < nvec; v0 += 32 * kVecPerLane) {
        uint4 hv[kRows][kVecPerLane], gv[kVecPerLane];
#pragma unroll
        for (int j = 0; j < kVecPerLane; ++j) {
            const int v = v0 + 32 * j;
#pragma unroll
            for (int i = 0; i < kRows; ++i)
                if (v < nvec && (i == 0 || src[i])) hv[i][j] = __ldcs(src[i] + v);
            if (v < nvec) gv[j] = __ldg(gvec + v);
        }
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            if (i > 0 && !src[i]) break;
#pragma unroll
            for (int j = 0; j < kVecPerLane; ++j) {
                const int v = v0 + 32 * j;
                if (v >= nvec) break;
                const uint4 h = hv[i][j];
                ss[i] = add_squares(h.w, add_squares(h.z, add_squares(h.y, add_squares(h.x, ss[i]))));
                // g*h of two bf16 values rounded once to bf16 (reading D1)
                dst[i * static_cast<size_t>(nvec) + v] =
                    make_uint4(mul_bf16x2(h.x, gv[j].x), mul_bf16x2(h.y, gv[j].y),
                               mul_bf16x2(h.z, gv[j].z), mul_bf16x2(h.w, gv[j].w));
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < kRows; ++i) ss[i] += __shfl_xor_sync(0xffffffffu, ss[i], o);
#pragma unroll
    for (int i = 0; i < kRows; ++i)
        if (lane == i && (i == 0 || src[i])) p.inv_rms[r + i] = 1.0f / sqrtf(ss[i] / static_cast<float>(p.d) + p.eps);
}

// Rows a warp claims at a time: one while every warp of the grid can have its own, several (each
// row's reads then overlap its predecessor's work) in larger passes.
__device__ __forceinline__ int rows_per_claim(int rows, int warps) {
    return max(1, min(8, rows / (2 * warps)));
}

// Claim and gather rows of the pass until none is left, starting with the claim made before; one
// warp.  Compact index -> position through `map`, or through the lists in global memory when
// num_words is 0.  The rows are counted once the warp has no more of them.
//
// kPlain (the plain step), or a row a claim: one at a time.  The general kernel, whose batches have tens
// of thousands, finds the positions of a claim's rows in as many lanes and keeps two rows in flight: one
// after another a row took a warp 0.78 us of waiting (131072 rows of d = 64, 256 entries: 201 us, now 123).
template <bool kPlain>
__device__ __forceinline__ void gather_rows(const NormParams &p, const MaskMap &map, int num_words,
                                            int rows, int sel, int layer0, int claim, int per_claim,
                                            int32_t *meta, int lane) {
    const int nvec = p.d >> 3;
    auto source = [&](int r) -> const uint4 * {  // null if out of bounds
        const int kr = r / sel;
        const int sr = r - kr * sel;
        int pos;
        if (kPlain || num_words > 0) {
            pos = map.position(sr, num_words);
        } else {
            const int q = p.sel_list ? p.sel_list[sr] : sr;
            pos = rpd_check(q >= 0 && q < p.BN, meta + kMetaStatus) ? p.pos_of_q[q] : -1;
        }
        if (!rpd_check(pos >= 0 && pos < p.BN, meta + kMetaStatus)) return nullptr;
        return reinterpret_cast<const uint4 *>(p.hidden + (static_cast<size_t>(layer0 + kr) * p.BN + pos) * p.d);
    };
    auto prefetch = [&](const uint4 *src) {
        if (!src) return;
#pragma unroll 1
        for (int v = lane * 8; v < nvec; v += 32 * 8) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + v));
    };
    int done = 0;
    while (claim * per_claim < rows) {
        const int r0 = claim * per_claim, r1 = min(rows, r0 + per_claim);
        int next = 0;
        if (lane == 0) next = atomicAdd(&meta[kMetaRowNext], 1);  // its latency hides behind the rows
        if (kPlain || per_claim == 1) {
            const uint4 *src[1] = {source(r0)};
            prefetch(src[0]);
#pragma unroll 1
            for (int r = r0; r < r1; ++r) {
                const uint4 *ahead = r + 1 < r1 ? source(r + 1) : nullptr;
                prefetch(ahead);
                if (src[0]) gather_row<1>(p, r, src, lane);  // warp-uniform
                src[0] = ahead;
            }
        } else {
            const uint4 *mine = lane < r1 - r0 ? source(r0 + lane) : nullptr;  // at most 8 rows
            auto of = [&](int r) {  // of row r, in every lane
                const unsigned long long a =
                    __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(mine), (r - r0) & 31);
                return reinterpret_cast<const uint4 *>(r < r1 ? a : 0ull);
            };
            prefetch(of(r0));
            prefetch(of(r0 + 1));
#pragma unroll 1
            for (int r = r0; r < r1; r += 2) {
                const uint4 *src[2] = {of(r), of(r + 1)};
                prefetch(of(r + 2));
                prefetch(of(r + 3));
                if (src[0]) gather_row<2>(p, r, src, lane);
            }
        }
        done += r1 - r0;
        claim = __shfl_sync(0xffffffffu, next, 0);
    }
    if (done > 0) {
        proxy_fence_global();  // u is read by TMA
        __syncwarp();
        if (lane == 0) counter_add_release(&meta[kMetaRowsDone], done);
    }
}

}  // namespace
}  // namespace rpd
