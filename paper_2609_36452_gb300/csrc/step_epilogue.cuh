// step_epilogue.cuh - what follows the contraction: the merge of the split statistics of each row
// (argmax, its probability, entropy; Eq. 1), and the scoring, candidate flags, entropy prefix
// scan and commitment of a canvas (§3).
//
// The head kernel runs both after its last tile: its CTAs claim blocks of rows to merge, and the
// one that completes the merge scores the canvas (a single one; several, and a long one, are scored by
// k_score_commit, a CTA each).
//
// Both parts are bound by latency: a handful of dependent trips to L2 and, because the head's
// stream has evicted the instructions by then, the fetching of their code.  So the code is kept
// short (rolled loops over shared memory rather than unrolled ones over registers), and loads
// that do not depend on one another are issued together.
#pragma once

#include "ptx.cuh"
#include "rpd_internal.h"
#include "step_common.cuh"

namespace rpd {
namespace {

// ------------------------------------------------------------------------------ merge

// Lanes per row: the smallest power of two keeping at most 8 partials per lane, at most a warp.
__device__ __forceinline__ int merge_lanes(int splits) {
    int gs = 1;
    while (gs < 32 && gs * 8 < splits) gs <<= 1;
    return gs;
}

// Merge the split partials of rows [block * groups, +groups) of the pass, groups = blockDim.x / gs,
// and store each row's argmax, its probability 1/s and the entropy H = ln s - ln2 * t / s (Eq. 1)
// at layer * masked + q.  A row is handled by a group of gs lanes: each folds every gs-th partial,
// then the lanes combine in a fixed order (the result does not depend on which CTA merges).
// `sel_list`: compact index of the pass's s-th position (null: s itself); `position`: canvas
// position of a compact index (only for vocabulary shards).
// kPlain: no list and no shards.
template <bool kPlain, typename Position>
__device__ __forceinline__ void merge_block(const MergeArgs &mg, const PassInfo &pass,
                                            const int32_t *sel_list, int block, int gs,
                                            const int32_t *status, Position position) {
    const int groups = blockDim.x / gs;
    const int gid = threadIdx.x / gs, gl = threadIdx.x % gs;
    const int row = block * groups + gid;
    const bool valid = row < pass.rows && rpd_check(pass.splits <= mg.max_splits, status);
    Stat acc{-INFINITY, 0.f, 0.f, 0x7fffffff};
    if (valid) {
        const float4 *part = mg.partials + static_cast<size_t>(row) * mg.max_splits;
#pragma unroll 1
        for (int g0 = gl; g0 < pass.splits; g0 += 4 * gs) {
            float4 v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)  // past the last: an empty partial
                v[j] = g0 + j * gs < pass.splits ? __ldcg(part + g0 + j * gs) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                acc = merge2(acc, Stat{v[j].x, v[j].y, v[j].z, __float_as_int(v[j].w)});
        }
    }
#pragma unroll 1
    for (int o = gs >> 1; o > 0; o >>= 1) {
        Stat other;
        other.m = __shfl_xor_sync(0xffffffffu, acc.m, o, gs);
        other.s = __shfl_xor_sync(0xffffffffu, acc.s, o, gs);
        other.t = __shfl_xor_sync(0xffffffffu, acc.t, o, gs);
        other.a = __shfl_xor_sync(0xffffffffu, acc.a, o, gs);
        const bool upper = gl & o;  // fixed operand order
        acc = merge2(upper ? other : acc, upper ? acc : other);
    }
    if (valid && gl == 0) {
        const int kr = row / pass.sel;
        const int s = row - kr * pass.sel;
        const int q = !kPlain && sel_list ? sel_list[s] : s;
        if (!kPlain && mg.shard_out) {
            mg.shard_out[static_cast<size_t>(pass.layer0 + kr) * mg.shard_stride + position(q)] =
                make_float4(acc.m, acc.s, acc.t, __int_as_float(acc.a + mg.v_offset));
        } else {
            const size_t out = static_cast<size_t>(pass.layer0 + kr) * pass.masked + q;
            mg.row_arg[out] = acc.a;
            mg.row_pmax[out] = 1.0f / acc.s;
            mg.row_H[out] = fmaxf(logf(acc.s) - kLn2 * (acc.t / acc.s), 0.f);
        }
    }
}

// ------------------------------------------------------------------------------ band

// Lazy projection, after the final layer's pass: the compact indices of the positions whose
// confidence lies in their canvas's stability band theta_c <= c < tau (Eq. 5 reads S_i only
// there), in order; the whole CTA.  `final_p`: the final layer's probabilities by compact index;
// `canvas(q)`: the canvas of compact index q; `warp_sum`: 32 ints of shared memory.  Returns how
// many there are.
template <typename Canvas>
__device__ __forceinline__ int select_band(const float *final_p, int masked, float theta_c,
                                           const float *tau, int32_t *sel_q, int *warp_sum, Canvas canvas) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    int carry = 0;
#pragma unroll 1
    for (int base = 0; base < masked; base += blockDim.x) {
        const int q = base + threadIdx.x;
        bool in = false;
        if (q < masked) {
            const float c = __ldcg(final_p + q);
            in = c >= theta_c && c < tau[canvas(q)];
        }
        const unsigned ballot = __ballot_sync(0xffffffffu, in);
        if (lane == 0) warp_sum[warp] = __popc(ballot);
        __syncthreads();
        int at = carry;
#pragma unroll 1
        for (int w = 0; w < nwarps; ++w) {
            if (w < warp) at += warp_sum[w];
            carry += warp_sum[w];
        }
        if (in) sel_q[at + __popc(ballot & ((1u << lane) - 1u))] = q;
        __syncthreads();
    }
    return carry;
}

// ------------------------------------------------------------------------------ score

struct ScanPair {
    float q;  // entropy of masked non-candidates
    int m;    // masked positions
};

// Shared memory of the scoring of one canvas: `header` and then 13 bytes per position.
struct ScoreSmem {
    ScanPair *scan;            // [33]
    int4 *sum;                 // [32]
    int *first_reject;
    unsigned long long *best;  // fallback candidate
    float *conf, *H;           // [N] c_i, H_i
    int *y;                    // [N] argmax of the final layer
    uint8_t *flags;            // [N]
};
constexpr int kScoreHeaderBytes = 1024;
constexpr int kFlagScored = 1, kFlagCandidate = 2, kFlagHigh = 4;

__host__ __device__ inline size_t score_smem_bytes(int N) {
    return kScoreHeaderBytes + 13 * static_cast<size_t>((N + 15) / 16 * 16);
}

__device__ __forceinline__ ScoreSmem carve_score(uint8_t *base, int N) {
    const int n = (N + 15) / 16 * 16;
    ScoreSmem s;
    s.sum = reinterpret_cast<int4 *>(base);
    s.scan = reinterpret_cast<ScanPair *>(s.sum + 32);
    s.best = reinterpret_cast<unsigned long long *>(s.scan + 34);
    s.first_reject = reinterpret_cast<int *>(s.best + 1);
    s.conf = reinterpret_cast<float *>(base + kScoreHeaderBytes);
    s.H = s.conf + n;
    s.y = reinterpret_cast<int *>(s.H + n);
    s.flags = reinterpret_cast<uint8_t *>(s.y + n);
    return s;
}
static_assert(32 * 16 + 34 * 8 + 8 + 4 <= kScoreHeaderBytes, "score header");

// Exclusive scan of (q, m) in thread order over the block, plus the block totals.
__device__ __forceinline__ ScanPair block_scan_pair(ScanPair v, ScanPair *sh, ScanPair &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    auto warp_scan = [lane](ScanPair x) {
#pragma unroll 1
        for (int o = 1; o < 32; o <<= 1) {
            const float tq = __shfl_up_sync(0xffffffffu, x.q, o);
            const int tm = __shfl_up_sync(0xffffffffu, x.m, o);
            if (lane >= o) {
                x.q += tq;
                x.m += tm;
            }
        }
        return x;
    };
    const ScanPair incl = warp_scan(v);
    if (lane == 31) sh[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const ScanPair w = lane < nwarps ? sh[lane] : ScanPair{0.f, 0};
        const ScanPair wi = warp_scan(w);
        sh[lane] = ScanPair{wi.q - w.q, wi.m - w.m};
        if (lane == 31) sh[32] = wi;
    }
    __syncthreads();
    total = sh[32];
    const ScanPair base = sh[warp];
    return ScanPair{base.q + incl.q - v.q, base.m + incl.m - v.m};
}

// Block-wide sums of four counters.
__device__ __forceinline__ int4 block_sum4(int4 v, int4 *sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    v.x = __reduce_add_sync(0xffffffffu, v.x);
    v.y = __reduce_add_sync(0xffffffffu, v.y);
    v.z = __reduce_add_sync(0xffffffffu, v.z);
    v.w = __reduce_add_sync(0xffffffffu, v.w);
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    int4 t = make_int4(0, 0, 0, 0);
#pragma unroll 1
    for (int w = 0; w < nwarps; ++w) {
        t.x += sh[w].x;
        t.y += sh[w].y;
        t.z += sh[w].z;
        t.w += sh[w].w;
    }
    return t;
}

constexpr int kLayerBatch = 4;  // window layers whose statistics are loaded together

// Scores and commits canvas b with the whole CTA (positions i = b * N ...):
//   y_i = argmax of the final layer, c_i its probability, H_i its entropy;
//   K_i = window layers, counted back from the final one, whose argmax is y_i (Eq. 2,
//         stopping at the first disagreement, App. A.2);
//   r_i = max over those layers of p(y_i) - c_i (Eq. 3; inside the suffix the layer argmax
//         is y_i, so p(y_i) is that layer's maximum probability);
//   S_i = min(K_i, K_max) - w r_i (Eq. 4);  cand_i per Eq. 5;
//   Q_i = sum over j < i of H_j for masked non-candidates (block-wide exclusive scan);
//   accept the candidates before the first candidate with Q > beta.  This equals the
//   sequential rule of §3.2: H >= 0, accepted candidates are excluded from E_i, so while
//   every earlier candidate was accepted E_i = Q_i, and after the first rejection every
//   later candidate sees at least that much entropy.
//   If nothing is accepted and something is masked, commit the most confident of the
//   first W masked positions (leftmost on ties, §3.2).  Then write the outputs and clear the
//   committed mask bits.  RPD-block skips the budget and takes the fallback over the active
//   block.
// `compact_index(i)`: compact index of canvas position i, negative if it is not scored (called
// with the position's mask byte).  `clear()`: whether the committed mask bits are cleared here.  The merged row statistics are read through L2 (ld.cg): other
// CTAs of the same grid may have written them.
template <typename CompactIndex, typename Clear>
__device__ __forceinline__ void score_canvas(const ScoreParams &p, int b, float tau, float beta,
                                             const PassInfo &pass, int status, int rows_total,
                                             const ScoreSmem &sm, CompactIndex compact_index, Clear clear) {
    const int N = p.N, K = p.K;
    const int nmt = pass.masked;
    const bool lazy_on = pass.lazy != 0;  // earlier layers exist only in the band
    uint8_t *mask = p.mask + static_cast<size_t>(b) * N;
    const bool dbg_layers = p.dbg.layer_argmax || p.dbg.layer_pmax;

    int n_cand = 0, n_masked_all = 0;
#pragma unroll 1
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const size_t pos = static_cast<size_t>(b) * N + i;
        const bool is_masked = mask[i] != 0;
        // Scored positions: every masked one, or (RPD-block) the active block's masked ones,
        // which are exactly those the compaction kept.
        const int q = compact_index(i, is_masked);
        int y = -1, ki = 0;
        bool cand = false, high = false;
        float conf = 0.f, H = 0.f, r = 0.f, s = 0.f;
        if (q >= 0) {
            // Backward over the window, a batch of layers at a time (loads issued together).
            H = __ldcg(p.row_H + static_cast<size_t>(K - 1) * nmt + q);
            float peak = 0.f;
            bool run = true;
            bool projected = true;  // lazy projection: earlier layers exist only in the band
#pragma unroll 1
            for (int k_hi = K; k_hi > 0; k_hi -= kLayerBatch) {
                if (!run && !dbg_layers) break;  // persistence settled; debug wants every layer
                int a_b[kLayerBatch];
                float p_b[kLayerBatch];
#pragma unroll
                for (int t = 0; t < kLayerBatch; ++t) {
                    const int k = max(k_hi - 1 - t, 0);
                    const size_t rk = static_cast<size_t>(k) * nmt + q;
                    a_b[t] = __ldcg(p.row_arg + rk);
                    p_b[t] = __ldcg(p.row_pmax + rk);
                }
#pragma unroll
                for (int t = 0; t < kLayerBatch; ++t) {
                    const int k = k_hi - 1 - t;
                    if (k < 0) break;
                    if (k == K - 1) {
                        y = a_b[t];
                        conf = p_b[t];
                        peak = conf;
                        ki = 1;
                        // outside the band K_i and r_i are not needed
                        projected = !lazy_on || (conf >= p.theta_c && conf < tau);
                        run = projected;
                    } else if (!projected) {
                        a_b[t] = -1;
                        p_b[t] = 0.f;
                    } else if (run) {
                        run = a_b[t] == y;
                        if (run) {
                            ++ki;
                            peak = fmaxf(peak, p_b[t]);
                        }
                    }
                    if (dbg_layers) {
                        const size_t o = (static_cast<size_t>(k) * p.B) * N + pos;
                        if (p.dbg.layer_argmax) p.dbg.layer_argmax[o] = a_b[t];
                        if (p.dbg.layer_pmax) p.dbg.layer_pmax[o] = p_b[t];
                    }
                }
            }
            r = peak - conf;
            s = static_cast<float>(min(ki, p.k_max)) - p.w * r;
            high = conf >= tau;
            cand = high || (conf >= p.theta_c && conf < tau && s >= p.theta_s);
            if (!projected) {  // reported as not evaluated
                ki = 0;
                r = 0.f;
                s = 0.f;
            }
            n_cand += cand;
        } else if (dbg_layers) {
#pragma unroll 1
            for (int k = 0; k < K; ++k) {
                const size_t o = (static_cast<size_t>(k) * p.B) * N + pos;
                if (p.dbg.layer_argmax) p.dbg.layer_argmax[o] = -1;
                if (p.dbg.layer_pmax) p.dbg.layer_pmax[o] = 0.f;
            }
        }
        n_masked_all += is_masked;  // (after the loads that do not need it)
        sm.conf[i] = conf;
        sm.H[i] = H;
        sm.y[i] = y;
        sm.flags[i] = static_cast<uint8_t>((q >= 0 ? kFlagScored : 0) | (cand ? kFlagCandidate : 0) |
                                           (high ? kFlagHigh : 0));
        if (p.dbg.conf) p.dbg.conf[pos] = conf;
        if (p.dbg.entropy) p.dbg.entropy[pos] = H;
        if (p.dbg.persist) p.dbg.persist[pos] = ki;
        if (p.dbg.drop) p.dbg.drop[pos] = r;
        if (p.dbg.stability) p.dbg.stability[pos] = s;
        if (p.dbg.candidate) p.dbg.candidate[pos] = cand;
    }
    if (threadIdx.x == 0) {
        *sm.first_reject = N;
        *sm.best = 0ull;
    }
    __syncthreads();

    // ------------------------------ entropy of masked non-candidates and masked ranks, scanned
    // (positions in blocked order across threads)
    const int items = (N + blockDim.x - 1) / blockDim.x;
    const int i0 = min(N, static_cast<int>(threadIdx.x) * items), i1 = min(N, i0 + items);
    ScanPair local{0.f, 0};  // (entropy of scored non-candidates, scored positions)
#pragma unroll 1
    for (int i = i0; i < i1; ++i) {
        const int f = sm.flags[i];
        local.m += f & kFlagScored;
        if ((f & (kFlagScored | kFlagCandidate)) == kFlagScored) local.q += sm.H[i];
    }
    ScanPair total;
    const ScanPair pre = block_scan_pair(local, sm.scan, total);  // synchronises the block
    if (p.block == 0) {  // RPD-block: no entropy budget
        float q = pre.q;
#pragma unroll 1
        for (int i = i0; i < i1; ++i) {
            const int f = sm.flags[i];
            if ((f & kFlagCandidate) && q > beta) {
                atomicMin(sm.first_reject, i);
                break;
            }
            if ((f & (kFlagScored | kFlagCandidate)) == kFlagScored) q += sm.H[i];
        }
    }
    __syncthreads();
    const int reject_at = *sm.first_reject;

    // accepted, accepted through c >= tau, candidates, masked positions of the canvas
    int4 cnt = make_int4(0, 0, n_cand, n_masked_all);
#pragma unroll 1
    for (int i = i0; i < min(i1, reject_at); ++i) {
        const int f = sm.flags[i];
        cnt.x += (f & kFlagCandidate) != 0;
        cnt.y += (f & (kFlagCandidate | kFlagHigh)) == (kFlagCandidate | kFlagHigh);
    }
    const int4 tot = block_sum4(cnt, sm.sum);
    const int fallback_window = p.block > 0 ? p.block : p.window;

    // ------------------------------------------------------------------------ fallback
    int fb_pos = -1;
    if (tot.x == 0 && total.m > 0) {  // uniform across the block
        int rank = pre.m;
        unsigned long long mine = 0ull;
#pragma unroll 1
        for (int i = i0; i < i1 && rank < fallback_window; ++i) {
            if (!(sm.flags[i] & kFlagScored)) continue;
            // c >= 0: its bit pattern orders like the value; ties -> lowest position
            const unsigned long long key =
                (static_cast<unsigned long long>(__float_as_uint(sm.conf[i])) << 32) |
                static_cast<unsigned long long>(0xFFFFFFFFu - static_cast<unsigned>(i));
            mine = key > mine ? key : mine;
            ++rank;
        }
        if (mine) atomicMax(sm.best, mine);
        __syncthreads();
        fb_pos = static_cast<int>(0xFFFFFFFFu - static_cast<unsigned>(*sm.best & 0xFFFFFFFFull));
    }

    // ------------------------------------------------------------------------- outputs
    const bool clear_now = clear();
#pragma unroll 1
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const size_t pos = static_cast<size_t>(b) * N + i;
        const bool commit = ((sm.flags[i] & kFlagCandidate) && i < reject_at) || i == fb_pos;
        p.out_commit[pos] = commit ? 1 : 0;
        if (commit) {
            p.out_token[pos] = sm.y[i];
            if (clear_now) mask[i] = 0;
        }
    }
    if (threadIdx.x == 0) {
        rpd_stats st;
        st.n_masked = tot.w;
        st.n_candidates = tot.z;
        st.n_high_conf = tot.y;
        st.n_stability = tot.x - tot.y;
        st.n_committed = tot.x + (fb_pos >= 0 ? 1 : 0);
        st.fallback_used = fb_pos >= 0 ? 1 : 0;
        st.fallback_pos = fb_pos;
        st.status = status;
        st.n_rows = rows_total;
        p.out_stats[b] = st;
    }
}

// The mask bits that score_canvas left (of a single canvas); one warp.
__device__ __forceinline__ void clear_committed(const ScoreParams &p, int lane) {
#pragma unroll 4
    for (int i = lane; i < p.N; i += 32)
        if (__ldcg(p.out_commit + i)) p.mask[i] = 0;
}

}  // namespace
}  // namespace rpd
