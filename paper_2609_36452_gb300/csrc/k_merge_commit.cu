// k_merge_commit.cu - the step's small kernels: the lazy projection's band selection, the scoring
// of several canvases or a long one, the merge of vocabulary shards and the decoding loop's stop test.
//
// k_band (one CTA; lazy projection of batches that the head kernel does not compact itself): selects
//   the positions whose final confidence lies in their canvas's stability band theta_c <= c < tau
//   (Eq. 5 reads S_i only there) and sets up the second pass over their earlier window layers.
//
// k_score_commit (one CTA per canvas): scores and commits several canvases, or one of more than
//   kFuseScoreMaxN positions (score_canvas in step_epilogue.cuh; any other single canvas is scored by
//   the head kernel itself).
#include "ptx.cuh"
#include "rpd_internal.h"
#include "step_common.cuh"
#include "step_epilogue.cuh"

namespace rpd {
namespace {

constexpr int kMergeThreads = 256;

// Merge of P vocabulary shards' statistics per (layer, masked position), shards in order.
__global__ void __launch_bounds__(kMergeThreads) k_merge_shards(ShardMergeParams p) {
    pdl_trigger();
    pdl_wait();
    const int nmt = p.meta[kMetaMasked];
    const long long total = static_cast<long long>(p.K) * nmt;
    for (long long r = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; r < total;
         r += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int k = static_cast<int>(r / nmt);
        const int q = static_cast<int>(r - static_cast<long long>(k) * nmt);
        const int pos = p.pos_of_q[q];
        Stat acc{-INFINITY, 0.f, 0.f, 0x7fffffff};
        for (int sh = 0; sh < p.P; ++sh) {
            const float4 v = p.gathered[(static_cast<size_t>(sh) * p.K + k) * p.BN + pos];
            acc = merge2(acc, Stat{v.x, v.y, v.z, __float_as_int(v.w)});
        }
        p.row_arg[r] = acc.a;
        p.row_pmax[r] = 1.0f / acc.s;
        p.row_H[r] = fmaxf(logf(acc.s) - kLn2 * (acc.t / acc.s), 0.f);
    }
}

constexpr int kBandThreads = 1024;

__global__ void __launch_bounds__(kBandThreads, 1) k_band(BandParams p) {
    __shared__ int warp_sum[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_trigger();  // successors may launch now; they wait for this grid before reading
    pdl_wait();
    const int nmt = p.meta[kMetaMasked];
    const bool lazy_on = p.meta[kMetaLazy] != 0;  // else the first pass covered every layer
    // 1. band positions, in compact order (the first pass is merged)
    const float *final_p = p.mg.row_pmax + static_cast<size_t>(p.K - 1) * nmt;
    const int carry = lazy_on ? select_band(final_p, nmt, p.theta_c, p.tau, p.sel_q, warp_sum,
                                            [&](int q) { return p.pos_of_q[q] / p.N; })
                              : 0;
    // 2. the second pass: the K-1 earlier window layers of the band positions
    const long long rows = static_cast<long long>(p.K - 1) * carry;
    if (warp == 0) {
        const HeadPlan hp = table_plan(rows, p.plan, p.plan_rows);
        if (lane == 0) {
            p.meta[kMetaSwapRows] = hp.swap_rows;
            p.meta[kMetaSplits] = hp.splits;
            p.meta[kMetaHeadMode] = hp.mode;
        }
    }
    if (tid == 0) {
        p.meta[kMetaRows] = static_cast<int>(rows);
        p.meta[kMetaSel] = carry;
        p.meta[kMetaLayer0] = 0;
        p.meta[kMetaRowsTotal] += static_cast<int>(rows);
    }
}

extern __shared__ __align__(16) uint8_t score_smem[];

__global__ void __launch_bounds__(kScoreThreads, 1) k_score_commit(const __grid_constant__ BatchScoreParams p) {
    pdl_trigger();  // successors may launch now; they wait for this grid before reading
    pdl_wait();
    const ScoreParams &c = p.canvas;
    const int b = blockIdx.x;
    PassInfo pass{};
    pass.masked = c.meta[kMetaMasked];
    pass.lazy = c.meta[kMetaLazy];
    const int published = c.meta[kMetaStepStatus];  // else one that a kernel since then latched
    const int32_t *q_of_pos = c.q_of_pos + static_cast<size_t>(b) * c.N;
    score_canvas(c, b, p.tau[b], p.budget[b], pass, published ? published : c.meta[kMetaStatus],
                 c.meta[kMetaRowsTotal], carve_score(score_smem, c.N),
                 [q_of_pos](int i, bool masked) {
                     const int q = q_of_pos[i];  // loaded with the mask byte
                     return masked ? q : -1;
                 },
                 [] { return true; });
}

}  // namespace

namespace {
// The stop test of the decoding loop: one thread counts the step and keeps the loop going
// while some canvas has more than floor(stop_frac * N) positions masked, fewer than max_steps
// steps have run and every canvas's step succeeded.
__global__ void k_loop_test(cudaGraphConditionalHandle handle, const rpd_stats *stats, int B, int N,
                            float stop_frac, int max_steps, int32_t *steps) {
    const int n = *steps + 1;
    *steps = n;
    const int limit = static_cast<int>(floorf(stop_frac * static_cast<float>(N)));
    bool ok = true, open = false;
    for (int b = 0; b < B; ++b) {
        ok = ok && stats[b].status == RPD_OK;
        open = open || stats[b].n_masked - stats[b].n_committed > limit;
    }
    cudaGraphSetConditional(handle, ok && open && n < max_steps ? 1u : 0u);
}
}  // namespace

cudaError_t launch_loop_test(cudaGraphConditionalHandle handle, const rpd_stats *stats, int B, int N,
                             float stop_frac, int max_steps, int32_t *steps, cudaStream_t s) {
    // a plain launch: it must see the finished step's statistics
    k_loop_test<<<1, 1, 0, s>>>(handle, stats, B, N, stop_frac, max_steps, steps);
    return cudaGetLastError();
}

cudaError_t launch_merge_shards(const ShardMergeParams &p, int grid, cudaStream_t s) {
    return launch_pdl(k_merge_shards, dim3(grid), dim3(kMergeThreads), 0, s, p);
}

cudaError_t launch_band(const BandParams &p, cudaStream_t s) {
    return launch_pdl(k_band, dim3(1), dim3(kBandThreads), 0, s, p);
}

cudaError_t launch_score_commit(const BatchScoreParams &p, cudaStream_t s) {
    const int N = p.canvas.N;
    const int threads = N >= kScoreThreads ? kScoreThreads : ((N + 31) / 32) * 32;
    const size_t smem = score_smem_bytes(N);
    if (smem > 48 * 1024) {  // set on the current device before every such launch
        cudaError_t e = cudaFuncSetAttribute(k_score_commit, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(smem));
        if (e != cudaSuccess) return e;
    }
    return launch_pdl(k_score_commit, dim3(p.canvas.B), dim3(threads), smem, s, p);
}

}  // namespace rpd
