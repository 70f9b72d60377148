// k_compact.cu - device-side compaction of the masked positions (App. A.6: only masked positions
// are projected) as a kernel of its own: for batches of more than kFusedMaxPositions canvas
// positions, and for the second half of a vocabulary-parallel step.  For everything smaller the
// head kernel compacts the mask itself (step_prologue.cuh).
//
// k_compact (one CTA): order-preserving compaction of mask[B][N] into compact indices
//   q = 0..NMT-1 (canvas-major, then position), the projected row
//   count R = K*NMT and the head kernel's tiling plan.  Nothing goes back to the host: later
//   kernels read these words from device memory.
#include "ptx.cuh"
#include "rpd_internal.h"
#include "step_common.cuh"

namespace rpd {
namespace {

constexpr int kCompactThreads = 1024;
constexpr int kCompactItems = 4;

__global__ void __launch_bounds__(kCompactThreads, 1) k_compact(CompactParams p) {
    __shared__ int warp_sum[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ int block_lo[kMaxBatch];  // RPD-block: first position of each canvas's active block
    pdl_trigger();  // successors may launch now; they wait for this grid before reading
    pdl_wait();
    const int total = p.B * p.N;
    if (p.block > 0) {
        for (int b = tid; b < p.B; b += kCompactThreads) block_lo[b] = p.N;
        __syncthreads();
        for (int i = tid; i < total; i += kCompactThreads)
            if (p.mask[i]) atomicMin(&block_lo[i / p.N], i % p.N);
        __syncthreads();
        for (int b = tid; b < p.B; b += kCompactThreads)
            block_lo[b] = block_lo[b] < p.N ? (block_lo[b] / p.block) * p.block : p.N;
        __syncthreads();
    }
    int carry = 0;
    for (int base = 0; base < total; base += kCompactThreads * kCompactItems) {
        const int i0 = base + tid * kCompactItems;
        int f[kCompactItems];
        int cnt = 0;
#pragma unroll
        for (int j = 0; j < kCompactItems; ++j) {
            const int i = i0 + j;
            f[j] = (i < total) ? (p.mask[i] != 0) : 0;
            if (f[j] && p.block > 0) {
                const int lo = block_lo[i / p.N], pos = i % p.N;
                f[j] = pos >= lo && pos < lo + p.block;
            }
            cnt += f[j];
        }
        const int incl = warp_inclusive_scan(cnt, lane);
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const int v = warp_sum[lane];
            const int vi = warp_inclusive_scan(v, lane);
            warp_sum[lane] = vi - v;  // exclusive prefix of warp totals
        }
        __syncthreads();
        int excl = carry + warp_sum[warp] + incl - cnt;
#pragma unroll
        for (int j = 0; j < kCompactItems; ++j) {
            const int i = i0 + j;
            if (i < total) {
                p.q_of_pos[i] = f[j] ? excl : -1;
                if (f[j]) p.pos_of_q[excl] = i;
                excl += f[j];
            }
        }
        // chunk total = exclusive prefix of the last warp + its inclusive total
        __syncthreads();
        if (tid == kCompactThreads - 1) warp_sum[0] = excl;  // running count after the chunk
        __syncthreads();
        carry = warp_sum[0];
        __syncthreads();
    }

    // First pass: every window layer of the scored positions, or only the final layer (lazy).
    // Automatic choice: lazy when its two passes (the final layer of every position, then
    // the earlier layers of an assumed band fraction) are estimated cheaper than one pass
    // over all layers.
    __shared__ int lazy_on;
    __shared__ HeadPlan plan;
    const long long all_rows = static_cast<long long>(p.K) * carry;
    if (warp == 0) {
        int lz = (p.lazy == 1 && p.K > 1) ? 1 : 0;
        if (p.lazy == 2 && p.K > 1) {
            const long long guess = static_cast<long long>(kLazyBandGuess * (p.K - 1) * carry);
            const float e_all = table_plan(all_rows, p.plan, p.plan_rows).est;
            const float e_fin = table_plan(carry, p.plan, p.plan_rows).est;
            const float e_band = table_plan(guess, p.plan, p.plan_rows).est;
            lz = (e_fin + e_band < e_all) ? 1 : 0;
        }
        const HeadPlan hp = table_plan(lz ? static_cast<long long>(carry) : all_rows, p.plan, p.plan_rows);
        if (lane == 0) {
            lazy_on = lz;
            plan = hp;
        }
    }
    __syncthreads();
    const long long rows = lazy_on ? static_cast<long long>(carry) : all_rows;
    const int mode = plan.mode, splits = plan.splits, swap_rows = plan.swap_rows;
    if (tid == 0) {
        p.meta[kMetaSwapRows] = swap_rows;
        p.meta[kMetaMasked] = carry;
        p.meta[kMetaRows] = static_cast<int>(rows);
        p.meta[kMetaSplits] = splits;
        p.meta[kMetaHeadMode] = mode;
        p.meta[kMetaSel] = carry;
        p.meta[kMetaLayer0] = lazy_on ? p.K - 1 : 0;
        p.meta[kMetaRowsTotal] = static_cast<int>(rows);
        p.meta[kMetaLazy] = lazy_on;
    }
}

}  // namespace

cudaError_t launch_compact(const CompactParams &p, cudaStream_t s) {
    return launch_pdl(k_compact, dim3(1), dim3(kCompactThreads), 0, s, p);
}

}  // namespace rpd
