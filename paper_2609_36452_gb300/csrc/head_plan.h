// head_plan.h - the choice of the head kernel's tiling and vocabulary split count for a
// projection pass of `rows` rows, and the order of its work units (host and device).  It changes no computed quantity, only
// how the contraction is laid out on the GPU.
//
// It is evaluated on the host: for passes of up to kStepPlanRows rows into an argument of the head
// kernel, for larger ones into a context's device table (every row count up to kPlanRows, then
// every 256th).  On the device a search over the split counts cost 4 to 9 us of every step's
// critical path.
#pragma once

#include <cmath>
#include <cstring>

#include "rpd_internal.h"

namespace rpd {

static_assert(sizeof(HeadPlan) == 16, "a plan is one 16-byte table entry");

__host__ __device__ inline unsigned float_bits(float x) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    unsigned u;
    std::memcpy(&u, &x, sizeof(u));
    return u;
#endif
}

__host__ __device__ inline float bits_float(unsigned u) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float x;
    std::memcpy(&x, &u, sizeof(x));
    return x;
#endif
}

// Smallest (time, g) over split counts g <= gmax of `tiles` x g work units on `slots` persistent
// pairs: waves x (tiles-per-unit x tile_cost + unit_cost), packed so that the smaller key is the
// smaller time, then the smaller g.  Of the counts with the same tiles per unit only the smallest can win.
__host__ __device__ inline unsigned long long best_split_key(float tile_cost, int tiles, int slots,
                                                             int num_n, int gmax, float unit_cost = 0.f) {
    unsigned long long key = ~0ull;
    for (int g = 1; g <= gmax;) {
        const int per = (num_n + g - 1) / g;
        const int waves = (tiles * g + slots - 1) / slots;
        const float cost = static_cast<float>(waves) * static_cast<float>(per) * tile_cost +
                           static_cast<float>(waves) * unit_cost;
        const unsigned long long k = (static_cast<unsigned long long>(float_bits(cost)) << 20) |
                                     static_cast<unsigned>(g);
        key = k < key ? k : key;
        if (per == 1) break;
        g = (num_n + per - 2) / (per - 1);
    }
    return key;
}

// Time of one "rows on N" tile (256 vocabulary entries x a group of `ng` rows on a CTA pair)
// in tile units (the measured calibration of rpd_internal.h).
__host__ __device__ inline float swap_tile_cost(int ng) {
    return ng <= kPairTileM ? kSwapTileBase + kSwapTilePerRow * static_cast<float>(ng)
                            : kSwapWideTileBase + kSwapWideTilePerRow * static_cast<float>(ng);
}

// Rows-on-N groups of a pass: as few as possible (every group streams the whole head through
// its SMs; measured on GB300, groups of 256 rows or fewer never beat pair tiles), equal,
// padded to a multiple of kSwapRowStep.
__host__ __device__ inline int swap_groups(long long rows) {
    return static_cast<int>((rows + kSwapMaxRows - 1) / kSwapMaxRows);
}
__host__ __device__ inline int swap_group_rows(long long rows, int groups) {
    const long long per = (rows + groups - 1) / groups;
    return static_cast<int>((per + kSwapRowStep - 1) / kSwapRowStep * kSwapRowStep);
}

// The plan from the best keys of both tilings: each estimate is the larger of its MMA time and
// the head streaming time scaled by the vocabulary share of its largest split (and, for pair
// tiles, by their slower streaming); the cheaper wins (equal estimates go to the one with less
// MMA work), or the one `force` names.
__host__ __device__ inline HeadPlan plan_from_keys(const HeadPlanInputs &in, unsigned long long key2,
                                                   unsigned long long key3, int ng3) {
    auto est_of = [&](float t, int g, float stream) {
        const float per = static_cast<float>((in.num_n + g - 1) / g);
        const float hbm = stream * in.hbm_tiles * per * static_cast<float>(g) / static_cast<float>(in.num_n);
        return t > hbm ? t : hbm;
    };
    const int g2 = static_cast<int>(key2 & 0xFFFFFull);
    const float t2 = bits_float(static_cast<unsigned>(key2 >> 20));
    const float e2 = est_of(t2, g2, kPairStreamFactor);
    HeadPlan pair{kHeadModePair, g2, 0, e2};
    if (key3 == ~0ull || in.force == RPD_TILING_PAIR) return pair;
    const int g3 = static_cast<int>(key3 & 0xFFFFFull);
    const float t3 = bits_float(static_cast<unsigned>(key3 >> 20));
    const float e3 = est_of(t3, g3, 1.f);
    const bool rows_n = in.force == RPD_TILING_ROWS_N || e3 < e2 || (e3 == e2 && t3 < t2);
    return rows_n ? HeadPlan{kHeadModeRowsN, 2 * g3, ng3, e3} : pair;
}

// The plan of a pass of `rows` rows.
__host__ __device__ inline HeadPlan plan_head(long long rows, const HeadPlanInputs &in) {
    if (rows <= 0 || in.pair_slots <= 0) return HeadPlan{kHeadModePair, 1, 0, 0.f};
    const int tiles2 = static_cast<int>((rows + kPairTileM - 1) / kPairTileM);
    const int gmax2 = in.num_n < in.max_splits ? in.num_n : in.max_splits;
    const unsigned long long key2 =
        best_split_key(kPairTileCost, tiles2, in.pair_slots, in.num_n, gmax2);
    const int gmax3 = in.num_n < in.max_splits / 2 ? in.num_n : in.max_splits / 2;
    const int groups = swap_groups(rows);
    const int ng = swap_group_rows(rows, groups);
    const unsigned long long key3 =
        gmax3 > 0 ? best_split_key(swap_tile_cost(ng), groups, in.pair_slots, in.num_n, gmax3)
                  : ~0ull;
    return plan_from_keys(in, key2, key3, ng);
}

// Row groups of a pass of more than one group, with their sizes weighed against pair tiles once
// more: plan_head has as few groups as possible, but smaller ones may fit the rows better (1068
// rows: five groups of 224 leave 52 rows of padding, five pair tiles 212).  Time per tile in pair
// tiles' time, at groups that share the head's tiles through L2 (measured with 2 to 6 groups of
// 96 to 512 rows at the LLaDA head, d = 4096; in the power-limited steady state, where the clock
// follows the work, the differences are larger: 1068 rows 732 us with pair tiles, 704 with groups of 224).
//
// The table is of d = 4096.  A tile's contraction grows with d, its epilogue does not, and that of a
// row group (which transposes its logits) costs more than a pair tile's: groups of 224 and 288 rows
// against pair tiles took 1.49, 1.40, 1.33, 1.22, 1.21, 1.09 times the table at d = 64, 128, 256, 512,
// 1024, 2048, which 0.08 per halving of d follows.  With the table alone 1088 rows of d = 64 at the
// LLaDA vocabulary took 122 us in groups, which pair tiles do in 90.
inline float group_tile_cost(int ng, int d) {
    // groups of 32, 64, ..., 512 rows
    constexpr float kCost[kSwapMaxRows / kSwapRowStep] = {0.70f, 0.70f, 0.72f, 0.74f, 0.79f, 0.85f,
                                                          0.94f, 1.05f, 1.22f, 1.41f, 1.57f, 1.68f,
                                                          1.95f, 2.05f, 2.16f, 2.30f};
    const float shallow = d < 4096 ? 1.f + 0.08f * std::log2(4096.f / static_cast<float>(d)) : 1.f;
    return kCost[ng / kSwapRowStep - 1] * shallow;
}
// What a unit of either tiling costs beside its tiles (the partials, and with row groups the
// combination of the sub-partitions and its barriers): about 1.2 and 3.2 us whatever the depth, in
// pair tiles' time, which is 21.5 us at d = 4096 and no less than 2.25 us.  Without it 1216 rows of
// d = 1024 and 8192 entries took 36.7 us in groups (32.1 in pair tiles), and 1568 rows of d = 256 at the
// LLaDA vocabulary 189 us in 247 ranges of two pair tiles (136 in 21 ranges).
inline float unit_cost(float at_4096, int d) { return at_4096 * std::fmin(4096.f / static_cast<float>(d), 9.5f); }
constexpr float kPairUnitCost = 0.055f, kGroupUnitCost = 0.15f;
// Up to 2048 rows: with more, pair tiles' padding is under an eighth.
constexpr int kRegroupMaxGroups = 8;

inline HeadPlan regroup_plan(const HeadPlan &plan, long long rows, const HeadPlanInputs &in) {
    const int gmax = (in.num_n < in.max_splits / 2 ? in.num_n : in.max_splits / 2);
    if (!in.regroup || in.force != RPD_TILING_AUTO || rows <= kSwapMaxRows || in.pair_slots <= 0 || gmax <= 0 ||
        rows > static_cast<long long>(kRegroupMaxGroups) * kPairTileM)
        return plan;
    const int tiles2 = static_cast<int>((rows + kPairTileM - 1) / kPairTileM);
    unsigned long long best = best_split_key(1.f, tiles2, in.pair_slots, in.num_n,
                                             in.num_n < in.max_splits ? in.num_n : in.max_splits,
                                             unit_cost(kPairUnitCost, in.d));
    HeadPlan chosen{kHeadModePair, static_cast<int>(best & 0xFFFFFull), 0, plan.est};
    for (int groups = swap_groups(rows); groups <= kRegroupMaxGroups; ++groups) {
        const int ng = swap_group_rows(rows, groups);
        const unsigned long long key =
            best_split_key(group_tile_cost(ng, in.d), groups, in.pair_slots, in.num_n, gmax,
                           unit_cost(kGroupUnitCost, in.d));
        if (key >> 20 >= best >> 20) continue;
        best = key;
        chosen = HeadPlan{kHeadModeRowsN, 2 * static_cast<int>(key & 0xFFFFFull), ng, plan.est};
    }
    return chosen;
}

// Pair tiles in whole waves over the CTA pairs and a rest of at most half a wave: the rest runs as
// half tiles (128 vocabulary entries), two to a tile, in about half a wave.  Every whole tile is then a
// unit of its own, and each row has two partials per vocabulary tile, which the scratch must hold
// (heads of up to 38912 entries on 152 SMs) and the merge must read.
//
// That pays where nothing but the rest is left to run: 200 rows over 20 and 30 tiles take 33.4 and 25.9
// us whole, 29.8 and 23.2 halved (d = 4096 and 2048; at d = 128, where a tile is mostly epilogue, 15.2 and
// 15.3).  After whole waves the units and partials cost most of what half a wave saves, or more:
//   d = 4096, several row tiles, 2.1 and 2.5 waves: 70.7 -> 68.6, 75.2 -> 74.3 us; 3.4 and 5.3 waves: 90.5 ->
//   92.4, 141.9 -> 144.8; one row tile (bound by reading the head), 1.4 waves: 53.5 -> 54.4;
//   d = 2048, 2.5 and 7.4 waves: 45.2 -> 45.8, 98.0 -> 104.4;  d = 512, 2.4 and 4.1: 26.8 -> 29.8, 33.0 -> 38.6;
//   d = 128, 2.5 and 7.4: 23.2 -> 25.3, 35.9 -> 49.2.
struct TailSplit {
    int whole, units;  // tiles in whole waves; work units in all
};
__host__ __device__ inline TailSplit tail_split(int tiles, int pairs) {
    const int rest = tiles % pairs;
    return TailSplit{tiles - rest, tiles + rest};
}
constexpr int kTailAfterWavesDepth = 4096;  // from this d on also after up to two whole waves

inline HeadPlan split_tail(const HeadPlan &plan, long long rows, const HeadPlanInputs &in) {
    if (!in.regroup || in.force != RPD_TILING_AUTO || plan.mode != kHeadModePair || in.pair_slots <= 0 ||
        rows <= 0 || 2 * in.num_n > in.max_splits)
        return plan;
    const long long tiles = (rows + kPairTileM - 1) / kPairTileM * in.num_n;
    const int rest = static_cast<int>(tiles % in.pair_slots);
    const bool after_waves = in.d >= kTailAfterWavesDepth && rows > kPairTileM && tiles < 3ll * in.pair_slots;
    if (rest == 0 || 2 * rest > in.pair_slots || (tiles >= in.pair_slots && !after_waves)) return plan;
    return HeadPlan{kHeadModePair, 2 * in.num_n, kSplitTail, plan.est};
}

// The kernel argument with the plans of every pass of up to kStepPlanRows rows; `plan(rows)`.
// (rows past max_rows, a multiple of 32, do not occur.)
template <typename Plan>
inline void fill_step_plan(StepPlan &p, int max_rows, Plan plan) {
    for (int i = 0; i < kStepPlanRows / 32 && 32 * i < max_rows; ++i) {
        const HeadPlan hp = plan(32 * (i + 1));
        p.splits[i] = hp.mode == kHeadModeRowsN ? -hp.splits : hp.splits;
        p.swap_rows[i] = static_cast<uint16_t>(hp.swap_rows);
        p.est[i] = hp.est;
    }
}

// Work units (row tile m, vocabulary split g) in the order the persistent CTAs take them:
// row tiles are grouped into bands of `band` tiles; inside a band m runs fastest, then g.
// The units running at the same time therefore share W tiles (each streamed from HBM once
// per band) and re-read at most `band` u tiles (kept in L2 while the band runs).  With few
// row tiles there is a single band and the order is plain (m fastest).
// With a split tail every unit is one tile, and those after the last whole wave are half tiles.
struct TileWalk {
    int num_m, num_n, splits, units, band;
    int whole;  // units before the half tiles
    __host__ __device__ __forceinline__ void init(int rows, int tile_rows, int V, int d, int g, bool tail, int pairs) {
        num_m = (rows + tile_rows - 1) / tile_rows;
        num_n = (V + kTileN - 1) / kTileN;
        splits = tail ? num_n : g;
        units = num_m * splits;
        whole = units;
        if (tail) {
            const TailSplit t = tail_split(units, pairs);
            whole = t.whole;
            units = t.units;
        }
        band = static_cast<int>(kBandBytes / 2) / tile_rows / d;
        band = band < num_m ? band : num_m;
        band = band > 1 ? band : 1;
    }
    // A unit's vocabulary range is given in half tiles [v0, v1); an odd one is a half tile.
    __host__ __device__ __forceinline__ void unit(int u, int &m, int &g, int &v0, int &v1) const {
        const int half = u - whole;  // of tile whole + half / 2
        if (half >= 0) u = whole + (half >> 1);
        const int per_band = band * splits;
        const int b = u / per_band;
        const int r = u - b * per_band;
        const int m0 = b * band;
        const int in_band = band < num_m - m0 ? band : num_m - m0;
        m = m0 + r % in_band;
        g = r / in_band;
        // at most a few hundred splits of at most 2^23 tiles: the products fit 32 bits
        v0 = 2 * static_cast<int>(static_cast<unsigned>(g) * num_n / splits);
        v1 = 2 * static_cast<int>(static_cast<unsigned>(g + 1) * num_n / splits);
        if (half >= 0) {
            v0 += half & 1;
            v1 = v0 + 1;
        }
    }
};

// The plan of a pass from plan_head's (a function of the multiple of 32 rows).
inline HeadPlan refine_plan(const HeadPlan &plan, long long rows, const HeadPlanInputs &in) {
    if (rows > static_cast<long long>(kRegroupMaxGroups) * kPairTileM) return plan;
    return split_tail(regroup_plan(plan, rows, in), rows, in);
}

#ifdef __CUDACC__
// A pass's plan from a step's kernel argument (0 <= rows <= kStepPlanRows).
__device__ inline HeadPlan step_plan(const StepPlan &p, long long rows) {
    if (rows <= 0) return HeadPlan{kHeadModePair, 1, 0, 0.f};
    const int i = static_cast<int>(rows - 1) / 32;
    return HeadPlan{p.splits[i] < 0 ? kHeadModeRowsN : kHeadModePair, abs(p.splits[i]), p.swap_rows[i], p.est[i]};
}

// A pass's plan from a context's tables: one entry per row count up to table_rows, then one per
// 256 rows (the plan of the most rows with that many pair tiles, its groups fitted to the rows).
__device__ inline HeadPlan table_plan(long long rows, const HeadPlan *table, int table_rows) {
    if (rows <= table_rows) return table[rows];
    HeadPlan hp = table[table_rows + (rows + kPairTileM - 1) / kPairTileM - table_rows / kPairTileM];
    if (hp.mode == kHeadModeRowsN) hp.swap_rows = swap_group_rows(rows, swap_groups(rows));
    return hp;
}
#endif

}  // namespace rpd
