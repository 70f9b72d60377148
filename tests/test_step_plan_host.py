"""The plans that a step passes to the head kernel (StepPlan, one entry per 32 rows) are those of
every row count up to its limit, the work units of each plan cover its pass exactly once, and the
search over split counts finds what trying each of them does, at the two models' heads, small and
ragged ones (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_36452_gb300", "csrc")

DRIVER = r"""
#include "head_plan.h"
#include <cstdio>
#include <cstdlib>
#include <vector>
// every split count in turn
static unsigned long long every_key(float cost1, int tiles, int slots, int num_n, int gmax) {
    unsigned long long key = ~0ull;
    for (int g = 1; g <= gmax; ++g) {
        const int per = (num_n + g - 1) / g, waves = (tiles * g + slots - 1) / slots;
        const float cost = static_cast<float>(waves) * static_cast<float>(per) * cost1;
        const unsigned long long k = (static_cast<unsigned long long>(rpd::float_bits(cost)) << 20) | unsigned(g);
        key = k < key ? k : key;
    }
    return key;
}
int main(int argc, char **argv) {
    const int V = atoi(argv[1]), d = atoi(argv[2]), sms = atoi(argv[3]), force = atoi(argv[4]);
    rpd::HeadPlanInputs in{};
    in.num_n = (V + 255) / 256;
    in.max_splits = 2 * in.num_n < 2 * sms ? 2 * in.num_n : 2 * sms;
    in.pair_slots = sms / 2;
    in.hbm_tiles = rpd::head_stream_in_tiles(V, d, sms);
    in.force = force;
    in.regroup = 1;
    in.d = d;
    if (argc > 5) {  // one pass's plan
        const rpd::HeadPlan a = rpd::refine_plan(rpd::plan_head(atoi(argv[5]), in), atoi(argv[5]), in);
        std::printf("%d %d %d\n", a.mode, a.splits, a.swap_rows);
        return 0;
    }
    auto plan = [&](int r) { return rpd::refine_plan(rpd::plan_head(r, in), r, in); };
    rpd::StepPlan sp;
    rpd::fill_step_plan(sp, rpd::kStepPlanRows, plan);
    int bad = 0;
    int tails = 0;
    for (int r = 1; r <= 4096; ++r) {  // refining keeps the plan's rules at every row count
        const rpd::HeadPlan a = plan(r);
        const bool rows_n = a.mode == rpd::kHeadModeRowsN, tail = !rows_n && a.swap_rows == rpd::kSplitTail;
        const int splits = rows_n || tail ? a.splits / 2 : a.splits;
        tails += tail;
        bad += splits < 1 || splits > in.num_n || a.splits > in.max_splits || a.est != rpd::plan_head(r, in).est;
        bad += !rows_n && a.swap_rows != (tail ? rpd::kSplitTail : 0);
        bad += tail && (a.splits != 2 * in.num_n || force != RPD_TILING_AUTO);
        if (r > 64 && r % 32 > 1) continue;
        // the units of the pass: every half tile of every row tile once, every partial of a row once
        const int ng = rows_n ? a.swap_rows : rpd::kPairTileM, tiles = (r + ng - 1) / ng;
        rpd::TileWalk tw;
        tw.init(r, ng, V, d, rows_n ? a.splits / 2 : a.splits, tail, in.pair_slots);
        bad += tw.num_m != tiles;
        std::vector<int> halves(static_cast<size_t>(tiles) * 2 * in.num_n), slots(static_cast<size_t>(tiles) * a.splits);
        for (int u = 0; u < tw.units; ++u) {
            int m, g, v0, v1;
            tw.unit(u, m, g, v0, v1);
            if (m < 0 || m >= tiles || v0 < 0 || v1 <= v0 || v1 > 2 * in.num_n) return !std::printf("1\n");
            bad += v0 + 1 == v1 ? !tail || u < tw.whole : (v0 | v1) & 1;  // half tiles in the tail only
            for (int v = v0; v < v1; ++v) ++halves[static_cast<size_t>(m) * 2 * in.num_n + v];
            const int first = rows_n ? 2 * g : tail ? v0 : g, n = rows_n ? 2 : tail ? v1 - v0 : 1;
            for (int s = first; s < first + n; ++s) {
                if (s >= a.splits) return !std::printf("1\n");
                ++slots[static_cast<size_t>(m) * a.splits + s];
            }
        }
        for (int h : halves) bad += h != 1;
        for (int s : slots) bad += s != 1;
        const int rest = tiles * in.num_n % in.pair_slots;  // two half tiles to each pair at most
        bad += tail && (rest == 0 || 2 * rest > in.pair_slots || tw.units - tw.whole != 2 * rest);
    }
    bad += (force != RPD_TILING_AUTO || 2 * in.num_n > in.max_splits) && tails > 0;
    for (int r = 1; r <= 4096; ++r) {
        const rpd::HeadPlan a = plan(r);
        const bool rows_n = a.mode == rpd::kHeadModeRowsN;
        bad += rows_n && (a.swap_rows % 32 || a.swap_rows < 32 || a.swap_rows > 512);
        bad += force == RPD_TILING_PAIR && rows_n;
        bad += force == RPD_TILING_ROWS_N && !rows_n && in.max_splits >= 2;
    }
    for (int r = 1; r <= rpd::kStepPlanRows; ++r) {
        const rpd::HeadPlan a = plan(r);
        const int i = (r - 1) / 32;
        const int splits = sp.splits[i] < 0 ? -sp.splits[i] : sp.splits[i];
        const int mode = sp.splits[i] < 0 ? rpd::kHeadModeRowsN : rpd::kHeadModePair;
        bad += a.mode != mode || a.splits != splits || a.swap_rows != sp.swap_rows[i] || a.est != sp.est[i];
    }
    for (int tiles = 1; tiles <= 130; ++tiles)
        for (int gmax = 1; gmax <= in.num_n && gmax <= in.max_splits; gmax = 3 * gmax + 1)
            bad += every_key(0.914f, tiles, in.pair_slots, in.num_n, gmax) !=
                   rpd::best_split_key(0.914f, tiles, in.pair_slots, in.num_n, gmax);
    std::printf("%d\n", bad);
    return 0;
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("needs a host C++ compiler and the CUDA headers")
    d = tmp_path_factory.mktemp("step_plan")
    src, exe = d / "plan.cpp", d / "plan"
    src.write_text(DRIVER)
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-I", inc, "-I", CSRC, "-I",
                        os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(exe)


@pytest.mark.parametrize("force", [0, 1, 2])
@pytest.mark.parametrize("V,d,sms", [(126464, 4096, 152), (152064, 3584, 152), (256, 64, 152),
                                     (4100, 256, 152), (15872, 4096, 148), (50257, 768, 2)])
def test_one_entry_per_32_rows_is_exact(driver, V, d, sms, force):
    out = subprocess.run([driver, str(V), str(d), str(sms), str(force)], capture_output=True, text=True, check=True)
    assert int(out.stdout) == 0


# Measured on GB300 (us a pass over every row of the head, in the steady state of a second of them):
# V, d, rows, in pair tiles, in several row groups.
MEASURED = [(126464, 64, 1088, 89.5, 121.9), (126464, 256, 1344, 119.8, 149.1), (126464, 512, 672, 82.8, 93.1),
            (126464, 1024, 1152, 197.2, 224.4), (126464, 3072, 1568, 796.1, 758.1), (126464, 4096, 1088, 741.7, 708.8),
            (152064, 3584, 896, 647.9, 624.0), (152064, 3584, 1088, 782.9, 754.5), (32000, 128, 1568, 48.6, 58.9),
            (32000, 512, 1344, 51.6, 59.3), (32000, 1024, 832, 48.2, 54.9), (32000, 2048, 576, 67.1, 62.9),
            (32000, 4096, 576, 123.7, 111.3), (8192, 128, 1472, 24.5, 34.1), (8192, 512, 1216, 27.9, 33.9),
            (8192, 1024, 1216, 32.1, 36.7), (8192, 4096, 1152, 68.3, 64.3), (8192, 4096, 1472, 75.4, 80.0)]


@pytest.mark.parametrize("V,d,rows,pair,groups", MEASURED)
def test_row_groups_where_they_were_measured_faster(driver, V, d, rows, pair, groups):
    out = subprocess.run([driver, str(V), str(d), "152", "0", str(rows)], capture_output=True, text=True, check=True)
    mode = int(out.stdout.split()[0])
    assert mode == (3 if groups < pair else 2)


def test_ranges_of_two_tiles_are_not_taken_for_a_wave_saved(driver):
    """1568 rows at V 126464: 247 ranges leave no pair idle, but took 189 us at d = 256 where 21 take 136."""
    out = subprocess.run([driver, "126464", "256", "152", "0", "1568"], capture_output=True, text=True, check=True)
    assert out.stdout.split()[:2] == ["2", "21"]


# The same for the last wave of pair tiles: V, d, rows, us with whole tiles throughout, us with its half tiles.
TAILS = [(5120, 4096, 200, 33.4, 29.8), (7680, 2048, 200, 25.9, 23.2), (5120, 1024, 200, 20.1, 18.6),
         (20480, 4096, 400, 70.7, 68.6), (24064, 4096, 400, 74.5, 73.4), (15872, 4096, 748, 75.2, 74.3),
         (28160, 128, 200, 20.0, 21.0), (28160, 4096, 200, 53.5, 54.4), (20480, 128, 400, 22.8, 24.4),
         (24064, 1024, 400, 31.1, 32.4), (24064, 2048, 400, 45.2, 45.8), (15872, 128, 748, 23.6, 26.4),
         (15872, 1024, 748, 31.5, 33.4), (26880, 512, 748, 33.0, 38.6), (35840, 128, 1000, 35.9, 49.2),
         (35840, 2048, 1000, 98.0, 104.4), (34560, 4096, 748, 141.9, 144.8), (32000, 4096, 480, 90.5, 92.4)]


@pytest.mark.parametrize("V,d,rows,whole,halved", TAILS)
def test_half_tiles_where_they_were_measured_faster(driver, V, d, rows, whole, halved):
    out = subprocess.run([driver, str(V), str(d), "152", "0", str(rows)], capture_output=True, text=True, check=True)
    assert (out.stdout.split()[2] == "1") == (halved < whole)
