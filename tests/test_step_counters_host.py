"""The counters that the head kernel's CTAs share are zero after every grid, also after two grids on
the same counters that overlapped: their CTAs leaving in every order around the first grid's zeroing,
`csrc/step_counters.h` compiled with the host C++ compiler (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_36452_gb300", "csrc")

DRIVER = r"""
#include "step_counters.h"
#include <cstdio>
#include <functional>
struct Words {
    int w[rpd::kMetaWords] = {};
    int zeroed = 0;                // stores of the zeroing that runs
    std::function<void(int)> hook; // called before each
    unsigned inc_wrap(int i, unsigned top) {
        const unsigned old = w[i];
        w[i] = old >= top ? 0 : old + 1;
        return old;
    }
    void zero(int i) {
        if (hook) hook(zeroed++);
        w[i] = 0;
    }
};
int resets;
void leave(Words &m, int grid) {  // a CTA that has used every counter
    for (int i : {rpd::kMetaUnitNext, rpd::kMetaRowNext, rpd::kMetaMergeNext, rpd::kMetaMergeDone, rpd::kMetaRowsDone,
                  rpd::kMetaUnitsDone, rpd::kMetaMaskRead, rpd::kMetaClearLater})
        ++m.w[i];
    if (rpd::last_to_leave(m, grid)) {
        ++resets;
        rpd::zero_counters(m);
    }
}
int main() {
    int bad = 0;
    const int grid = 6;
    // of the second grid, `before` CTAs leave before the first one's last, `inside` more during the
    // k-th store of the first zeroing
    for (int before = 0; before <= grid; ++before)
        for (int k = 0; k < 10; ++k)
            for (int inside = 0; before + inside <= grid; ++inside) {
                Words m;
                int left = 0;  // CTAs that have left, of 2 * grid
                auto go = [&](int n) { while (n-- > 0) { ++left; leave(m, grid); } };
                bool nested = false;
                m.hook = [&](int store) {
                    if (store != k || nested) return;
                    nested = true;
                    go(inside < 2 * grid - left ? inside : 2 * grid - left);
                };
                go(before + grid);
                go(2 * grid - left);
                m.hook = nullptr;
                for (int i = 0; i < rpd::kMetaWords; ++i) bad += m.w[i] != 0;
                for (int call = 0; call < 2; ++call) {  // the calls after them
                    resets = 0;
                    for (int c = 0; c < grid; ++c) {
                        leave(m, grid);
                        bad += resets != (c == grid - 1);
                    }
                    for (int i = 0; i < rpd::kMetaWords; ++i) bad += m.w[i] != 0;
                }
            }
    std::printf("%d\n", bad);
    return 0;
}
"""


def test_counters_recover_from_overlapping_grids(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("needs a host C++ compiler and the CUDA headers")
    src, exe = tmp_path / "counters.cpp", tmp_path / "counters"
    src.write_text(DRIVER)
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-I", inc, "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                        str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert int(subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout) == 0
