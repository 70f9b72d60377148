// step_common.cuh - device routines shared by the step's kernels: warp scans and the combination
// of softmax statistics (the head-tiling plan is in head_plan.h).
#pragma once

#include "head_plan.h"
#include "ptx.cuh"
#include "rpd_internal.h"

namespace rpd {
namespace {

__device__ __forceinline__ int warp_inclusive_scan(int v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Running softmax statistics of one row over part of the vocabulary, in log2 units:
// m = max x, s = sum 2^(x-m), t = sum 2^(x-m) (x-m), a = argmax (lowest index).
struct Stat {
    float m, s, t;
    int a;
};

// Combine two partials: m = max, alpha = 2^(m_j - m), s = sum alpha s_j,
// t = sum alpha (t_j + (m_j - m) s_j); the argmax is the lowest index attaining m.
__device__ __forceinline__ Stat merge2(const Stat &x, const Stat &y) {
    if (y.s <= 0.f) return x;
    if (x.s <= 0.f) return y;
    Stat r;
    r.m = fmaxf(x.m, y.m);
    const float dx = x.m - r.m, dy = y.m - r.m;
    const float ax = ex2(dx), ay = ex2(dy);
    r.s = ax * x.s + ay * y.s;
    r.t = ax * fmaf(dx, x.s, x.t) + ay * fmaf(dy, y.s, y.t);
    r.a = (x.m > y.m) ? x.a : (y.m > x.m) ? y.a : min(x.a, y.a);
    return r;
}

constexpr float kLn2 = 0.6931471805599453f;

}  // namespace
}  // namespace rpd
