// step_counters.h - the counters through which the head kernel's CTAs share out a pass, and how the
// grid leaves them for the next one (host and device).
#pragma once

#include "rpd_internal.h"

namespace rpd {

// Counts a CTA that is done with the counters; true for the last one of the grid, which zeroes them.
// The count wraps to zero by itself: if two grids on the same counters have overlapped (which a caller
// must not let happen: both steps are meaningless), it is zero again once both have left, whoever
// zeroed what in between, and the CTA that leaves last of all leaves every counter at zero.  A store of
// zero instead can erase an arrival of the other grid, and then no later step finds its last CTA.
template <typename Words>
__host__ __device__ inline bool last_to_leave(Words &w, int grid) {
    return w.inc_wrap(kMetaExit, static_cast<unsigned>(grid) - 1u) == static_cast<unsigned>(grid) - 1u;
}

template <typename Words>
__host__ __device__ inline void zero_counters(Words &w) {
    w.zero(kMetaUnitNext);
    w.zero(kMetaRowNext);
    w.zero(kMetaMergeNext);
    w.zero(kMetaMergeDone);
    w.zero(kMetaRowsDone);
    w.zero(kMetaUnitsDone);
    w.zero(kMetaMaskRead);
    w.zero(kMetaClearLater);
}

}  // namespace rpd
