// Walking the rows that an ascending list of kept rows leaves out (the dropped rows of dX, which become +0.0).
#pragma once

#include "sbp_common.cuh"

namespace sbp {

// First position p of the ascending list rows[0, n) with rows[p] >= value (n if there is none), found by one warp: 32
// probes a step, so four dependent loads for a list of a million.
__device__ __forceinline__ int64_t warp_lower_bound(const int32_t* rows, int64_t n, int64_t value, int lane) {
    int64_t lo = 0, hi = n;                                  // the answer lies in [lo, hi]
    while (hi > lo) {
        const int64_t step = (hi - lo + 31) / 32;
        const int64_t at = lo + (int64_t)lane * step;
        const bool below = at < hi && (int64_t)__ldg(rows + at) < value;
        const int c = __popc(__ballot_sync(0xffffffffu, below));       // probes 0 .. c - 1 are below
        if (c == 0) return lo;
        const int64_t last = lo + (int64_t)(c - 1) * step;
        if (step == 1) return last + 1;
        lo = last + 1;
        if (last + step < hi) hi = last + step;
    }
    return lo;
}

// One warp visits rows [lo, hi) in windows of 32 and calls f(base, todo) for each window that has dropped rows: bit d of
// todo is set when row base + d is not in the list rows[0, n) (nullptr: the identity list 0, 1, ..., n - 1).
// Splitting the rows themselves, and not the gaps between kept rows, evens the work out for every mask: with whole frames
// kept a single gap can hold half of a clip.
template <typename F>
__device__ __forceinline__ void warp_visit_dropped_rows(const int32_t* rows, int64_t n, int64_t lo, int64_t hi, int lane, F f) {
    int64_t p = 0;
    if (rows == nullptr) {
        if (lo < n) lo = n;                                  // all of [0, n) is kept
        if (lo >= hi) return;
    } else {
        if (lo >= hi) return;
        p = warp_lower_bound(rows, n, lo, lane);
    }
    for (int64_t base = lo; base < hi; base += 32) {
        uint32_t kept = 0u;
        if (rows != nullptr) {
            const int64_t d = (p + lane < n) ? (int64_t)__ldg(rows + p + lane) - base : 32;
            kept = __reduce_or_sync(0xffffffffu, (d >= 0 && d < 32) ? (1u << d) : 0u);
            p += __popc(kept);
        }
        uint32_t todo = ~kept;
        if (hi - base < 32) todo &= (1u << (hi - base)) - 1u;
        if (todo) f(base, todo);
    }
}

}  // namespace sbp
