// Lower window bound of the text-anchored mode on a compacted cache (Eq. 2 with the window rule
// "query at row qpos sees text anchor p iff qpos - window < p"): the anchors are strictly
// increasing, so the visible text anchors of a query are a contiguous run of the compacted cache
// and one index per query -- its first visible compact row -- describes it.
#pragma once
#include "common.cuh"

namespace sparrow {

// First index j in [0, n_text) with anchor[j] > bound (n_text if none); at most 32 halvings.
inline int first_anchor_above(const int32_t* anchor, int n_text, long long bound)
{
    int lo = 0, hi = n_text;
    for (int step = 0; step < 32 && lo < hi; ++step) {
        const int mid = lo + (hi - lo) / 2;
        if ((long long)anchor[mid] > bound) hi = mid; else lo = mid + 1;
    }
    return lo;
}

// The same by a whole warp: 32 probes at a time instead of one, so a search over 448 anchors waits for memory
// twice instead of nine times.  A drafting round of six steps, each an append, these bounds and the window
// attention, launches kept ahead: 61.6 -> 56.2 us, with the address arithmetic of the row movers below 64 bits.
__device__ __forceinline__ int first_anchor_above_warp(const int32_t* anchor, int n_text, long long bound)
{
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = n_text;
    for (int round = 0; round < 8 && lo < hi; ++round) {
        const int step = (hi - lo + 31) / 32;
        const long long at = (long long)lo + (long long)(lane + 1) * step - 1;
        const bool above = at >= hi || (long long)ld_behind(anchor + at) > bound;
        const int below = __popc(~__ballot_sync(0xffffffffu, above));         // probes that are not above: lanes 0, 1, ... in sorted anchors
        const long long next_hi = (long long)lo + (long long)(below + 1) * step - 1;
        lo = min((long long)hi, (long long)lo + (long long)below * step);
        if (next_hi < hi) hi = (int)next_hi;
    }
    return lo;
}

// One warp per (sequence, query token).  anchor_idx [B][n_anchor]: text anchors first, then the
// T_tree rows of the draft tree; the queries are its last T_new nodes.
__global__ void window_bounds_kernel(const int32_t* anchor_idx, int n_anchor, int window, int T_tree, int T_new,
                                     int batch, int32_t* first_visible)
{
    let_dependents_launch();
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= batch * T_new) return;
    const int b = i / T_new, t = i - b * T_new;
    const int32_t* a = anchor_idx + (size_t)b * n_anchor;
    const int n_text = n_anchor - T_tree;
    wait_for_predecessors();
    int first = 0;
    if (window > 0) first = first_anchor_above_warp(a, n_text, (long long)ld_behind(a + n_anchor - T_new + t) - window);
    if ((threadIdx.x & 31) == 0) first_visible[i] = first;
}

}  // namespace sparrow
