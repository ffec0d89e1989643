// walk.cuh -- sharing the rows that a warp walks over its lanes.
#pragma once

#include "tc_internal.cuh"

namespace tc {

// The 32 entries a warp holds and the steps (32 ids each) of its walk: the
// steps of all entries are shared out evenly over the warp's eight groups of
// four lanes, so short and long rows keep every lane busy.
struct Walk {
    uint32_t i, left, iters;  // the group's entry, its steps, the steps of the longest group
    uint32_t skip;            // steps of entry i that belong to the groups before
};
__device__ __forceinline__ Walk share_steps(uint32_t steps) {
    const unsigned lane = lane_id();
    uint32_t incl = steps;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (unsigned)o) incl += y;
    }
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    Walk w;
    w.iters = (total + 7) / 8;
    const uint32_t c = min((lane >> 2) * w.iters, total);
    w.left = min(w.iters, total - c);
    w.i = 0;  // the entry of step c: the first whose inclusive count passes it
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (__shfl_sync(0xFFFFFFFFu, incl, w.i + o - 1) <= c) w.i += o;
    w.skip = c - __shfl_sync(0xFFFFFFFFu, incl - steps, w.i);
    return w;
}

}  // namespace tc
