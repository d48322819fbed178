// Walking the lists of several nodes at once (node -> communities).
#pragma once

#include "common.cuh"

// f(l) for every entry l of the lists mlist[mptr[u]..mptr[u+1]) of the nodes u
// in nodes[e0, e1), at most 32 nodes.  The lists are laid end to end: the lanes
// take 32 entries of several lists at a time, and the next ones are loaded
// while these are handled (lists are often shorter than a warp is wide, and one
// at a time each costs three dependent loads).  Long lists are walked one at a
// time: finding an entry's list takes seven shuffles, which share the pipe of
// the shared-memory tables behind f (11,541 and 11,926 communities of some 3,000
// of 300,000 nodes, lists of 115 and 134: 152 -> 126 ms a call; no difference
// between 24, 64 and 160 as the line on graphs with short lists).  After every
// 32 * AHEAD entries the lanes ask done(); if it is true for any of them the warp
// leaves, and true is returned to all.  Warp-collective.
template <class F, class D>
__device__ __forceinline__ bool visit_lists(const i32 *nodes, i64 e0, i64 e1, const i64 *mptr, const i32 *mlist, F f,
                                            D done) {
    constexpr int AHEAD = 4;  // entries a lane has in flight
    constexpr int LONG_LISTS = 64;  // entries a list, on average
    const int lane = threadIdx.x & 31;
    i64 lo = 0, n = 0;
    if (e0 + lane < e1) {
        const i32 u = nodes[e0 + lane];
        lo = mptr[u];
        n = mptr[u + 1] - lo;
    }
    const bool giant = __any_sync(FULL_MASK, n > 1 << 25);  // the sums below would not fit
    const int len = giant ? 0 : (int)n;
    int incl = len;  // node i's entries are incl - len .. incl of the whole
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL_MASK, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(FULL_MASK, incl, 31);
    if (giant || total >= LONG_LISTS * (int)(e1 - e0)) {
        for (int i = 0; i < (int)(e1 - e0); ++i) {
            const i64 b = __shfl_sync(FULL_MASK, lo, i), m = __shfl_sync(FULL_MASK, n, i);
            for (i64 t0 = 0; t0 < m; t0 += 32 * AHEAD) {
                i32 l[AHEAD];
#pragma unroll
                for (int j = 0; j < AHEAD; ++j) {
                    const i64 t = t0 + 32 * j + lane;
                    l[j] = t < m ? mlist[b + t] : -1;
                }
#pragma unroll
                for (int j = 0; j < AHEAD; ++j)
                    if (l[j] >= 0) f(l[j]);
                if (__any_sync(FULL_MASK, done())) return true;
            }
        }
        return false;
    }
    const i64 first = lo - (incl - len);  // entry t of the whole is mlist[first + t]
    for (int t0 = 0; t0 < total; t0 += 32 * AHEAD) {
        i32 l[AHEAD];
#pragma unroll
        for (int j = 0; j < AHEAD; ++j) {
            l[j] = -1;
            if (t0 + 32 * j >= total) continue;
            const int t = t0 + 32 * j + lane;
            int i = 0;  // first node whose list ends beyond t
#pragma unroll
            for (int step = 16; step; step >>= 1)
                if (__shfl_sync(FULL_MASK, incl, i + step - 1) <= t) i += step;
            const i64 b = __shfl_sync(FULL_MASK, first, i);
            if (t < total) l[j] = mlist[b + t];
        }
#pragma unroll
        for (int j = 0; j < AHEAD; ++j)
            if (l[j] >= 0) f(l[j]);
        if (__any_sync(FULL_MASK, done())) return true;
    }
    return false;
}
