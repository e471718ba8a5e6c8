// The row (tail) of every edge of a warp's range of consecutive edges, found without a search per
// edge.  The warp holds the starts of the rows that have an edge among 32 rows at a time, one a lane
// (ascending), so the rows that start within the 32 edges of a step are a bit mask, and a lane's row
// is the count of starts up to it.  A run of rows without edges is passed by a search: a graph from the
// layout ends each partition with one (R-MAT of 4.2 M vertices, 65 M edges: the predecessor pass of an
// 8-source solve 1.03 -> 0.81 ms against window after window).
#pragma once

#include "common.cuh"

namespace sssp {

struct RowWalk {
    const uint32_t* row_ptr;
    uint32_t V;
    uint32_t* row;    // shared, 32 words of the warp: the window's rows with an edge
    uint32_t* start;  // shared, 32 words of the warp
    uint32_t r0, p, end, seen;  // first row of the window, start of the lane's row, edge after the window, rows passed

    __device__ __forceinline__ bool window() {  // false: no row with an edge
        const uint32_t lane = threadIdx.x & 31u, r = r0 + lane;
        const uint32_t a = __ldg(&row_ptr[min(r, V)]), b = __ldg(&row_ptr[min(r + 1u, V)]);
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, b > a), k = __popc(m & ((1u << lane) - 1u));
        __syncwarp();
        if (b > a) row[k] = r, start[k] = a;
        __syncwarp();
        p = lane < (uint32_t)__popc(m) ? start[lane] : 0xFFFFFFFFu;
        end = __shfl_sync(0xFFFFFFFFu, b, 31);
        seen = 0;
        return m != 0u;
    }

    // to the row that holds edge e: a 32-way search of row_ptr
    __device__ __forceinline__ void seek(uint32_t e) {
        const uint32_t lane = threadIdx.x & 31u;
        uint32_t lo = 0, len = V;  // last row r with row_ptr[r] <= e
        while (len > 1u) {
            const uint32_t step = (len + 31u) / 32u, i = lane * step;
            const bool le = i < len && __ldg(&row_ptr[lo + i]) <= e;
            const uint32_t k = 31u - (uint32_t)__clz(__ballot_sync(0xFFFFFFFFu, le) | 1u);
            lo += k * step;
            len = min(step, len - k * step);
        }
        r0 = lo;
        window();
        seen = __popc(__ballot_sync(0xFFFFFFFFu, p < e));
    }

    // the row of edge eb + lane (of those below e1); called with ascending steps of 32
    __device__ __forceinline__ uint32_t step(uint32_t eb, uint32_t e1) {
        const uint32_t lane = threadIdx.x & 31u;
        uint32_t u = 0;
        for (;;) {
            const uint32_t at = __reduce_or_sync(0xFFFFFFFFu, p - eb < 32u ? 1u << (p - eb) : 0u);
            // (a lane at or past the window's end finds its row in a later window, and overwrites this)
            const uint32_t k = seen + __popc(at & (0xFFFFFFFFu >> (31u - lane)));
            if (k) u = row[k - 1u];
            seen += __popc(at);
            if (end >= min(eb + 32u, e1)) return u;
            r0 += 32u;
            if (r0 >= V) return u;  // (the last row ends before e1: an edge count that is too large)
            if (!window()) seek(end);
        }
    }
};

}  // namespace sssp
