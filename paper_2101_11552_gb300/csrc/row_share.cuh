// Work split of the row reductions: equal shares of edges and row ends for
// every CTA and, inside it, for every warp.
#pragma once

#include "common.cuh"

namespace tfg {

#ifndef TFG_ROW_COST
#define TFG_ROW_COST 6
#endif
// Work coordinate of row t: the edges before it plus kRowCost for each row.
// Ending a row costs as many instructions as several edges; with one unit a
// row, warps with the short rows of a skewed graph finish last.  Measured on
// the fp32 ten-hop propagation (169,343 nodes, mean in-degree 6.9, F = 41):
// 807 us with 1, 677 with 4, 646 with 6, 625 with 8; wide features on 19,717
// nodes go the other way (64.5, 62.9 to 65.6, 66.7, 67.5 us).
constexpr int64_t kRowCost = TFG_ROW_COST;

// Last row t in [lo, hi] whose coordinate rowptr[t] + kRowCost * t is at most
// q, found by the whole warp (lo's coordinate is): 32 probes a round, 4 rounds
// for a million rows, where a scalar binary search takes 20 dependent loads.
__device__ __forceinline__ int64_t warp_last_row_at(const int32_t *rowptr, int64_t lo, int64_t hi,
                                                    int64_t q) {
    const int lane = threadIdx.x & 31;
    while (lo < hi) {
        const int64_t step = (hi - lo + 31) / 32;
        const int64_t p = lo + (lane + 1) * step;                   // probes in (lo, hi]
        const bool le = p <= hi && static_cast<int64_t>(__ldg(rowptr + p)) + kRowCost * p <= q;
        const int c = __popc(lane_ballot(le));             // monotone: lanes 0 .. c - 1
        const int64_t top = lo + (c + 1) * step - 1;
        lo += c * step;
        hi = top < hi ? top : hi;
    }
    return lo;
}

// The share of one warp.  A CTA of WARPS warps owns whole rows holding an equal
// share of the work coordinate; inside it every warp owns an equal range of it,
// so a hub row is shared by the warps it spans.  min_work: the least a warp
// should have; a small graph leaves the last CTAs without work.
template <int WARPS>
struct WarpShare {
    int32_t ta, tb;       // the rows [ta, tb) end here; row tb is open at the end
    int32_t ka, kb;       // the edges [ka, kb)
    bool head_split;      // row ta was begun by an earlier warp

    // Collective over the CTA.  False: the CTA has no work (it returns).
    __device__ __forceinline__ bool init(const int32_t *rowptr, int64_t n, int min_work, int64_t (&s_row)[2]) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const int64_t total = static_cast<int64_t>(__ldg(rowptr + n)) + kRowCost * n;
        int64_t nb = (total + WARPS * min_work - 1) / (WARPS * min_work);
        nb = min64(nb, gridDim.x);
        const int64_t b = blockIdx.x;
        if (b >= nb) return false;
        const int64_t w = (total + nb - 1) / nb;
        if (warp < 2) {   // first row whose coordinate is at or past (b + warp) * w
            const int64_t at = (b + warp) * w;
            int64_t r = 0;
            if (at > 0) r = at >= total ? n : warp_last_row_at(rowptr, 0, n, at - 1) + 1;
            if (lane == 0) s_row[warp] = r;
        }
        __syncthreads();
        const int64_t r0 = s_row[0], r1 = s_row[1];
        if (r0 >= r1) return false;                                 // uniform over the CTA
        const int64_t q0 = static_cast<int64_t>(__ldg(rowptr + r0)) + kRowCost * r0;
        const int64_t q1 = static_cast<int64_t>(__ldg(rowptr + r1)) + kRowCost * r1;
        const int64_t per = (q1 - q0 + WARPS - 1) / WARPS;
        const int64_t qa = min64(q1, q0 + warp * per), qb = min64(q1, qa + per);
        const int64_t a = warp_last_row_at(rowptr, r0, r1, qa);
        const int64_t c = warp_last_row_at(rowptr, a, r1, qb);
        ta = static_cast<int32_t>(a);
        tb = static_cast<int32_t>(c);
        // a boundary inside the row-end cost of a row lies after its last edge
        ka = static_cast<int32_t>(a < n ? min64(qa - kRowCost * a, __ldg(rowptr + a + 1)) : qa - kRowCost * a);
        kb = static_cast<int32_t>(c < n ? min64(qb - kRowCost * c, __ldg(rowptr + c + 1)) : qb - kRowCost * c);
        head_split = ka > __ldg(rowptr + a);
        return true;
    }
};

}  // namespace tfg
