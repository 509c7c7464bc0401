// Row walk with a policy: the attention passes' version of the walk that
// aggregate_rows (agg.cuh) makes.  Equal shares of edges and row ends per warp
// (row_share.cuh), edges taken in windows of 32 whose ids are requested a window
// ahead and staged in shared memory, rows taking their edges from the window
// one after the other, parts of a row shared by several warps merged in warp
// order after the CTA's one barrier.
//
// A policy P holds one lane's state of one row and provides
//   kLpr, kState          lanes per row, floats a lane parks for another warp
//   open(t, k, beg)       start row t at edge k; its first edge is beg (loads what the
//                         row needs, clears the state)
//   clear()               the empty state
//   add<CHECK>(ids, cnt)  edges ids[0 .. cnt) (whole warp; ids in shared memory,
//                         readable up to 32 entries past them)
//   join()                combine the warp's lane groups (every lane ends with
//                         the state of the warp's edges)
//   park(slot) / merge(slot)  this lane's state to / combined with a parked one,
//                         float q of lane sub at slot[q * kLpr + sub]
//   close(t, beg, end, shared)  write row t, whose edges are [beg, end); shared:
//                         it was held by several warps
//   after(w, t, beg, end)  called by every warp of the CTA for each shared row t,
//                         closed by warp w, when wants_after() says so
#pragma once

#include "row_share.cuh"

namespace tfg {

template <int WARPS>
struct WalkShared {
    int64_t row[2];
    int32_t tail_row[WARPS], head_row[WARPS];
    int32_t ids[WARPS][64];
};

constexpr int kWalkMinWork = 8;   // work (edges + kRowCost per row) a warp should have, at least

// Gathers in flight per lane in a partial window of G lane groups: about 8 edges
// a step, so that a row of a few edges does not pay for empty slots (100,000
// nodes, 4 x 8 bf16, G = 4: 138 us with 4, 108 with 2).
__host__ __device__ constexpr int walk_part(int g) { return g >= 8 ? 1 : (g >= 4 ? 2 : 4); }

// parts: [2 * WARPS][kState * kLpr] floats of shared memory
template <int WARPS, class P>
__device__ __forceinline__ void walk_rows(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ col,
                                          int64_t n, P &p, WalkShared<WARPS> &s, float *parts) {
    WarpShare<WARPS> sh;
    if (!sh.init(rowptr, n, kWalkMinWork, s.row)) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int32_t *ids = s.ids[warp];
    constexpr int kSlot = P::kState * P::kLpr;
    if (lane == 0) s.head_row[warp] = -1;
    const int32_t kb = sh.kb, tb = sh.tb;
    uint32_t ahead = static_cast<uint32_t>(sh.ka);          // the window after the staged one
    auto col_at = [&](uint32_t k) { return k + lane < static_cast<uint32_t>(kb) ? ld_stream(col + k + lane) : 0; };
    int32_t c1 = col_at(ahead);
    auto next_window = [&]() {
        __syncwarp();                                       // the previous window's reads are done
        ids[lane] = c1;
        __syncwarp();
        ahead += 32;
        c1 = col_at(ahead);
    };
    int32_t t = sh.ta, rwin;
    int tl = 0;                                             // row t is lane tl of the row ends held
    auto row_window = [&]() {
        const int64_t r = static_cast<int64_t>(t) + lane;
        rwin = r < n ? __ldg(rowptr + r + 1) : 0;
        tl = 0;
    };
    row_window();
    next_window();
    int32_t k = sh.ka, rbeg = __ldg(rowptr + t);
    int j = 0;                                              // position in the staged window
    for (;;) {
        const bool closes = t < tb;
        const int32_t rend = closes ? lane_get(rwin, tl) : kb;
        int rem = rend - k;
        k = rend;
        if (closes || rem > 0) {
            p.open(t, rend - rem, rbeg);
            while (rem > 0) {
                if (j == 32) {
                    next_window();
                    j = 0;
                }
                const int cnt = min(rem, 32 - j);
                if (cnt == 32) p.template add<false>(ids, 32);
                else p.template add<true>(ids + j, cnt);
                rem -= cnt;
                j += cnt;
            }
            p.join();
        } else {
            p.clear();
        }
        if (!closes) break;
        if (t == sh.ta && sh.head_split) {                  // parts of it sit with earlier warps
            p.park(parts + (WARPS + warp) * kSlot);
            if (lane == 0) s.head_row[warp] = t;
        } else {
            p.close(t, rbeg, rend, false);
        }
        rbeg = rend;
        ++t;
        if (++tl == 32) row_window();
    }
    p.park(parts + warp * kSlot);                           // this warp's part of row tb
    if (lane == 0) s.tail_row[warp] = tb;
    __syncthreads();
    const int32_t hr = s.head_row[warp];
    if (hr >= 0) {                                          // earlier parts in warp order, then ours
        int first = warp;
        while (first > 0 && s.tail_row[first - 1] == hr) --first;
        const int32_t beg = __ldg(rowptr + hr);
        p.open(hr, beg, beg);
        for (int w = first; w < warp; ++w) p.merge(parts + w * kSlot);
        p.merge(parts + (WARPS + warp) * kSlot);
        p.close(hr, beg, __ldg(rowptr + hr + 1), true);
    }
    if (p.wants_after()) {
        __syncthreads();
        for (int w = 0; w < WARPS; ++w) {
            const int32_t r = s.head_row[w];
            if (r >= 0) p.after(w, r, __ldg(rowptr + r), __ldg(rowptr + r + 1));
        }
    }
}

// One CTA per SM of a policy's warps, a column of CTAs per feature tile.  Args has
// rowptr, col, n, width() (features of a row) and statistics() (whether the warps'
// statistics are wanted).  A policy is built from (args, the tile's first feature,
// kHeld floats a lane of its warp's shared memory or, when kHeld is 0, the warp's
// parking slot, which is free until the walk ends, the warps' statistics in
// shared memory).
template <class Policy, class Args>
__global__ void __launch_bounds__(Policy::kWarps * 32, 1) row_walk(Args a) {
    extern __shared__ __align__(16) float s_parts[];
    __shared__ WalkShared<Policy::kWarps> s_walk;
    const uint32_t f = a.width();
    for (uint32_t ft = blockIdx.y * Policy::kTile; ft < f; ft += gridDim.y * Policy::kTile) {
        float *held = s_parts + 2 * Policy::kWarps * Policy::kState * Policy::kLpr;
        const int warp = threadIdx.x >> 5;
        float *own = Policy::kHeld > 0 ? held + warp * 32 * Policy::kHeld : s_parts + warp * Policy::kState * Policy::kLpr;
        Policy p(a, ft, own, held + Policy::kWarps * 32 * Policy::kHeld);
        walk_rows<Policy::kWarps>(a.rowptr, a.col, a.n, p, s_walk, s_parts);
        __syncthreads();                   // before the next tile reuses the shared memory
    }
}

template <class Policy, class Args>
cudaError_t launch_walk(const Args &a, cudaStream_t s) {
    constexpr int parts = Policy::kWarps * (2 * Policy::kState * Policy::kLpr + 32 * Policy::kHeld) *
                          static_cast<int>(sizeof(float));
    constexpr int stats = Policy::kWarps * Policy::kLpr * Policy::kHeadsPerLane * static_cast<int>(sizeof(float2));
    const int smem = parts + (a.statistics() ? stats : 0);
    if (smem > 32 * 1024) {   // with the static part above the 48 KB every launch may use
        const cudaError_t err = cudaFuncSetAttribute(row_walk<Policy, Args>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     parts + stats);
        if (err != cudaSuccess) return err;
    }
    const int64_t tiles = (static_cast<int64_t>(a.width()) + Policy::kTile - 1) / Policy::kTile;
    const dim3 grid(static_cast<unsigned>(min64(a.n, static_cast<int64_t>(sm_count()))),
                    static_cast<unsigned>(min64(tiles, 65535)));
    row_walk<Policy, Args><<<grid, Policy::kWarps * 32, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace tfg
