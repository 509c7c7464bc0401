// Backward of the message aggregation: the gradient with respect to the node
// features x of out = aggregate(x) (the paper keeps graph construction and
// mini-batching differentiable, Sections 2.1.1 and 2.1.3, so gradients flow
// through the aggregation to the features).  For a sum with edge weights w,
// out[t] = sum over edges e = (s -> t) of w_e x[s], so
//
//   grad_x[s] = sum over edges e = (s -> t) of w_e grad_out[t]
//
// -- the same aggregation over the transposed graph.  The caller builds the
// CSR grouped by SOURCE (the radix build keyed on row 0 of edge_index: rows
// are sources, col holds targets, perm the original edge ids); the sum then
// runs on the ordinary aggregation kernels:
//
//   sum    weights w_e                      (edge_weight[perm], or 1)
//   mean   weights w_e / in_degree(t)       (the forward divides by the count)
//   GCN    dinv[s] * dinv[t] on the fly, plus fill * dinv[s]^2 grad_out[s]:
//          the symmetric normalisation is its own transpose, so the GCN
//          kernel runs unchanged on the source-grouped CSR with the forward's
//          dinv
//
// Max: the forward with argmax records, per (t, f), the original id of the
// first edge (in original order) attaining the maximum; the backward gives
// w_e grad_out[t, f] to that edge's source only.  It walks the source-grouped
// CSR, so each grad_x[s, f] is a sum in a fixed order (no atomics, bitwise
// reproducible).
#include "max_walk.cuh"

namespace tfg {
namespace {

// w_src[k] = (edge_weight ? edge_weight[perm_src[k]] : 1) / (mean ? max(deg[col_src[k]], 1) : 1)
__global__ void transposed_weights(const int32_t *__restrict__ perm_src,
                                   const int32_t *__restrict__ col_src,
                                   const float *__restrict__ edge_weight,
                                   const int32_t *__restrict__ in_degree, int64_t e,
                                   float *__restrict__ w_src) {
    const int64_t k = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (k >= e) return;
    float w = edge_weight ? __ldg(edge_weight + __ldg(perm_src + k)) : 1.f;
    if (in_degree) w = w / static_cast<float>(max(__ldg(in_degree + __ldg(col_src + k)), 1));
    w_src[k] = w;
}

// ---- max backward on long rows ----------------------------------------------
// The kernel walks CSR rows in 32-edge chunks: one coalesced load brings the
// chunk's indices and lanes pass them on by shuffle.  Each CTA owns a
// work-balanced range of rows (balanced_rows); its warps take rows from a shared
// counter.  A row longer than kMxHeavyDeg is set aside and then split over all the
// CTA's warps in contiguous edge segments, whose sums are added in segment order.
constexpr int kMxWarps = 8;
constexpr int kMxThreads = kMxWarps * 32;
constexpr int64_t kMxHeavyDeg = 1024;
constexpr int kMxMaxHeavy = 64;
// The kernel waits on the chain edge id -> mark -> row slices, so resident warps
// count more than edges in flight, and a thread keeps lanes instead of ids and
// weights for the edges in flight.  114.6M edges F = 128 / 20M edges F = 256 / 20M
// edges F = 96, us: 8 CTAs an SM and 2 edges 2929 / 1716 / 613, 8 and 1 3267 / 2016 /
// 740, 8 and 3 3263 / 1894 / 710, 6 and 2 3021 / 1822 / 636, 4 and 4 3124 / 1835 / 672
// (4 and 4 with ids and weights held 3445 / 1988 / 771).  The row walk with marks (a
// list of the window's marked pairs, eight read at once) took 3628 and 800 for the
// first and the last.
#ifndef TFG_MXB_DEPTH
#define TFG_MXB_DEPTH 2        // marked out-edges in flight per warp
#endif
#ifndef TFG_MXB_MINB
#define TFG_MXB_MINB 8         // with marks: resident CTAs per SM (32 registers per thread)
#endif

// Two ways to find the (edge, feature) pairs that contribute, with the same
// sums in the same order:
//  * every out-edge: a lane requests its slice of the argmax row and of the
//    gradient row of t together (one round trip, D edges in flight) and
//    adds where the argmax names the edge;
//  * win marks (MASKED): the features are cut into at most 8 groups, and bit
//    j of mark[e] is set when edge e is the argmax of some (t, f) with f in
//    group j.  A chunk's edges with no bit set are skipped, and for the
//    others only the lanes whose group bit is set read their slices.  On
//    long rows few edges win anything and a winner wins few features, so
//    most row reads disappear; the marks take a byte per edge and stay in
//    L2.  A bit can come from another row's argmax naming the edge: the
//    argmax check decides, as in the full walk.
template <int VEC, bool MASKED>
struct MaxBwd {
    float acc[VEC];

    __device__ void init() {
#pragma unroll
        for (int q = 0; q < VEC; ++q) acc[q] = 0.f;
    }

    // A chunk's loads: its target ids and edge ids, then (given the edge
    // ids) its marks and weights.  Requesting the next chunk's ids and marks
    // before this chunk's rows measured slower (more registers, spills).
    struct Chunk {
        int c;
        int32_t ec;
    };
    static __device__ __forceinline__ Chunk ids(const MaxBwdArgs &a, uint32_t base, uint32_t k1, int lane) {
        Chunk r{0, 0};
        if (base + lane < k1) {
            r.c = ld_stream(a.col + base + lane);
            r.ec = __ldg(a.perm + base + lane);
        }
        return r;
    }
    static __device__ __forceinline__ uint32_t mark_of(const MaxBwdArgs &a, uint32_t base, uint32_t k1,
                                                       int lane, int32_t ec) {
        const bool mine = base + lane < k1;
        if constexpr (MASKED)
            return mine && static_cast<uint64_t>(ec) < static_cast<uint64_t>(a.e) ? __ldg(a.mark + ec) : 0u;
        return mine ? 0xffu : 0u;
    }
    static __device__ __forceinline__ float weight_of(const MaxBwdArgs &a, uint32_t mk, int32_t ec) {
        return a.w ? (mk != 0 ? __ldg(a.w + ec) : 0.f) : 1.f;
    }

    __device__ void scan(const MaxBwdArgs &a, uint32_t k0, uint32_t k1, uint32_t fl, int lane) {
        constexpr int D = MASKED ? TFG_MXB_DEPTH : 4;
        const uint32_t f = a.width();
        const uint32_t my_bit =
            MASKED ? 1u << (fl / static_cast<uint32_t>(a.group)) : 0xffu;
        for (uint32_t base = k0; base < k1; base += 32) {
            const Chunk ch = ids(a, base, k1, lane);
            const int c = ch.c;
            const int32_t ec = ch.ec;
            const uint32_t mk = mark_of(a, base, k1, lane, ec);
            const float wc = weight_of(a, mk, ec);
            const bool win = mk != 0;
            // the chunk's edges that may contribute, D at a time in chunk order
            for (uint32_t m = lane_ballot(win); m != 0;) {
                int at[D];                                  // the edges' lanes in the chunk
                int32_t am[D][VEC];                         // -2: no edge's id
                float gv[D][VEC];
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    const bool any = m != 0;
                    at[d] = any ? __ffs(m) - 1 : 0;
                    m &= m - 1;
                    const uint32_t t = static_cast<uint32_t>(lane_get(c, at[d]));
                    const bool ok = any && (lane_get(mk, at[d]) & my_bit) != 0;   // per lane
                    const uint64_t from = static_cast<uint64_t>(t) * f + fl;
                    if constexpr (VEC == 4) {
                        const int4 v = ok ? __ldg(reinterpret_cast<const int4 *>(a.argmax + from)) : make_int4(-2, -2, -2, -2);
                        const float4 w4 = ok ? __ldg(reinterpret_cast<const float4 *>(a.grad_out + from))
                                             : make_float4(0.f, 0.f, 0.f, 0.f);
                        am[d][0] = v.x; am[d][1] = v.y; am[d][2] = v.z; am[d][3] = v.w;
                        gv[d][0] = w4.x; gv[d][1] = w4.y; gv[d][2] = w4.z; gv[d][3] = w4.w;
                    } else {
                        am[d][0] = ok ? __ldg(a.argmax + from) : -2;
                        gv[d][0] = ok ? __ldg(a.grad_out + from) : 0.f;
                    }
                }
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    const int32_t ed = lane_get(ec, at[d]);
                    const float we = a.w ? lane_get(wc, at[d]) : 1.f;
#pragma unroll
                    for (int q = 0; q < VEC; ++q)
                        if (am[d][q] == ed) acc[q] = fmaf(we, gv[d][q], acc[q]);
                }
            }
        }
    }

    // the sum over a later segment of the same row
    __device__ void merge(const float *v) {
#pragma unroll
        for (int q = 0; q < VEC; ++q) acc[q] += v[q];
    }

    __device__ void store(float *to) const {
#pragma unroll
        for (int q = 0; q < VEC; ++q) to[q] = acc[q];
    }
};

// One row by one warp, feature tiles of 32 * VEC.
template <int VEC, bool MASKED>
__device__ void max_warp_row(const MaxBwdArgs &a, int64_t s, int lane) {
    const int64_t beg = a.rowptr[s], end = a.rowptr[s + 1];
    for (int64_t f0 = lane * VEC, ft = 0; ft < a.f; ft += 32 * VEC, f0 += 32 * VEC) {
        MaxBwd<VEC, MASKED> st;
        st.init();
        st.scan(a, beg, end, f0 < a.f ? f0 : 0, lane);
        if (f0 < a.f) st.store(a.grad_x + s * a.f + f0);
    }
}

// One long row by all warps of the CTA: warp w takes the w-th of kMxWarps
// contiguous edge segments; warp 0 adds the other segments to its own, in segment
// order.  Every thread of the CTA calls this.
template <int VEC, bool MASKED>
__device__ void max_cta_row(const MaxBwdArgs &a, int64_t s, float *s_val) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t beg = a.rowptr[s], d = a.rowptr[s + 1] - beg;
    const int64_t k0 = beg + d * warp / kMxWarps, k1 = beg + d * (warp + 1) / kMxWarps;
    for (int64_t f0 = lane * VEC, ft = 0; ft < a.f; ft += 32 * VEC, f0 += 32 * VEC) {
        MaxBwd<VEC, MASKED> st;
        st.init();
        st.scan(a, k0, k1, f0 < a.f ? f0 : 0, lane);
        if (warp > 0) st.store(s_val + (warp * 32 + lane) * VEC);
        __syncthreads();
        if (warp == 0) {
            for (int w = 1; w < kMxWarps; ++w) st.merge(s_val + (w * 32 + lane) * VEC);
            if (f0 < a.f) st.store(a.grad_x + s * a.f + f0);
        }
        __syncthreads();
    }
}

template <int VEC, bool MASKED>
__global__ void __launch_bounds__(kMxThreads, MASKED ? TFG_MXB_MINB : 4) max_bwd_kernel(MaxBwdArgs a) {
    __shared__ int s_next, s_nheavy;
    __shared__ int64_t s_heavy[kMxMaxHeavy];
    __shared__ float s_val[kMxThreads * VEC];
    int64_t r0, r1;
    balanced_rows(a.rowptr, a.n, gridDim.x, blockIdx.x, r0, r1);
    const int64_t nrows = r1 - r0;
    if (threadIdx.x == 0) {
        s_next = 0;
        s_nheavy = 0;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (;;) {
        int i = 0;
        if (lane == 0) i = atomicAdd(&s_next, 1);
        i = lane_get(i, 0);
        if (i >= nrows) break;
        const int64_t s = r0 + i;
        if (a.rowptr[s + 1] - a.rowptr[s] > kMxHeavyDeg) {
            int slot = 0;
            if (lane == 0) slot = atomicAdd(&s_nheavy, 1);
            slot = lane_get(slot, 0);
            if (slot < kMxMaxHeavy) {
                if (lane == 0) s_heavy[slot] = s;
                continue;
            }
        }
        max_warp_row<VEC, MASKED>(a, s, lane);
    }
    __syncthreads();
    const int nh = min(s_nheavy, kMxMaxHeavy);
    for (int h = 0; h < nh; ++h) max_cta_row<VEC, MASKED>(a, s_heavy[h], s_val);
}

bool aligned(const void *p, uintptr_t b) { return reinterpret_cast<uintptr_t>(p) % b == 0; }

// Win marks of the max backward.  Every (t, f) has one winning edge (none
// for a row without edges); a row of in-degree d has at most min(d, F)
// distinct winners, so on long rows most out-edges win nothing and a
// winner wins few features.  Two launches write the marks: zero them, then
// for each e = argmax[t, f] set bit f / group of mark[e] (atomicOr on the
// word holding the byte).  Ids outside [0, E) are ignored.
__global__ void max_marks_zero(uint8_t *__restrict__ mark, int64_t bytes) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t i0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t n16 = reinterpret_cast<uintptr_t>(mark) % 16 == 0 ? bytes / 16 : 0;
    uint4 *m16 = reinterpret_cast<uint4 *>(mark);
    for (int64_t i = i0; i < n16; i += stride) m16[i] = make_uint4(0, 0, 0, 0);
    for (int64_t i = n16 * 16 + i0; i < bytes; i += stride) mark[i] = 0;
}

__global__ void max_marks_set(const int32_t *__restrict__ argmax, int64_t n, int64_t f, int64_t e,
                              int group, uint8_t *__restrict__ mark) {
    uint32_t *words = reinterpret_cast<uint32_t *>(mark);   // 4-byte aligned (checked by the caller)
    // rows t over the grid, features over the threads of a block
    for (int64_t t = blockIdx.x; t < n; t += gridDim.x)
        for (int64_t c = threadIdx.x; c < f; c += blockDim.x) {
            const int32_t k = __ldg(argmax + t * f + c);
            if (static_cast<uint64_t>(k) >= static_cast<uint64_t>(e)) continue;
            const uint32_t bit = 1u << static_cast<uint32_t>(c / group);
            atomicOr(words + (k >> 2), bit << (8 * (k & 3)));
        }
}

}  // namespace

size_t backward_workspace_bytes(int mode, int64_t e) {
    if (mode != TFG_SUM && mode != TFG_MEAN) return 0;
    return (sizeof(float) * static_cast<size_t>(e) + 255) & ~size_t(255);
}

cudaError_t launch_aggregate_backward(int mode, const int32_t *rowptr_src, const int32_t *col_src,
                                      const int32_t *perm_src, const float *edge_weight,
                                      const int32_t *in_degree, const float *grad_out, int64_t n,
                                      int64_t e, int64_t f, float *grad_x, void *ws,
                                      cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    float *w_src = nullptr;
    if (e > 0 && (edge_weight || mode == TFG_MEAN)) {
        w_src = static_cast<float *>(ws);
        transposed_weights<<<ceil_div(e, 256), 256, 0, s>>>(
            perm_src, col_src, edge_weight, mode == TFG_MEAN ? in_degree : nullptr, e, w_src);
        const cudaError_t err = cudaGetLastError();
        if (err != cudaSuccess) return err;
    }
    return launch_aggregate(0, rowptr_src, e > 0 ? col_src : nullptr, w_src, nullptr, grad_out,
                            TFG_F32, n, f, 0, 0.f, grad_x, s);
}

// The win marks pay when most edges win nothing in a row tile of kMxbSpan
// features: an edge into a row of in-degree d wins a given feature with
// probability about 1 / d, so it is visited in a tile with probability
// about 1 - exp(-span / d), span = min(F, kMxbSpan).  They are used when
// the mean in-degree E / N is at least span.  Measured: 114.6M edges, mean
// in-degree 492, bf16: 1.7-2x faster for F = 128-2048, 1.4x at F = 4096;
// 12.0M edges over the same nodes (mean in-degree 51.5, F = 128): 0.94 ms
// for the marked walk + 0.15 ms for the marks against 0.91 ms unmarked
// (ncu, serialised); 1.17M edges, mean in-degree 6.9: 2-60 % slower for F =
// 8-128.
#ifndef TFG_MXB_SPAN
#define TFG_MXB_SPAN 128
#endif
constexpr int64_t kMxbSpan = TFG_MXB_SPAN;

size_t max_backward_workspace_bytes(int64_t n, int64_t e, int64_t f) {
    if (n <= 0 || e <= 0 || f <= 0 || e < n * (f < kMxbSpan ? f : kMxbSpan)) return 0;
    return (static_cast<size_t>(e) + 255) & ~size_t(255);
}

// Features per mark bit: at most 8 groups, each a multiple of 4 features so
// that a lane's 16-byte slice lies in one group.
int mark_group(int64_t f) { return static_cast<int>(((f + 7) / 8 + 3) / 4 * 4); }

// Rows long enough for win marks take the row-per-warp kernel, with the marks when
// a workspace is given and over every out-edge when not: the same sums in the same
// order either way.  Shorter rows take the row walk.
cudaError_t launch_max_backward(const int32_t *rowptr_src, const int32_t *col_src,
                                const int32_t *perm_src, const int32_t *argmax,
                                const float *edge_weight, const float *grad_out, int64_t n,
                                int64_t e, int64_t f, float *grad_x, void *ws, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const bool v4 = f % 4 == 0 && aligned(argmax, 16) && aligned(grad_out, 16) && aligned(grad_x, 16);
    const int group = mark_group(f);
    MaxBwdArgs a{rowptr_src, col_src, perm_src, argmax, edge_weight, grad_out, n, f, e, grad_x, nullptr, group};
    if (col_src == nullptr || max_backward_workspace_bytes(n, e, f) == 0) {
        if (v4) return launch_walk<MaxBySource<4, 1>>(a, s);
        if (f <= 32) return launch_walk<MaxBySource<1, 1>>(a, s);
        if (f <= 64) return launch_walk<MaxBySource<1, 2>>(a, s);
        return launch_walk<MaxBySource<1, 4>>(a, s);
    }
    const int grid = balanced_grid(n, 0, 1);   // the kernel reads rowptr[N] for the split
    if (ws == nullptr) {
        if (v4) max_bwd_kernel<4, false><<<grid, kMxThreads, 0, s>>>(a);
        else max_bwd_kernel<1, false><<<grid, kMxThreads, 0, s>>>(a);
        return cudaGetLastError();
    }
    uint8_t *mark = static_cast<uint8_t *>(ws);
    a.mark = mark;
    const int mark_grid = sm_count() * 8;
    max_marks_zero<<<mark_grid, 256, 0, s>>>(mark, e);
    max_marks_set<<<mark_grid, f >= 256 ? 256 : 128, 0, s>>>(argmax, n, f, e, group, mark);
    if (v4) max_bwd_kernel<4, true><<<grid, kMxThreads, 0, s>>>(a);
    else max_bwd_kernel<1, true><<<grid, kMxThreads, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace tfg
