// Fused gather * weight * reduce over a CSR grouped by target: the message
// aggregation of tf_geometric (Fig. 1) with the reducer of Fig. 5b, which the
// paper implements as tf.math.unsorted_segment_* over the edge list
// (Section 2.1.2).  Grouping by target first turns the scatter-reduce into
// owner-computes row reductions: no atomics, a fixed summation order, and
// bit-identical results from run to run.
//
// One kernel for every layout and degree, aggregate_rows:
//  * One CTA of 28 warps per SM owns whole rows holding an equal share of edges
//    and row ends, and every warp an equal share of the CTA's (row_share.cuh),
//    so a hub row is shared by as many of the 28 warps as it needs: with four
//    CTAs of 8 warps an SM's hub row had 8 warps at its disposal and the
//    kernel waited for it.  A row that a warp finishes is written at once,
//    unless earlier warps hold parts of it: then its owner (the warp holding
//    its last edge) parks its own part in shared memory, and after the CTA's
//    one barrier adds the earlier warps' parts and its own in warp order.  No
//    global scratch, a fixed summation order.
//  * A warp walks its edges in windows of 32.  The ids are requested two windows
//    ahead and the weights (dinv[src], a dependent gather) one window ahead;
//    the window's (id, weight) pairs are staged in shared memory, and its rows
//    take their edges from it one after the other, so short rows share the
//    cost of a window.  What a row's end needs (its own row, x0, dinv) is
//    requested before the row's gathers.
//  * A row's edges are split among G = 32 / LPR lane groups, each covering the
//    row's features with LPR lanes (16-byte slices, or T single features a lane
//    in rows without 16-byte slices); D gathers are in flight per lane in full
//    windows, P in partial ones; the groups' sums are combined by a butterfly.
//  * Sums are blocked per window, so an fp32 chain is at most 32 / (G * CH) + degree / 32
//    additions long, CH the chains a lane keeps: two in rows of 17 to 31 slices, one
//    otherwise.  Slots without an edge are not loaded: an infinity in an unrelated row
//    never meets a zero weight.
//  * GCN mode without w_csr forms the weight on the fly:  out[t] = dinv[t] *
//    (sum_k dinv[col[k]] * x[col[k]] + fill * dinv[t] * x[t]), so no per-edge
//    weight array is read.  With w_csr it adds fill * dinv[t]^2 * x[t] to the
//    weighted sum.
//  * APPNP mode (one propagation step, Klicpera et al., the APPNP model the
//    paper lists in Section 2.2 and Table 1) is GCN mode with an epilogue:
//    out[t] = (1 - alpha) * gcn(h)[t] + alpha * x0[t], x0 read in its own
//    storage type X0T.  alpha = 0 is one SGC step.
//
// What bounds it.  Long rows: the gather from L2 (114.6M edges, mean in-degree
// 492: 1.62 ms for 256-byte bf16 rows against 1.27 ms for the bare gather; 2.77
// ms for 512-byte fp32 rows, 21 TB/s).  Short rows: instructions per row (1,024
// molecule graphs, mean in-degree 5, F = 128 fp32: 45 us, 250 instructions a
// row, issue 54 %).  Against the two kernels this one replaced (merge-path over
// 8-warp CTAs, and a row per warp from a shared counter): GCN bf16 1.74 -> 1.62
// ms and fp32 3.02 -> 2.77 ms at 114.6M edges; 169,343 nodes of mean in-degree
// 6.9, F = 41, ten hops 1,530 -> 646 us; sum + mean + max of 19,717 nodes,
// F = 256, 287 -> 66 us; 60,000 nodes, 900,000 edges, F = 100 weighted, two
// passes 244 -> 83 us; 2,708 nodes, F = 64, 11.4 us in two launches -> 6.4 us.
//
// Shared by aggregate.cu (one-hop entry points) and propagate.cu (multi-hop);
// each translation unit instantiates the variants it launches.
#pragma once
#include <math_constants.h>

#include "row_share.cuh"

namespace tfg {
namespace {

// Tuning knobs (compile-time; the defaults are the measured best on GB300).
// Warps of a CTA, one CTA per SM: 28 (72 registers a thread) against 24 and 32
// at 114.6M edges: bf16 1.617 / 1.693 / 1.611 ms, fp32 2.77 / 2.83 / 2.84 ms;
// 900,000 edges, F = 100: 41 / 42 / 41 us a pass.
#ifndef TFG_AGG_WARPS
#define TFG_AGG_WARPS 28
#endif
// 16-byte fp32 gathers in flight per lane in full windows (bf16, whose 8
// features a slice take twice the registers, keeps 4): 8 against 4 at 114.6M
// edges 2.77 / 2.99 ms.
#ifndef TFG_AGG_DEPTH
#define TFG_AGG_DEPTH 8
#endif
// Gathers in flight per lane in partial windows of rows of 8 lanes (4 or more lane
// groups): 2 against 4, two passes over 100,000 nodes and 1.5M edges, F = 32 fp32,
// 92.8 / 95.9 us.
#ifndef TFG_AGG_PART4
#define TFG_AGG_PART4 2
#endif
constexpr int kAggWarps = TFG_AGG_WARPS;
// 16-byte bf16 rows with two chains, whose registers are short: 24 against 28, GCN of
// 23.3M edges, F = 136 / 200 / 248: 757 / 867 / 971 us against 835 / 979 / 1100 (one
// chain 711 / 804 / 886); 169,343 nodes of mean in-degree 6.9: 117 / 138 / 154 us against
// 123 / 146 / 161 (105 / 123 / 135).
#ifndef TFG_AGG_WARPS_CHAINS
#define TFG_AGG_WARPS_CHAINS 24
#endif
__host__ __device__ constexpr int agg_warps(int vec, int chains) {
    return vec == 8 && chains > 1 ? TFG_AGG_WARPS_CHAINS : kAggWarps;
}
// Work (edges + kRowCost per row) a warp should have, at least: 8 against 32 on
// 2,708 nodes and 13,264 edges: 6.4 / 8.0 us.
constexpr int kAggMinWork = 8;

struct AggArgs {
    const int32_t *rowptr;
    const int32_t *col;
    const float *w;     // CSR-order weights or null
    const float *dinv;  // GCN mode
    const void *x;
    float *out;
    int64_t n;
    int64_t f;
    int mean;
    int add_self;
    float fill;
    const void *x0;     // APPNP mode: the teleport features x0 [N, F]
    float alpha;        // APPNP mode: teleport weight
    float beta;         // APPNP mode: 1 - alpha, rounded once on the host
};

enum Kind { kSumLike = 0, kMax = 1, kGcn = 2, kAppnp = 3 };

// KIND: kSumLike (mean by the runtime flag), kMax, kGcn, kAppnp.
template <typename XT, int VEC, int LPR, int T, int KIND, typename X0T>
struct RowAgg {
    using V = VecLoad<XT, VEC>;
    using V0 = VecLoad<X0T, VEC>;
    static constexpr bool kIsMax = KIND == kMax, kGcnLike = KIND == kGcn || KIND == kAppnp, kX0 = KIND == kAppnp;
    static constexpr int G = 32 / LPR;
    static constexpr int kTile = LPR * VEC * T;               // features of one pass
    static constexpr int D0 = T > 1 || VEC == 8 ? 4 : TFG_AGG_DEPTH;
    static constexpr int D = D0 * G > 32 ? 32 / G : D0;       // gathers in flight per lane, full windows
    static constexpr int P = G >= 4 ? TFG_AGG_PART4 : 4;       // the same, partial windows: about 8 edges a step
    static_assert(32 % (G * D) == 0 && G * P <= 32, "steps of G * D slots must tile the 32-edge window");

    static __device__ __forceinline__ float combine(float a, float b) { return kIsMax ? fmaxf(a, b) : a + b; }
    static __device__ __forceinline__ float identity() { return kIsMax ? -CUDART_INF_F : 0.f; }

    // part += w * row (max: where ok); the slots of a partial window that hold no
    // edge carry zero weight and a zero row, so they add an exact zero.
    template <bool CHECK>
    static __device__ __forceinline__ void axpy(float (&part)[VEC], float w, const typename V::Raw &raw, bool ok) {
        float v[VEC];
        V::widen(raw, v);
        if constexpr (kIsMax) {
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                const float p = w * v[q];
                part[q] = fmaxf(part[q], !CHECK || ok ? p : -CUDART_INF_F);
            }
        } else if constexpr (VEC % 2 == 0) {
            const float2 w2 = make_float2(w, w);
#pragma unroll
            for (int q = 0; q < VEC; q += 2) {
                const float2 r = fma2(make_float2(v[q], v[q + 1]), w2, make_float2(part[q], part[q + 1]));
                part[q] = r.x;
                part[q + 1] = r.y;
            }
        } else {
#pragma unroll
            for (int q = 0; q < VEC; ++q) part[q] = fmaf(w, v[q], part[q]);
        }
    }

    // the sum of the chains of a window, in the first (pairs through fma2: times one is exact)
    template <int CH>
    static __device__ __forceinline__ void join_chains(float (&part)[CH][T][VEC]) {
        if constexpr (CH > 1) {
            static_assert(CH == 2 && !kIsMax, "one chain or two, of sums");
            const float2 one = make_float2(1.f, 1.f);
#pragma unroll
            for (int i = 0; i < T; ++i)
#pragma unroll
                for (int q = 0; q < VEC; q += 2) {
                    const float2 r = fma2(make_float2(part[1][i][q], part[1][i][q + 1]), one,
                                          make_float2(part[0][i][q], part[0][i][q + 1]));
                    part[0][i][q] = r.x;
                    part[0][i][q + 1] = r.y;
                }
        }
    }

    // Final values of VEC features: dt * (acc + fill dt self), with given edge
    // weights acc + fill dt^2 self; acc / deg for a mean; 0 for an empty max.
    static __device__ __forceinline__ void finish(const AggArgs &a, float c1, float c2, int32_t deg, float (&r)[VEC],
                                                  const typename V::Raw &self, const typename V0::Raw &x0) {
        if constexpr (kIsMax) {
#pragma unroll
            for (int q = 0; q < VEC; ++q) r[q] = deg == 0 ? 0.f : r[q];
        } else if constexpr (kGcnLike) {
            float xt[VEC];
            V::widen(self, xt);
#pragma unroll
            for (int q = 0; q < VEC; ++q) r[q] = c2 * fmaf(c1, xt[q], r[q]);
            if constexpr (kX0) {
                V0::widen(x0, xt);
#pragma unroll
                for (int q = 0; q < VEC; ++q) r[q] = fmaf(a.alpha, xt[q], a.beta * r[q]);
            }
        } else if (a.mean && deg > 0) {
#pragma unroll
            for (int q = 0; q < VEC; ++q) r[q] /= static_cast<float>(deg);
        }
    }
    static __device__ __forceinline__ void write(float *o, const float (&r)[VEC]) {
        if constexpr (VEC % 4 == 0) {
#pragma unroll
            for (int q = 0; q < VEC; q += 4)
                *reinterpret_cast<float4 *>(o + q) = make_float4(r[q], r[q + 1], r[q + 2], r[q + 3]);
        } else {
#pragma unroll
            for (int q = 0; q < VEC; ++q) o[q] = r[q];
        }
    }
    static __device__ __forceinline__ void factors(const AggArgs &a, float dt, float &c1, float &c2) {
        c1 = a.add_self ? a.fill * dt : 0.f;
        c2 = dt;
        if (a.w) {
            c1 *= dt;
            c2 = 1.f;
        }
    }
};

// CH: chains of additions a lane keeps within a window, edge by edge in turn.
template <typename XT, int VEC, int LPR, int T, int CH, int KIND, typename X0T>
__global__ void __launch_bounds__(agg_warps(VEC, CH) * 32, 1) aggregate_rows(AggArgs a) {
    using S = RowAgg<XT, VEC, LPR, T, KIND, X0T>;
    using V = typename S::V;
    using V0 = typename S::V0;
    constexpr int G = S::G, D = S::D, P = S::P;
    constexpr int W = agg_warps(VEC, CH);
    static_assert(D % CH == 0 && P % CH == 0, "steps give every chain the same number of edges");
    extern __shared__ __align__(16) float s_parts[];          // tails [warp][kTile], heads [warp][kTile]
    __shared__ int64_t s_row[2];
    __shared__ int32_t s_tail_row[W], s_head_row[W];
    __shared__ __align__(16) float2 s_stage[W][64];    // a window's (id, weight) pairs, and room to read past them
    WarpShare<W> sh;
    if (!sh.init(a.rowptr, a.n, kAggMinWork, s_row)) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane % LPR, g = lane / LPR;
    float2 *stage = s_stage[warp];
    const uint32_t f = static_cast<uint32_t>(a.f);
    const uint32_t row_bytes = f * static_cast<uint32_t>(sizeof(XT));
    const int32_t kb = sh.kb, tb = sh.tb;
    const bool self = S::kGcnLike && a.add_self;

    for (uint32_t ft = blockIdx.y * S::kTile; ft < f; ft += gridDim.y * S::kTile) {
        // this lane's features: f0 + i * LPR * VEC, i < T; past F they are not touched
        const uint32_t f0 = ft + sub * VEC;
        const int own = f0 < f ? min(T, static_cast<int>((f - f0 + LPR * VEC - 1) / (LPR * VEC))) : 0;
        const char *xb = reinterpret_cast<const char *>(static_cast<const XT *>(a.x) + (own > 0 ? f0 : 0));
        auto row = [&](uint32_t id) { return reinterpret_cast<const XT *>(xb + static_cast<uint64_t>(id) * row_bytes); };
        // T = 1: lanes past F read (and never use) the row's first features
        auto load = [&](typename V::Raw (&r)[T], const XT *p, bool ok) {
#pragma unroll
            for (int i = 0; i < T; ++i) {
                const bool on = T == 1 ? ok : (ok && i < own);
                r[i] = on ? V::raw(p + i * LPR * VEC) : V::zero();
            }
        };
        if (lane == 0) s_head_row[warp] = -1;
        // Windows of 32 edges: ids requested two windows ahead, weights one.
        uint32_t ahead = static_cast<uint32_t>(sh.ka);      // the window after the staged one
        auto col_at = [&](uint32_t k) { return k + lane < static_cast<uint32_t>(kb) ? ld_stream(a.col + k + lane) : 0; };
        auto weight_at = [&](uint32_t k, int32_t id) {
            if (k + lane >= static_cast<uint32_t>(kb)) return 0.f;
            if (a.w) return ld_stream(a.w + k + lane);
            return S::kGcnLike ? __ldg(a.dinv + id) : 1.f;
        };
        int32_t c1 = col_at(ahead), c2 = col_at(ahead + 32);
        float w1 = weight_at(ahead, c1);
        auto next_window = [&]() {
            __syncwarp();                                  // the previous window's reads are done
            stage[lane] = make_float2(__int_as_float(c1), w1);
            __syncwarp();
            ahead += 32;
            c1 = c2;
            w1 = weight_at(ahead, c1);
            c2 = col_at(ahead + 32);
        };
        // row ends and dinv of 32 rows
        int32_t t = sh.ta, rwin;
        float dwin = 0.f;
        int tl = 0;                                        // row t is lane tl of them
        auto row_window = [&]() {
            const int64_t r = static_cast<int64_t>(t) + lane;
            rwin = r < a.n ? __ldg(a.rowptr + r + 1) : 0;
            if (S::kGcnLike) dwin = r < a.n ? __ldg(a.dinv + r) : 0.f;
            tl = 0;
        };
        row_window();
        next_window();

        float acc[T][VEC];
        int32_t k = sh.ka, rbeg = __ldg(a.rowptr + t);
        int j = 0;                                         // position in the staged window
        // edges [j, j + cnt) of the staged window into part
        auto some = [&](float (&part)[CH][T][VEC], int cnt) {
            const float2 *sp = stage + j + g;
            int m = cnt - g;                               // this group's are sp[0], sp[G], ... below m
#pragma unroll 1
            for (int e = 0; e < cnt; e += G * P) {
                typename V::Raw raw[P][T];
                float w[P];
#pragma unroll
                for (int u = 0; u < P; ++u) {
                    const float2 iw = sp[u * G];
                    const bool ok = m > u * G;
                    w[u] = ok ? iw.y : 0.f;
                    load(raw[u], row(static_cast<uint32_t>(__float_as_int(iw.x))), ok);
                }
#pragma unroll
                for (int u = 0; u < P; ++u)
#pragma unroll
                    for (int i = 0; i < T; ++i) S::template axpy<true>(part[u % CH][i], w[u], raw[u][i], m > u * G);
                sp += G * P;
                m -= G * P;
            }
        };
        auto clear = [&](float (&v)[CH][T][VEC]) {
#pragma unroll
            for (int c = 0; c < CH; ++c)
#pragma unroll
                for (int i = 0; i < T; ++i)
#pragma unroll
                    for (int q = 0; q < VEC; ++q) v[c][i][q] = S::identity();
        };
        for (;;) {
            const bool closes = t < tb;
            const int32_t rend = closes ? lane_get(rwin, tl) : kb;
            typename V::Raw xt[T];
            typename V0::Raw x0t[T];
            if (S::kGcnLike) load(xt, row(static_cast<uint32_t>(t)), self && closes);   // what the row end
            if (S::kX0) {                                                                // needs besides the sum
                const X0T *p = static_cast<const X0T *>(a.x0) + static_cast<uint64_t>(static_cast<uint32_t>(t)) * f + (own > 0 ? f0 : 0);
#pragma unroll
                for (int i = 0; i < T; ++i) x0t[i] = closes && i < own ? V0::raw(p + i * LPR * VEC) : V0::zero();
            }
            int rem = rend - k;
            k = rend;
            if (j == 32 && rem > 0) {
                next_window();
                j = 0;
            }
            if (rem <= 32 - j) {                           // the rest of the row lies in this window
                float part[CH][T][VEC];
                clear(part);
                some(part, rem);
                S::join_chains(part);
#pragma unroll
                for (int i = 0; i < T; ++i)
#pragma unroll
                    for (int q = 0; q < VEC; ++q) acc[i][q] = part[0][i][q];
                j += rem;
            } else {
#pragma unroll
                for (int i = 0; i < T; ++i)
#pragma unroll
                    for (int q = 0; q < VEC; ++q) acc[i][q] = S::identity();
                while (rem > 0) {
                    if (j == 32) {
                        next_window();
                        j = 0;
                    }
                    const int cnt = min(rem, 32 - j);
                    float part[CH][T][VEC];                // sums are blocked per window
                    clear(part);
                    if (cnt == 32) {
#pragma unroll
                        for (int e = 0; e < 32; e += G * D) {
                            typename V::Raw raw[D][T];
                            float w[D];
#pragma unroll
                            for (int u = 0; u < D; ++u) {
                                const float2 iw = stage[e + u * G + g];
                                w[u] = iw.y;
                                load(raw[u], row(static_cast<uint32_t>(__float_as_int(iw.x))), true);
                            }
#pragma unroll
                            for (int u = 0; u < D; ++u)
#pragma unroll
                                for (int i = 0; i < T; ++i) S::template axpy<false>(part[u % CH][i], w[u], raw[u][i], true);
                        }
                    } else {
                        some(part, cnt);
                    }
                    S::join_chains(part);
#pragma unroll
                    for (int i = 0; i < T; ++i)
#pragma unroll
                        for (int q = 0; q < VEC; ++q) acc[i][q] = S::combine(acc[i][q], part[0][i][q]);
                    rem -= cnt;
                    j += cnt;
                }
            }
#pragma unroll
            for (int s = LPR; s < 32; s <<= 1)
#pragma unroll
                for (int i = 0; i < T; ++i)
#pragma unroll
                    for (int q = 0; q < VEC; ++q)
                        acc[i][q] = S::combine(acc[i][q], lane_xor(acc[i][q], s));
            if (!closes) break;
            float c1f = 0.f, c2f = 1.f;
            if (S::kGcnLike) S::factors(a, lane_get(dwin, tl), c1f, c2f);
            if (t == sh.ta && sh.head_split) {             // parts of it sit with earlier warps
                if (g == 0) {
#pragma unroll
                    for (int i = 0; i < T; ++i)
#pragma unroll
                        for (int q = 0; q < VEC; ++q)
                            s_parts[(W + warp) * S::kTile + (i * LPR + sub) * VEC + q] = acc[i][q];
                }
                if (lane == 0) s_head_row[warp] = t;
            } else if (g == 0) {
                float *o = a.out + static_cast<uint64_t>(static_cast<uint32_t>(t)) * f + f0;
#pragma unroll
                for (int i = 0; i < T; ++i) {
                    S::finish(a, c1f, c2f, rend - rbeg, acc[i], xt[i], x0t[i]);
                    if (i < own) S::write(o + i * LPR * VEC, acc[i]);
                }
            }
            rbeg = rend;
            ++t;
            if (++tl == 32) row_window();
        }
        // the part of row tb held here (empty when the share ends on a row end)
        if (g == 0) {
#pragma unroll
            for (int i = 0; i < T; ++i)
#pragma unroll
                for (int q = 0; q < VEC; ++q) s_parts[warp * S::kTile + (i * LPR + sub) * VEC + q] = acc[i][q];
        }
        if (lane == 0) s_tail_row[warp] = tb;
        __syncthreads();
        const int32_t hr = s_head_row[warp];
        if (hr >= 0 && g == 0) {                           // earlier parts in warp order, then ours
            int first = warp;
            while (first > 0 && s_tail_row[first - 1] == hr) --first;
            const int32_t deg = __ldg(a.rowptr + hr + 1) - __ldg(a.rowptr + hr);
            float c1f = 0.f, c2f = 1.f;
            if (S::kGcnLike) S::factors(a, __ldg(a.dinv + hr), c1f, c2f);
            typename V::Raw xt[T];
            load(xt, row(static_cast<uint32_t>(hr)), self);
            const uint64_t at0 = static_cast<uint64_t>(static_cast<uint32_t>(hr)) * f + f0;
#pragma unroll
            for (int i = 0; i < T; ++i) {
                if (i >= own) continue;
                const int at = (i * LPR + sub) * VEC;
                float r[VEC];
#pragma unroll
                for (int q = 0; q < VEC; ++q) r[q] = S::identity();
                for (int s = first; s < warp; ++s)
#pragma unroll
                    for (int q = 0; q < VEC; ++q) r[q] = S::combine(r[q], s_parts[s * S::kTile + at + q]);
#pragma unroll
                for (int q = 0; q < VEC; ++q) r[q] = S::combine(r[q], s_parts[(W + warp) * S::kTile + at + q]);
                typename V0::Raw x0t = V0::zero();
                if (S::kX0) x0t = V0::raw(static_cast<const X0T *>(a.x0) + at0 + i * LPR * VEC);
                S::finish(a, c1f, c2f, deg, r, xt[i], x0t);
                S::write(a.out + at0 + i * LPR * VEC, r);
            }
        }
        __syncthreads();                                   // before the next tile reuses the parts
    }
}

template <typename XT, int VEC, int LPR, int T, int KIND, typename X0T, int CH = 1>
cudaError_t launch_rows(const AggArgs &a, cudaStream_t s) {
    using S = RowAgg<XT, VEC, LPR, T, KIND, X0T>;
    auto *kernel = aggregate_rows<XT, VEC, LPR, T, CH, KIND, X0T>;
    const int64_t tiles = (a.f + S::kTile - 1) / S::kTile;
    constexpr int threads = agg_warps(VEC, CH) * 32;
    constexpr int smem = 2 * agg_warps(VEC, CH) * S::kTile * static_cast<int>(sizeof(float));
    if constexpr (smem > 32 * 1024) {   // with the static part above the 48 KB every launch may use
        const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (err != cudaSuccess) return err;
    }
    const dim3 grid(static_cast<unsigned>(min64(a.n, static_cast<int64_t>(sm_count()))),
                    static_cast<unsigned>(min64(tiles, 65535)));
    kernel<<<grid, threads, smem, s>>>(a);
    return cudaGetLastError();
}

// Rows in whole 16-byte slices: LPR lanes, the fewest that cover the row (wider
// rows are cut into tiles of 32 lanes, a CTA column per tile).
template <typename XT, int VEC, int KIND, typename X0T = XT>
cudaError_t launch_rows_vec(const AggArgs &a, cudaStream_t s) {
    const int64_t slices = a.f / VEC;
    if (slices <= 8) return launch_rows<XT, VEC, 8, 1, KIND, X0T>(a, s);
    if (slices <= 16) return launch_rows<XT, VEC, 16, 1, KIND, X0T>(a, s);
    if constexpr (KIND != kMax) {
        if (slices < 32) return launch_rows<XT, VEC, 32, 1, KIND, X0T, 2>(a, s);
    }
    return launch_rows<XT, VEC, 32, 1, KIND, X0T>(a, s);
}

// Any other row: one feature per lane, T features a lane in one walk, so that
// the fewest lanes idle and the edges are walked once per 128 features.
template <typename XT, int KIND, typename X0T = XT>
cudaError_t launch_rows_scalar(const AggArgs &a, cudaStream_t s) {
    if (a.f <= 8) return launch_rows<XT, 1, 8, 1, KIND, X0T>(a, s);
    if (a.f <= 16) return launch_rows<XT, 1, 16, 1, KIND, X0T>(a, s);
    if (a.f <= 32) return launch_rows<XT, 1, 16, 2, KIND, X0T>(a, s);
    if (a.f <= 48) return launch_rows<XT, 1, 16, 3, KIND, X0T>(a, s);
    const int64_t passes = (a.f + 127) / 128, per = (a.f + passes - 1) / passes;
    if (per <= 64) return launch_rows<XT, 1, 32, 2, KIND, X0T>(a, s);
    if (per <= 96) return launch_rows<XT, 1, 32, 3, KIND, X0T>(a, s);
    return launch_rows<XT, 1, 32, 4, KIND, X0T>(a, s);
}

}  // namespace
}  // namespace tfg
