// The three edge passes of the additive (GAT) attention as row-walk policies:
// forward, backward by target, backward by source.  Lane layout as in the
// aggregation: LPR lanes cover a row in 16-byte slices (T = 1, a slice lies in one
// head), or with T single features a lane, feature i * LPR + sub in turn; G = 32 /
// LPR lane groups take every G-th edge.  Every lane forms the logits of its own
// heads (NH of them: 1 when all its features share a head), so no weight passes
// between lanes.  Logits are in base-2 units.
#pragma once
#include <math_constants.h>

#include "row_walk.cuh"

namespace tfg {

struct GatArgs {
    const int32_t *rowptr, *col;         // CSR of the pass
    const void *x;
    int64_t n;
    int heads, channels;
    float slope;
    const float *s_src, *s_dst;          // base-2 node scores [N, H]
    float *out, *alpha;                  // forward
    const float *fwd_out, *grad_out;     // backward by target
    float4 *stats;                       // [N, H]: (s_dst, m, 1 / den, beta)
    float *ds_dst, *ds_src, *grad_x;
    const float *a_src, *a_dst;          // backward by source
    __host__ __device__ uint32_t width() const { return static_cast<uint32_t>(heads) * static_cast<uint32_t>(channels); }
    __host__ __device__ bool statistics() const { return alpha != nullptr; }
};

namespace {

// What bounds it: instructions on short rows (169,343 nodes, mean in-degree 6.9, 8
// x 16 fp32: forward 106, by target 135, by source 168 us, against 36-45 us for
// the gathered bytes at the L2 rate), the gathers and the weights' arithmetic on
// long ones (by source at 114.6M edges, 8 x 16 bf16: 640 bytes an edge, 4.97 ms, 14.8
// TB/s; 7.9-8.0 ms in a row-per-warp kernel).  One head of 41 channels on the first graph,
// alpha written: 199 us; 1,753 in a row-per-warp kernel whose hub rows one warp walked.
//
// Tuning knobs.  Warps per CTA (one CTA per SM).  By target: 28 against 24 and 32 on the
// first graph, forward 107 / 112 / 100 us, backward 135 / 149 / 131, 3 x 32 fp32 over 10M
// edges 345 / 353 / 335 (odd widths of several heads, which spill at 28, spill more
// at 32); rows of 4 lanes take 32: 4 x 8 bf16, 100,000 nodes of mean degree 29, 90 us a call
// against 94.  By source: 168 us with 28, 185 with 24, 181 with 32; 4M edges of mean degree
// 40 245 / 264 / 257.
#ifndef TFG_GW_WARPS
#define TFG_GW_WARPS 28
#endif
#ifndef TFG_GW_SRC_WARPS
#define TFG_GW_SRC_WARPS 28
#endif
// Gathers in flight per lane: 4 against 2, 8 x 16 fp32 calls on the first graph 143 / 180
// us; rows of 8 slices and fewer the same with either.
#ifndef TFG_GW_DEPTH
#define TFG_GW_DEPTH 4
#endif
// The same by source: 168 / 216 us; over 114.6M edges 4.97 / 8.7 ms.
#ifndef TFG_GW_SRC_DEPTH
#define TFG_GW_SRC_DEPTH 4
#endif
// By source with 32-byte gradient slices (VEC = 8: half the lanes a row, so an edge's
// weight is formed by half as many lanes, and twice the bytes a load; its full windows are
// unrolled, 10.1 ms a call against 10.5 rolled): 114.6M edges 4.98 ms with 16 warps, 20
// 5.25, 12 5.46.
#ifndef TFG_GW_SRC8_WARPS
#define TFG_GW_SRC8_WARPS 16
#endif
#ifndef TFG_GW_SRC8_DEPTH
#define TFG_GW_SRC8_DEPTH 4
#endif

template <int VEC>
__device__ __forceinline__ void gw_axpy(float (&acc)[VEC], float w, const float (&v)[VEC]) {
    if constexpr (VEC % 2 == 0) {
        const float2 w2 = make_float2(w, w);
#pragma unroll
        for (int q = 0; q < VEC; q += 2) {
            const float2 r = fma2(make_float2(v[q], v[q + 1]), w2, make_float2(acc[q], acc[q + 1]));
            acc[q] = r.x;
            acc[q + 1] = r.y;
        }
    } else {
#pragma unroll
        for (int q = 0; q < VEC; ++q) acc[q] = fmaf(w, v[q], acc[q]);
    }
}

template <int VEC>
__device__ __forceinline__ void gw_load(const float *p, float (&r)[VEC]) {
    if constexpr (VEC % 4 == 0) {
#pragma unroll
        for (int q = 0; q < VEC; q += 4) {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(p + q));
            r[q] = v.x; r[q + 1] = v.y; r[q + 2] = v.z; r[q + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int q = 0; q < VEC; ++q) r[q] = __ldg(p + q);
    }
}

template <int VEC>
__device__ __forceinline__ void gw_store(float *p, const float (&r)[VEC]) {
    if constexpr (VEC % 4 == 0) {
#pragma unroll
        for (int q = 0; q < VEC; q += 4)
            *reinterpret_cast<float4 *>(p + q) = make_float4(r[q], r[q + 1], r[q + 2], r[q + 3]);
    } else {
#pragma unroll
        for (int q = 0; q < VEC; ++q) p[q] = r[q];
    }
}

// A lane's share of a dot product.  Eight features are two fours added, as two lanes of
// four would be by the first exchange of a head's sum: the sum over a head has the same
// bits in either slice width (and in gw_spread_sums), so that a difference of two equal
// products is zero whichever pass formed each.
template <int VEC>
__device__ __forceinline__ float gw_dot(const float (&a)[VEC], const float (&b)[VEC]) {
    static_assert(VEC == 4 || VEC == 8, "whole 16-byte slices");
    float r[VEC / 4];
#pragma unroll
    for (int i = 0; i < VEC / 4; ++i) {
        float2 d = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 4 * i; q < 4 * i + 4; q += 2)
            d = fma2(make_float2(a[q], a[q + 1]), make_float2(b[q], b[q + 1]), d);
        r[i] = d.x + d.y;
    }
    return VEC == 8 ? r[0] + r[VEC / 4 - 1] : r[0];
}

// Sum over the lanes of a head (a power of two: LH, or hl where LH = 0), to each of them.
template <int LH>
__device__ __forceinline__ float gw_head_sum(float v, int hl) {
    if constexpr (LH > 0) {
#pragma unroll
        for (int o = 1; o < LH; o <<= 1) v += lane_xor(v, o);
    } else {
        for (int o = 1; o < hl; o <<= 1) v += lane_xor(v, o);
    }
    return v;
}

// The head sums of D values, spread over the LH lanes of the head: in log2(LH) exchanges
// each lane gives away one half of its values and takes its neighbour's other half, so
// that D - 1 values are exchanged instead of D log2(LH).  The lane ends with the first
// max(1, D / LH) entries of v complete; w and b follow their values.  lane: the lane's
// place in the head.  Lanes left with the same value (LH > D): all but the first get w = 0.
template <int LH, int D>
__device__ __forceinline__ void gw_spread_sums(float (&v)[D], float (&w)[D], float (&b)[D], int lane) {
    int n = D;
#pragma unroll
    for (int o = 1; o < LH; o <<= 1) {
        const bool up = (lane & o) != 0;
        if (n > 1) {
            n /= 2;
#pragma unroll
            for (int i = 0; i < D / 2; ++i) {
                if (i >= n) continue;
                const float give = up ? v[i] : v[n + i];
                v[i] = (up ? v[n + i] : v[i]) + lane_xor(give, o);
                w[i] = up ? w[n + i] : w[i];
                b[i] = up ? b[n + i] : b[i];
            }
        } else {
            v[0] += lane_xor(v[0], o);
            w[0] = up ? 0.f : w[0];
        }
    }
}

// 2^(m_old - m_new) for base-2 maxima; 0 for an empty state (m_old = -inf).
__device__ __forceinline__ float gw_rescale(float m_old, float m_new) {
    return m_old == -CUDART_INF_F ? 0.f : exp2f(m_old - m_new);
}

// A lane's place in a row of heads * channels features.
template <int VEC, int LPR, int T, int NH>
struct GatLane {
    int sub, g, own;                 // own: features i < own of this lane exist
    uint32_t f, f0;
    int head[NH];
    __device__ __forceinline__ void place(uint32_t ft, int heads, int channels) {
        const int lane = threadIdx.x & 31;
        sub = lane % LPR;
        g = lane / LPR;
        f = static_cast<uint32_t>(heads) * static_cast<uint32_t>(channels);
        f0 = ft + sub * VEC;
        own = f0 < f ? min(T, static_cast<int>((f - f0 + LPR * VEC - 1) / (LPR * VEC))) : 0;
#pragma unroll
        for (int i = 0; i < NH; ++i) head[i] = i < own ? static_cast<int>((f0 + i * LPR * VEC) / channels) : 0;
    }
};

// Softmax passes by target.  TARGET_BWD = false: out = sum of alpha x, and alpha
// if wanted.  TARGET_BWD = true (one slice a lane, T = 1): the row's statistics for the
// source pass and
//   ds_dst = sum of alpha phi (dalpha - beta),  dalpha = <grad_out[t], x[src]>,
// phi the LeakyReLU's slope at the edge.  A lane keeps its own slice's share of dalpha and
// of beta = <grad_out[t], out[t]>, subtracts them edge by edge, and the shares are added
// over the lanes of the head once a row: an edge costs what it does in the forward, and
// the difference, which cancels where an edge has most of its row's weight (to nothing
// where t has one in-edge), is taken before anything is rounded to a larger sum.
// CH: chains of additions a lane keeps within a window, edge by edge in turn: two in
// rows of more than 16 slices, whose 32 lanes leave one lane group.  softmax_fast adds a
// window's weights on 32 / H score lanes and rescales once a window, a lane here after every
// step of D edges; with one chain the walk's error against 64 bits was 1-5 % above
// it, with two it is 1-4 % below, and the walk is faster: 8 x 16 fp32 on 169,343 nodes 157
// us against 186, on 100,000 nodes of mean in-degree 24 168 against 188.
template <typename XT, int VEC, int LPR, int T, int NH, bool TARGET_BWD, int CH = 1>
struct GatByTarget {
    using V = VecLoad<XT, VEC>;
    static constexpr int kWarps = LPR == 4 ? 32 : TFG_GW_WARPS, kLpr = LPR, G = 32 / LPR;
    static constexpr int kTile = LPR * VEC * T, kHeadsPerLane = T;
    static constexpr int kSums = TARGET_BWD ? 1 : T * VEC;      // dz, or acc
    static constexpr int kState = kSums + 2 * NH, kHeld = 0;
    static_assert(!TARGET_BWD || (T == 1 && NH == 1), "the backward has one slice a lane");
    static constexpr int kStepFull = TFG_GW_DEPTH * G > 32 ? 32 / G : TFG_GW_DEPTH;   // gathers in flight per lane
    static_assert(32 % (G * kStepFull) == 0, "a full window is read in whole steps");
    static constexpr int kStepPart = walk_part(G) < kStepFull ? walk_part(G) : kStepFull;   // the same, a window's rest
    const GatArgs &a;
    GatLane<VEC, LPR, T, NH> at;
    const char *xb;
    uint32_t row_bytes;
    float *scratch;                      // [warp][heads of the tile] (m, den), for alpha
    float sd[NH], m[NH], den[NH], acc[T][VEC];
    float gt[TARGET_BWD ? VEC : 1], beta, dz;   // backward: this slice of grad_out[t], its share of beta and of the sum

    __device__ __forceinline__ GatByTarget(const GatArgs &args, uint32_t ft, float *, float *scr) : a(args), scratch(scr) {
        at.place(ft, a.heads, a.channels);
        xb = reinterpret_cast<const char *>(static_cast<const XT *>(a.x) + (at.own > 0 ? at.f0 : 0));
        row_bytes = at.f * static_cast<uint32_t>(sizeof(XT));
    }
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            m[i] = -CUDART_INF_F;
            den[i] = 0.f;
        }
        dz = 0.f;
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int q = 0; q < VEC; ++q) acc[i][q] = 0.f;
    }
    __device__ __forceinline__ void open(int32_t t, int32_t, int32_t) {
#pragma unroll
        for (int i = 0; i < NH; ++i)
            sd[i] = __ldg(a.s_dst + static_cast<uint64_t>(static_cast<uint32_t>(t)) * a.heads + at.head[i]);
        if constexpr (TARGET_BWD) {
            float o[VEC];
#pragma unroll
            for (int q = 0; q < VEC; ++q) gt[q] = o[q] = 0.f;
            if (at.own > 0) {
                const uint64_t row = static_cast<uint64_t>(static_cast<uint32_t>(t)) * at.f + at.f0;
                gw_load(a.grad_out + row, gt);
                gw_load(a.fwd_out + row, o);
            }
            beta = gw_dot(gt, o);
        }
        clear();
    }
    // a window's sums
    struct Window {
        float part[CH][T][VEC], dpart[CH][NH], zpart[CH];
    };
    // D edges of the group, sp[0], sp[G], ... (CHECK: those below left)
    template <int D, bool CHECK>
    __device__ __forceinline__ void step(const int32_t *sp, int left, Window &s) {
        static_assert(D % CH == 0, "a step gives every chain the same number of edges");
        typename V::Raw raw[D][T];
        float z[D][NH];
#pragma unroll
        for (int u = 0; u < D; ++u) {
            const uint32_t id = static_cast<uint32_t>(sp[u * G]);
            const bool ok = !CHECK || left > u * G;
            const XT *row = reinterpret_cast<const XT *>(xb + static_cast<uint64_t>(id) * row_bytes);
#pragma unroll
            for (int i = 0; i < NH; ++i)
                z[u][i] = ok ? __ldg(a.s_src + static_cast<uint64_t>(id) * a.heads + at.head[i]) : 0.f;
#pragma unroll
            for (int i = 0; i < T; ++i)
                raw[u][i] = (T == 1 ? ok : ok && i < at.own) ? V::raw(row + i * LPR * VEC) : V::zero();
        }
        float l[D][NH], w[D][NH];
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            float top = m[i];
#pragma unroll
            for (int u = 0; u < D; ++u) {
                z[u][i] += sd[i];
                l[u][i] = z[u][i] > 0.f ? z[u][i] : a.slope * z[u][i];
                if (CHECK && left <= u * G) l[u][i] = -CUDART_INF_F;
                top = fmaxf(top, l[u][i]);
            }
            if (top > m[i]) {                           // a new running maximum: rescale the sums so far
                const float sc = gw_rescale(m[i], top);
                den[i] *= sc;
                dz *= sc;
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    s.dpart[c][i] *= sc;
                    s.zpart[c] *= sc;
                }
#pragma unroll
                for (int j = 0; j < T; ++j) {
                    if (TARGET_BWD || (NH > 1 && j != i)) continue;
#pragma unroll
                    for (int q = 0; q < VEC; ++q) {
                        acc[j][q] *= sc;
#pragma unroll
                        for (int c = 0; c < CH; ++c) s.part[c][j][q] *= sc;
                    }
                }
                m[i] = top;
            }
#pragma unroll
            for (int u = 0; u < D; ++u) {
                const float p = !CHECK || left > u * G ? exp2f(l[u][i] - m[i]) : 0.f;
                s.dpart[u % CH][i] += p;
                w[u][i] = TARGET_BWD && z[u][i] <= 0.f ? a.slope * p : p;
            }
        }
#pragma unroll
        for (int u = 0; u < D; ++u)
#pragma unroll
            for (int i = 0; i < T; ++i) {
                float v[VEC];
                V::widen(raw[u][i], v);
                if constexpr (TARGET_BWD) {
                    const float diff = gw_dot(gt, v) - beta;
                    s.zpart[u % CH] = fmaf(w[u][0], !CHECK || left > u * G ? diff : 0.f, s.zpart[u % CH]);
                } else {
                    gw_axpy(s.part[u % CH][i], w[u][NH > 1 ? i : 0], v);
                }
            }
    }
    template <bool CHECK>
    __device__ __forceinline__ void add(const int32_t *ids, int cnt) {
        Window s;                                           // sums are blocked per window
#pragma unroll
        for (int c = 0; c < CH; ++c) {
#pragma unroll
            for (int i = 0; i < T; ++i)
#pragma unroll
                for (int q = 0; q < VEC; ++q) s.part[c][i][q] = 0.f;
#pragma unroll
            for (int i = 0; i < NH; ++i) s.dpart[c][i] = 0.f;
            s.zpart[c] = 0.f;
        }
        const int32_t *sp = ids + at.g;
#pragma unroll 1
        for (; cnt >= G * kStepFull; cnt -= G * kStepFull, sp += G * kStepFull) step<kStepFull, false>(sp, 0, s);
#pragma unroll 1
        for (; CHECK && cnt > 0; cnt -= G * kStepPart, sp += G * kStepPart) step<kStepPart, true>(sp, cnt - at.g, s);
#pragma unroll
        for (int i = 0; i < NH; ++i) den[i] += CH == 1 ? s.dpart[0][i] : s.dpart[0][i] + s.dpart[CH - 1][i];
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                if (CH > 1) s.part[0][i][q] += s.part[CH - 1][i][q];
                acc[i][q] += s.part[0][i][q];
            }
        dz += CH == 1 ? s.zpart[0] : s.zpart[0] + s.zpart[CH - 1];
    }
    // this state and (sums, m, den) of another, element by element
    template <class Get>
    __device__ __forceinline__ void fold(Get get) {
        float sa[NH], sb[NH];
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            const float m2 = get(m[i], kSums + i), mm = fmaxf(m[i], m2);
            sa[i] = gw_rescale(m[i], mm);
            sb[i] = gw_rescale(m2, mm);
            den[i] = den[i] * sa[i] + get(den[i], kSums + NH + i) * sb[i];
            m[i] = mm;
        }
        if constexpr (TARGET_BWD) {
            dz = dz * sa[0] + get(dz, 0) * sb[0];
            return;
        }
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int q = 0; q < VEC; ++q)
                acc[i][q] = acc[i][q] * sa[NH > 1 ? i : 0] + get(acc[i][q], i * VEC + q) * sb[NH > 1 ? i : 0];
    }
    // the lane groups: their largest maximum first, one rescale, then plain sums
    __device__ __forceinline__ void join() {
        if constexpr (G > 1) {
#pragma unroll
            for (int i = 0; i < NH; ++i) {
                float top = m[i];
#pragma unroll
                for (int o = LPR; o < 32; o <<= 1) top = fmaxf(top, lane_xor(top, o));
                const float sc = gw_rescale(m[i], top);
                den[i] *= sc;
                dz *= sc;
#pragma unroll
                for (int j = 0; j < T; ++j) {
                    if (TARGET_BWD || (NH > 1 && j != i)) continue;
#pragma unroll
                    for (int q = 0; q < VEC; ++q) acc[j][q] *= sc;
                }
                m[i] = top;
            }
#pragma unroll
            for (int o = LPR; o < 32; o <<= 1) {
#pragma unroll
                for (int i = 0; i < NH; ++i) den[i] += lane_xor(den[i], o);
                if constexpr (TARGET_BWD) {
                    dz += lane_xor(dz, o);
                } else {
#pragma unroll
                    for (int i = 0; i < T; ++i)
#pragma unroll
                        for (int q = 0; q < VEC; ++q) acc[i][q] += lane_xor(acc[i][q], o);
                }
            }
        }
    }
    __device__ __forceinline__ void merge(const float *slot) {
        fold([&](float, int q) { return slot[q * LPR + at.sub]; });
    }
    __device__ __forceinline__ void park(float *slot) const {
        if (at.g != 0) return;
        if constexpr (TARGET_BWD) {
            slot[at.sub] = dz;
        } else {
#pragma unroll
            for (int i = 0; i < T; ++i)
#pragma unroll
                for (int q = 0; q < VEC; ++q) slot[(i * VEC + q) * LPR + at.sub] = acc[i][q];
        }
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            slot[(kSums + i) * LPR + at.sub] = m[i];
            slot[(kSums + NH + i) * LPR + at.sub] = den[i];
        }
    }
    __device__ __forceinline__ void close(int32_t t, int32_t beg, int32_t end, bool shared) {
        const uint64_t row = static_cast<uint64_t>(static_cast<uint32_t>(t)) * at.f + at.f0;
        const bool any = end > beg;
        if constexpr (!TARGET_BWD) {
            if (at.g == 0) {
#pragma unroll
                for (int i = 0; i < T; ++i) {
                    if (i >= at.own) continue;
                    float r[VEC];
#pragma unroll
                    for (int q = 0; q < VEC; ++q) r[q] = any ? acc[i][q] / den[NH > 1 ? i : 0] : 0.f;
                    gw_store(a.out + row + i * LPR * VEC, r);
                }
            }
            if (a.alpha) {
                const int warp = threadIdx.x >> 5;
                put_statistics(warp);
                if (!shared) weights(warp, t, beg, end, threadIdx.x & 31, 32);
            }
        } else {
            const float d = gw_head_sum<0>(dz, a.channels / VEC), b = gw_head_sum<0>(beta, a.channels / VEC);
            if (at.g == 0 && at.own > 0 && at.f0 % a.channels == 0) {
                const uint64_t th = static_cast<uint64_t>(static_cast<uint32_t>(t)) * a.heads + at.head[0];
                a.ds_dst[th] = any ? d / den[0] : 0.f;
                a.stats[th] = make_float4(sd[0], m[0], any ? 1.f / den[0] : 0.f, b);
            }
        }
    }
    // alpha of the row's edges: after the row (by its warp), or for a row that
    // several warps held by all warps of the CTA together
    __device__ __forceinline__ bool wants_after() const { return !TARGET_BWD && a.alpha != nullptr; }
    __device__ __forceinline__ void after(int w, int32_t t, int32_t beg, int32_t end) {
        weights(w, t, beg, end, threadIdx.x, kWarps * 32);
    }
    // heads whose first feature lies in this tile
    __device__ __forceinline__ int first_head() const {
        return static_cast<int>((at.f0 - at.sub * VEC + a.channels - 1) / a.channels);
    }
    __device__ __forceinline__ float2 *statistics(int w) const {
        return reinterpret_cast<float2 *>(scratch) + w * (LPR * T);
    }
    __device__ __forceinline__ void put_statistics(int warp) {
        const int h0 = first_head();
        __syncwarp();
        if (at.g == 0) {
#pragma unroll
            for (int i = 0; i < T; ++i)
                if (i < at.own && (at.f0 + i * LPR * VEC) % a.channels == 0)
                    statistics(warp)[static_cast<int>((at.f0 + i * LPR * VEC) / a.channels) - h0] =
                        make_float2(m[NH > 1 ? i : 0], den[NH > 1 ? i : 0]);
        }
        __syncwarp();
    }
    // threads id, id + stride, ... over (edge, head): coalesced, four in flight
    __device__ __forceinline__ void weights(int w, int32_t t, int32_t beg, int32_t end, int id, int stride) {
        const uint32_t ft = at.f0 - at.sub * VEC;
        const int h0 = first_head();
        const int nh = static_cast<int>((min(ft + LPR * VEC * T, at.f) + a.channels - 1) / a.channels) - h0;
        const float *sdt = a.s_dst + static_cast<uint64_t>(static_cast<uint32_t>(t)) * a.heads + h0;
        const float *ssh = a.s_src + h0;
        const int64_t total = static_cast<int64_t>(end - beg) * nh;
        for (int64_t i0 = id; i0 < total; i0 += 4 * stride) {
            int64_t at_e[4];
            int h[4];
            uint64_t src[4];
            float z[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t i = min64(i0 + u * stride, total - 1), e = nh == 1 ? i : i / nh;
                h[u] = static_cast<int>(i - e * nh);
                at_e[u] = beg + e;
                src[u] = static_cast<uint32_t>(__ldg(a.col + at_e[u]));
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) z[u] = __ldg(ssh + src[u] * a.heads + h[u]) + __ldg(sdt + h[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (i0 + u * stride >= total) break;
                const float2 st = statistics(w)[h[u]];
                const float l = z[u] > 0.f ? z[u] : a.slope * z[u];
                a.alpha[at_e[u] * a.heads + h0 + h[u]] = exp2f(l - st.x) / st.y;
            }
        }
    }
};

// Backward by source (CSR by source: ids are targets).  grad_x = P + ds_src a_src +
// ds_dst a_dst with P = sum of alpha grad_out[t] over the out-edges, and
//   ds_src = sum of alpha phi (dalpha - beta).
// The lanes of a head finish dalpha edge by edge (gw_spread_sums), so that beta of the
// target is subtracted before anything is summed, as in the pass by target.  Every lane
// forms alpha of its head from the target's statistics.  LH: lanes of a head.
template <typename XT, int VEC, int LPR, int LH>
struct GatBySource {
    using V = VecLoad<float, VEC>;
    static constexpr int kWarps = VEC == 8 ? TFG_GW_SRC8_WARPS : TFG_GW_SRC_WARPS, kLpr = LPR, G = 32 / LPR;
    static constexpr int kTile = LPR * VEC, kHeadsPerLane = 1;
    static constexpr int kState = VEC + 1, kHeld = 0;
    static constexpr int kDepth = VEC == 8 ? TFG_GW_SRC8_DEPTH : TFG_GW_SRC_DEPTH;
    static constexpr int D = kDepth * G > 32 ? 32 / G : kDepth;
    static_assert(32 % (G * D) == 0, "a full window is read in whole steps");
    static constexpr int kOwnSums = D > LH ? D / LH : 1;         // edges of a step whose sums a lane ends with
    static constexpr int kUnroll = VEC == 8 ? 32 / (G * D) : 1;      // steps of a full window unrolled
    const GatArgs &a;
    GatLane<VEC, LPR, 1, 1> at;
    const char *gb;
    uint32_t row_bytes;
    float ss, ds, xs[VEC], P[VEC];           // ds: this lane's share

    __device__ __forceinline__ GatBySource(const GatArgs &args, uint32_t ft, float *, float *) : a(args) {
        at.place(ft, a.heads, a.channels);
        gb = reinterpret_cast<const char *>(a.grad_out + (at.own > 0 ? at.f0 : 0));
        row_bytes = at.f * 4u;
    }
    __device__ __forceinline__ uint64_t element(int32_t s) const {   // feature f0 of row s
        return static_cast<uint64_t>(static_cast<uint32_t>(s)) * at.f + at.f0;
    }
    __device__ __forceinline__ void clear() {
        ds = 0.f;
#pragma unroll
        for (int q = 0; q < VEC; ++q) P[q] = 0.f;
    }
    __device__ __forceinline__ void open(int32_t s, int32_t, int32_t) {
        ss = __ldg(a.s_src + static_cast<uint64_t>(static_cast<uint32_t>(s)) * a.heads + at.head[0]);
#pragma unroll
        for (int q = 0; q < VEC; ++q) xs[q] = 0.f;
        if (at.own > 0) VecLoad<XT, VEC>::load(static_cast<const XT *>(a.x) + element(s), xs);
        clear();
    }
    template <bool CHECK>
    __device__ __forceinline__ void add(const int32_t *ids, int cnt) {
        float p[VEC], part = 0.f;
#pragma unroll
        for (int q = 0; q < VEC; ++q) p[q] = 0.f;
        const int32_t *sp = ids + at.g;
        int left = cnt - at.g;
#pragma unroll CHECK ? 1 : kUnroll
        for (int e = 0; e < (CHECK ? cnt : 32); e += G * D) {
            typename V::Raw raw[D];
            float4 st[D];
#pragma unroll
            for (int u = 0; u < D; ++u) {
                const uint32_t id = static_cast<uint32_t>(sp[u * G]);
                const bool ok = !CHECK || left > u * G;
                const float *row = reinterpret_cast<const float *>(gb + static_cast<uint64_t>(id) * row_bytes);
                st[u] = ok ? __ldg(a.stats + static_cast<uint64_t>(id) * a.heads + at.head[0])
                           : make_float4(0.f, 0.f, 0.f, 0.f);
                if constexpr (VEC == 8) raw[u] = CHECK ? V::raw(ok, row) : V::raw(row);
                else raw[u] = ok ? V::raw(row) : V::zero();
            }
            float dots[D], af[D], beta[D];
#pragma unroll
            for (int u = 0; u < D; ++u) {
                const float z = ss + st[u].x;
                const float l = z > 0.f ? z : a.slope * z;
                float al = exp2f(l - st[u].y) * st[u].z;
                if (CHECK) al = left > u * G ? al : 0.f;
                af[u] = z > 0.f ? al : a.slope * al;
                beta[u] = st[u].w;
                float v[VEC];
                V::widen(raw[u], v);
                gw_axpy(p, al, v);
                dots[u] = gw_dot(xs, v);
            }
            gw_spread_sums<LH>(dots, af, beta, at.sub);
#pragma unroll
            for (int u = 0; u < D; ++u)
                if (u < kOwnSums) part = fmaf(af[u], dots[u] - beta[u], part);
            sp += G * D;
            left -= G * D;
        }
        ds += part;
#pragma unroll
        for (int q = 0; q < VEC; ++q) P[q] += p[q];
    }
    template <class Get>
    __device__ __forceinline__ void fold(Get get) {
#pragma unroll
        for (int q = 0; q < VEC; ++q) P[q] += get(P[q], q);
        ds += get(ds, VEC);
    }
    __device__ __forceinline__ void join() {
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) fold([&](float mine, int) { return lane_xor(mine, o); });
    }
    __device__ __forceinline__ void merge(const float *slot) {
        fold([&](float, int q) { return slot[q * LPR + at.sub]; });
    }
    __device__ __forceinline__ void park(float *slot) const {
        if (at.g != 0) return;
#pragma unroll
        for (int q = 0; q < VEC; ++q) slot[q * LPR + at.sub] = P[q];
        slot[VEC * LPR + at.sub] = ds;
    }
    __device__ __forceinline__ bool wants_after() const { return false; }
    __device__ __forceinline__ void after(int, int32_t, int32_t, int32_t) {}
    __device__ __forceinline__ void close(int32_t s, int32_t, int32_t, bool) {
        const float dz = gw_head_sum<LH>(ds, LH);
        if (at.g != 0 || at.own == 0) return;
        const uint64_t sh = static_cast<uint64_t>(static_cast<uint32_t>(s)) * a.heads + at.head[0];
        const float dd = __ldg(a.ds_dst + sh);
        float as[VEC], ad[VEC], r[VEC];
        gw_load(a.a_src + at.f0, as);
        gw_load(a.a_dst + at.f0, ad);
#pragma unroll
        for (int q = 0; q < VEC; ++q) r[q] = P[q] + dz * as[q] + dd * ad[q];
        gw_store(a.grad_x + element(s), r);
        if (at.f0 % a.channels == 0) a.ds_src[sh] = dz;
    }
};

}  // namespace
}  // namespace tfg
