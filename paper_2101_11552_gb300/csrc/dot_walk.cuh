// The three edge passes of the dot-product attention as row-walk policies
// (row_walk.cuh): forward, backward by target, backward by source.  A row's head
// is LH lanes of VEC features (LH a power of two; LH = 0 takes the count at run
// time), which finish a dot product with a butterfly, so every lane of a head
// holds the same logit; LPR lanes cover whole heads of a row (wider rows loop
// over tiles), G = 32 / LPR lane groups take every G-th edge.  Logits are in base-2
// units (scale2 = scale log2 e).
#pragma once
#include <math_constants.h>

#include "row_walk.cuh"

namespace tfg {

struct DotArgs {
    const int32_t *rowptr, *col;          // CSR of the pass
    const void *q, *k, *v;
    int64_t n;
    int heads, channels, lh;
    float scale, scale2;
    float *out, *alpha;                   // forward
    const float *fwd_out, *grad_out;      // backward
    float4 *stats;                        // [N, H]: (m, 1 / den, beta, 0)
    float *grad_q, *grad_k, *grad_v;
    __host__ __device__ uint32_t width() const { return static_cast<uint32_t>(heads) * static_cast<uint32_t>(channels); }
    __host__ __device__ bool statistics() const { return alpha != nullptr; }
};

namespace {

// What bounds it: instructions on short rows (169,343 nodes, mean in-degree 6.9, 8
// x 16 fp32: forward 166, by target 206, by source 253 us); on long ones (114.6M
// edges, 8 x 16 bf16) the gathers, 896 bytes an edge by source (7.5 ms, 13.7 TB/s)
// and 512 by target (5.4 ms, 11 TB/s), with one CTA of few, register-rich warps.
// Before: a row per warp, the lanes of a head a run-time count and every slot
// tested, 141 instructions for two edges by source: 12.4 ms, by target 8.9 ms.
//
// Tuning knobs, measured there: by target 20 warps 5.54 ms, 16 5.66, 24 6.29; four
// steps of a full window unrolled 5.35, one 5.54.  By source 16 warps with 4 edges
// in flight 7.6 ms, 20 with 2 8.8, 12 with 4 9.1; before the earlier windows' sums
// waited in shared memory 8.9.  Forward (short rows; fp32) 24 warps 166 us, 20 183.
#ifndef TFG_DW_FWD_WARPS
#define TFG_DW_FWD_WARPS 24
#endif
#ifndef TFG_DW_TGT_WARPS
#define TFG_DW_TGT_WARPS 20
#endif
#ifndef TFG_DW_SRC_WARPS
#define TFG_DW_SRC_WARPS 16
#endif
// The same in bf16 rows with two chains, whose registers are short: forward and
// backward of 6 x 32 over 10M edges 3689 us with 20 and 16, by target 16 3501, by
// source 12 3639, 14 3849 (one chain 3291); 169,343 nodes 987 / 961 / 945 / 1027 (839).
#ifndef TFG_DW_TGT_WARPS_CHAINS
#define TFG_DW_TGT_WARPS_CHAINS 16
#endif
#ifndef TFG_DW_SRC_WARPS_CHAINS
#define TFG_DW_SRC_WARPS_CHAINS 12
#endif
#ifndef TFG_DW_DEPTH
#define TFG_DW_DEPTH 4        // edges in flight per lane group, full windows
#endif
#ifndef TFG_DW_UNROLL
#define TFG_DW_UNROLL 4       // by target: steps of a full window unrolled
#endif

template <int VEC>
__device__ __forceinline__ float dw_dot(const float (&a)[VEC], const float (&b)[VEC]) {
    float2 d = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < VEC; i += 2) d = fma2(make_float2(a[i], a[i + 1]), make_float2(b[i], b[i + 1]), d);
    return d.x + d.y;
}
template <int VEC>
__device__ __forceinline__ void dw_axpy(float (&acc)[VEC], float w, const float (&v)[VEC]) {
    const float2 w2 = make_float2(w, w);
#pragma unroll
    for (int i = 0; i < VEC; i += 2) {
        const float2 r = fma2(make_float2(v[i], v[i + 1]), w2, make_float2(acc[i], acc[i + 1]));
        acc[i] = r.x;
        acc[i + 1] = r.y;
    }
}
template <int VEC>
__device__ __forceinline__ void dw_load(const float *p, float (&r)[VEC]) {
#pragma unroll
    for (int i = 0; i < VEC; i += 4) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(p + i));
        r[i] = v.x; r[i + 1] = v.y; r[i + 2] = v.z; r[i + 3] = v.w;
    }
}
template <int VEC>
__device__ __forceinline__ void dw_store(float *p, const float (&r)[VEC], float w) {
#pragma unroll
    for (int i = 0; i < VEC; i += 4)
        *reinterpret_cast<float4 *>(p + i) = make_float4(r[i] * w, r[i + 1] * w, r[i + 2] * w, r[i + 3] * w);
}
template <int VEC>
__device__ __forceinline__ void dw_clear(float (&r)[VEC]) {
#pragma unroll
    for (int i = 0; i < VEC; ++i) r[i] = 0.f;
}
__device__ __forceinline__ float dw_rescale(float m_old, float m_new) {
    return m_old == -CUDART_INF_F ? 0.f : exp2f(m_old - m_new);
}

// A lane's place and the sum over its head's lanes.
template <typename XT, int VEC, int LPR, int LH>
struct DotLane {
    using V = VecLoad<XT, VEC>;
    int sub, g, head, lh;
    bool own;                             // the lane holds features
    uint32_t f, f0, row_bytes;
    __device__ __forceinline__ DotLane(const DotArgs &a, uint32_t ft) {
        const int lane = threadIdx.x & 31;
        sub = lane % LPR;
        g = lane / LPR;
        f = static_cast<uint32_t>(a.heads) * static_cast<uint32_t>(a.channels);
        own = ft + sub * VEC < f;
        f0 = own ? ft + sub * VEC : 0;    // lanes past F read (and never store) feature 0
        head = static_cast<int>(f0 / a.channels);
        lh = LH > 0 ? LH : a.lh;
        row_bytes = f * static_cast<uint32_t>(sizeof(XT));
    }
    __device__ __forceinline__ float head_sum(float v) const {
        if constexpr (LH > 0) {
#pragma unroll
            for (int o = 1; o < LH; o <<= 1) v += lane_xor(v, o);
        } else {
            for (int o = 1; o < lh; o <<= 1) v += lane_xor(v, o);
        }
        return v;
    }
    __device__ __forceinline__ const char *base(const void *p) const {
        return reinterpret_cast<const char *>(static_cast<const XT *>(p) + f0);
    }
    __device__ __forceinline__ const XT *row(const char *b, uint32_t id) const {
        return reinterpret_cast<const XT *>(b + static_cast<uint64_t>(id) * row_bytes);
    }
    __device__ __forceinline__ uint64_t at(int32_t r) const {   // element f0 of row r
        return static_cast<uint64_t>(static_cast<uint32_t>(r)) * f + f0;
    }
    __device__ __forceinline__ uint64_t stat(uint32_t r, int heads) const {
        return static_cast<uint64_t>(r) * heads + head;
    }
};

// Within a window a lane adds its edges in CH chains, edge by edge in turn: two in rows
// of 17 to 31 slices, whose 32 lanes leave one lane group.  The chains' sum, in the first.
template <int CH, int N>
__device__ __forceinline__ void dw_join_chains(float (&acc)[CH][N]) {
    if constexpr (CH > 1) {
        static_assert(CH == 2, "one chain or two");
#pragma unroll
        for (int i = 0; i < N; ++i) acc[0][i] += acc[1][i];
        dw_clear(acc[1]);
    }
}

// Sums are blocked per window of 32 edges.  The sums of a row's earlier windows wait
// in shared memory (element q of a lane at q * 32), so that the registers hold
// one set of accumulators and more rows in flight; a row of one window never
// goes there.
template <int N>
struct DotHeld {
    float *at;
    bool begun, used;
    __device__ __forceinline__ explicit DotHeld(float *warp_slots) : at(warp_slots + (threadIdx.x & 31)) {}
    __device__ __forceinline__ void clear() { begun = used = false; }
    // before a window: the previous window's sums join the earlier ones
    __device__ __forceinline__ void next(float (&acc)[N]) {
        if (begun) {
#pragma unroll
            for (int q = 0; q < N; ++q) {
                at[q * 32] = (used ? at[q * 32] : 0.f) + acc[q];
                acc[q] = 0.f;
            }
            used = true;
        }
        begun = true;
    }
    __device__ __forceinline__ void scale(float sc) {
        if (used) {
#pragma unroll
            for (int q = 0; q < N; ++q) at[q * 32] *= sc;
        }
    }
    __device__ __forceinline__ void last(float (&acc)[N]) {
        if (used) {
#pragma unroll
            for (int q = 0; q < N; ++q) acc[q] += at[q * 32];
            used = false;
        }
    }
};

// Softmax over the in-edges of a target.  BWD = false: acc = sum of p v[src];
// BWD = true: acc = sum of p (dalpha - beta) k[src], dalpha = <grad_out[t], v[src]>.
template <typename XT, int VEC, int LPR, int LH, bool BWD, int CH = 1>
struct DotByTarget {
    using L = DotLane<XT, VEC, LPR, LH>;
    using V = VecLoad<XT, VEC>;
    static constexpr int kWarps = !BWD ? TFG_DW_FWD_WARPS
                                       : (VEC == 8 && CH > 1 ? TFG_DW_TGT_WARPS_CHAINS : TFG_DW_TGT_WARPS);
    static constexpr int kLpr = LPR, G = 32 / LPR;
    static constexpr int kTile = LPR * VEC, kHeadsPerLane = 1;
    static constexpr int kState = VEC + 2, kHeld = VEC;
    static constexpr int kStepFull = TFG_DW_DEPTH * G > 32 ? 32 / G : TFG_DW_DEPTH, kUnroll = TFG_DW_UNROLL;
    static_assert(32 % (G * kStepFull) == 0, "a full window is read in whole steps");
    static constexpr int kStepPart = walk_part(G) < kStepFull ? walk_part(G) : kStepFull;
    const DotArgs &a;
    L ln;
    const char *kb, *vb;
    float2 *scratch;                      // [warp][heads of the tile] (m, den), for alpha
    DotHeld<VEC> held;                    // the sums of the row's earlier windows
    float qv[VEC], gt[BWD ? VEC : 1], beta, m, den, acc[CH][VEC];

    __device__ __forceinline__ DotByTarget(const DotArgs &args, uint32_t ft, float *hold, float *scr)
        : a(args), ln(args, ft), scratch(reinterpret_cast<float2 *>(scr)), held(hold) {
        kb = ln.base(a.k);
        vb = ln.base(a.v);
        beta = 0.f;
    }
    __device__ __forceinline__ void clear() {
        m = -CUDART_INF_F;
        den = 0.f;
#pragma unroll
        for (int c = 0; c < CH; ++c) dw_clear(acc[c]);
        held.clear();
    }
    __device__ __forceinline__ void load_query(int32_t t) {
        V::load(static_cast<const XT *>(a.q) + ln.at(t), qv);
        if (!ln.own) dw_clear(qv);
    }
    __device__ __forceinline__ void open(int32_t t, int32_t, int32_t) {
        load_query(t);
        if constexpr (BWD) {
            float ov[VEC];
            dw_load(a.grad_out + ln.at(t), gt);
            dw_load(a.fwd_out + ln.at(t), ov);
            if (!ln.own) dw_clear(gt);
            beta = ln.head_sum(dw_dot(gt, ov));
        }
        clear();
    }
    // D edges of the group, sp[0], sp[G], ... (CHECK: those below left)
    template <int D, bool CHECK>
    __device__ __forceinline__ void step(const int32_t *sp, int left, float (&dpart)[CH]) {
        static_assert(D % CH == 0, "a step gives every chain the same number of edges");
        typename V::Raw rk[D], rv[D];
#pragma unroll
        for (int u = 0; u < D; ++u) {
            const uint32_t id = static_cast<uint32_t>(sp[u * G]);
            const bool ok = !CHECK || left > u * G;
            rk[u] = ok ? V::raw(ln.row(kb, id)) : V::zero();
            rv[u] = ok ? V::raw(ln.row(vb, id)) : V::zero();
        }
        float l[D], w[D], top = m;
#pragma unroll
        for (int u = 0; u < D; ++u) {
            float x[VEC];
            V::widen(rk[u], x);
            l[u] = ln.head_sum(dw_dot(qv, x)) * a.scale2;
            if (CHECK && left <= u * G) l[u] = -CUDART_INF_F;
            top = fmaxf(top, l[u]);
            if constexpr (BWD) {
                V::widen(rv[u], x);
                w[u] = ln.head_sum(dw_dot(gt, x)) - beta;
            }
        }
        if (top > m) {                                           // a new running maximum: rescale the sums so far
            const float sc = dw_rescale(m, top);
            den *= sc;
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                dpart[c] *= sc;
#pragma unroll
                for (int i = 0; i < VEC; ++i) acc[c][i] *= sc;
            }
            held.scale(sc);
            m = top;
        }
#pragma unroll
        for (int u = 0; u < D; ++u) {
            const float p = !CHECK || left > u * G ? exp2f(l[u] - m) : 0.f;
            dpart[u % CH] += p;
            float x[VEC];
            V::widen(BWD ? rk[u] : rv[u], x);
            dw_axpy(acc[u % CH], !BWD ? p : (!CHECK || left > u * G ? p * w[u] : 0.f), x);
        }
    }
    template <bool CHECK>
    __device__ __forceinline__ void add(const int32_t *ids, int cnt) {
        dw_join_chains(acc);
        held.next(acc[0]);                                       // sums are blocked per window
        float dpart[CH] = {};
        const int32_t *sp = ids + ln.g;
        if (!CHECK) {                                            // a full window
#pragma unroll kUnroll
            for (int e = 0; e < 32; e += G * kStepFull) step<kStepFull, false>(sp + e, 0, dpart);
            den += CH == 1 ? dpart[0] : dpart[0] + dpart[CH - 1];
            return;
        }
#pragma unroll 1
        for (; cnt >= G * kStepFull; cnt -= G * kStepFull, sp += G * kStepFull) step<kStepFull, false>(sp, 0, dpart);
#pragma unroll 1
        for (; CHECK && cnt > 0; cnt -= G * kStepPart, sp += G * kStepPart) step<kStepPart, true>(sp, cnt - ln.g, dpart);
        den += CH == 1 ? dpart[0] : dpart[0] + dpart[CH - 1];
    }
    template <class Get>
    __device__ __forceinline__ void fold(Get get) {
        const float m2 = get(m, VEC), mm = fmaxf(m, m2);
        const float sa = dw_rescale(m, mm), sb = dw_rescale(m2, mm);
        den = den * sa + get(den, VEC + 1) * sb;
#pragma unroll
        for (int i = 0; i < VEC; ++i) acc[0][i] = acc[0][i] * sa + get(acc[0][i], i) * sb;
        m = mm;
    }
    __device__ __forceinline__ void join() {
        dw_join_chains(acc);
        held.last(acc[0]);
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) fold([&](float mine, int) { return lane_xor(mine, o); });
    }
    __device__ __forceinline__ void merge(const float *slot) {
        fold([&](float, int i) { return slot[i * LPR + ln.sub]; });
    }
    __device__ __forceinline__ void park(float *slot) const {
        if (ln.g != 0) return;
#pragma unroll
        for (int i = 0; i < VEC; ++i) slot[i * LPR + ln.sub] = acc[0][i];
        slot[VEC * LPR + ln.sub] = m;
        slot[(VEC + 1) * LPR + ln.sub] = den;
    }
    __device__ __forceinline__ void close(int32_t t, int32_t beg, int32_t end, bool shared) {
        const bool any = end > beg;
        if (ln.g == 0 && ln.own) {
            if constexpr (BWD) {
                dw_store(a.grad_q + ln.at(t), acc[0], any ? a.scale / den : 0.f);
                if (ln.sub % ln.lh == 0)
                    a.stats[ln.stat(static_cast<uint32_t>(t), a.heads)] =
                        make_float4(m, any ? 1.f / den : 0.f, beta, 0.f);
            } else {
                float r[VEC];
#pragma unroll
                for (int i = 0; i < VEC; ++i) r[i] = any ? acc[0][i] / den : 0.f;
                dw_store(a.out + ln.at(t), r, 1.f);
            }
        }
        if (!BWD && a.alpha) {
            const int warp = threadIdx.x >> 5;
            __syncwarp();
            if (ln.g == 0 && ln.sub % ln.lh == 0) statistics(warp)[ln.sub / ln.lh] = make_float2(m, den);
            __syncwarp();
            if (!shared) weights(warp, t, beg, end, ln.g, G);
        }
    }
    // alpha: every logit again, one writer per (edge, head); a row that several
    // warps held is done by all warps of the CTA
    __device__ __forceinline__ float2 *statistics(int w) const { return scratch + w * LPR; }
    __device__ __forceinline__ bool wants_after() const { return !BWD && a.alpha != nullptr; }
    __device__ __forceinline__ void after(int w, int32_t t, int32_t beg, int32_t end) {
        load_query(t);
        weights(w, t, beg, end, (threadIdx.x >> 5) * G + ln.g, kWarps * G);
    }
    __device__ __forceinline__ void weights(int w, int32_t, int32_t beg, int32_t end, int first, int stride) {
        const float2 st = statistics(w)[ln.sub / ln.lh];
        const int64_t steps = (static_cast<int64_t>(end) - beg + stride - 1) / stride;   // the same for every lane
        for (int64_t i = 0; i < steps; ++i) {
            const int64_t e = beg + i * stride + first;
            const bool ok = e < end;
            const uint32_t src = ok ? static_cast<uint32_t>(__ldg(a.col + e)) : 0u;
            float x[VEC];
            V::load(ln.row(kb, src), x);
            const float l = ln.head_sum(dw_dot(qv, x)) * a.scale2;
            if (ok && ln.own && ln.sub % ln.lh == 0) a.alpha[e * a.heads + ln.head] = exp2f(l - st.x) / st.y;
        }
    }
};

// Backward by source (CSR by source: ids are targets), from the targets'
// statistics: grad_k = scale sum of alpha (dalpha - beta) q[t], grad_v = sum of
// alpha grad_out[t].
// WIDE (VEC = 8): 32-byte gradient slices, one load each instead of two that each
// touch every sector: 114.6M edges 7.49 ms against 7.59.
template <typename XT, int VEC, int LPR, int LH, bool WIDE, int CH = 1>
struct DotSource {
    using L = DotLane<XT, VEC, LPR, LH>;
    using V = VecLoad<XT, VEC>;
    static constexpr int kWarps = VEC == 8 && CH > 1 ? TFG_DW_SRC_WARPS_CHAINS : TFG_DW_SRC_WARPS, kLpr = LPR, G = 32 / LPR;
    static constexpr int kTile = LPR * VEC, kHeadsPerLane = 1;
    static constexpr int kState = 2 * VEC, kHeld = 2 * VEC;
    static constexpr int kStepFull = TFG_DW_DEPTH * G > 32 ? 32 / G : TFG_DW_DEPTH;
    static_assert(32 % (G * kStepFull) == 0, "a full window is read in whole steps");
    static constexpr int kStepPart = walk_part(G) < kStepFull ? walk_part(G) : kStepFull;
    const DotArgs &a;
    L ln;
    const char *qb, *gb;
    DotHeld<2 * VEC> held;
    float ks[VEC], vs[VEC], dkv[CH][2 * VEC];  // grad_k's and grad_v's sums

    __device__ __forceinline__ DotSource(const DotArgs &args, uint32_t ft, float *hold, float *)
        : a(args), ln(args, ft), held(hold) {
        qb = ln.base(a.q);
        gb = reinterpret_cast<const char *>(a.grad_out + ln.f0);
    }
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int c = 0; c < CH; ++c) dw_clear(dkv[c]);
        held.clear();
    }
    __device__ __forceinline__ void open(int32_t s, int32_t, int32_t) {
        V::load(static_cast<const XT *>(a.k) + ln.at(s), ks);
        V::load(static_cast<const XT *>(a.v) + ln.at(s), vs);
        clear();
    }
    template <int D, bool CHECK>
    __device__ __forceinline__ void step(const int32_t *sp, int left) {
        static_assert(D % CH == 0, "a step gives every chain the same number of edges");
        typename V::Raw rq[D];
        float gr[D][VEC];
        float4 st[D];
#pragma unroll
        for (int u = 0; u < D; ++u) {
            const uint32_t id = static_cast<uint32_t>(sp[u * G]);
            const bool ok = !CHECK || left > u * G;
            const float *gp = reinterpret_cast<const float *>(gb + static_cast<uint64_t>(id) * (ln.f * 4u));
            rq[u] = ok ? V::raw(ln.row(qb, id)) : V::zero();
            if constexpr (WIDE) {
                const Row32 g8 = CHECK ? ld_row32(ok, gp) : ld_row32(gp);
#pragma unroll
                for (int i = 0; i < VEC; ++i) gr[u][i] = g8.v[i];
            } else
#pragma unroll
            for (int i = 0; i < VEC; i += 4) {
                const float4 g4 = ok ? __ldg(reinterpret_cast<const float4 *>(gp + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
                gr[u][i] = g4.x; gr[u][i + 1] = g4.y; gr[u][i + 2] = g4.z; gr[u][i + 3] = g4.w;
            }
            st[u] = ok ? __ldg(a.stats + ln.stat(id, a.heads)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < D; ++u) {
            float *pk = dkv[u % CH], *pv = dkv[u % CH] + VEC;
            float qv[VEC];
            V::widen(rq[u], qv);
            const float l = ln.head_sum(dw_dot(qv, ks)) * a.scale2;
            const float da = ln.head_sum(dw_dot(gr[u], vs));
            const bool ok = !CHECK || left > u * G;
            const float al = ok ? exp2f(l - st[u].x) * st[u].y : 0.f;
            const float wk = ok ? al * (da - st[u].z) : 0.f;
            const float2 wk2 = make_float2(wk, wk), al2 = make_float2(al, al);
#pragma unroll
            for (int i = 0; i < VEC; i += 2) {
                const float2 x = fma2(make_float2(qv[i], qv[i + 1]), wk2, make_float2(pk[i], pk[i + 1]));
                const float2 y = fma2(make_float2(gr[u][i], gr[u][i + 1]), al2, make_float2(pv[i], pv[i + 1]));
                pk[i] = x.x; pk[i + 1] = x.y;
                pv[i] = y.x; pv[i + 1] = y.y;
            }
        }
    }
    template <bool CHECK>
    __device__ __forceinline__ void add(const int32_t *ids, int cnt) {
        dw_join_chains(dkv);
        held.next(dkv[0]);
        const int32_t *sp = ids + ln.g;
#pragma unroll 1
        for (; cnt >= G * kStepFull; cnt -= G * kStepFull, sp += G * kStepFull) step<kStepFull, false>(sp, 0);
#pragma unroll 1
        for (; CHECK && cnt > 0; cnt -= G * kStepPart, sp += G * kStepPart) step<kStepPart, true>(sp, cnt - ln.g);
    }
    template <class Get>
    __device__ __forceinline__ void fold(Get get) {
#pragma unroll
        for (int i = 0; i < 2 * VEC; ++i) dkv[0][i] += get(dkv[0][i], i);
    }
    __device__ __forceinline__ void join() {
        dw_join_chains(dkv);
        held.last(dkv[0]);
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) fold([&](float mine, int) { return lane_xor(mine, o); });
    }
    __device__ __forceinline__ void merge(const float *slot) {
        fold([&](float, int i) { return slot[i * LPR + ln.sub]; });
    }
    __device__ __forceinline__ void park(float *slot) const {
        if (ln.g != 0) return;
#pragma unroll
        for (int i = 0; i < 2 * VEC; ++i) slot[i * LPR + ln.sub] = dkv[0][i];
    }
    __device__ __forceinline__ bool wants_after() const { return false; }
    __device__ __forceinline__ void after(int, int32_t, int32_t, int32_t) {}
    __device__ __forceinline__ void close(int32_t s, int32_t, int32_t, bool) {
        if (ln.g != 0 || !ln.own) return;
        float dk[VEC], dv[VEC];
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            dk[i] = dkv[0][i];
            dv[i] = dkv[0][VEC + i];
        }
        dw_store(a.grad_k + ln.at(s), dk, a.scale);
        dw_store(a.grad_v + ln.at(s), dv, 1.f);
    }
};

template <typename XT, int VEC, int LPR, int LH, int CH>
using DotBySource = DotSource<XT, VEC, LPR, LH, VEC == 8, CH>;
// gradient rows that are not 32-byte aligned: one kernel a row width, heads at run time
template <typename XT, int VEC, int LPR, int LH, int CH>
using DotBySourceNarrow = DotSource<XT, VEC, LPR, 0, false, CH>;

// lh (a power of two up to 32, at most the lanes of a row) picks the kernel with
// that many lanes per head.  PASS<XT, VEC, LPR, LH, CH> is the policy.
template <template <typename, int, int, int, int> class PASS, typename XT, int VEC, int LPR, int CH = 1>
cudaError_t launch_dot_lanes(const DotArgs &a, cudaStream_t s) {
    switch (a.lh) {
        case 1: return launch_walk<PASS<XT, VEC, LPR, 1, CH>>(a, s);
        case 2: return launch_walk<PASS<XT, VEC, LPR, 2, CH>>(a, s);
        case 4: return launch_walk<PASS<XT, VEC, LPR, 4, CH>>(a, s);
        case 8: return launch_walk<PASS<XT, VEC, LPR, 8, CH>>(a, s);
        default: return launch_walk<PASS<XT, VEC, LPR, 0, CH>>(a, s);
    }
}
template <template <typename, int, int, int, int> class PASS, typename XT, int VEC>
cudaError_t launch_dot_pass(const DotArgs &a, cudaStream_t s) {
    const int64_t slices = static_cast<int64_t>(a.heads) * a.channels / VEC;
    if (slices >= 32) return launch_dot_lanes<PASS, XT, VEC, 32>(a, s);
    if (slices > 16 || a.lh > 16) return launch_dot_lanes<PASS, XT, VEC, 32, 2>(a, s);
    if (slices > 8 || a.lh > 8) return launch_dot_lanes<PASS, XT, VEC, 16>(a, s);
    return launch_dot_lanes<PASS, XT, VEC, 8>(a, s);
}

}  // namespace
}  // namespace tfg
