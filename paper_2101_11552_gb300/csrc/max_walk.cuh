// Max aggregation with argmax as a row-walk policy (row_walk.cuh).
//
// The running maximum of a feature keeps the CSR POSITION of its edge; the
// original id is looked up once per row (perm) when the result is written.  The
// row's first edge is taken whatever its value (NaN included); after that only a
// strictly larger value replaces the maximum, so ties keep the earliest edge and a
// NaN is only ever held from the first edge.  States of lane groups and of warps
// that share a row combine by max_combine, which depends only on values and
// positions: the larger value wins, equal values go to the smaller position, and
// a NaN held from the row's first edge wins over everything.  That is exactly what
// one pass over the row in order gives.
#pragma once
#include <cuda_bf16.h>
#include <math_constants.h>

#include "row_walk.cuh"

namespace tfg {

struct MaxFwdArgs {
    const int32_t *rowptr, *col, *perm;
    const float *w;              // CSR order, or null
    const void *x;
    int64_t n, f;
    float *out;
    int32_t *argmax;
    __host__ __device__ uint32_t width() const { return static_cast<uint32_t>(f); }
    __host__ __device__ bool statistics() const { return false; }
};

namespace {

// Measured at 114.6M edges, F = 128 bf16: packed with argmax 1.64 ms (32 warps; 28
// 1.69, 24 1.75; a row per warp with widened compares 4.70 ms; the bare gather of
// the rows 1.27), on 20M edges F = 96 fp32 548 us with 28 warps, 574 with 20; on
// short rows (169,343 nodes, mean in-degree 6.9, F = 128 fp32) 107 us with 28, 117
// with 24.
#ifndef TFG_MW_WARPS
#define TFG_MW_WARPS 28
#endif
#ifndef TFG_MW_PACKED_WARPS
#define TFG_MW_PACKED_WARPS 32
#endif
#ifndef TFG_MW_DEPTH
#define TFG_MW_DEPTH 4
#endif

__device__ __forceinline__ void max_combine(float &b, int32_t &p, float ob, int32_t op,
                                            int32_t row_beg) {
    if (op < 0) return;
    const bool mine_first_nan = p == row_beg && isnan(b);
    const bool other_first_nan = op == row_beg && isnan(ob);
    bool take;
    if (p < 0 || other_first_nan) take = true;
    else if (mine_first_nan) take = false;
    else take = ob > b || (ob == b && op < p);
    if (take) {
        b = ob;
        p = op;
    }
}

// PACKED (bf16 rows without weights, 16-byte slices): the maxima stay bf16 pairs
// and the positions 16-bit pairs relative to `base`, so two features cost one
// compare and two selects instead of two widenings, two compares and four
// selects; every 65,000 edges of a row the state moves to full positions.
// ARG = false (PACKED only): no argmax; a NaN is passed over, as fmaxf does.
template <typename XT, int VEC, int LPR, int T, bool PACKED, bool ARG = true>
struct MaxByTarget {
    static_assert(ARG || PACKED, "without argmax only the packed form is used");
    using V = VecLoad<XT, VEC>;
    static constexpr int kWarps = PACKED ? TFG_MW_PACKED_WARPS : TFG_MW_WARPS, kLpr = LPR, G = 32 / LPR;
    static constexpr int kTile = LPR * VEC * T, kHeadsPerLane = T;
    static constexpr int kState = (ARG ? 2 : 1) * T * VEC, kHeld = 0;
    static constexpr int kStepFull = TFG_MW_DEPTH * G > 32 ? 32 / G : TFG_MW_DEPTH;
    static_assert(32 % (G * kStepFull) == 0, "a full window is read in whole steps");
    static constexpr int kStepPart = walk_part(G) < kStepFull ? walk_part(G) : kStepFull;
    static constexpr int kPairs = PACKED ? VEC / 2 : 1;
    static constexpr int kReach = 65000;          // edges that 16-bit positions cover
    static constexpr uint32_t kLowest = 0xff80ff80u, kNone = 0xffffffffu;
    const MaxFwdArgs &a;
    int sub, g, own;
    uint32_t f0, row_bytes;
    const char *xb;
    float *slot;                                  // the warp's own parking slot, free until the walk ends
    float b[T][VEC];
    int32_t p[T][VEC];
    uint32_t pb[kPairs], pp[kPairs];
    int32_t k, base, rbeg;                        // next edge's position, PACKED's origin, the row's first edge
    bool first, spilt;

    __device__ __forceinline__ MaxByTarget(const MaxFwdArgs &args, uint32_t ft, float *hold, float *) : a(args), slot(hold) {
        const int lane = threadIdx.x & 31;
        sub = lane % LPR;
        g = lane / LPR;
        const uint32_t f = a.width();
        f0 = ft + sub * VEC;
        own = f0 < f ? min(T, static_cast<int>((f - f0 + LPR * VEC - 1) / (LPR * VEC))) : 0;
        xb = reinterpret_cast<const char *>(static_cast<const XT *>(a.x) + (own > 0 ? f0 : 0));
        row_bytes = f * static_cast<uint32_t>(sizeof(XT));
    }
    __device__ __forceinline__ const XT *row(uint32_t id) const {
        return reinterpret_cast<const XT *>(xb + static_cast<uint64_t>(id) * row_bytes);
    }
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                b[i][q] = -CUDART_INF_F;
                p[i][q] = -1;
            }
        clear_packed();
        spilt = false;
    }
    __device__ __forceinline__ void clear_packed() {
#pragma unroll
        for (int q = 0; q < kPairs; ++q) {
            pb[q] = kLowest;
            pp[q] = kNone;
        }
    }
    __device__ __forceinline__ void open(int32_t, int32_t at, int32_t row_beg) {
        clear();
        k = base = at;
        rbeg = row_beg;
        first = ARG && at == row_beg;
    }
    static __device__ __forceinline__ uint32_t word(const uint4 &r, int q) {
        return q == 0 ? r.x : (q == 1 ? r.y : (q == 2 ? r.z : r.w));
    }
    static __device__ __forceinline__ void take(uint32_t &best, uint32_t &pos, uint32_t v, uint32_t at) {
        __nv_bfloat162 x, y;
        memcpy(&x, &v, 4);
        memcpy(&y, &best, 4);
        if constexpr (!ARG) {
            const __nv_bfloat162 z = __hmax2(x, y);
            memcpy(&best, &z, 4);
            return;
        }
        const uint32_t m = __hgt2_mask(x, y);             // false for NaN, as v > best is
        best = (v & m) | (best & ~m);
        pos = (at & m) | (pos & ~m);
    }
    template <int D, bool CHECK>
    __device__ __forceinline__ void step(const int32_t *sp, int left, int32_t at) {
        typename V::Raw raw[D][T];
        float w[D];
#pragma unroll
        for (int u = 0; u < D; ++u) {
            const uint32_t id = static_cast<uint32_t>(sp[u * G]);
            const bool ok = !CHECK || left > u * G;
            if (!PACKED) w[u] = a.w && ok ? __ldg(a.w + at + u * G) : 1.f;
            const XT *r = row(id);
#pragma unroll
            for (int i = 0; i < T; ++i)
                raw[u][i] = (T == 1 ? ok : ok && i < own) ? V::raw(r + i * LPR * VEC) : V::zero();
            if constexpr (PACKED) {
                if (CHECK && !ok) raw[u][0] = make_uint4(kLowest, kLowest, kLowest, kLowest);
            }
        }
#pragma unroll
        for (int u = 0; u < D; ++u) {
            if constexpr (PACKED) {
                const uint32_t at2 = static_cast<uint32_t>(at + u * G - base) * 0x10001u;
#pragma unroll
                for (int q = 0; q < kPairs; ++q) take(pb[q], pp[q], word(raw[u][0], q), at2);
            } else {
                const bool ok = !CHECK || left > u * G;
#pragma unroll
                for (int i = 0; i < T; ++i) {
                    float v[VEC];
                    V::widen(raw[u][i], v);
#pragma unroll
                    for (int q = 0; q < VEC; ++q) {
                        const float m = a.w ? w[u] * v[q] : v[q];
                        if (ok && m > b[i][q]) {
                            b[i][q] = m;
                            p[i][q] = at + u * G;
                        }
                    }
                }
            }
        }
    }
    template <bool CHECK>
    __device__ __forceinline__ void add(const int32_t *ids, int cnt) {
        if (PACKED && ARG && k - base > kReach - 32) spill();
        if (first) {                                      // the row's first edge, whatever its value
            first = false;
            if (g == 0) {
                const XT *r = row(static_cast<uint32_t>(ids[0]));
                const float w0 = a.w ? __ldg(a.w + k) : 1.f;
#pragma unroll
                for (int i = 0; i < T; ++i) {
                    if (T > 1 && i >= own) continue;
                    const typename V::Raw raw = V::raw(r + i * LPR * VEC);
                    if constexpr (PACKED) {
#pragma unroll
                        for (int q = 0; q < kPairs; ++q) {
                            pb[q] = word(raw, q);
                            pp[q] = 0;                    // base is the row's first position
                        }
                    } else {
                        float v[VEC];
                        V::widen(raw, v);
#pragma unroll
                        for (int q = 0; q < VEC; ++q) {
                            b[i][q] = a.w ? w0 * v[q] : v[q];
                            p[i][q] = k;
                        }
                    }
                }
            }
        }
        const int32_t *sp = ids + g;
        int32_t at = k + g;
        k += cnt;
        if (!CHECK) {                                     // a full window
#pragma unroll
            for (int e = 0; e < 32; e += G * kStepFull) step<kStepFull, false>(sp + e, 0, at + e);
            return;
        }
#pragma unroll 1
        for (; cnt >= G * kStepFull; cnt -= G * kStepFull, sp += G * kStepFull, at += G * kStepFull) step<kStepFull, false>(sp, 0, at);
#pragma unroll 1
        for (; cnt > 0; cnt -= G * kStepPart, sp += G * kStepPart, at += G * kStepPart) step<kStepPart, true>(sp, cnt - g, at);
    }
    template <class GetB, class GetP>
    __device__ __forceinline__ void fold(GetB get_b, GetP get_p) {
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                const float ob = get_b(b[i][q], i * VEC + q);
                if constexpr (!ARG) {
                    b[i][q] = fmaxf(b[i][q], ob);
                    continue;
                }
                const int32_t op = get_p(p[i][q], i * VEC + q);
                max_combine(b[i][q], p[i][q], ob, op, rbeg);
            }
    }
    // the packed state as values and positions, the lane groups combined
    __device__ __forceinline__ void unpack_and_join() {
        if constexpr (PACKED) {
#pragma unroll
            for (int q = 0; q < kPairs; ++q) {
                b[0][2 * q] = bf16_lo(pb[q]);
                b[0][2 * q + 1] = bf16_hi(pb[q]);
                if constexpr (!ARG) continue;
                const uint32_t lo = pp[q] & 0xffffu, hi = pp[q] >> 16;
                p[0][2 * q] = lo == 0xffffu ? -1 : base + static_cast<int32_t>(lo);
                p[0][2 * q + 1] = hi == 0xffffu ? -1 : base + static_cast<int32_t>(hi);
            }
        }
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1)
            fold([&](float mine, int) { return lane_xor(mine, o); },
                 [&](int32_t mine, int) { return lane_xor(mine, o); });
    }
    __device__ __forceinline__ void spill() {             // warp-uniform, rare
        unpack_and_join();
        if (spilt) merge(slot);
        park(slot);
        __syncwarp();
        spilt = true;
        clear_packed();
        base = k;
    }
    __device__ __forceinline__ void join() {
        unpack_and_join();
        if (PACKED && spilt) {
            merge(slot);
            spilt = false;
            __syncwarp();
        }
    }
    __device__ __forceinline__ void merge(const float *from) {
        fold([&](float, int q) { return from[q * LPR + sub]; },
             [&](int32_t, int q) { return __float_as_int(from[(T * VEC + q) * LPR + sub]); });
    }
    __device__ __forceinline__ void park(float *to) const {
        if (g != 0) return;
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                to[(i * VEC + q) * LPR + sub] = b[i][q];
                if (ARG) to[(T * VEC + i * VEC + q) * LPR + sub] = __int_as_float(p[i][q]);
            }
    }
    __device__ __forceinline__ bool wants_after() const { return false; }
    __device__ __forceinline__ void after(int, int32_t, int32_t, int32_t) {}
    __device__ __forceinline__ void close(int32_t t, int32_t beg, int32_t end, bool) {
        if (g != 0) return;
        const uint64_t at = static_cast<uint64_t>(static_cast<uint32_t>(t)) * a.width() + f0;
#pragma unroll
        for (int i = 0; i < T; ++i) {
            if (i >= own) continue;
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                if constexpr (ARG) {
                    p[i][q] = p[i][q] < 0 ? -1 : __ldg(a.perm + p[i][q]);
                    b[i][q] = p[i][q] < 0 ? 0.f : b[i][q];
                } else {
                    b[i][q] = end > beg ? b[i][q] : 0.f;
                }
            }
            float *o = a.out + at + i * LPR * VEC;
            int32_t *r = ARG ? a.argmax + at + i * LPR * VEC : nullptr;
            if constexpr (VEC % 4 == 0) {                 // out and argmax 16-byte aligned
#pragma unroll
                for (int q = 0; q < VEC; q += 4) {
                    *reinterpret_cast<float4 *>(o + q) = make_float4(b[i][q], b[i][q + 1], b[i][q + 2], b[i][q + 3]);
                    if constexpr (ARG) *reinterpret_cast<int4 *>(r + q) = make_int4(p[i][q], p[i][q + 1], p[i][q + 2], p[i][q + 3]);
                }
            } else {
#pragma unroll
                for (int q = 0; q < VEC; ++q) {
                    o[q] = b[i][q];
                    if constexpr (ARG) r[q] = p[i][q];
                }
            }
        }
    }
};

// ---- backward -------------------------------------------------------------
struct MaxBwdArgs {
    const int32_t *rowptr, *col, *perm;   // CSR by source (col holds targets)
    const int32_t *argmax;
    const float *w;                       // original edge order, or null
    const float *grad_out;
    int64_t n, f, e;
    float *grad_x;
    const uint8_t *mark;                  // max_bwd_kernel: bit j of mark[e] when edge e wins a feature of group j
    int group;                            // features per group, a multiple of 4
    __host__ __device__ uint32_t width() const { return static_cast<uint32_t>(f); }
    __host__ __device__ bool statistics() const { return false; }
};

// 32 warps against 28 on the two graphs below: F = 128 164 / 165 us, F = 41 79 / 89;
// four slices a lane (F > 64 in single floats) spill at 32 warps and take 28.
#ifndef TFG_MXA_WARPS
#define TFG_MXA_WARPS 32
#endif
#ifndef TFG_MXA_DEPTH
#define TFG_MXA_DEPTH 4        // edges in flight per warp
#endif

// grad_x[s, f] = sum over the out-edges e = (s -> t) of s, in CSR (= original)
// order, of w_e grad_out[t, f] where argmax[t, f] == e: a lane requests its slices
// of row t of argmax and of the gradient together and adds where the argmax names
// the edge.  On short rows an edge wins about one feature in its target's
// in-degree, so every row is read, and equal shares of edges and row ends keep the
// warps busy to the end: 169,343 nodes of mean degree 6.9, F = 128 fp32, 164 us
// against 234 with a warp per row; 100,000 nodes, 1.5M edges, F = 41, 79 against 230.
template <int VEC, int T>
struct MaxBySource {
    static constexpr int kWarps = T > 2 ? 28 : TFG_MXA_WARPS, kLpr = 32, D = TFG_MXA_DEPTH;
    static_assert(32 % D == 0, "a full window is read in whole steps");
    static constexpr int kTile = 32 * VEC * T, kHeadsPerLane = 1;
    static constexpr int kState = T * VEC, kHeld = 0;
    const MaxBwdArgs &a;
    int lane, own;
    uint32_t f, f0;
    int32_t k;                            // the next edge's position
    float acc[T][VEC];

    __device__ __forceinline__ MaxBySource(const MaxBwdArgs &args, uint32_t ft, float *, float *) : a(args) {
        lane = threadIdx.x & 31;
        f = a.width();
        f0 = ft + lane * VEC;
        own = f0 < f ? min(T, static_cast<int>((f - f0 + 32 * VEC - 1) / (32 * VEC))) : 0;
    }
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int q = 0; q < VEC; ++q) acc[i][q] = 0.f;
    }
    __device__ __forceinline__ void open(int32_t, int32_t at, int32_t) {
        clear();
        k = at;
    }
    struct Slice {
        int32_t am[T][VEC];
        float g[T][VEC];
    };
    // the first n slices of row t; the others hold no edge's id
    __device__ __forceinline__ void load(Slice &s, uint32_t t, int n) const {
        const uint64_t o = static_cast<uint64_t>(t) * f + f0;
#pragma unroll
        for (int i = 0; i < T; ++i) {
            const bool on = i < n;
            if constexpr (VEC == 4) {
                const int4 v = on ? __ldg(reinterpret_cast<const int4 *>(a.argmax + o + i * 32 * VEC)) : make_int4(-2, -2, -2, -2);
                const float4 g4 = on ? __ldg(reinterpret_cast<const float4 *>(a.grad_out + o + i * 32 * VEC))
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
                s.am[i][0] = v.x; s.am[i][1] = v.y; s.am[i][2] = v.z; s.am[i][3] = v.w;
                s.g[i][0] = g4.x; s.g[i][1] = g4.y; s.g[i][2] = g4.z; s.g[i][3] = g4.w;
            } else {
                s.am[i][0] = on ? __ldg(a.argmax + o + i * 32 * VEC) : -2;
                s.g[i][0] = on ? __ldg(a.grad_out + o + i * 32 * VEC) : 0.f;
            }
        }
    }
    // this slice's terms of edge e (never -2)
    __device__ __forceinline__ void take(const Slice &s, int32_t e, float w) {
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int q = 0; q < VEC; ++q) acc[i][q] = s.am[i][q] == e ? fmaf(w, s.g[i][q], acc[i][q]) : acc[i][q];
    }
    template <bool CHECK>
    __device__ __forceinline__ void add(const int32_t *ids, int cnt) {
        const int64_t at = k;
        k += cnt;
#pragma unroll 1
        for (int e = 0; e < cnt; e += D) {
            Slice s[D];
            int32_t ed[D];
            float w[D];
#pragma unroll
            for (int u = 0; u < D; ++u) {
                const bool ok = !CHECK || e + u < cnt;
                ed[u] = ok ? __ldg(a.perm + at + e + u) : -1;
                load(s[u], static_cast<uint32_t>(ids[e + u]), ok ? own : 0);
            }
#pragma unroll
            for (int u = 0; u < D; ++u) w[u] = a.w && (!CHECK || e + u < cnt) ? __ldg(a.w + ed[u]) : 1.f;
#pragma unroll
            for (int u = 0; u < D; ++u) take(s[u], ed[u], w[u]);
        }
    }
    __device__ __forceinline__ void join() {}
    __device__ __forceinline__ void merge(const float *slot) {
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int q = 0; q < VEC; ++q) acc[i][q] += slot[(i * VEC + q) * 32 + lane];
    }
    __device__ __forceinline__ void park(float *slot) const {
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int q = 0; q < VEC; ++q) slot[(i * VEC + q) * 32 + lane] = acc[i][q];
    }
    __device__ __forceinline__ bool wants_after() const { return false; }
    __device__ __forceinline__ void after(int, int32_t, int32_t, int32_t) {}
    __device__ __forceinline__ void close(int32_t s, int32_t, int32_t, bool) {
        float *o = a.grad_x + static_cast<uint64_t>(static_cast<uint32_t>(s)) * f + f0;
#pragma unroll
        for (int i = 0; i < T; ++i) {
            if (i >= own) continue;
            if constexpr (VEC == 4)
                *reinterpret_cast<float4 *>(o + i * 32 * VEC) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
            else o[i * 32 * VEC] = acc[i][0];
        }
    }
};

}  // namespace
}  // namespace tfg
