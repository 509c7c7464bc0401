// Edge-softmax (GAT) aggregation: the map-reduce workflow of tf_geometric
// Fig. 5a (Section 2.1.2) fused with the attention-weighted sum it feeds.
//
//   node scores  s_src[n,h] = <x[n,h,:], a_src[h,:]>, s_dst likewise  (prologue)
//   map          l = LeakyReLU(s_src[src,h] + s_dst[t,h])
//   reduce       m = max over row t of l; den = sum over row t of exp(l - m)
//   map          alpha = exp(l - m) / den
//   aggregate    out[t,h,:] = sum over row t of alpha * x[src,h,:]
//
// The paper's workflow runs map, reduce and map as separate passes over the
// edges.  Here a row is read in a single pass with the running-maximum form of
// the softmax: when an edge raises the row maximum m of a head, the running
// denominator and weighted sum are rescaled by exp(m_old - m_new), which leaves
// alpha and out mathematically unchanged.  Two forms: softmax_fast (this file)
// on graphs of long rows whose layout it takes, the row walk of gat_walk.cuh
// otherwise.  Sums are blocked per 32 edges to keep fp32 chains short, in a
// fixed order (deterministic).  With alpha requested, a second pass over a row
// writes its normalised weights.
//
// Logits are kept in base-2 units: the node scores are multiplied by log2(e)
// once, and since LeakyReLU(c v) = c LeakyReLU(v) for c > 0 every logit,
// maximum and difference is log2(e) times its natural-log value, so
// exp(l - m) = exp2f(l2 - m2).  exp2f is the CUDA math library's base-2
// exponential (documented maximum error 2 ulp over its whole range), so the
// relative error of each weight is set by the fp32 rounding of the logits,
// not by an approximate exponential.
#include <math_constants.h>

#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "gat_walk.cuh"

namespace tfg {
namespace {

constexpr int kSmThreads = 256;
#ifndef TFG_SM_UNROLL
#define TFG_SM_UNROLL 4   // gathers in flight per lane (tuning knob)
#endif
constexpr int kSmUnroll = TFG_SM_UNROLL;
#ifndef TFG_SM_FULL_CHUNKS
#define TFG_SM_FULL_CHUNKS 1   // separate code for full 32-edge chunks (no slot tests)
#endif
constexpr bool kSmFullChunks = TFG_SM_FULL_CHUNKS != 0;
constexpr float kLog2e = 1.4426950408889634f;   // log2(e): natural-log units -> base-2 units

// Compensated dot product (the "Dot2" scheme of Ogita, Rump and Oishi,
// "Accurate sum and dot product", SIAM J. Sci. Comput. 2005): each product
// is split exactly into p + e with one fma, each running sum into s + e with
// the error-free two-sum, and the collected errors are added at the end.  The
// result is as accurate as a dot product in twice the working precision,
// rounded once -- node scores feed every logit, so their error would become a
// relative error in every attention weight.
struct Dot2 {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float a, float b) {
        const float p = a * b;
        const float pe = fmaf(a, b, -p);       // a * b = p + pe exactly
        const float t = s + p;
        const float z = t - s;
        const float se = (s - (t - z)) + (p - z);  // s + p = t + se exactly
        s = t;
        c += pe + se;
    }
    __device__ __forceinline__ float value() const { return s + c; }
};

// One thread per (node, head), VEC channels a load (VEC > 1: channels a multiple
// of VEC, x, a_src and a_dst 16-byte aligned); the additions run channel by
// channel whatever VEC is.  Single-channel loads made the kernel LSU-bound:
// 169,343 nodes x 8 x 16 fp32 55 us against 13 us for its 87 MB.
template <typename XT, int VEC>
__global__ void node_scores(const XT *__restrict__ x, int64_t n, int heads, int channels,
                            const float *__restrict__ a_src, const float *__restrict__ a_dst,
                            float *__restrict__ s_src, float *__restrict__ s_dst) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n * heads) return;
    const int h = static_cast<int>(i % heads);
    const XT *xr = x + i * channels;
    const float *as = a_src + h * channels, *ad = a_dst + h * channels;
    Dot2 a, b;
#pragma unroll 2
    for (int c = 0; c < channels; c += VEC) {
        float xv[VEC], av[VEC], bv[VEC];
        VecLoad<XT, VEC>::load(xr + c, xv);
        gw_load(as + c, av);
        gw_load(ad + c, bv);
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
            a.add(xv[q], av[q]);
            b.add(xv[q], bv[q]);
        }
    }
    s_src[i] = a.value() * kLog2e;
    s_dst[i] = b.value() * kLog2e;
}

__device__ __forceinline__ float leaky(float v, float slope) { return v > 0.f ? v : slope * v; }

// Fast form for the common layout: H divides 32, every lane's VEC features
// lie in one head, and one feature tile covers the row (F <= LPR * VEC).
// One pass over the row in 32-edge chunks:
//  * score lanes: lane (se, sh) = (lane / H, lane % H) evaluates the logit of
//    edge slot se and head sh -- each (edge, head) logit and exponential is
//    computed once.  The chunk's maximum per head (butterfly over the lanes
//    of a head) updates the running maximum m; when m rises, the sums so far
//    are rescaled by exp(m_old - m_new) (a warp-uniform branch, taken a few
//    times per row).  p = exp(l - m) then feeds the denominator.
//  * feature lanes: group g = lane / LPR gathers every G-th edge, fetches the
//    p of its (edge, head) from the score lane holding it with one shuffle,
//    and accumulates p * x into fp32 per-chunk partials.
//
// BWD: the backward by target, as in GatByTarget: a feature lane adds p times the
// LeakyReLU's slope at the edge times its share of dalpha - beta; out is then the
// forward's output, and grad_out, stats and ds_dst are set (114.6M edges, 8 x 16 bf16:
// 2.74 ms against 3.44 ms for a pass that finished <grad_out[t], x[src]> per edge with a
// butterfly).
template <typename XT, int VEC, int LPR, int H, bool BWD>
__device__ __forceinline__ void fast_row(const int32_t *__restrict__ rowptr,
                                         const int32_t *__restrict__ col,
                                         const XT *__restrict__ x, int channels, float slope,
                                         const float *__restrict__ s_src,
                                         const float *__restrict__ s_dst, float *__restrict__ out,
                                         float *__restrict__ alpha, const float *__restrict__ grad_out,
                                         float4 *__restrict__ stats, float *__restrict__ ds_dst,
                                         int64_t t, int lane) {
    using V = VecLoad<XT, VEC>;
    constexpr int G = 32 / LPR;     // edges per feature step
    constexpr int ES = 32 / H;      // edges per score step
    constexpr int R = 32 / ES;      // score steps per 32-edge chunk (= H)
    static_assert(ES % G == 0, "score step must hold whole feature steps");
    // a step's slots e + u * G + g must stay inside one 32-edge chunk (full
    // chunks take no slot test, and p[k0 / ES] must stay inside p[R])
    static_assert(G * kSmUnroll <= 32 && 32 % (G * kSmUnroll) == 0,
                  "steps of G * kSmUnroll slots must tile the 32-edge chunk");
    const int se = lane / H, sh = lane % H;
    const int g = lane / LPR, sub = lane % LPR;
    const int f = H * channels;
    const int f0 = sub * VEC;
    const bool fok = f0 < f;
    const int fh = fok ? f0 / channels : 0;
    const char *xb = reinterpret_cast<const char *>(x + (fok ? f0 : 0));
    const uint32_t row_bytes = static_cast<uint32_t>(f) * static_cast<uint32_t>(sizeof(XT));
    // row slice of node src, addressed in bytes (one wide multiply-add per gather)
    auto gather = [&](uint32_t src) {
        return V::raw(reinterpret_cast<const XT *>(xb + static_cast<uint64_t>(src) * row_bytes));
    };
    const int64_t beg = rowptr[t], end = col ? rowptr[t + 1] : rowptr[t];
    const float sd = __ldg(s_dst + t * H + sh);

    // one pass over the row, 32 edges at a time: the score lanes form the
    // chunk's logits, the running maximum m of each head absorbs the chunk's
    // maximum (earlier sums are rescaled by exp(m_old - m_new) when it rises),
    // then p = exp(l - m) weights the chunk's gathered rows
    float m = -CUDART_INF_F, den = 0.f, acc[VEC];
#pragma unroll
    for (int q = 0; q < VEC; ++q) acc[q] = 0.f;
    float gt[VEC], beta = 0.f, dz = 0.f;             // BWD: the lane's slice of grad_out[t], its shares of beta and ds_dst
    if constexpr (BWD) {
        float ov[VEC];
#pragma unroll
        for (int q = 0; q < VEC; ++q) gt[q] = ov[q] = 0.f;
        if (fok) {
            gw_load(grad_out + t * f + f0, gt);
            gw_load(out + t * f + f0, ov);
        }
        beta = gw_dot(gt, ov);
    }
    // The next chunk's column ids are requested one chunk ahead, and its node scores
    // gathered while this chunk's rows are summed (114.6M edges: 2.29 ms; ids alone
    // ahead 2.40-2.50, neither 2.44-2.57).
    int cnext = (col && beg + lane < end) ? ld_stream(col + beg + lane) : 0;   // lane j: edge j of the next chunk
    float sv[R];     // s_src of the chunk about to run, for (edge r * ES + se, head sh)
#pragma unroll
    for (int r = 0; r < R; ++r)
        sv[r] = __ldg(s_src + static_cast<int64_t>(lane_get(cnext, r * ES + se)) * H + sh);
    // one 32-edge chunk with its column ids in c (lane j: edge base + j; an id of
    // the row past cnt); FULL chunks (all 32 slots used) skip every slot test
    auto chunk = [&](auto full_tag, int c, int cnt) {
        constexpr bool FULL = decltype(full_tag)::value;
        // the first step's row gathers need only the column ids: issue them
        // before the scores so that their latency overlaps the score work
        typename V::Raw raw0[kSmUnroll];
#pragma unroll
        for (int u = 0; u < kSmUnroll; ++u)
            raw0[u] = gather(static_cast<uint32_t>(lane_get(c, (u * G + g) & 31)));
        float p[R];
        float cm = -CUDART_INF_F;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int k = r * ES + se;
            p[r] = (FULL || k < cnt) ? leaky(sv[r] + sd, slope) : -CUDART_INF_F;
            cm = fmaxf(cm, p[r]);
        }
#pragma unroll
        for (int o = H; o < 32; o <<= 1) cm = fmaxf(cm, lane_xor(cm, o));
        const bool rises = cm > m;
        if (lane_any(rises)) {   // warp-uniform; rare after the first chunks
            const float sc = rises ? (m == -CUDART_INF_F ? 0.f : exp2f(m - cm)) : 1.f;
            den *= sc;
            const float fsc = lane_get(sc, fh);   // lane fh scores head fh
            if constexpr (BWD) {
                dz *= fsc;
            } else {
#pragma unroll
                for (int q = 0; q < VEC; ++q) acc[q] *= fsc;
            }
            m = fmaxf(m, cm);
        }
        float den_part = 0.f;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int k = r * ES + se;
            p[r] = (FULL || k < cnt) ? exp2f(p[r] - m) : 0.f;
            den_part += p[r];
            if (BWD) p[r] = sv[r] + sd > 0.f ? p[r] : slope * p[r];
        }
        den += den_part;
        // the next chunk's node scores, requested before this chunk's rows
#pragma unroll
        for (int r = 0; r < R; ++r)
            sv[r] = __ldg(s_src + static_cast<int64_t>(lane_get(cnext, r * ES + se)) * H + sh);
        float part[VEC], zpart = 0.f;
#pragma unroll
        for (int q = 0; q < VEC; ++q) part[q] = 0.f;
#pragma unroll
        for (int e = 0; e < 32; e += G * kSmUnroll) {
            if (!FULL && e >= cnt) break;   // warp-uniform
            typename V::Raw raw[kSmUnroll];
            float pw[kSmUnroll];
#pragma unroll
            for (int u = 0; u < kSmUnroll; ++u) {
                const int k0 = e + u * G;              // edge of group 0 in this step
                const int k = k0 + g;
                // p of (edge k, head fh) sits in lane (k % ES) * H + fh, register k / ES
                pw[u] = lane_get(p[k0 / ES], ((k0 % ES) + g) * H + fh);
                if (e == 0) raw[u] = raw0[u];
                else raw[u] = gather(static_cast<uint32_t>(lane_get(c, k & 31)));
            }
#pragma unroll
            for (int u = 0; u < kSmUnroll; ++u) {
                float v[VEC];
                V::widen(raw[u], v);
                if constexpr (BWD) {
                    zpart = fmaf(pw[u], gw_dot(gt, v) - beta, zpart);
                } else if constexpr (VEC % 2 == 0) {
                    const float2 w2 = make_float2(pw[u], pw[u]);
#pragma unroll
                    for (int q = 0; q < VEC; q += 2) {
                        const float2 r2 = fma2(make_float2(v[q], v[q + 1]), w2,
                                               make_float2(part[q], part[q + 1]));
                        part[q] = r2.x;
                        part[q + 1] = r2.y;
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < VEC; ++q) part[q] = fmaf(pw[u], v[q], part[q]);
                }
            }
        }
        if constexpr (BWD) {
            dz += zpart;
        } else {
#pragma unroll
            for (int q = 0; q < VEC; ++q) acc[q] += part[q];
        }
    };
    for (int64_t base = beg; base < end; base += 32) {
        const int cnt = static_cast<int>(min64(32, end - base));
        const int c = cnext;
        cnext = (base + 32 + lane < end) ? ld_stream(col + base + 32 + lane) : 0;
        // slots without an edge have zero weight: they read the row of the chunk's last
        // edge, since an infinity in another node's row would come through it
        if (kSmFullChunks && cnt == 32) chunk(std::true_type{}, c, 32);
        else chunk(std::false_type{}, lane_get(c, min(lane, cnt - 1)), cnt);
    }
#pragma unroll
    for (int o = H; o < 32; o <<= 1) den += lane_xor(den, o);
#pragma unroll
    for (int o = LPR; o < 32; o <<= 1) {
        if constexpr (BWD) {
            dz += lane_xor(dz, o);
        } else {
#pragma unroll
            for (int q = 0; q < VEC; ++q) acc[q] += lane_xor(acc[q], o);
        }
    }
    const float dh = lane_get(den, fh);   // lane fh holds head fh's denominator
    if constexpr (BWD) {
        const float mh = lane_get(m, fh), sdh = lane_get(sd, fh);
        const int hl = channels / VEC;               // lanes of a head, a power of two
        const float d = gw_head_sum<0>(dz, hl), b = gw_head_sum<0>(beta, hl);
        if (lane < LPR && fok && f0 % channels == 0) {
            ds_dst[t * H + fh] = end > beg ? d / dh : 0.f;
            stats[t * H + fh] = make_float4(sdh, mh, end > beg ? 1.f / dh : 0.f, b);
        }
        return;
    }
    if (lane < LPR && fok) {
        float *o = out + t * f + f0;
#pragma unroll
        for (int q = 0; q < VEC; ++q) o[q] = end > beg ? acc[q] / dh : 0.f;
    }
    if (alpha) {
        for (int64_t base = beg; base < end; base += 32) {
            const int cnt = static_cast<int>(min64(32, end - base));
            const int c = lane < cnt ? __ldg(col + base + lane) : 0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int k = r * ES + se;
                const int src = lane_get(c, k);
                if (k < cnt) {
                    const float l = leaky(__ldg(s_src + static_cast<int64_t>(src) * H + sh) + sd, slope);
                    alpha[(base + k) * H + sh] = exp2f(l - m) / den;
                }
            }
        }
    }
}

// Graphs of a mean in-degree below this take the row walk (gat_walk.cuh), whose
// warps share hub rows and whose windows cross row ends; longer rows take
// softmax_fast, whose score lanes evaluate each (edge, head) once.  Measured, walk /
// softmax_fast, us a call: block-model graphs of 100,000 nodes, mean degree 16, 32, 64 and
// 100, 8 x 16 bf16 115 / 140, 155 / 182, 230 / 254, 308 / 334; 8 x 16 fp32 114 / 149, 166 /
// 208, 270 / 311, 376 / 432; 4 x 8 bf16 79 / 97, 99 / 119, 133 / 172, 163 / 234; 114.6M
// edges, mean 492, 8 x 16 bf16 2.59 / 2.24 ms.  So the two meet between 100 and 492; the
// line stands where they met before the walk's partial steps and has not been moved since.
// Where hubs hold a large part of the edges the walk is faster at every degree
// (preferential attachment, mean 64, 8 x 16 bf16 247 / 675), but E and N do not tell.
#ifndef TFG_SM_WALK_DEGREE
#define TFG_SM_WALK_DEGREE 32
#endif
constexpr int64_t kWalkMaxDegree = TFG_SM_WALK_DEGREE;

// Measured on the 114.6M-edge graph (bf16, 8 heads x 16), ids and scores
// requested one chunk ahead: 3 CTAs per SM with 4 gathers in flight per lane
// 2.29 ms; 4 CTAs 2.31 ms; 3 CTAs with 8 in flight 2.52 ms.  Without the
// early requests: 4 CTAs / 4 in flight 2.44-2.50 ms, 3 / 8 2.62 ms, 2 / 8 3.48 ms.
#ifndef TFG_SMF_BLOCKS
#define TFG_SMF_BLOCKS 3     // resident CTAs per SM of softmax_fast
#endif

template <typename XT, int VEC, int LPR, int H>
__global__ void __launch_bounds__(kSmThreads, TFG_SMF_BLOCKS)
softmax_fast(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ col,
             const XT *__restrict__ x, int64_t n, int channels, float slope,
             const float *__restrict__ s_src, const float *__restrict__ s_dst,
             float *__restrict__ out, float *__restrict__ alpha) {
    for_each_row(rowptr, n, [&](int64_t t, int lane) {
        fast_row<XT, VEC, LPR, H, false>(rowptr, col, x, channels, slope, s_src, s_dst, out, alpha, nullptr,
                                         nullptr, nullptr, t, lane);
    });
}

template <typename XT, int VEC, int LPR, int H>
__global__ void __launch_bounds__(kSmThreads, TFG_SMF_BLOCKS)
softmax_fast_bwd(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ col,
                 const XT *__restrict__ x, int64_t n, int channels, float slope,
                 const float *__restrict__ s_src, const float *__restrict__ s_dst,
                 float *__restrict__ out, const float *__restrict__ grad_out, float4 *__restrict__ stats,
                 float *__restrict__ ds_dst) {
    for_each_row(rowptr, n, [&](int64_t t, int lane) {
        fast_row<XT, VEC, LPR, H, true>(rowptr, col, x, channels, slope, s_src, s_dst, out, nullptr, grad_out,
                                        stats, ds_dst, t, lane);
    });
}

constexpr int kFastBwdHeads = 8;       // the backward's most: 16 score steps a chunk and its sums spill
constexpr int64_t kSmMinWork = 2048;   // edges + rows per CTA, at least

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

// Launch softmax_fast (or its backward) when the layout allows it; false means
// "take the walk".
template <typename XT, int VEC, int LPR>
bool launch_fast_lpr(const GatArgs &a, int64_t e, bool bwd, cudaStream_t s) {
    constexpr int G = 32 / LPR;
    const int grid = balanced_grid(a.n, e, kSmMinWork);
    const XT *xp = static_cast<const XT *>(a.x);
#define TFG_FAST(HH)                                                                              \
    if (a.heads == HH) {                                                                          \
        if constexpr ((32 / HH) % G == 0) {                                                       \
            if (bwd) {                                                                            \
                if constexpr (HH <= kFastBwdHeads)                                                \
                    softmax_fast_bwd<XT, VEC, LPR, HH><<<grid, kSmThreads, 0, s>>>(               \
                        a.rowptr, a.col, xp, a.n, a.channels, a.slope, a.s_src, a.s_dst,          \
                        const_cast<float *>(a.fwd_out), a.grad_out, a.stats, a.ds_dst);           \
            } else                                                                                \
                softmax_fast<XT, VEC, LPR, HH><<<grid, kSmThreads, 0, s>>>(                       \
                    a.rowptr, a.col, xp, a.n, a.channels, a.slope, a.s_src, a.s_dst, a.out, a.alpha); \
            return true;                                                                          \
        }                                                                                         \
        return false;                                                                             \
    }
    TFG_FAST(1)
    TFG_FAST(2)
    TFG_FAST(4)
    TFG_FAST(8)
    TFG_FAST(16)
#undef TFG_FAST
    return false;
}

template <typename XT, int VEC>
bool launch_fast(const GatArgs &a, int64_t e, bool bwd, cudaStream_t s) {
    const int64_t f = static_cast<int64_t>(a.heads) * a.channels;
    if (a.channels % VEC != 0 || f > 32 * VEC || e < kWalkMaxDegree * a.n) return false;
    if (bwd && a.heads > kFastBwdHeads) return false;
    const int64_t chunks = f / VEC;
    if (chunks > 16) return launch_fast_lpr<XT, VEC, 32>(a, e, bwd, s);
    if (chunks > 8) return launch_fast_lpr<XT, VEC, 16>(a, e, bwd, s);
    return launch_fast_lpr<XT, VEC, 8>(a, e, bwd, s);
}

// Scratch of tfg_edge_softmax_aggregate_noalloc: the node scores s_src and
// s_dst of up to kNoAllocNodeHeads (node, head) pairs each, 16 MiB in all,
// resident on every GPU that loads the library for as long as it stays
// loaded.  Every call overwrites the part it uses, so nothing needs clearing.
constexpr int64_t kNoAllocNodeHeads = int64_t(1) << 21;
static __device__ __align__(256) float g_noalloc_scores[2 * kNoAllocNodeHeads];

}  // namespace

int64_t noalloc_softmax_max_node_heads() { return kNoAllocNodeHeads; }

// Device address of the scratch array on the current device.  Host code
// cannot use the array's name as a device pointer, so the address is looked
// up once per device with that device current (the lookup may load the
// module, which is why the first call on a device must not be captured into
// a CUDA graph) and cached.
cudaError_t noalloc_softmax_scratch(void **ptr, size_t *bytes) {
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static void *addr[kMaxDevices] = {};
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (addr[dev] == nullptr) {
        void *p = nullptr;
        err = cudaGetSymbolAddress(&p, g_noalloc_scores);
        if (err != cudaSuccess) return err;
        addr[dev] = p;
    }
    *ptr = addr[dev];
    *bytes = sizeof(g_noalloc_scores);
    return cudaSuccess;
}

cudaError_t launch_node_scores(const void *x, int x_dtype, int64_t n, int heads, int channels,
                               const float *a_src, const float *a_dst, float *s_src, float *s_dst,
                               cudaStream_t s) {
    const int grid = ceil_div(n * heads, 256);
    const uint16_t *xh = static_cast<const uint16_t *>(x);
    const float *xf = static_cast<const float *>(x);
    auto a16 = [](const void *p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; };
    const bool aligned = a16(x) && a16(a_src) && a16(a_dst);
    if (x_dtype == TFG_BF16 && aligned && channels % 8 == 0)
        node_scores<uint16_t, 8><<<grid, 256, 0, s>>>(xh, n, heads, channels, a_src, a_dst, s_src, s_dst);
    else if (x_dtype == TFG_BF16)
        node_scores<uint16_t, 1><<<grid, 256, 0, s>>>(xh, n, heads, channels, a_src, a_dst, s_src, s_dst);
    else if (aligned && channels % 4 == 0)
        node_scores<float, 4><<<grid, 256, 0, s>>>(xf, n, heads, channels, a_src, a_dst, s_src, s_dst);
    else
        node_scores<float, 1><<<grid, 256, 0, s>>>(xf, n, heads, channels, a_src, a_dst, s_src, s_dst);
    return cudaGetLastError();
}

namespace {
// 16-byte slices (or 8-byte bf16 ones) that lie in one head: one slice per lane, the
// fewest lanes that cover the row (4 x 8 bf16, 100,000 nodes of mean degree 23: 84 us with
// 4 lanes, 90 with 8).
template <typename XT, int VEC>
cudaError_t walk_vec(const GatArgs &a, cudaStream_t s) {
    const int64_t slices = static_cast<int64_t>(a.heads) * a.channels / VEC;
    if (slices <= 4) return launch_walk<GatByTarget<XT, VEC, 4, 1, 1, false>>(a, s);
    if (slices <= 8) return launch_walk<GatByTarget<XT, VEC, 8, 1, 1, false>>(a, s);
    if (slices <= 16) return launch_walk<GatByTarget<XT, VEC, 16, 1, 1, false>>(a, s);
    return launch_walk<GatByTarget<XT, VEC, 32, 1, 1, false, 2>>(a, s);
}
template <typename XT, int LPR, int T>
cudaError_t walk_lanes(const GatArgs &a, cudaStream_t s) {
    if (T == 1 || a.heads == 1) return launch_walk<GatByTarget<XT, 1, LPR, T, 1, false>>(a, s);
    return launch_walk<GatByTarget<XT, 1, LPR, T, T, false>>(a, s);
}
template <typename XT>
cudaError_t walk_scalar(const GatArgs &a, cudaStream_t s) {
    const int64_t f = static_cast<int64_t>(a.heads) * a.channels;
    if (f <= 8) return walk_lanes<XT, 8, 1>(a, s);
    if (f <= 16) return walk_lanes<XT, 16, 1>(a, s);
    if (f <= 32) return walk_lanes<XT, 16, 2>(a, s);
    if (f <= 48) return walk_lanes<XT, 16, 3>(a, s);
    const int64_t passes = (f + 127) / 128, per = (f + passes - 1) / passes;
    if (per <= 64) return walk_lanes<XT, 32, 2>(a, s);
    if (per <= 96) return walk_lanes<XT, 32, 3>(a, s);
    return walk_lanes<XT, 32, 4>(a, s);
}
}  // namespace

size_t softmax_workspace_bytes(int64_t n, int heads) {
    return 2 * align256(sizeof(float) * size_t(n > 0 ? n : 1) * size_t(heads));
}

// Softmax statistics and ds_dst of the backward (attention_backward.cu), when
// softmax_fast takes the layout; false means "take the walk".
bool launch_softmax_fast_bwd(const GatArgs &a, int x_dtype, int64_t e, cudaStream_t s) {
    return x_dtype == TFG_BF16 ? launch_fast<uint16_t, 8>(a, e, true, s) : launch_fast<float, 4>(a, e, true, s);
}

cudaError_t launch_edge_softmax(const int32_t *rowptr, const int32_t *col, const void *x,
                                int x_dtype, int64_t n, int64_t e, int heads, int channels,
                                const float *a_src, const float *a_dst, float slope, float *out,
                                float *alpha, void *ws, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    float *s_src = static_cast<float *>(ws);
    float *s_dst = reinterpret_cast<float *>(static_cast<char *>(ws) +
                                             align256(sizeof(float) * size_t(n) * size_t(heads)));
    const cudaError_t err = launch_node_scores(x, x_dtype, n, heads, channels, a_src, a_dst, s_src, s_dst, s);
    if (err != cudaSuccess) return err;
    const bool aligned = (reinterpret_cast<uintptr_t>(x) % 16 == 0) &&
                         (reinterpret_cast<uintptr_t>(out) % 16 == 0);
    const GatArgs a{rowptr, col, x, n, heads, channels, slope, s_src, s_dst, out, alpha};
    if (x_dtype == TFG_BF16) {
        if (aligned && launch_fast<uint16_t, 8>(a, e, false, s)) return cudaGetLastError();
        if (aligned && channels % 8 == 0) return walk_vec<uint16_t, 8>(a, s);
        if (aligned && channels % 4 == 0) return walk_vec<uint16_t, 4>(a, s);
        return walk_scalar<uint16_t>(a, s);
    }
    if (aligned && launch_fast<float, 4>(a, e, false, s)) return cudaGetLastError();
    if (aligned && channels % 4 == 0) return walk_vec<float, 4>(a, s);
    return walk_scalar<float>(a, s);
}

}  // namespace tfg
