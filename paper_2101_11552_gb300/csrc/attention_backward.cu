// Backward of the GAT edge-softmax aggregation (Fig. 5a workflow): the
// gradients with respect to the node features x and the attention vectors
// a_src, a_dst, given grad_out = dL/dout and the forward's output out.  The
// paper keeps graph construction and mini-batching differentiable (Sections
// 2.1.1 and 2.1.3); with alpha the softmax weights of the forward:
//
//   dalpha[e,h] = <grad_out[t,h,:], x[s,h,:]>                 (e = s -> t)
//   beta[t,h]   = sum over e into t of alpha dalpha = <grad_out[t,h,:], out[t,h,:]>
//   dz[e,h]     = alpha (dalpha - beta[t,h]) * (z > 0 ? 1 : slope)
//   grad_x[s,h,:] = sum over e out of s of alpha grad_out[t,h,:]
//                   + ds_src[s,h] a_src[h,:] + ds_dst[s,h] a_dst[h,:]
//   ds_src[s,h] = sum over e out of s of dz,   ds_dst[t,h] = sum over e into t of dz
//   grad_a_src[h,c] = sum_v ds_src[v,h] x[v,h,c],  grad_a_dst likewise.
//
// Kernels:
//   node_scores         s_src, s_dst in base-2 units, as in the forward
//   by target           (whole 16-byte slices per head, F <= 128) softmax_fast's
//                       backward on long rows, GatByTarget's walk otherwise: one
//                       online pass gives the softmax statistics and ds_dst
//   by source           (the same layouts) GatBySource's walk: alpha from the
//                       statistics, grad_x and ds_src
//   bwd_targets,        the same two passes for any other layout, one warp per
//   bwd_sources         row: lanes cover the features in tiles of 32, a head's dot
//                       products finished by a butterfly over its lanes per edge
//   bwd_vectors_*       grad_a_src / grad_a_dst: per-block column sums, then
//                       the blocks' sums added in a fixed order (deterministic)
// The same file holds the backward of the dot-product form (below).
#include <math_constants.h>

#include "dot_walk.cuh"
#include "gat_walk.cuh"

namespace tfg {
namespace {

constexpr int kBwThreads = 256;
constexpr int kBwWarps = kBwThreads / 32;
constexpr int kBwMaxTiles = 8;                 // F <= 256
constexpr int kBwRowsPerBlock = 512;           // node rows per block of the vector sums
constexpr int kBwUnroll = 4;                   // in-edges whose rows are in flight together
constexpr int kBwUnrollSrc = 2;                // out-edges whose target rows are in flight

__device__ __forceinline__ float bw_leaky(float v, float slope) { return v > 0.f ? v : slope * v; }

// Sum of v over the lanes holding the same head.  Heads of C <= 32 channels
// are aligned groups of C lanes inside a 32-feature tile; heads of C >= 32
// channels span whole tiles, whose full-warp sums are added over the tiles
// of the head.  Every lane of a head receives the head's sum.
template <int NT>
__device__ __forceinline__ void head_sums(float (&v)[NT], int channels) {
    if (channels <= 32) {
#pragma unroll
        for (int i = 0; i < NT; ++i)
            for (int o = 1; o < channels; o <<= 1) v[i] += lane_xor(v[i], o);
    } else {
#pragma unroll
        for (int i = 0; i < NT; ++i)
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) v[i] += lane_xor(v[i], o);
        const int per = channels / 32;             // tiles per head
        float tot[NT];
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            tot[i] = 0.f;
#pragma unroll
            for (int j = 0; j < NT; ++j)
                if (j / per == i / per) tot[i] += v[j];
        }
#pragma unroll
        for (int i = 0; i < NT; ++i) v[i] = tot[i];
    }
}

struct BwArgs {
    const int32_t *rowptr, *col;          // CSR by target
    const int32_t *rowptr_src, *col_src;  // CSR by source (col_src holds targets)
    const void *x;
    int64_t n;
    int heads, channels;
    float slope;
    const float *a_src, *a_dst;
    const float *out, *grad_out;
    const float *s_src, *s_dst;           // base-2 node scores
    float *m, *den, *beta, *ds_dst, *ds_src;   // [N, H] each
    float *grad_x;
};

// Per target t: the forward's softmax statistics (running maximum in base-2
// units and denominator), beta = <grad_out[t], out[t]> per head, and
// ds_dst[t] = sum of dz over the in-edges.
template <typename XT, int NT>
__global__ void __launch_bounds__(kBwThreads) bwd_targets(BwArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t t = static_cast<int64_t>(blockIdx.x) * kBwWarps + (threadIdx.x >> 5);
    if (t >= a.n) return;
    const int f = a.heads * a.channels;
    const XT *x = static_cast<const XT *>(a.x);
    float g[NT], sd[NT], beta[NT];
    int hd[NT];
    bool ok[NT];
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        const int fi = 32 * i + lane;
        ok[i] = fi < f;
        hd[i] = ok[i] ? fi / a.channels : 0;
        g[i] = ok[i] ? a.grad_out[t * f + fi] : 0.f;
        beta[i] = ok[i] ? g[i] * a.out[t * f + fi] : 0.f;
        sd[i] = __ldg(a.s_dst + t * a.heads + hd[i]);
    }
    head_sums<NT>(beta, a.channels);
    const int32_t beg = a.rowptr[t], end = a.rowptr[t + 1];
    // pass 1: maximum and denominator of each head's logits (base 2)
    float m[NT], den[NT];
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        m[i] = -CUDART_INF_F;
        den[i] = 0.f;
    }
    // (ids of 32 edges loaded together, kBwUnroll edges' scores in flight)
    for (int32_t k0 = beg; k0 < end; k0 += 32) {
        const int cnt = min(32, end - k0);
        const int c = lane < cnt ? __ldg(a.col + k0 + lane) : 0;
        for (int j = 0; j < cnt; j += kBwUnroll) {
            float l[kBwUnroll][NT];
#pragma unroll
            for (int u = 0; u < kBwUnroll; ++u) {
                const int64_t s = lane_get(c, (j + u) & 31);
#pragma unroll
                for (int i = 0; i < NT; ++i)
                    l[u][i] = bw_leaky(__ldg(a.s_src + s * a.heads + hd[i]) + sd[i], a.slope);
            }
#pragma unroll
            for (int u = 0; u < kBwUnroll; ++u) {
                if (j + u >= cnt) break;                 // warp-uniform
#pragma unroll
                for (int i = 0; i < NT; ++i) {
                    if (l[u][i] > m[i]) {
                        den[i] = (m[i] == -CUDART_INF_F ? 0.f : den[i] * exp2f(m[i] - l[u][i]));
                        m[i] = l[u][i];
                    }
                    den[i] += exp2f(l[u][i] - m[i]);
                }
            }
        }
    }
    // pass 2: dz of every in-edge, summed into ds_dst
    // (sums blocked per 32 edges to keep fp32 chains short)
    float dsd[NT];
#pragma unroll
    for (int i = 0; i < NT; ++i) dsd[i] = 0.f;
    for (int32_t k0 = beg; k0 < end; k0 += 32) {
        const int cnt = min(32, end - k0);
        const int c = lane < cnt ? __ldg(a.col + k0 + lane) : 0;
        float part[NT];
#pragma unroll
        for (int i = 0; i < NT; ++i) part[i] = 0.f;
        for (int j = 0; j < cnt; j += kBwUnroll) {
            float d[kBwUnroll][NT], z[kBwUnroll][NT];
#pragma unroll
            for (int u = 0; u < kBwUnroll; ++u) {
                const int64_t s = lane_get(c, (j + u) & 31);
#pragma unroll
                for (int i = 0; i < NT; ++i) {
                    float xv[1] = {0.f};
                    if (ok[i]) VecLoad<XT, 1>::load(x + s * f + 32 * i + lane, xv);
                    d[u][i] = g[i] * xv[0];
                    z[u][i] = __ldg(a.s_src + s * a.heads + hd[i]) + sd[i];
                }
            }
#pragma unroll
            for (int u = 0; u < kBwUnroll; ++u) {
                if (j + u >= cnt) break;                 // warp-uniform
                head_sums<NT>(d[u], a.channels);
#pragma unroll
                for (int i = 0; i < NT; ++i) {
                    const float alpha = exp2f(bw_leaky(z[u][i], a.slope) - m[i]) / den[i];
                    part[i] += alpha * (d[u][i] - beta[i]) * (z[u][i] > 0.f ? 1.f : a.slope);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < NT; ++i) dsd[i] += part[i];
    }
    // one lane per head writes the head's values
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        const int fi = 32 * i + lane;
        if (ok[i] && fi % a.channels == 0) {
            const int64_t o = t * a.heads + hd[i];
            a.m[o] = m[i];
            a.den[o] = den[i];
            a.beta[o] = beta[i];
            a.ds_dst[o] = dsd[i];
        }
    }
}

// Per source s: alpha of every out-edge from the statistics of its target,
// the weighted sum of the targets' gradients, ds_src, and grad_x[s].
template <typename XT, int NT>
__global__ void __launch_bounds__(kBwThreads) bwd_sources(BwArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t s = static_cast<int64_t>(blockIdx.x) * kBwWarps + (threadIdx.x >> 5);
    if (s >= a.n) return;
    const int f = a.heads * a.channels;
    const XT *x = static_cast<const XT *>(a.x);
    float xs[NT], ss[NT], acc[NT], dss[NT];
    int hd[NT];
    bool ok[NT];
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        const int fi = 32 * i + lane;
        ok[i] = fi < f;
        hd[i] = ok[i] ? fi / a.channels : 0;
        float xv[1] = {0.f};
        if (ok[i]) VecLoad<XT, 1>::load(x + s * f + fi, xv);
        xs[i] = xv[0];
        ss[i] = __ldg(a.s_src + s * a.heads + hd[i]);
        acc[i] = 0.f;
        dss[i] = 0.f;
    }
    const int32_t beg = a.rowptr_src[s], end = a.rowptr_src[s + 1];
    for (int32_t k0 = beg; k0 < end; k0 += 32) {          // sums blocked per 32 edges
        const int cnt = min(32, end - k0);
        const int c = lane < cnt ? __ldg(a.col_src + k0 + lane) : 0;
        float pa[NT], pd[NT];
#pragma unroll
        for (int i = 0; i < NT; ++i) pa[i] = pd[i] = 0.f;
        for (int j = 0; j < cnt; j += kBwUnrollSrc) {
            float gt[kBwUnrollSrc][NT], zt[kBwUnrollSrc][NT], mt[kBwUnrollSrc][NT],
                dt[kBwUnrollSrc][NT], bt[kBwUnrollSrc][NT];
#pragma unroll
            for (int u = 0; u < kBwUnrollSrc; ++u) {
                const int64_t t = lane_get(c, (j + u) & 31);
#pragma unroll
                for (int i = 0; i < NT; ++i) {
                    const int64_t th = t * a.heads + hd[i];
                    gt[u][i] = ok[i] ? __ldg(a.grad_out + t * f + 32 * i + lane) : 0.f;
                    zt[u][i] = ss[i] + __ldg(a.s_dst + th);
                    mt[u][i] = __ldg(a.m + th);
                    dt[u][i] = __ldg(a.den + th);
                    bt[u][i] = __ldg(a.beta + th);
                }
            }
#pragma unroll
            for (int u = 0; u < kBwUnrollSrc; ++u) {
                if (j + u >= cnt) break;                 // warp-uniform
                float d[NT];
#pragma unroll
                for (int i = 0; i < NT; ++i) d[i] = gt[u][i] * xs[i];
                head_sums<NT>(d, a.channels);
#pragma unroll
                for (int i = 0; i < NT; ++i) {
                    const float z = zt[u][i];
                    const float alpha = exp2f(bw_leaky(z, a.slope) - mt[u][i]) / dt[u][i];
                    pa[i] = fmaf(alpha, gt[u][i], pa[i]);
                    pd[i] += alpha * (d[i] - bt[u][i]) * (z > 0.f ? 1.f : a.slope);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            acc[i] += pa[i];
            dss[i] += pd[i];
        }
    }
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        const int fi = 32 * i + lane;
        if (!ok[i]) continue;
        const float dsd = __ldg(a.ds_dst + s * a.heads + hd[i]);
        a.grad_x[s * f + fi] = acc[i] + dss[i] * __ldg(a.a_src + fi) + dsd * __ldg(a.a_dst + fi);
        if (fi % a.channels == 0) a.ds_src[s * a.heads + hd[i]] = dss[i];
    }
}

size_t bw_align(size_t b) { return (b + 255) & ~size_t(255); }

int bw_blocks(int64_t n) { return static_cast<int>((n + kBwRowsPerBlock - 1) / kBwRowsPerBlock); }

// ---------------------------------------------------------------------------
// Backward of the dot-product attention (l = scale <q[t], k[s]> per head):
//   dalpha = <grad_out[t,h,:], v[s,h,:]>,  beta[t,h] = <grad_out[t,h,:], out[t,h,:]>
//   dl = alpha (dalpha - beta)
//   grad_q[t] = scale sum over e into t of dl k[s];  grad_k[s] = scale sum over
//   e out of s of dl q[t];  grad_v[s] = sum over e out of s of alpha grad_out[t].
// Logits are recomputed in base-2 units (scale2 = scale log2 e) with the same
// lane layout in both kernels, so both see the same weights.
// ---------------------------------------------------------------------------
struct DotBwArgs {
    const int32_t *rowptr, *col, *rowptr_src, *col_src;
    const void *q, *k, *v;
    int64_t n;
    int heads, channels;
    float scale, scale2;
    const float *out, *grad_out;
    float *m, *den, *beta;                // [N, H] each
    float *grad_q, *grad_k, *grad_v;
};

template <typename XT, int NT>
__device__ __forceinline__ void load_row(const XT *base, int64_t row, int f, int lane,
                                         const bool (&ok)[NT], float (&r)[NT]) {
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        float xv[1] = {0.f};
        if (ok[i]) VecLoad<XT, 1>::load(base + row * f + 32 * i + lane, xv);
        r[i] = xv[0];
    }
}

// Per target t: the softmax statistics, beta and grad_q[t].
template <typename XT, int NT>
__global__ void __launch_bounds__(kBwThreads) dot_bwd_targets(DotBwArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t t = static_cast<int64_t>(blockIdx.x) * kBwWarps + (threadIdx.x >> 5);
    if (t >= a.n) return;
    const int f = a.heads * a.channels;
    const XT *qp = static_cast<const XT *>(a.q), *kp = static_cast<const XT *>(a.k),
             *vp = static_cast<const XT *>(a.v);
    bool ok[NT];
    int hd[NT];
    float qt[NT], g[NT], beta[NT], m[NT], den[NT], dq[NT];
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        const int fi = 32 * i + lane;
        ok[i] = fi < f;
        hd[i] = ok[i] ? fi / a.channels : 0;
        g[i] = ok[i] ? a.grad_out[t * f + fi] : 0.f;
        beta[i] = ok[i] ? g[i] * a.out[t * f + fi] : 0.f;
        m[i] = -CUDART_INF_F;
        den[i] = 0.f;
        dq[i] = 0.f;
    }
    load_row<XT, NT>(qp, t, f, lane, ok, qt);
    head_sums<NT>(beta, a.channels);
    const int32_t beg = a.rowptr[t], end = a.rowptr[t + 1];
    for (int32_t k = beg; k < end; ++k) {                 // pass 1: maximum and denominator
        float kr[NT];
        load_row<XT, NT>(kp, __ldg(a.col + k), f, lane, ok, kr);
        float l[NT];
#pragma unroll
        for (int i = 0; i < NT; ++i) l[i] = qt[i] * kr[i];
        head_sums<NT>(l, a.channels);
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            const float l2 = l[i] * a.scale2;
            if (l2 > m[i]) {
                den[i] = (m[i] == -CUDART_INF_F ? 0.f : den[i] * exp2f(m[i] - l2));
                m[i] = l2;
            }
            den[i] += exp2f(l2 - m[i]);
        }
    }
    for (int32_t k0 = beg; k0 < end; k0 += 32) {          // pass 2: grad_q (blocked sums)
        const int32_t k1 = min(end, k0 + 32);
        float part[NT];
#pragma unroll
        for (int i = 0; i < NT; ++i) part[i] = 0.f;
        for (int32_t k = k0; k < k1; ++k) {
            const int64_t s = __ldg(a.col + k);
            float kr[NT], vr[NT], l[NT], d[NT];
            load_row<XT, NT>(kp, s, f, lane, ok, kr);
            load_row<XT, NT>(vp, s, f, lane, ok, vr);
#pragma unroll
            for (int i = 0; i < NT; ++i) {
                l[i] = qt[i] * kr[i];
                d[i] = g[i] * vr[i];
            }
            head_sums<NT>(l, a.channels);
            head_sums<NT>(d, a.channels);
#pragma unroll
            for (int i = 0; i < NT; ++i) {
                const float alpha = exp2f(l[i] * a.scale2 - m[i]) / den[i];
                part[i] = fmaf(a.scale * alpha * (d[i] - beta[i]), kr[i], part[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < NT; ++i) dq[i] += part[i];
    }
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        const int fi = 32 * i + lane;
        if (!ok[i]) continue;
        a.grad_q[t * f + fi] = dq[i];
        if (fi % a.channels == 0) {
            const int64_t o = t * a.heads + hd[i];
            a.m[o] = m[i];
            a.den[o] = den[i];
            a.beta[o] = beta[i];
        }
    }
}

// Per source s: grad_k[s] and grad_v[s] from the out-edges' weights.
template <typename XT, int NT>
__global__ void __launch_bounds__(kBwThreads) dot_bwd_sources(DotBwArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t s = static_cast<int64_t>(blockIdx.x) * kBwWarps + (threadIdx.x >> 5);
    if (s >= a.n) return;
    const int f = a.heads * a.channels;
    const XT *qp = static_cast<const XT *>(a.q), *kp = static_cast<const XT *>(a.k),
             *vp = static_cast<const XT *>(a.v);
    bool ok[NT];
    int hd[NT];
    float ks[NT], vs[NT], dk[NT], dv[NT];
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        const int fi = 32 * i + lane;
        ok[i] = fi < f;
        hd[i] = ok[i] ? fi / a.channels : 0;
        dk[i] = dv[i] = 0.f;
    }
    load_row<XT, NT>(kp, s, f, lane, ok, ks);
    load_row<XT, NT>(vp, s, f, lane, ok, vs);
    const int32_t beg = a.rowptr_src[s], end = a.rowptr_src[s + 1];
    for (int32_t k0 = beg; k0 < end; k0 += 32) {          // sums blocked per 32 edges
        const int32_t k1 = min(end, k0 + 32);
        float pk[NT], pv[NT];
#pragma unroll
        for (int i = 0; i < NT; ++i) pk[i] = pv[i] = 0.f;
        for (int32_t k = k0; k < k1; ++k) {
            const int64_t t = __ldg(a.col_src + k);
            float qr[NT], gr[NT], l[NT], d[NT];
            load_row<XT, NT>(qp, t, f, lane, ok, qr);
#pragma unroll
            for (int i = 0; i < NT; ++i) {
                gr[i] = ok[i] ? __ldg(a.grad_out + t * f + 32 * i + lane) : 0.f;
                l[i] = qr[i] * ks[i];
                d[i] = gr[i] * vs[i];
            }
            head_sums<NT>(l, a.channels);
            head_sums<NT>(d, a.channels);
#pragma unroll
            for (int i = 0; i < NT; ++i) {
                const int64_t th = t * a.heads + hd[i];
                const float alpha = exp2f(l[i] * a.scale2 - __ldg(a.m + th)) / __ldg(a.den + th);
                pk[i] = fmaf(a.scale * alpha * (d[i] - __ldg(a.beta + th)), qr[i], pk[i]);
                pv[i] = fmaf(alpha, gr[i], pv[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            dk[i] += pk[i];
            dv[i] += pv[i];
        }
    }
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        if (!ok[i]) continue;
        a.grad_k[s * f + 32 * i + lane] = dk[i];
        a.grad_v[s * f + 32 * i + lane] = dv[i];
    }
}

template <typename XT, int NT>
cudaError_t launch_dot_bw(const DotBwArgs &a, cudaStream_t s) {
    const int rows = ceil_div(a.n, kBwWarps);
    dot_bwd_targets<XT, NT><<<rows, kBwThreads, 0, s>>>(a);
    dot_bwd_sources<XT, NT><<<rows, kBwThreads, 0, s>>>(a);
    return cudaGetLastError();
}

template <typename XT>
cudaError_t launch_dot_bw_tiles(const DotBwArgs &a, cudaStream_t s) {
    switch (ceil_div(static_cast<int64_t>(a.heads) * a.channels, 32)) {
        case 1: return launch_dot_bw<XT, 1>(a, s);
        case 2: return launch_dot_bw<XT, 2>(a, s);
        case 3: return launch_dot_bw<XT, 3>(a, s);
        case 4: return launch_dot_bw<XT, 4>(a, s);
        case 5: return launch_dot_bw<XT, 5>(a, s);
        case 6: return launch_dot_bw<XT, 6>(a, s);
        case 7: return launch_dot_bw<XT, 7>(a, s);
        default: return launch_dot_bw<XT, 8>(a, s);
    }
}

// Column sums of ds[v, head(f)] * x[v, f] over a block of rows, for both
// vectors: part[b][0:F] (a_src) and part[b][F:2F] (a_dst).  The block's threads
// are F / VEC columns of VEC features times as many rows as fit; the rows'
// sums are added in row order.  (One thread per feature walking 512 rows left
// the loads in flight to a chain of fmas: 79 us for 169,343 x 128 fp32.)
template <typename XT, int VEC>
__global__ void __launch_bounds__(kBwThreads) bwd_vectors_partial(const XT *__restrict__ x,
                                                                  int64_t n, int heads,
                                                                  int channels,
                                                                  const float *__restrict__ ds_src,
                                                                  const float *__restrict__ ds_dst,
                                                                  float *__restrict__ part) {
    __shared__ float s_sum[2][kBwThreads * VEC];
    const int f = heads * channels, cols = f / VEC, rows = kBwThreads / cols;
    const int c = threadIdx.x % cols, r = threadIdx.x / cols, h = c * VEC / channels;
    const int64_t v0 = static_cast<int64_t>(blockIdx.x) * kBwRowsPerBlock;
    const int64_t v1 = min64(n, v0 + kBwRowsPerBlock);
    float s1[VEC], s2[VEC];
#pragma unroll
    for (int q = 0; q < VEC; ++q) s1[q] = s2[q] = 0.f;
    if (r < rows) {
#pragma unroll 4
        for (int64_t v = v0 + r; v < v1; v += rows) {
            float xv[VEC];
            VecLoad<XT, VEC>::load(x + v * f + c * VEC, xv);
            const float d1 = __ldg(ds_src + v * heads + h), d2 = __ldg(ds_dst + v * heads + h);
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                s1[q] = fmaf(d1, xv[q], s1[q]);
                s2[q] = fmaf(d2, xv[q], s2[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
            s_sum[0][r * f + c * VEC + q] = s1[q];
            s_sum[1][r * f + c * VEC + q] = s2[q];
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * f; i += kBwThreads) {
        const float *p = s_sum[i < f ? 0 : 1] + (i < f ? i : i - f);
        float sum = 0.f;
        for (int k = 0; k < rows; ++k) sum += p[k * f];
        part[static_cast<int64_t>(blockIdx.x) * 2 * f + i] = sum;
    }
}

// The blocks' sums, 32 columns a block: warp w adds blocks w, w + 8, ..., then
// the warps' sums are added in warp order.
__global__ void __launch_bounds__(kBwThreads) bwd_vectors_final(const float *__restrict__ part,
                                                                int blocks, int f,
                                                                float *__restrict__ ga_src,
                                                                float *__restrict__ ga_dst) {
    __shared__ float s_sum[kBwWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, fi = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (fi < 2 * f) {
#pragma unroll 8
        for (int b = warp; b < blocks; b += kBwWarps) s += __ldg(part + static_cast<int64_t>(b) * 2 * f + fi);
    }
    s_sum[warp][lane] = s;
    __syncthreads();
    if (warp > 0 || fi >= 2 * f) return;
    for (int w = 1; w < kBwWarps; ++w) s += s_sum[w][lane];
    if (fi < f) ga_src[fi] = s;
    else ga_dst[fi - f] = s;
}

// nb: blocks of kBwRowsPerBlock rows (bw_blocks)
template <typename XT>
cudaError_t launch_vectors(const XT *x, int64_t n, int heads, int channels, const float *ds_src,
                           const float *ds_dst, int nb, float *part, float *ga_src, float *ga_dst,
                           cudaStream_t s) {
    const int f = heads * channels;
    if (channels % 4 == 0 && reinterpret_cast<uintptr_t>(x) % (4 * sizeof(XT)) == 0)
        bwd_vectors_partial<XT, 4><<<nb, kBwThreads, 0, s>>>(x, n, heads, channels, ds_src, ds_dst, part);
    else
        bwd_vectors_partial<XT, 1><<<nb, kBwThreads, 0, s>>>(x, n, heads, channels, ds_src, ds_dst, part);
    bwd_vectors_final<<<ceil_div(2 * f, 32), kBwThreads, 0, s>>>(part, nb, f, ga_src, ga_dst);
    return cudaGetLastError();
}

template <typename XT, int VEC>
cudaError_t walk_targets(const GatArgs &a, cudaStream_t s) {
    const int slices = a.heads * a.channels / VEC;
    if (slices <= 8) return launch_walk<GatByTarget<XT, VEC, 8, 1, 1, true>>(a, s);
    if (slices <= 16) return launch_walk<GatByTarget<XT, VEC, 16, 1, 1, true>>(a, s);
    return launch_walk<GatByTarget<XT, VEC, 32, 1, 1, true, 2>>(a, s);
}
// 32-byte gradient slices pay on long rows only: they take fewer, register-rich warps.
// Forward + backward with 32- / 16-byte slices, us: 10M edges of mean degree 100, 8 x 16
// bf16 1241 / 1287, fp32 1418 / 1470, 4 x 32 bf16 1163 / 1223; 4M edges of mean degree 40
// 730 / 725, 784 / 788, 693 / 694.
#ifndef TFG_GW_WIDE_DEGREE
#define TFG_GW_WIDE_DEGREE 64
#endif
// lanes of a head: a power of two up to the lanes of a row
template <typename XT, int VEC, int LPR, int LH = 1>
cudaError_t walk_sources_lanes(const GatArgs &a, cudaStream_t s) {
    if constexpr (LH < LPR) {
        if (a.channels / VEC > LH) return walk_sources_lanes<XT, VEC, LPR, 2 * LH>(a, s);
    }
    return launch_walk<GatBySource<XT, VEC, LPR, LH>>(a, s);
}
template <typename XT>
cudaError_t walk_sources(const GatArgs &a, int64_t e, cudaStream_t s) {
    const int slices = a.heads * a.channels / 4;
    if (e >= TFG_GW_WIDE_DEGREE * a.n && slices > 8 && a.channels % 8 == 0 && reinterpret_cast<uintptr_t>(a.grad_out) % 32 == 0) {
        if (slices <= 16) return walk_sources_lanes<XT, 8, 8>(a, s);
        return walk_sources_lanes<XT, 8, 16>(a, s);
    }
    if (slices <= 8) return walk_sources_lanes<XT, 4, 8>(a, s);
    if (slices <= 16) return walk_sources_lanes<XT, 4, 16>(a, s);
    return walk_sources_lanes<XT, 4, 32>(a, s);
}

template <typename XT, int NT>
cudaError_t launch_bw(const BwArgs &a, float *part, float *ga_src, float *ga_dst,
                      cudaStream_t s) {
    const int rows = ceil_div(a.n, kBwWarps);
    bwd_targets<XT, NT><<<rows, kBwThreads, 0, s>>>(a);
    bwd_sources<XT, NT><<<rows, kBwThreads, 0, s>>>(a);
    return launch_vectors(static_cast<const XT *>(a.x), a.n, a.heads, a.channels, a.ds_src, a.ds_dst,
                          bw_blocks(a.n), part, ga_src, ga_dst, s);
}

template <typename XT>
cudaError_t launch_bw_tiles(const BwArgs &a, float *part, float *ga_src, float *ga_dst,
                            cudaStream_t s) {
    const int nt = ceil_div(static_cast<int64_t>(a.heads) * a.channels, 32);
    switch (nt) {
        case 1: return launch_bw<XT, 1>(a, part, ga_src, ga_dst, s);
        case 2: return launch_bw<XT, 2>(a, part, ga_src, ga_dst, s);
        case 3: return launch_bw<XT, 3>(a, part, ga_src, ga_dst, s);
        case 4: return launch_bw<XT, 4>(a, part, ga_src, ga_dst, s);
        case 5: return launch_bw<XT, 5>(a, part, ga_src, ga_dst, s);
        case 6: return launch_bw<XT, 6>(a, part, ga_src, ga_dst, s);
        case 7: return launch_bw<XT, 7>(a, part, ga_src, ga_dst, s);
        default: return launch_bw<XT, 8>(a, part, ga_src, ga_dst, s);
    }
}

}  // namespace

bool attention_backward_layout_ok(int heads, int channels) {
    const int64_t f = static_cast<int64_t>(heads) * channels;
    const bool heads_fit = channels <= 32 ? (32 % channels == 0) : (channels % 32 == 0);
    return heads >= 1 && channels >= 1 && f <= 32 * kBwMaxTiles && heads_fit;
}

size_t attention_backward_workspace_bytes(int64_t n, int heads, int channels) {
    const size_t nh = bw_align(sizeof(float) * size_t(n > 0 ? n : 1) * size_t(heads));
    const size_t f = static_cast<size_t>(heads) * channels;
    return 8 * nh + bw_align(sizeof(float) * 2 * f * size_t(bw_blocks(n > 0 ? n : 1)));
}

size_t dot_attention_backward_workspace_bytes(int64_t n, int heads) {
    return 4 * bw_align(sizeof(float) * size_t(n > 0 ? n : 1) * size_t(heads));
}

cudaError_t launch_dot_walk_targets(const DotArgs &a, int x_dtype, cudaStream_t s);
cudaError_t launch_dot_walk_sources(const DotArgs &a, int x_dtype, cudaStream_t s);

cudaError_t launch_dot_softmax_backward(const int32_t *rowptr, const int32_t *col,
                                        const int32_t *rowptr_src, const int32_t *col_src,
                                        const void *q, const void *k, const void *v, int x_dtype,
                                        int64_t n, int64_t e, int heads, int channels, float scale,
                                        const float *out, const float *grad_out, float *grad_q,
                                        float *grad_k, float *grad_v, void *ws, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const size_t nh = bw_align(sizeof(float) * size_t(n) * size_t(heads));
    char *w = static_cast<char *>(ws);
    auto a16 = [](const void *p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; };
    const int vec = x_dtype == TFG_BF16 ? 8 : 4;
    const int lh = channels / vec;
    if (a16(q) && a16(k) && a16(v) && a16(out) && a16(grad_out) && a16(grad_q) && a16(grad_k) &&
        a16(grad_v) && channels % vec == 0 && lh >= 1 && lh <= 32 && (lh & (lh - 1)) == 0) {
        // workspace: the [N, H] float4 statistics (4 * nh bytes)
        DotArgs da{rowptr, col, q, k, v, n, heads, channels, lh, scale, scale * 1.4426950408889634f, nullptr,
                   nullptr, out, grad_out, reinterpret_cast<float4 *>(w), grad_q, grad_k, grad_v};
        const cudaError_t err = launch_dot_walk_targets(da, x_dtype, s);
        if (err != cudaSuccess) return err;
        da.rowptr = rowptr_src;
        da.col = col_src;
        return launch_dot_walk_sources(da, x_dtype, s);
    }
    DotBwArgs a{rowptr, col, rowptr_src, col_src, q, k, v, n, heads, channels, scale,
                scale * 1.4426950408889634f, out, grad_out,
                reinterpret_cast<float *>(w), reinterpret_cast<float *>(w + nh),
                reinterpret_cast<float *>(w + 2 * nh), grad_q, grad_k, grad_v};
    return x_dtype == TFG_BF16 ? launch_dot_bw_tiles<uint16_t>(a, s) : launch_dot_bw_tiles<float>(a, s);
}

// edge_softmax.cu's node-score launcher (the same scores as the forward)
cudaError_t launch_node_scores(const void *x, int x_dtype, int64_t n, int heads, int channels,
                               const float *a_src, const float *a_dst, float *s_src, float *s_dst,
                               cudaStream_t s);

bool launch_softmax_fast_bwd(const GatArgs &a, int x_dtype, int64_t e, cudaStream_t s);

cudaError_t launch_edge_softmax_backward(const int32_t *rowptr, const int32_t *col,
                                         const int32_t *rowptr_src, const int32_t *col_src,
                                         const void *x, int x_dtype, int64_t n, int64_t e,
                                         int heads, int channels, const float *a_src,
                                         const float *a_dst,
                                         float slope, const float *out, const float *grad_out,
                                         float *grad_x, float *grad_a_src, float *grad_a_dst,
                                         void *ws, cudaStream_t s) {
    const size_t f = static_cast<size_t>(heads) * channels;
    if (n <= 0) {   // no nodes: the vector gradients are zero
        cudaError_t err = cudaMemsetAsync(grad_a_src, 0, sizeof(float) * f, s);
        if (err == cudaSuccess) err = cudaMemsetAsync(grad_a_dst, 0, sizeof(float) * f, s);
        return err;
    }
    // workspace: s_src, s_dst, four [N, H] buffers (the fast form's float4
    // statistics, or m, den, beta and ds_dst), two more, the vector partials
    const size_t nh = bw_align(sizeof(float) * size_t(n) * size_t(heads));
    char *w = static_cast<char *>(ws);
    float *buf[8];
    for (int i = 0; i < 8; ++i) buf[i] = reinterpret_cast<float *>(w + i * nh);
    float *part = reinterpret_cast<float *>(w + 8 * nh);
    cudaError_t err = launch_node_scores(x, x_dtype, n, heads, channels, a_src, a_dst, buf[0],
                                         buf[1], s);
    if (err != cudaSuccess) return err;
    auto a16 = [](const void *p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; };
    const bool aligned = a16(x) && a16(out) && a16(grad_out) && a16(grad_x) && a16(a_src) &&
                         a16(a_dst);
    // Whole 16-byte gradient slices in one head each, a power of two of them per
    // head, and one feature tile per row: softmax_fast's backward or the walk by
    // target, then the walk by source.
    const int hl4 = channels / 4;
    if (aligned && channels % 4 == 0 && (hl4 & (hl4 - 1)) == 0 && f <= 128) {
        GatArgs ga{rowptr, col, x, n, heads, channels, slope, buf[0], buf[1], nullptr, nullptr, out,
                   grad_out, reinterpret_cast<float4 *>(buf[2]), buf[6], buf[7], grad_x, a_src, a_dst};
        const bool bf16 = x_dtype == TFG_BF16;
        if (launch_softmax_fast_bwd(ga, x_dtype, e, s)) err = cudaGetLastError();
        else if (bf16) err = channels % 8 == 0 ? walk_targets<uint16_t, 8>(ga, s) : walk_targets<uint16_t, 4>(ga, s);
        else err = walk_targets<float, 4>(ga, s);
        if (err != cudaSuccess) return err;
        ga.rowptr = rowptr_src;
        ga.col = col_src;
        err = bf16 ? walk_sources<uint16_t>(ga, e, s) : walk_sources<float>(ga, e, s);
        if (err != cudaSuccess) return err;
        if (bf16)
            return launch_vectors(static_cast<const uint16_t *>(x), n, heads, channels, buf[7], buf[6],
                                  bw_blocks(n), part, grad_a_src, grad_a_dst, s);
        return launch_vectors(static_cast<const float *>(x), n, heads, channels, buf[7], buf[6],
                              bw_blocks(n), part, grad_a_src, grad_a_dst, s);
    }
    BwArgs a{rowptr, col, rowptr_src, col_src, x, n, heads, channels, slope, a_src, a_dst,
             out, grad_out, buf[0], buf[1], buf[2], buf[3], buf[4], buf[5], buf[6], grad_x};
    return x_dtype == TFG_BF16 ? launch_bw_tiles<uint16_t>(a, part, grad_a_src, grad_a_dst, s)
                               : launch_bw_tiles<float>(a, part, grad_a_src, grad_a_dst, s);
}

}  // namespace tfg
