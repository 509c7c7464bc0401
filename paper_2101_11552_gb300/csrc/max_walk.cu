// Max aggregation with argmax: the dispatch of max_walk.cuh.
#include "max_walk.cuh"

namespace tfg {
namespace {

template <typename XT, int VEC, bool PACKED, bool ARG = true>
cudaError_t max_vec(const MaxFwdArgs &a, cudaStream_t s) {
    const int64_t slices = a.f / VEC;
    if (slices <= 8) return launch_walk<MaxByTarget<XT, VEC, 8, 1, PACKED, ARG>>(a, s);
    if (slices <= 16) return launch_walk<MaxByTarget<XT, VEC, 16, 1, PACKED, ARG>>(a, s);
    return launch_walk<MaxByTarget<XT, VEC, 32, 1, PACKED, ARG>>(a, s);
}

// Rows without 16-byte slices, and any row when out or argmax is not 16-byte aligned.
// Single features a lane against a row per warp that read 8- or 16-byte slices whatever
// the outputs' alignment, 114.6M edges: bf16 F = 100 4.21 / 5.39 ms, F = 20 1.35 / 5.29; fp32
// F = 128 with misaligned outputs 4.87 / 5.47; 169,343 nodes of mean in-degree 6.9, bf16 F =
// 100 126 / 181 us, F = 44 120 / 127.
template <typename XT>
cudaError_t max_scalar(const MaxFwdArgs &a, cudaStream_t s) {
    if (a.f <= 8) return launch_walk<MaxByTarget<XT, 1, 8, 1, false>>(a, s);
    if (a.f <= 16) return launch_walk<MaxByTarget<XT, 1, 16, 1, false>>(a, s);
    if (a.f <= 32) return launch_walk<MaxByTarget<XT, 1, 16, 2, false>>(a, s);
    if (a.f <= 48) return launch_walk<MaxByTarget<XT, 1, 16, 3, false>>(a, s);
    const int64_t passes = (a.f + 127) / 128, per = (a.f + passes - 1) / passes;
    if (per <= 64) return launch_walk<MaxByTarget<XT, 1, 32, 2, false>>(a, s);
    if (per <= 96) return launch_walk<MaxByTarget<XT, 1, 32, 3, false>>(a, s);
    return launch_walk<MaxByTarget<XT, 1, 32, 4, false>>(a, s);
}

bool aligned16(const void *p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

}  // namespace

cudaError_t launch_max_argmax(const int32_t *rowptr, const int32_t *col, const int32_t *perm,
                              const float *w, const void *x, int x_dtype, int64_t n, int64_t f,
                              float *out, int32_t *argmax, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const MaxFwdArgs a{rowptr, col, perm, w, x, n, f, out, argmax};
    const bool aligned = aligned16(x) && aligned16(out) && aligned16(argmax);
    if (x_dtype == TFG_BF16) {
        if (aligned && f % 8 == 0) return w ? max_vec<uint16_t, 8, false>(a, s) : max_vec<uint16_t, 8, true>(a, s);
        return max_scalar<uint16_t>(a, s);
    }
    if (aligned && f % 4 == 0) return max_vec<float, 4, false>(a, s);
    return max_scalar<float>(a, s);
}

// Max of bf16 rows without weights in 16-byte slices (x and out aligned, f a
// multiple of 8): the packed form without argmax.
cudaError_t launch_max_packed(const int32_t *rowptr, const int32_t *col, const void *x, int64_t n, int64_t f,
                              float *out, cudaStream_t s) {
    const MaxFwdArgs a{rowptr, col, nullptr, nullptr, x, n, f, out, nullptr};
    return max_vec<uint16_t, 8, true, false>(a, s);
}

}  // namespace tfg
