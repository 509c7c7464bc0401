// Backward of the dot-product attention by source (dot_walk.cuh): grad_k and
// grad_v from the targets' statistics.
#include "dot_walk.cuh"

namespace tfg {

cudaError_t launch_dot_walk_sources(const DotArgs &a, int x_dtype, cudaStream_t s) {
    if (x_dtype == TFG_BF16) {
        if (reinterpret_cast<uintptr_t>(a.grad_out) % 32 != 0) return launch_dot_pass<DotBySourceNarrow, uint16_t, 8>(a, s);
        return launch_dot_pass<DotBySource, uint16_t, 8>(a, s);
    }
    return launch_dot_pass<DotBySource, float, 4>(a, s);
}

}  // namespace tfg
