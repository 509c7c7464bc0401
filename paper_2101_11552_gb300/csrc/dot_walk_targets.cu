// Backward of the dot-product attention by target (dot_walk.cuh): the softmax
// statistics and grad_q.
#include "dot_walk.cuh"

namespace tfg {
namespace {
template <typename XT, int VEC, int LPR, int LH, int CH>
using DotTargets = DotByTarget<XT, VEC, LPR, LH, true, CH>;
}  // namespace

cudaError_t launch_dot_walk_targets(const DotArgs &a, int x_dtype, cudaStream_t s) {
    if (x_dtype == TFG_BF16) return launch_dot_pass<DotTargets, uint16_t, 8>(a, s);
    return launch_dot_pass<DotTargets, float, 4>(a, s);
}

}  // namespace tfg
