// Walking kernel, at most 32 instances: one instance per engine and estimate.
#include "walk_kernel.cuh"

namespace maaso {

template <int Warps>
static cudaError_t launch_fixed_speed(const EvalParams& P, int grid, bool overlap, cudaStream_t stream) {
    const bool opt = (P.flags & MAASO_FLAG_PRED_OPTIMISTIC) != 0;
    if (P.flags & MAASO_FLAG_INSTANCE_QUEUES)
        return opt ? launch_walk<true, 2, true, false, false, Warps>(P, grid, overlap, stream) : launch_walk<false, 2, true, false, false, Warps>(P, grid, overlap, stream);
    return opt ? launch_walk<true, 1, false, false, false, Warps>(P, grid, overlap, stream) : launch_walk<false, 1, false, false, false, Warps>(P, grid, overlap, stream);
}
template <bool Apart>
static cudaError_t launch_dynamic(const EvalParams& P, int grid, bool overlap, cudaStream_t stream) {
    const bool opt = (P.flags & MAASO_FLAG_PRED_OPTIMISTIC) != 0;
    if (P.walk_rcp)
        return opt ? launch_walk<true, 0, false, false, true, kWalkWarps, Apart>(P, grid, overlap, stream)
                   : launch_walk<false, 0, false, false, true, kWalkWarps, Apart>(P, grid, overlap, stream);
    return opt ? launch_walk<true, 0, false, false, false, kWalkWarps, Apart>(P, grid, overlap, stream)
               : launch_walk<false, 0, false, false, false, kWalkWarps, Apart>(P, grid, overlap, stream);
}
cudaError_t launch_eval_walk(const EvalParams& P, int grid, bool overlap, cudaStream_t stream) {
    if (P.flags & (MAASO_FLAG_ENGINE_FROZEN | MAASO_FLAG_INSTANCE_QUEUES))
        return P.walk_warps == (uint32_t)kWalkWarpsFew ? launch_fixed_speed<kWalkWarpsFew>(P, grid, overlap, stream) : launch_fixed_speed<kWalkWarps>(P, grid, overlap, stream);
    return P.apart ? launch_dynamic<true>(P, grid, overlap, stream) : launch_dynamic<false>(P, grid, overlap, stream);
}

}  // namespace maaso
