// Walking kernel, more than 32 instances: one instance per engine and estimate.
#include "walk_kernel.cuh"

namespace maaso {

cudaError_t launch_eval_walk_big(const EvalParams& P, int grid, cudaStream_t stream) {
    const bool opt = (P.flags & MAASO_FLAG_PRED_OPTIMISTIC) != 0;
    if (P.flags & MAASO_FLAG_INSTANCE_QUEUES)
        return opt ? launch_walk<true, 2, true, true, false>(P, grid, false, stream) : launch_walk<false, 2, true, true, false>(P, grid, false, stream);
    if (P.flags & MAASO_FLAG_ENGINE_FROZEN)
        return opt ? launch_walk<true, 1, false, true, false>(P, grid, false, stream) : launch_walk<false, 1, false, true, false>(P, grid, false, stream);
    if (P.walk_rcp_big) return opt ? launch_walk<true, 0, false, true, true>(P, grid, false, stream) : launch_walk<false, 0, false, true, true>(P, grid, false, stream);
    return opt ? launch_walk<true, 0, false, true, false>(P, grid, false, stream) : launch_walk<false, 0, false, true, false>(P, grid, false, stream);
}

}  // namespace maaso
