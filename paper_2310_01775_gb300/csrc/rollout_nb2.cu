// Rollout kernels for scenes of 2 block(s), one instantiation per team width.
#include "rollout_kernels.cuh"

namespace stamp {

cudaError_t launch_rollout_nb2(const SimConst& sc, const RolloutArgs& a, int lanes, bool adjoint,
                               cudaStream_t st) {
    return rollout::launch_lanes<2>(sc, a, lanes, adjoint, st);
}

cudaError_t launch_rollout_batch_nb2(const SimConst& sc, const BatchArgs& b, int lanes, int cta,
                                     bool adjoint, cudaStream_t st) {
    return rollout::launch_batch_lanes<2>(sc, b, lanes, cta, adjoint, st);
}

}  // namespace stamp
