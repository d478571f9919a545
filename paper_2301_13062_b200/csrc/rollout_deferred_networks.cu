// The deferred-restart rollout kernel (rollout_deferred.cuh) for the 4-16-16-2 network.
#include "rollout_deferred.cuh"

namespace cp {

// p.w holds every weight twice (launch_rollout_deferred has paired them).
cudaError_t launch_rollout_deferred_deep(RolloutParams &p, bool contracted, cudaStream_t s) {
    return launch_limit<7, false>(p, 3, contracted, s);
}

}  // namespace cp
