// The lane-split network rollout (rollout_lanes.cuh) for the 4-16-16-2 network, both arithmetics.
#include "rollout_lanes.cuh"

namespace cp {

cudaError_t launch_lanes_deep(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s) {
    return contracted ? launch_lanes_net<7, true>(p, g, streams, s) : launch_lanes_net<7, false>(p, g, streams, s);
}

}  // namespace cp
