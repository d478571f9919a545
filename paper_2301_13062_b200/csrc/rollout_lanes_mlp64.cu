// The lane-split network rollout (rollout_lanes.cuh) for the 4-64-2 network, both arithmetics.
#include "rollout_lanes.cuh"

namespace cp {

cudaError_t launch_lanes_mlp64(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s) {
    return contracted ? launch_lanes_net<5, true>(p, g, streams, s) : launch_lanes_net<5, false>(p, g, streams, s);
}

}  // namespace cp
