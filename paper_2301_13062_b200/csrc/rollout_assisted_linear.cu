// The producer-assisted kernel (rollout_assisted.cuh) for the linear policies.
#include "rollout_assisted.cuh"

namespace cp {

void launch_assisted_linear(const RolloutParams &p, int policy, bool contracted, cudaStream_t s) {
    if (policy == 1) launch_assisted_chunk<1, false>(p, contracted, s);
    else launch_assisted_chunk<6, false>(p, contracted, s);
}

}  // namespace cp
