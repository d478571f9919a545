// The producer-assisted kernel (rollout_assisted.cuh) for the linear policies.
#include "rollout_assisted.cuh"

namespace cp {

void launch_assisted_linear(const RolloutParams &p, int policy, bool two, bool contracted, cudaStream_t s) {
    if (policy == 1) launch_assisted_pairs<1, false>(p, two, contracted, s);
    else launch_assisted_pairs<6, false>(p, two, contracted, s);
}

}  // namespace cp
