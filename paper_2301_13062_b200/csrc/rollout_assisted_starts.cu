// The producer-assisted kernel (rollout_assisted.cuh) for supplied start states.
#include "rollout_assisted.cuh"

namespace cp {

void launch_assisted_starts(const RolloutParams &p, int policy, bool contracted, cudaStream_t s) {
    if (policy == 0) launch_assisted_chunk<0, true>(p, contracted, s);
    else if (policy == 1) launch_assisted_chunk<1, true>(p, contracted, s);
    else launch_assisted_chunk<6, true>(p, contracted, s);
}

}  // namespace cp
