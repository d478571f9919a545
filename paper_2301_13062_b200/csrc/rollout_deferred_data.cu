// The deferred-restart rollout kernel (rollout_deferred.cuh) for calls that bring their random values as
// data: supplied actions, supplied start states, or both.
#include "rollout_deferred.cuh"

namespace cp {

namespace {

template <int POLICY, bool START_IN, bool LIMIT, bool RD>
cudaError_t launch_data(RolloutParams &p, int k, bool contracted, cudaStream_t s) {
    unsigned block;
    const unsigned grid = deferred_grid(p, false, block, s);
    if (grid == 0) return cudaErrorInvalidConfiguration;
    if (contracted)
        rollout_deferred_kernel<POLICY, 6, false, LIMIT, RD, true, START_IN><<<grid, block, 0, s>>>(p);
    else if (k <= 2)
        rollout_deferred_kernel<POLICY, 2, false, LIMIT, RD, false, START_IN><<<grid, block, 0, s>>>(p);
    else if (k <= 4)
        rollout_deferred_kernel<POLICY, 4, false, LIMIT, RD, false, START_IN><<<grid, block, 0, s>>>(p);
    else
        rollout_deferred_kernel<POLICY, 6, false, LIMIT, RD, false, START_IN><<<grid, block, 0, s>>>(p);
    count_launch();
    return cudaGetLastError();
}

template <int POLICY, bool START_IN>
cudaError_t launch_data_limit(RolloutParams &p, int k, bool contracted, cudaStream_t s) {
    const bool rd = p.reward_stream != nullptr;
    if (p.max_steps)
        return rd ? launch_data<POLICY, START_IN, true, true>(p, k, contracted, s)
                  : launch_data<POLICY, START_IN, true, false>(p, k, contracted, s);
    return rd ? launch_data<POLICY, START_IN, false, true>(p, k, contracted, s)
              : launch_data<POLICY, START_IN, false, false>(p, k, contracted, s);
}

}  // namespace

// policy: 3 supplied actions, 0 hashed ones, 1 / 6 a linear policy (its weights paired)
cudaError_t launch_rollout_deferred_data(RolloutParams &p, int policy, int k, bool contracted, cudaStream_t s) {
    if (!p.start_in) return launch_data_limit<3, false>(p, k, contracted, s);
    switch (policy) {
        case 0: return launch_data_limit<0, true>(p, k, contracted, s);
        case 1: return launch_data_limit<1, true>(p, k, contracted, s);
        case 3: return launch_data_limit<3, true>(p, k, contracted, s);
        default: return launch_data_limit<6, true>(p, k, contracted, s);
    }
}

}  // namespace cp
