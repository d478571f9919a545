// The producer-assisted kernel (rollout_assisted.cuh) for hashed and supplied actions, and the entry
// that picks the instance for a call. The linear policies and the supplied start states are
// instantiated in files of their own (build time).
#include "rollout_assisted.cuh"

namespace cp {

void launch_assisted_linear(const RolloutParams &p, int policy, bool contracted, cudaStream_t s);
void launch_assisted_starts(const RolloutParams &p, int policy, bool contracted, cudaStream_t s);

bool rollout_assisted_applies(const RolloutParams &p, int policy, bool streams) {
    (void)streams;
    // supplied actions replace whatever policy was named
    if (policy != 0 && policy != 1 && policy != 6 && !p.action_bits_in) return false;
    if (g_tuning.rollout_coop == 4) return true;
    if (g_tuning.rollout_coop != 0 || g_tuning.rollout_ept != 0) return false;
    // supplied start states: every row is fetched, so short launches, which have no time to hide that
    // behind, keep the general kernel (a linear policy, 20,011 envs x 16: 9.2 us against 11.1, x 64 with
    // the reward plane and done bits 19 against 21, x 400 107 against 100)
    if (p.start_in && p.T < 96u) return false;
    // a linear policy, short launches with more than a warp's pair per SM: the first chunk of start states is
    // hashed before anything is stepped (general kernel / this, us: 45,000 envs x 2, 4, 8 steps 2.7 / 3.1,
    // 3.2 / 3.7, 4.6 / 4.8, 9,000 x 3 2.9 / 3.1); with the action bits or the trajectory among the outputs,
    // which the general kernel tests for one by one, only the largest lose, up to three steps (45,000 x 2
    // 1.12 of the general kernel's time, x 4 1.00, 37,000 x 2 0.99)
    const bool linear = policy == 1 || policy == 6, tested = p.action_bits || p.trajectory;
    if (linear && p.T <= (tested ? 3u : 8u) && (p.n + 31) / 32 > (int64_t)sm_count() * (tested ? 8 : 1)) return false;
    // up to ten pairs per SM (at 20 KB of shared memory each; an eleventh would wait for a second
    // wave). Measured against the general kernel's best shape, ms per launch:
    // x 5,000 steps 9,472 envs 0.25 / 0.61, 18,944 envs 0.45 / 0.61, 28,416 envs 0.57 / 0.74,
    // 37,888 envs 0.70 / 0.74; x 4,000 steps 47,360 envs (ten pairs per SM) 0.72 / 0.83,
    // 56,832 envs (twelve) 0.88 / 0.82. The linear policies (whose larger batches the deferred kernel
    // has taken before this test) and supplied start states gain as far or further, us per launch of
    // 500 steps: one linear policy per environment 4,099 envs 80.7 / 35.6, 20,011 91 / 66, 32,768 93 /
    // 81, with all per-step outputs 173 / 46, 189 / 116, 189 / 130; supplied actions and start states
    // 4,099 envs 134 / 81, 16,384 282 / 62, 47,000 282 / 132.
    return (p.n + 31) / 32 <= (int64_t)sm_count() * 10;
}

cudaError_t launch_rollout_assisted(RolloutParams &p, int policy, bool contracted, cudaStream_t s) {
    p.n_tasks = (p.n + 31) / 32;
    if (p.action_bits_in) policy = 0;
    if (p.start_in)
        launch_assisted_starts(p, policy, contracted, s);
    else if (policy == 0)
        launch_assisted_chunk<0, false>(p, contracted, s);
    else
        launch_assisted_linear(p, policy, contracted, s);
    count_launch();
    return cudaGetLastError();
}

}  // namespace cp
