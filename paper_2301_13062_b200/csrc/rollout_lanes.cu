// The lane-split network rollout (rollout_lanes.cuh): the 4-16-2 network, and the entry that picks
// the instance for a call. The other networks are in files of their own (build time).
#include "rollout_lanes.cuh"

namespace cp {

cudaError_t launch_lanes_mlp32(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s);
cudaError_t launch_lanes_mlp64(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s);
cudaError_t launch_lanes_deep(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s);

// Up to two warps per scheduler at four lanes per environment (9,472 environments on 148 SMs); beyond
// that the general kernel's one lane per environment keeps the schedulers busy with fewer
// instructions. us per launch of 128 steps, general kernel / this one:
//     environments        1,024         4,096         8,192        12,000
//     4-16-2            56.3 / 37.7   58.4 / 43.9   58.4 / 52.2   58.4 / 62.5
//     4-32-2            82.9 / 47.9   89.1 / 56.4   89.1 / 68.6   89.0 / 87.0
//     4-64-2           138.2 / 64.5  146.3 / 84.8  146.4 /115.7  146.5 /207.8
//     4-16-16-2        103.3 / 64.5  107.5 / 72.6  107.4 / 91.1  107.4 /115.7
//     with all four per-step outputs:
//     4-16-2            80.9 / 56.1   82.8 / 56.2   83.0 / 66.4   82.9 / 82.5
//     4-64-2           164.9 /103.4  172.9 /103.4  172.9 /138.1  173.1 /258.0
// One warp per scheduler where the gain is smaller than its fixed costs: launches of a few steps (8,192
// environments x 4 steps with outputs: 4-64-2 11.2 / 13.3) and the 4-32-2 network with per-step outputs
// (8,192 x 128, reward plane and done bits: 95.0 / 97.2).
// More lanes for the smallest batches, as long as every warp has a scheduler to itself (1,024
// environments at 4 / 8 / 16 lanes: 4-16-2 44.0 / 37.9, 4-32-2 56.0 / 54.3 / 47.9, 4-64-2 83.1 / 66.6 /
// 64.5; with per-step outputs four lanes are as good or better everywhere: 4-64-2 103.3 / 120.6).
int rollout_lanes_for(const RolloutParams &p, int policy, bool streams) {
    if (p.action_bits_in || !(policy == 2 || policy == 4 || policy == 5 || policy == 7)) return 0;
    // a forced shape keeps the other kernels
    if (g_tuning.rollout_coop || g_tuning.rollout_ept || g_tuning.rollout_block || g_tuning.rollout_ctas_per_sm) return 0;
    const int64_t schedulers = (int64_t)sm_count() * 4;
    const int64_t warps4 = (p.n + 7) / 8, warps8 = (p.n + 3) / 4, warps16 = (p.n + 1) / 2;
    if (warps4 > schedulers * (p.T < 32u || (streams && policy == 4) ? 1 : 2)) return 0;
    if (streams || warps8 > schedulers) return 4;
    return (policy == 4 || policy == 5) && warps16 <= schedulers ? 16 : 8;
}

cudaError_t launch_rollout_lanes(RolloutParams &p, int policy, int g, bool streams, bool contracted, cudaStream_t s) {
    switch (policy) {
        case 2: return contracted ? launch_lanes_net<2, true>(p, g, streams, s) : launch_lanes_net<2, false>(p, g, streams, s);
        case 4: return launch_lanes_mlp32(p, g, streams, contracted, s);
        case 5: return launch_lanes_mlp64(p, g, streams, contracted, s);
        default: return launch_lanes_deep(p, g, streams, contracted, s);
    }
}

}  // namespace cp
