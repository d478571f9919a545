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
// environments x 4 steps with outputs: 4-64-2 11.2 / 13.3), the 4-32-2 network with per-step outputs
// (8,192 x 128, reward plane and done bits: 95.0 / 97.2), and the 4-16-2 one with those two outputs or in the
// contracted arithmetic (9,000 x 32: 15.0 / 16.4 and 12.8 / 16.5).
// Launches of one to seven steps do not earn back the loads of a lane's weights, which differ from lane to
// lane (1,000 environments x 1, 2, 3, 4 steps: 4-16-2 1.04, 0.96, 0.93, 0.91 of the general kernel's time,
// 4-16-16-2 1.17, 1.03, 0.96, 0.93). The general kernel has an instance for the reward plane and done bits
// without tests, against which the small networks need longer (4-32-2 1.17, 1.10, 1.05, 1.02, at 8 steps
// 0.98), and its contracted tanh is so much cheaper that the 4-16-2 network only gains without outputs at
// one warp per scheduler and eight lanes, or where it has to test for other outputs (1,000 x 128: 0.81, 0.79;
// with reward plane and done bits 1.04, 4,600 without outputs 1.04 at 32 steps).
// More lanes for the smallest batches, as long as every warp has a scheduler to itself (1,024
// environments at 4 / 8 / 16 lanes: 4-16-2 44.0 / 37.9, 4-32-2 56.0 / 54.3 / 47.9, 4-64-2 83.1 / 66.6 /
// 64.5; with per-step outputs four lanes are as good or better everywhere: 4-64-2 103.3 / 120.6).
int rollout_lanes_for(const RolloutParams &p, int policy, bool streams, bool contracted) {
    if (p.action_bits_in || !(policy == 2 || policy == 4 || policy == 5 || policy == 7)) return 0;
    // a forced shape keeps the other kernels
    if (g_tuning.rollout_coop || g_tuning.rollout_ept || g_tuning.rollout_block || g_tuning.rollout_ctas_per_sm) return 0;
    const int64_t schedulers = (int64_t)sm_count() * 4;
    const int64_t warps4 = (p.n + 7) / 8, warps8 = (p.n + 3) / 4, warps16 = (p.n + 1) / 2;
    // reward plane and done bits alone
    const bool plain = p.reward_stream && p.done_bits && !p.action_bits && !p.trajectory;
    const bool one_warp = p.T < 32u || (streams && policy == 4) || (policy == 2 && (plain || contracted));
    if (warps4 > schedulers * (one_warp ? 1 : 2)) return 0;
    uint32_t from = !contracted ? 3u : policy == 7 ? 6u : 4u;
    if (plain && (policy == 2 || policy == 4)) from = 8u;
    if (contracted && policy == 2) {
        if (plain || (!streams && warps8 > schedulers)) return 0;
        if (streams) from = 6u;
    }
    if (p.T < from) return 0;
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
