// The lane-split network rollout (rollout_lanes.cuh): the 4-16-2 network, and the entry that picks
// the instance for a call. The other networks are in files of their own (build time).
#include "rollout_lanes.cuh"

namespace cp {

cudaError_t launch_lanes_mlp32(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s);
cudaError_t launch_lanes_mlp64(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s);
cudaError_t launch_lanes_deep(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s);

// Up to two and a half warps per scheduler at four lanes per environment (11,840 environments on 148
// SMs); beyond that the general kernel's one lane per environment keeps the schedulers busy with fewer
// instructions. us per launch of 500 steps, general kernel / this one:
//     environments        1,000          4,096          8,192         14,000
//     4-16-2           139 / 86       141 / 92       143 / 113      143 / 143
//     4-32-2           172 / 101      174 / 121      174 / 148      176 / 187
//     4-64-2           269 / 120      272 / 147      272 / 181      272 / 246
//     4-16-16-2        248 / 127      250 / 133      250 / 176      250 / 232
//     with all four per-step outputs:
//     4-16-2           225 / 152      228 / 152      229 / 176      229 / 209
//     4-64-2           362 / 168      365 / 168      365 / 221      367 / 280
// One warp per scheduler for launches below 32 steps (8,192 environments x 4 steps: 4-16-16-2 6.2 / 8.2, x 16
// 12.3 / 12.3, x 32 20.5 / 18.4), and for the two smaller networks with reward plane and done bits alone, for
// which the general kernel has an instance without tests (500 steps, 4,096 / 8,192 / 11,000 environments, this over
// that: 4-16-2 0.89 / 1.02 / 1.21, 4-32-2 0.86 / 1.00 / 1.19; 4-16-16-2, two warps, 0.67 / 0.85 / 1.12, 4-64-2
// 0.56 / 0.73 / 0.93).
// Launches of one to seven steps do not earn back the loads of a lane's weights, which differ from lane to
// lane; the two smaller networks with reward plane and done bits alone need eight steps.
// Eight lanes for the smallest batches, as long as every warp has a scheduler to itself (500 steps, 1,000
// environments at four / eight lanes: 4-16-2 92 / 86, 4-32-2 119 / 101, 4-64-2 147 / 120, 4-16-16-2 133 / 127, but
// contracted 152 / 187; with per-step outputs four are better everywhere: 4-64-2 168 / 190).
int rollout_lanes_for(const RolloutParams &p, int policy, bool streams, bool contracted) {
    if (p.action_bits_in || !is_network(policy)) return 0;
    // a forced shape keeps the other kernels
    if (g_tuning.rollout_coop || g_tuning.rollout_ept || g_tuning.rollout_block || g_tuning.rollout_ctas_per_sm) return 0;
    const int64_t schedulers = (int64_t)sm_count() * 4;
    const int64_t warps4 = (p.n + 7) / 8, warps8 = (p.n + 3) / 4;
    // reward plane and done bits alone
    const bool plain = p.reward_stream && p.done_bits && !p.action_bits && !p.trajectory;
    const bool small_plain = plain && (policy == 2 || policy == 4);
    if (2 * warps4 > schedulers * (p.T < 32u || small_plain ? 2 : plain && policy == 7 ? 4 : 5)) return 0;
    uint32_t from = !contracted ? 3u : policy == 7 || (policy == 2 && streams) ? 6u : 4u;
    if (small_plain) from = 8u;
    if (p.T < from) return 0;
    return streams || warps8 > schedulers || (policy == 7 && contracted) ? 4 : 8;
}

cudaError_t launch_rollout_lanes(RolloutParams &p, int policy, int g, bool streams, bool contracted, cudaStream_t s) {
    screen_bound(p, policy);
    switch (policy) {
        case 2: return contracted ? launch_lanes_net<2, true>(p, g, streams, s) : launch_lanes_net<2, false>(p, g, streams, s);
        case 4: return launch_lanes_mlp32(p, g, streams, contracted, s);
        case 5: return launch_lanes_mlp64(p, g, streams, contracted, s);
        default: return launch_lanes_deep(p, g, streams, contracted, s);
    }
}

}  // namespace cp
