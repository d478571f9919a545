// The lane-split network rollout (rollout_lanes.cuh): the 4-16-2 network, and the entry that picks
// the instance for a call. The other networks are in files of their own (build time).
#include "rollout_lanes.cuh"

namespace cp {

cudaError_t launch_lanes_mlp32(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s);
cudaError_t launch_lanes_mlp64(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s);
cudaError_t launch_lanes_deep(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s);

// Four lanes per environment: one warp per scheduler up to 4,736 environments on 148 SMs, two up to 9,472, three
// up to 14,208 (the time only changes from one to the next: 9,473 and 14,001 take the same); beyond that the general
// kernel's one lane per environment keeps the schedulers busy with fewer instructions. us per launch of 500 steps,
// general kernel / this one, canonical:
//     environments        1,000          4,096          8,192         14,001         16,001
//     4-16-2            127 / 81       128 / 79       127 / 95       127 / 121      128 / 155
//     4-32-2            165 / 87       166 / 90       165 / 115      166 / 148      166 / 193
//     4-64-2            271 / 100      278 / 133      278 / 177      281 / 236      282 / 345
//     4-16-16-2         241 / 119      244 / 131      245 / 174      245 / 228      245 / 343
//     with all four per-step outputs:
//     4-16-2            213 / 143      214 / 143      214 / 171      215 / 203      214 / 253
//     4-32-2            261 / 149      262 / 149      263 / 181      263 / 235      263 / 298
//     4-64-2            365 / 167      372 / 170      373 / 216      376 / 284      376 / 427
//     4-16-16-2         323 / 190      327 / 190      327 / 247      328 / 324      327 / 490
// Two warps from 32 steps on (this kernel's time over the general one's, 8,192 environments, at 16 and 100 steps: 4-16-2
// 0.99 and 0.79, contracted 1.03 and 0.85, 4-16-16-2 0.95 and 0.75, with reward and done bits 1.07 and 0.89). Not
// for the two smaller networks with reward plane and done bits alone, for which the general kernel has an instance
// without tests: 6,001 environments at 32, 128, 500 steps: 4-16-2 1.15, 1.06, 1.04, 4-32-2 1.04, 0.96, 0.94.
// Three warps (14,001 environments at 32, 64, 128, 500 steps): 4-64-2 in every form from 32 steps on (0.73 to 0.92); 4-32-2
// from 64 (1.06, 0.98, 0.93, 0.89), contracted from 32 (0.97, 0.89, 0.84, 0.80); 4-16-2 from 128 (1.10, 1.03, 0.99, 0.95;
// contracted 1.11, 1.05, 1.00, 0.95; all outputs 1.04, 0.99, 0.97, 0.94), contracted with outputs from 32 (0.97, 0.92, 0.89,
// 0.84); 4-16-16-2 from 128 without outputs (1.08, 1.01, 0.97, 0.93) and contracted with them from 32 (0.99, 0.94,
// 0.91, 0.88), but not the other way round (contracted 1.18, 1.11, 1.07, 1.03; all outputs 1.10, 1.04, 1.02, 0.99), and
// these three not with reward plane and done bits alone (1.08 to 1.34).
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
    int most = p.T >= 32u && !small_plain ? 2 : 1;  // warps per scheduler
    const uint32_t three_from = policy == 5 || (contracted && (streams || policy == 4)) ? 32u : policy == 4 ? 64u : 128u;
    if (p.T >= three_from && (policy == 5 || !plain) && (policy != 7 || streams == contracted)) most = 3;
    if (warps4 > schedulers * most) return 0;
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
