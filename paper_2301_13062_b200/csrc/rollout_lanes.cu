// The lane-split network rollout (rollout_lanes.cuh): the 4-16-2 network, and the entry that picks
// the instance for a call. The other networks are in files of their own (build time).
#include "rollout_lanes.cuh"
#include <algorithm>

namespace cp {

cudaError_t launch_lanes_mlp32(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s);
cudaError_t launch_lanes_mlp64(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s);
cudaError_t launch_lanes_deep(RolloutParams &p, int g, bool streams, bool contracted, cudaStream_t s);

// How many lanes an environment gets, and from how many steps on. A warp of this kernel takes its step's latency
// whatever it holds, until its scheduler has a second one: so as many lanes as leave every scheduler its one warp,
// and more warps where that is still quicker than the general kernel. Four lanes for up to 4,736 environments on 148 SMs
// (more measured the same or slower, but for the smallest batches without outputs: 1,000 environments x 300, time of four
// lanes over eight, 4-32-2 1.04, 4-64-2 1.20, 4-16-16-2 1.10, contracted 4-16-16-2 0.69, 4-16-2 0.95; below twelve steps, 33 to
// 2,368 environments at 3, 4, 5, 8 steps, 4-64-2 0.94-0.98, 0.94-0.99, 0.95-0.99, 0.97-1.00, 4-16-16-2 0.93-0.99, 0.95-1.00,
// 0.95-1.00, 0.97-1.01), two and one beyond them.
// us per launch, general kernel / this one, canonical, 300 steps without outputs, then with reward and done bits, then
// with all four:
//     environments         4,096                  9,001                  18,900                 37,800
//     4-16-2        78 / 41  82 / 49 129 / 50   78 / 49  99 / 62 129 / 64   88 / 62  99 / 76 140 / 80   103 / 96 115 / 109 155 / 115
//     4-32-2        97 / 51 117 / 60 145 / 60   97 / 64 117 / 80 145 / 82  108 / 88 119 / 108 166 / 109  (see below)
//     4-64-2       163 / 62 165 / 72 219 / 72  164 / 88 165 / 111 220 / 111     (see below)
//     4-16-16-2    144 / 68 165 / 84 194 / 85  144 / 101 165 / 120 195 / 119    (see below)
// Time of the general kernel over this one's around the lines, at the step counts given ("plain": reward and done bits alone,
// for which the general kernel has an instance without tests; "tested": action bits or trajectory too):
//   one warp per scheduler: 4 lanes without outputs x 3 1.03-1.05, contracted x 4 1.05, plain x 6 1.04-1.19, 4-64-2 plain x 3
//     0.99-1.33, x 4 1.07-1.41 (the others x 4 0.89-1.06); 2 lanes 4-16-2 x 6 1.05-1.08, plain x 8 1.05-1.08, 4-32-2 x 6 0.90-1.06,
//     x 8 0.97-1.12, plain x 8 0.93-1.04, x 12 1.04-1.13; 1 lane x 24 1.03-1.15, tested x 6 1.04
//   two: 4-16-2 x 64 1.01-1.04, plain canonical x 96 1.01 (contracted never more than 1.01), tested x 12 1.03; 4-32-2 x 24
//     0.95-1.03, contracted 1.01-1.09, plain x 48 1.00-1.04; 4-64-2 x 16 1.06-1.34; 4-16-16-2 x 24 1.06-1.29
//   three: 4-16-2 tested x 48 1.05-1.09 (otherwise at most 1.00); 4-32-2 x 64 1.05-1.10 (plain at most 1.00);
//     4-64-2 x 32 1.04-1.15; 4-16-16-2 x 64 1.00-1.09 (plain canonical at most 0.96)
//   the larger networks by one lane, one / two / three warps: 4-32-2 tested x 8 1.13-1.15, 1.09-1.12, 1.01 (x 32 1.31,
//     1.20, 1.08; four warps 1.01-1.03; without outputs 0.94-1.08, plain 0.91-1.07); 4-64-2 tested x 8 1.12-1.15,
//     1.07-1.10, 1.06, x 128 1.33, 1.19, 1.09, and 1.05-1.12 at 75,000 to 300,000 (sixteen warps x 8 to 100 1.01-1.10;
//     seventeen to 53, 303,200 to 1,000,003 environments, 1.02-1.16 too, which still go to the general
//     kernel); without outputs and plain x 32 1.00-1.10, 1.01-1.06, 1.00-1.04 (75,000 0.96-1.01); 4-16-16-2 tested x 8
//     1.06, 1.03, 1.03, x 128 1.25, 1.11, 1.04 (four 1.00; without 0.74-1.03)
// Launches shorter than that do not earn back the loads of a lane's weights. Supplied start states without outputs keep
// four lanes (14,001 x 200, 4-32-2, four over two 0.93). With outputs one lane and two fetch every step's row, of which
// the general kernel fetches the finished environments' part: all at about the same steps where the call begins the
// episodes, some in every step where it takes up a batch in the middle of them, which costs it more. From the beginning /
// from the middle: 2 lanes x 8 0.86-1.04 / 1.08-1.30, x 16 1.05-1.25 / 1.28-1.53; 1 lane 4-16-2 tested, one warp x 16
// 0.80-1.06 / 1.00-1.30, x 24 0.95-1.17 / 1.11-1.30, two (23,001 to 37,800 environments) x 32 0.84-1.04 / 0.95-1.17, x 64
// 0.96-1.23 / 1.06-1.24, three x 40 0.94 / 1.00, x 64 0.99-1.57 / 1.38; plain, one x 24 0.85-1.10 / 1.08, x 64 1.00-1.23
// / 1.11-1.43, two x 64 0.90-1.10 / 1.16, x 128 0.95-1.29 / 1.16-1.28; on the first batches with two warps (18,945)
// tested x 64 0.90-0.94, x 128 0.91-1.01 / 1.11, plain x 128 0.91 / 0.94-0.99, x 192 0.94 / 0.99, x 300 1.55 / 1.75;
// 4-64-2 tested, one to three x 8 0.92-0.98 / 0.97-1.06, x 24 0.99-1.05 / 1.02-1.12, four (75,001) x 32 0.94, x 64 1.08,
// five to sixteen x 8 0.95-1.13 / 0.95-1.16; plain, one x 32 0.98 / 1.05, x 64 1.01-1.05 / 1.04-1.09, two and three x 32
// 0.94-1.00 / 0.98-1.02, x 128 0.98-1.11 / 0.97-1.17; 4-32-2 and 4-16-16-2 tested, one x 8 0.84-1.01 / 1.03-1.15, x 24
// 1.02-1.10 / 1.15-1.28, two and three x 8 0.85-0.98 / 0.97-1.12, 4-32-2 x 32 0.94-1.10 / 1.02-1.21, 4-16-16-2 x 40
// 0.97-1.06 / 1.02-1.11, x 64 1.00-1.19 / 1.04-1.11.
int rollout_lanes_for(const RolloutParams &p, int policy, bool streams, bool contracted) {
    if (p.action_bits_in || !is_network(policy)) return 0;
    // a forced shape keeps the other kernels
    if (g_tuning.rollout_coop || g_tuning.rollout_ept || g_tuning.rollout_block || g_tuning.rollout_ctas_per_sm) return 0;
    const int64_t schedulers = (int64_t)sm_count() * 4;
    auto warps = [&](int lanes) {  // on the fullest scheduler
        return (int)std::min<int64_t>(64, ((p.n * lanes + 31) / 32 + schedulers - 1) / schedulers);
    };
    const bool tested = p.action_bits || p.trajectory, plain = streams && !tested;
    const bool middle = p.init_planes;  // the batch comes from the middle of its episodes
    int g = 4;
    if (p.start_in && !streams) g = 4;
    else if (policy == 5) g = warps(4) <= 3 ? 4 : 1;
    else if (policy == 7) g = warps(4) <= 2 || !tested ? 4 : 1;
    else if (warps(4) > 1) g = warps(2) == 1 || (policy == 4 && !tested) ? 2 : 1;
    const int w = warps(g);
    uint32_t from = 0u;  // steps; 0: the general kernel
    if (g == 4) {
        if (w == 1) from = plain ? (policy == 5 ? 3u : 6u) : contracted ? 4u : 3u;
        else if (w == 2) from = policy == 5 ? 16u : policy == 7 ? 24u : 32u;
        else if (w == 3) from = policy == 2 ? 128u : policy == 4 ? (contracted ? 32u : 64u) : policy == 5 ? 32u : plain && !contracted ? 0u : 64u;
    } else if (g == 2) {
        if (w == 1) from = (plain ? 8u : 6u) + (policy == 4 && !middle ? 2u : 0u);
        else if (w == 2) from = plain ? 48u : contracted ? 24u : 32u;
        else if (w == 3) from = plain ? 0u : 64u;
    } else if (policy == 2) {
        if (w == 1) from = tested ? 6u : 24u;
        else if (w == 2) from = tested ? 12u : !plain ? 64u : contracted ? 0u : 96u;
        else if (w == 3) from = tested ? 48u : 0u;
    } else if (policy == 5) {
        if (tested && w <= 16) from = 8u;
        else if (w <= 3) from = 32u;
    } else {  // tested
        if (w <= 3) from = w <= 2 ? 8u : 32u;
    }
    if (from && p.start_in && streams && g <= 2) {
        uint32_t least = 0u;
        if (g == 2) least = middle ? 0u : 16u;
        else if (policy == 2 && w == 2 && p.n * 20 < schedulers * 32 * 23) least = middle ? 128u : 256u;
        else if (policy == 2 && tested) least = middle ? (w == 1 ? 16u : 32u) : w == 1 ? 24u : 64u;
        else if (middle) least = 0u;
        else if (policy == 2) least = w == 1 ? 48u : 128u;
        else if (policy == 5) least = tested ? (w <= 3 ? 24u : w == 4 ? 64u : 8u) : w == 1 ? 64u : 128u;
        else least = w == 1 ? 24u : policy == 4 ? 32u : 48u;
        from = std::max(from, least);
    }
    if (from == 0u || p.T < from) return 0;
    return !streams && policy != 2 && !(policy == 7 && contracted) && warps(8) == 1 && (policy == 4 || p.T >= 12u) ? 8 : g;
}

cudaError_t launch_rollout_lanes(RolloutParams &p, int policy, int g, bool streams, bool contracted, cudaStream_t s) {
    if (g == 1 && policy != 2) screen_units(p, policy);
    else screen_bound(p, policy, g);
    switch (policy) {
        case 2: return contracted ? launch_lanes_net<2, true>(p, g, streams, s) : launch_lanes_net<2, false>(p, g, streams, s);
        case 4: return launch_lanes_mlp32(p, g, streams, contracted, s);
        case 5: return launch_lanes_mlp64(p, g, streams, contracted, s);
        default: return launch_lanes_deep(p, g, streams, contracted, s);
    }
}

}  // namespace cp
