// The deferred-restart rollout kernel (rollout_deferred.cuh) for hashed actions, the linear
// policies and the 4-16-2 network, and the entry that picks the instance for a call.
#include "rollout_deferred.cuh"

namespace cp {

bool rollout_deferred_applies(const RolloutParams &p, int policy, bool streams) {
    // per-step outputs: none, or exactly the reward plane + done bitmask
    const bool outputs_ok = !streams || (p.reward_stream && p.done_bits && !p.action_bits && !p.trajectory);
    if (!outputs_ok) return false;
    if (p.action_bits_in) return true;  // supplied actions replace whatever policy was named
    if (p.start_in) return policy == 0 || policy == 1 || policy == 6;
    return policy == 0 || policy == 1 || policy == 2 || policy == 6;
}

cudaError_t launch_rollout_deferred(RolloutParams &p, int policy, bool contracted, cudaStream_t s) {
    // measured on 1,048,576 x 500 at K = 3 / 4 / 6 / 8: hashed actions (22-step episodes) 0.996 /
    // 0.987 / 0.965 / 0.987 ms, the linear policy (80-step episodes) 0.945 / 0.924 / 0.907 / 0.908 ms
    // The network policies' trips are long, so waiting costs more and a restart pass less. 4-16-2,
    // 4,194,304 x 200 at K = 2 / 3 / 4: 4,842 / 4,915 / 5,170 us for a policy of 20-step episodes, 4,438 / 4,438 /
    // 4,559 for one of 9-step episodes, 4,174 / 4,199 / 4,268 and 4,288 / 4,249 / 4,371 for ones of 200 and 16.
    // Short launches (chunked rollouts of a batch in place) pay the ragged end on every call, so
    // the passes come closer together (us per step of 1,048,576 envs at K = 2 / 4 / 6, hashed
    // actions: T = 16: 3.39 / 3.65 / 4.03, T = 64: 2.41 / 2.38 / 2.45, T = 256: 2.17 / 2.02 / 2.00;
    // below 12 steps the general kernel is as fast or faster and keeps the call).
    // 8 trips between passes, which the shared linear policy once had from 384 steps on, suit a policy
    // whose episodes last 80 steps (1,048,576 x 400, with the reward plane and done bits, K = 6 / 8:
    // 835 / 833 us) and cost most policies drawn at random, which push one way and fall after 9 or 10
    // steps (1,009 / 1,359 us, without outputs 902 / 1,154). 5 and 10 trips fit such episodes
    // better (981, 935) and others worse (31-step mixtures 949 at 6; 1,080, 1,199). Choosing in the
    // kernel, by counting the waiting slots every second trip or after every pass, cost 6 to 14 % of
    // every launch.
    // One wave of two 64-env warps per scheduler leaves issue slots for passes that come closer together (hashed
    // actions without outputs, 50,000 and 75,000 x 500 at K = 4 / 6: 82.1 / 86.2 us; with one warp, 37,888, 57.1 /
    // 55.5, with more, 100,003, 120.4 / 119.0).
    const int64_t warps64 = (p.n + 63) / 64, sms = sm_count();
    const bool two_warps = policy == 0 && !p.start_in && !p.reward_stream && warps64 > sms * 4 && warps64 <= sms * 8;
    const int by_length = p.T < 48u ? 2 : p.T < 192u || two_warps ? 4 : 6;
    const int k = g_tuning.rollout_defer > 0 ? g_tuning.rollout_defer : (policy == 2 ? 2 : by_length);
    // the action hash folds the time's upper half into the lower one: nothing to do below 2^16
    const bool short_times = (uint64_t)p.t0 + p.T <= 65536u;
    // shared weights twice: one packed operand for both slots
    if (policy == 1)
        for (int i = 9; i >= 0; --i) p.w[2 * i] = p.w[2 * i + 1] = p.w[i];
    else if (policy == 2)
        screen_units(p, 2);
    if (p.action_bits_in || p.start_in) return launch_rollout_deferred_data(p, p.action_bits_in ? 3 : policy, k, contracted, s);
    switch (policy) {
        case 0: return short_times ? launch_limit<0, true>(p, k, contracted, s) : launch_limit<0, false>(p, k, contracted, s);
        case 1: return launch_limit<1, false>(p, k, contracted, s);
        case 2: return launch_limit<2, false>(p, k, contracted, s);
        default: return launch_limit<6, false>(p, k, contracted, s);
    }
}

}  // namespace cp
