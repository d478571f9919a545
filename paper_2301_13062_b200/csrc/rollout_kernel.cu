// The rollout kernels in the canonical arithmetic (every operation rounded once, in the order
// of the per-op ladder), and the entry the C ABI calls.
#include "rollout_kernel.cuh"

namespace cp {

// Do two ranges share memory? (A null pointer's shares none.)
static bool share_memory(const void *a, int64_t a_bytes, const void *b, int64_t b_bytes) {
    const char *x = static_cast<const char *>(a), *y = static_cast<const char *>(b);
    return x && y && x < y + b_bytes && y < x + a_bytes;
}

// A call may write its per-step outputs over the actions or start states it reads (the done bits of a
// recording where its actions were): the kernels that step a warp's environments together have read
// a row by the time they write it. The deferred-restart kernel has not: it clears the done bits before
// the first step, and its environments read rows that the warp's reward rows have passed.
static bool outputs_over_data(const RolloutParams &p) {
    const int64_t T = p.T, word_rows = T * ((p.n + 31) / 32) * 4, env_rows = T * p.n * 4;
    return share_memory(p.done_bits, word_rows, p.action_bits_in, word_rows) ||
           share_memory(p.done_bits, word_rows, p.start_in, 4 * env_rows) ||
           share_memory(p.reward_stream, env_rows, p.action_bits_in, word_rows) ||
           share_memory(p.reward_stream, env_rows, p.start_in, 4 * env_rows);
}

cudaError_t launch_rollout(RolloutParams &p, int policy, bool streams, bool contracted, cudaStream_t s) {
    // Supplied actions replace whatever policy was named: from here on the call is the same with and
    // without one (3, the name the kernels have for it). A network named beside them used to bring its own
    // spacing of the restart passes and its weights, paired, into the launch.
    if (p.action_bits_in) policy = 3;
    // a network policy on a batch that leaves schedulers idle, or with outputs that the deferred kernel
    // does not write: its hidden units spread over several lanes (rollout_lanes.cu)
    if (const int lanes = rollout_lanes_for(p, policy, streams)) return launch_rollout_lanes(p, policy, lanes, streams, contracted, s);
    // The deferred-restart kernel (rollout_deferred.cu) by default: from one 64-env warp per
    // scheduler on (37,888 envs on 148 SMs) for hashed actions and the linear policies, from seven
    // warps per SM on (66,304 envs) for the tanh networks, launches of at least a dozen steps,
    // per-step outputs none or reward plane + done bits. Measured at T = 500, this kernel against
    // the kernels below: hashed actions 37,888 envs 0.093 / 0.096 ms, 65,536 0.098 / 0.142,
    // 131,072 0.163 / 0.251; linear policy 47,360 0.088 / 0.100, 131,072 0.154 / 0.212; network
    // 56,832 0.483 / 0.427, 75,776 0.483 / 0.545. rollout_coop = 5 forces it wherever it
    // applies, any other forced shape keeps the other kernels.
    // Calls that bring actions or start states as data: beyond the batches of the helper-warp kernel
    // below, and from 96 steps on (general kernel / this one, us: supplied actions 60,000 x 140 44 / 35,
    // 200,003 x 250 147 / 120, with supplied start states too 85 / 58 and 290 / 140; but 100,000 x 64
    // 30 / 32 and 31 / 35, 1,048,576 x 16 46 / 61). With the reward plane and done bits, supplied
    // actions alone gain from 66,304 envs on (47,360 x 250 68 / 71, 70,000 x 140 49 / 45).
    const int64_t warps32 = (p.n + 31) / 32, warps64 = (p.n + 63) / 64, sms = sm_count();
    const bool data = p.action_bits_in || p.start_in;
    const bool network = policy == 2 || policy == 4 || policy == 5 || policy == 7;
    const bool enough = data ? warps32 > sms * 10 && (!streams || p.start_in || warps64 >= sms * 7) && p.T >= 96u
                             : warps64 >= sms * (network ? 7 : 4) && p.T >= 12u;
    const bool by_default = g_tuning.rollout_coop == 0 && g_tuning.rollout_ept == 0 && enough;
    if ((by_default || g_tuning.rollout_coop == 5) && rollout_deferred_applies(p, policy, streams) && !outputs_over_data(p))
        return launch_rollout_deferred(p, policy, contracted, s);
    // very small batches, unless a network acts: a helper warp per stepping warp (rollout_assisted.cu)
    if (rollout_assisted_applies(p, policy, streams)) return launch_rollout_assisted(p, policy, contracted, s);
    if (contracted) return launch_rollout_contracted(p, policy, streams, s);
    return launch_rollout_arith<false>(p, policy, streams, s);
}

}  // namespace cp
