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
    // a network policy on a batch that leaves schedulers idle: its hidden units spread over several lanes
    // (rollout_lanes.cu)
    if (const int lanes = rollout_lanes_for(p, policy, streams, contracted))
        return launch_rollout_lanes(p, policy, lanes, streams, contracted, s);
    // The deferred-restart kernel (rollout_deferred.cu) by default: from one 64-env warp per
    // scheduler on (37,825 envs on 148 SMs) for hashed actions and the linear policies, launches of at
    // least a dozen steps, per-step outputs none or reward plane + done bits. Measured at T = 500, this kernel
    // against the general one: hashed actions 65,536 envs 0.098 / 0.142 ms, 131,072 0.163 / 0.251; linear policy
    // 47,360 0.088 / 0.100, 131,072 0.154 / 0.212. Against the helper warps, hashed actions and the shared linear
    // policy gain from 33,089 environments on (three and a half 64-env warps per SM), in launches of 192 steps and more
    // (this kernel's time over theirs, 33,100 envs x 200 / 500: 0.85 / 0.75 and 0.72 / 0.69, with reward and done bits
    // 1.01 / 0.88 and 0.78 / 0.72, contracted 0.77 / 0.69 and 0.62 / 0.60, 1.02 / 0.88 and 0.77 / 0.72; 37,800 x 96 16.4 / 18.4
    // and 24.6 / 20.7 us; 28,000 x 500 with outputs 74 / 64; one linear policy each 70 / 74, but with outputs 92 / 84).
    // The networks' trips are short next to their waits since the estimate decides (policy_screen.cuh). Time of the general
    // kernel over this one's for 4-16-2, each weight loaded once for both environments of a thread, without outputs, contracted,
    // with reward and done bits, contracted, two policies each: x 128, 230,000 envs 1.06-1.08, 1.11-1.12, 1.00-1.02, 1.03-1.04;
    // 303,000 (one wave of four CTAs per SM) 1.10, 1.13, 1.03, 1.05; 310,000 (a second one) 1.00, 1.03, 0.93, 0.95; 480,000
    // 1.03, 1.07, 0.97, 1.00; x 48 to 128, 600,000 1.09-1.12, 1.13-1.15, 1.05-1.08, 1.07-1.09; x 100, 2,000,003 1.10, 1.14, 1.04,
    // 1.07, 4,200,001 1.11, 1.15, 1.06, 1.08; x 32 from states, 200,000 1.00, 1.04, 0.95, 0.97; x 24, 600,000 1.02, 1.07, 0.97,
    // 0.99; below one wave 120,000 x 128 1.03, 1.02, 1.00, 0.99, 90,000 x 128 1.00, 0.98, 0.96, 0.94. The larger networks, which the
    // special-function unit binds in either kernel, were tried in the same form: 4-32-2, 4-64-2 and 4-16-16-2 at 300,000 and
    // 1,000,003 0.98 to 1.05, at 75,000 and 100,000 0.88 to 1.03: they have no instance of it.
    // rollout_coop = 5 forces it wherever it applies, any other forced shape keeps the other kernels.
    // Calls that bring actions or start states as data: beyond the batches of the helper-warp kernel
    // below, and where every sort of data that was tried gains or nearly (time of this kernel over the
    // general kernel's; random actions / actions that end every episode after ten steps / those of a
    // balancing policy in every third environment):
    //   actions alone, T = 96, 128, 192: 48,000 envs 0.91 / 1.04 / 1.05, 0.88 / 1.00 / 1.02, 0.89 / 0.89 /
    //   0.92; 60,000 0.79 / 0.89 / 0.91 at 96, 100,003 0.91 / 1.05 / 1.06, 200,003 0.86 / 0.85 / 0.92;
    //   with reward plane and done bits, T = 96, 160, 192: 100,003 envs 1.04 / 1.16 / 1.19, 1.02 / 1.13 /
    //   1.13, 0.94 / 0.95 / 0.96; 200,003 0.91 / 0.92 / 0.97 at 96; below 66,304 envs nothing gained;
    //   in the contracted arithmetic 70,000 and 100,003 envs 0.81-0.87 at 128 already;
    //   start states of 10- to 20-step episodes, T = 96, 128: 48,000 envs 0.92-1.28, 0.74-1.06; 60,000
    //   0.82-1.07, 0.68-0.82; 100,003 0.78-1.01, 0.76-0.97; 200,003 0.52-0.71 at 96;
    //   with a step limit of 1, 5, 8, 12, 13, 16 at T = 250 (every episode costs whole blocks of trips): 200,003
    //   envs 2.87, 0.99, 1.31, 0.70, 0.96, 0.82, 100,003 envs with outputs 4.47, 1.25, 1.41, 0.82, 1.16, 0.92.
    // Start states whose episodes last one to three steps lose (see kMany), and nothing here can see
    // them. With the reward plane and start states of 2 GB and more the time depends on where
    // the memory lies (500,000 x 250, general kernel 746 us, this one 435 or 984 in different processes;
    // 1,048,576 x 128 687, 456 or 787; up to 1.6 GB always the lower one), so those stay there too.
    const int64_t warps32 = (p.n + 31) / 32, warps64 = (p.n + 63) / 64, sms = sm_count();
    const bool data = p.action_bits_in || p.start_in;
    uint32_t from = 96u;
    if (p.start_in && warps64 < sms * 7) from = 128u;
    if (!p.start_in && streams && warps64 < sms * 20) from = contracted ? 128u : 192u;
    const bool streams_gain = !streams || (p.start_in ? p.n * (int64_t)p.T <= 100000000 : warps64 >= sms * 7);
    int64_t least = sms * 4;  // 64-env warps
    // (4-16-2: whole waves, or several)
    const bool waves = streams ? p.T >= 96u && warps64 >= sms * 64
                               : p.T >= 64u && (warps64 >= sms * 48 || (warps64 >= sms * 17 && warps64 <= sms * 32));
    if (policy == 2) least = waves ? 0 : sms * 448;
    if ((policy == 0 || policy == 1) && p.T >= 192u) least = sms * 7 / 2;
    const bool enough = data ? p.T >= from && warps32 > sms * 10 && streams_gain && !(p.max_steps && p.max_steps < 12u)
                             : warps64 >= least && p.T >= 12u;
    const bool by_default = g_tuning.rollout_coop == 0 && g_tuning.rollout_ept == 0 && enough;
    if ((by_default || g_tuning.rollout_coop == 5) && rollout_deferred_applies(p, policy, streams) && !outputs_over_data(p))
        return launch_rollout_deferred(p, policy, contracted, s);
    // very small batches, unless a network acts: a helper warp per stepping warp (rollout_assisted.cu)
    if (rollout_assisted_applies(p, policy, streams)) return launch_rollout_assisted(p, policy, contracted, s);
    if (contracted) return launch_rollout_contracted(p, policy, streams, s);
    return launch_rollout_arith<false>(p, policy, streams, s);
}

}  // namespace cp
