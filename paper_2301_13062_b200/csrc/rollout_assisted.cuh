// Rollout for batches far too small to fill the chip (the paper's own shape, 2,048 environments
// x 10,000 steps, Sec. V-A, is 64 warps on 592 warp schedulers): there a step's LATENCY is what
// is paid, and every instruction the stepping warp does not have to issue shortens it.
//
// Everything random in a rollout depends on (seed, env, time) only, never on the trajectory. So
// each stepping warp ("consumer") gets a helper warp ("producer") on another scheduler of the
// same SM, on the smallest batches one on each of the three others, that hashes, a chunk of steps ahead, the action force and the start state of every
// step for the consumer's 32 environments into shared memory. The consumer's step is then two
// shared-memory loads, the dynamics, the termination test and four selects: about 60 instead
// of 110 instructions, with no integer hashing in its dependency chain. Same hashes, same
// dynamics function, same bits as the general kernel.
//
// Synchronisation: one hardware barrier per consumer/producer pair (bar.sync with the pair's own
// id, the threads of its two or four warps), once per chunk, double-buffered. All warps of a pair execute exactly
// 1 + ceil(T / chunk) barriers, a number fixed by the launch parameters alone; there is no flag,
// no spin and no dependence on data, so neither warp can wait for an arrival that does not come.
//
// Scope: hashed or supplied actions (the producer turns the caller's action words into forces) and
// the linear policies (the consumer evaluates them, the producer hashes start states alone); hashed
// or supplied start states (the producer fetches every row, a chunk ahead: a consumer that fetched
// a finished environment's row itself would wait for memory on most steps); either arithmetic,
// with or without an episode step limit and per-step output streams. The network policies have a
// kernel of their own (rollout_lanes.cuh).
#pragma once
#include "cartpole_device.cuh"
#include "cartpole_internal.h"

namespace cp {

namespace {

// Steps per hand-over: 40 KB of shared memory per pair (640 bytes per step, two buffers) while at most five
// pairs share an SM, 20 KB beyond that. (2,048 x 10,000 at 8, 16, 32 steps: 0.543, 0.512, 0.481 ms; 500 steps on
// 17,000 environments, supplied actions, 32 / 16 steps: 41.0 / 45.0 us; on 27,000, where five pairs
// of 32 steps fill an SM and the sixth waits, 71.5 / 63.5.) Nothing is stepped before the first hand-over, so a launch
// of 32 to 63 steps takes the short one, and one of 24 to 127 with at most two pairs per SM, where the helpers have
// schedulers to themselves. 32 over 16 steps per hand-over, all policies, without outputs, with reward and done bits
// and with all outputs, at T = 17, 24, 32, 48, 64, 96, 128, 200, 500: 3,001 to 9,001 environments 0.96-1.00, 1.02-1.08,
// 1.08-1.16, 1.06-1.13, 1.03-1.09, 1.01-1.06, 0.99-1.05, 0.95-1.03, 0.92-1.01; 11,001 to 18,001 0.96-0.99, 0.98-1.03,
// 1.01-1.09, 1.00-1.05, 0.94-1.02, 0.94-1.03, 0.95-1.08, 0.95-1.07, 0.94-1.06. The contracted arithmetic, whose step is
// shorter, waits for its helper sooner: up to 9,001 environments 0.98-1.12 at 50 steps, 0.94-1.03 at 150, so up to 95
// there, and 0.94-1.06 at 50 steps on 14,001 and 23,001, so never beyond two pairs.
constexpr int kLongChunk = 32, kShortChunk = 16;
inline bool long_chunks(const RolloutParams &p, bool contracted) {
    const int64_t sms = sm_count();
    if (p.n_tasks <= sms * 2) return p.T < 24u || p.T >= (contracted ? 96u : 128u);
    return p.n_tasks <= sms * 5 && (contracted || p.T < 32u || p.T >= 64u);
}

// Steps per trip of the consumer's loop over a chunk. Measured on 2,048 x 10,000 (ms per launch):
// 1: 0.666, 2: 0.481, 3: 0.487, 4: 0.503, 8: 0.504, 16: 0.506, whole chunk: 0.506.
constexpr int kStepUnroll = 2;
// The same with the cart one step behind (CartBehind), whose steps overlap. 2,048 x 10,000 with three helpers: 1: 543, 2: 425,
// 4: 389, 8: 388 us; with one, reward and done bits, x 500 (us) 40.9, 29.7, 27.5, 27.8.
constexpr int kBehindUnroll = 4;

template <int CHUNK>
struct PairBuffers {
    float4 start[2][CHUNK][32];  // start state of time t + 1, for the env of each lane
    float force[2][CHUNK][32];   // +-F of the action at time t
};

// One hand-over among a stepping warp and its HELPERS: barrier 1 for pair 0, barrier 2 for pair 1 (immediates: a register
// id makes the kernel claim all sixteen barriers).
template <int PAIRS, int HELPERS>
__device__ __forceinline__ void pair_barrier(uint32_t pair) {
    __syncwarp();
    if (PAIRS == 1 || pair == 0u)
        asm volatile("bar.sync 1, %0;" ::"n"(32 * (1 + HELPERS)) : "memory");
    else
        asm volatile("bar.sync 2, %0;" ::"n"(32 * (1 + HELPERS)) : "memory");
}

// Pairs per CTA: one, but two, whose first two warps step, for supplied start states, whose helpers fetch instead of
// hashing: without per-step outputs always (500 steps with supplied actions, 27,000 environments two / one: 88.1 /
// 92.2 us, 45,000 130.9 / 138.5), and with the reward plane and done bits, in the contracted arithmetic up to 256 steps
// also with all outputs, beyond five pairs per SM where the fullest SM gets no more pairs that way (two_pairs). Time of
// one over two there, actions supplied, hashed and by a policy per environment, 96, 200, 500 steps: reward and done bits,
// 26,001 environments 1.05-1.08, 1.05-1.09, 1.03-1.07, 36,001 1.00-1.03, 1.01-1.05, 1.00-1.04, 45,001 0.99-1.04, 1.04-1.08,
// 1.03-1.07; all outputs, contracted 26,001 1.06-1.08, 1.07-1.09, 0.94-1.01, 45,001 1.06-1.07, 1.03-1.05, 0.92-0.97, canonical
// 0.94-0.98, 1.01-1.02, 0.96-0.97 and 1.02-1.04, 1.00-1.02, 0.93-0.98. Where the fullest SM gets more, 33,100, 0.94-1.03, and
// below five pairs 3,001 to 23,001 0.74-1.07 (mean 0.95). One shared linear policy with reward and done bits: canonical
// 0.94-1.03, one pair; contracted 26,001 and 45,001 x 200 1.05-1.06.
template <int POLICY, bool START_IN, bool CONTRACT, int STREAMS>
constexpr bool kMayPair = START_IN && (STREAMS == 1 ? POLICY != 1 || CONTRACT : STREAMS == 3 && CONTRACT && POLICY != 1);
template <int STREAMS>
bool two_pairs(const RolloutParams &p) {
    const int64_t sms = sm_count(), pairs = p.n_tasks, ctas = (pairs + 1) / 2;
    return pairs > sms * 5 && (ctas + sms - 1) / sms * 2 == (pairs + sms - 1) / sms && (STREAMS != 3 || p.T <= 256u);
}

// Which warp of a CTA of one pair steps (0 or 1; of four, 0 to 3). A warp's place among an SM's warps decides which of the four
// schedulers it has: a CTA of two warps has schedulers 0 and 1 or 2 and 3. The first warp stepping
// everywhere, schedulers 0 and 2 would have every stepping warp, whose step is the longer one, and 1 and 3 the
// helpers; so the roles change places from one group of four warp places to the next. The place is read, not
// assumed: whatever it is, the result is the same.
// us per launch of 500 steps, roles by place against two pairs per CTA with a fixed place each (start states
// hashed in two operations fewer on both sides): hashed actions 12,000 environments 39.9 / 47.1, with
// all outputs 55.3 / 65.6, 27,000 57.5 / 59.4, 77.9 / 82.0; one linear policy each, all outputs, 17,000 57.4 / 75.9,
// 33,000 106.5 / 118.8.
template <int HELPERS>
__device__ __forceinline__ uint32_t stepping_warp(uint32_t &shared) {
    if (threadIdx.x == 0) {
        uint32_t place;
        asm volatile("mov.u32 %0, %%warpid;" : "=r"(place));
        shared = (place >> 2) & (uint32_t)HELPERS;
    }
    __syncthreads();
    return shared;
}

// Instances that take the role, which comes from shared memory, once more from a lane of the warp, as a value that the
// compiler sees to be the same for all lanes. With / without, 150 and 400 or 500 steps, 2,001 to 30,001 environments:
// a policy per environment and the shared linear one, action bits among the outputs 0.90-0.96, all outputs canonical
// 0.90-1.04, contracted 0.88-1.14; reward and done bits, a policy per environment 0.89-1.00, hashed and supplied actions
// canonical 0.93-1.01, contracted 0.93-1.03, the shared linear policy 0.98-1.09; without outputs 0.95-1.05.
template <int POLICY, bool START_IN, bool CONTRACT, int STREAMS>
constexpr bool kUniformRole = !START_IN && (POLICY == 0 ? STREAMS == 1 && !CONTRACT
                                                        : STREAMS == 2 || (STREAMS == 3 && !CONTRACT) || (STREAMS == 1 && POLICY == 6));

// Where the consumer's per-step outputs go (only read when STREAMS; NULL = not wanted): one pointer
// per output, advanced by a row per step.
struct StreamCursor {
    float *rew, *traj;     // this lane's environment in the row
    uint32_t *done, *act;  // the warp's word in the row
    int64_t n, words;
    bool valid;
};

// POLICY: 0 the producer supplies the forces (hashed or the caller's actions), 1 the shared linear
// policy, 6 one linear policy per environment (own).
template <int POLICY, bool KNOWN_SMALL, bool LIMIT, bool CONTRACT, int STREAMS, int CHUNK>
__device__ __forceinline__ void consume_step(const RolloutParams &p, const PairBuffers<CHUNK> &buf, uint32_t b,
                                             int s, uint32_t lane, uint32_t t1, const LinearW &own, StreamCursor &sc,
                                             State &z, uint32_t &cnt, uint32_t &begin) {
    const float4 fresh = buf.start[b][s][lane];
    float force;
    if (POLICY == 0) force = buf.force[b][s][lane];
    else force = force_from_signbit(linear_action(POLICY == 1 ? *reinterpret_cast<const LinearW *>(p.w) : own, z));
    bool done = CONTRACT ? euler_step_contracted<KNOWN_SMALL>(z, force) : euler_step<KNOWN_SMALL>(z, force);
    if (LIMIT) done |= (t1 - begin) >= p.max_steps;
    // selects, not a branch: nothing diverges in the stepping warp (measured equal or up to 4 % faster)
    cnt += done ? 1u : 0u;
    begin = done ? t1 : begin;
    z.x = done ? fresh.x : z.x;
    z.xd = done ? fresh.y : z.xd;
    z.th = done ? fresh.z : z.th;
    z.thd = done ? fresh.w : z.thd;
    // Same layout and meaning as the general kernel's streams. STREAMS 1: exactly the reward plane and
    // the done bits, 3: all four, no tests (each run-time test is a branch in the one warp whose
    // latency is the launch's time); 2: any combination.
    if (STREAMS == 1 || STREAMS == 3 || (STREAMS == 2 && sc.done)) {
        const uint32_t m = __ballot_sync(0xffffffffu, done && sc.valid);
        if (lane == 0u) *sc.done = m;
        sc.done += sc.words;
    }
    if (STREAMS == 3 || (STREAMS == 2 && sc.act)) {
        const uint32_t m = __ballot_sync(0xffffffffu, force > 0.0f && sc.valid);
        if (lane == 0u) *sc.act = m;
        sc.act += sc.words;
    }
    if (STREAMS == 1 || STREAMS == 3 || (STREAMS == 2 && sc.rew)) {
        if (sc.valid) *sc.rew = 1.0f;
        sc.rew += sc.n;
    }
    if (STREAMS == 3 || (STREAMS == 2 && sc.traj)) {
        const float v[4] = {z.x, z.xd, z.th, z.thd};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (sc.valid) *sc.traj = v[q];
            sc.traj += sc.n;
        }
    }
}

// The same step with the cart's velocity one step behind. The chain that a step waits for is the pole's: rates, angular
// acceleration, rates. The cart's acceleration comes after it (seven operations more) and is needed only by the next step's
// position, so the next step computes it first, while its own angular acceleration is under way; in one step after the
// other a loop's end waited for it. For actions that are not the state's, without the trajectory among the outputs, and
// up to two pairs per SM, where latency is the time: hashed actions, 500 steps, before / after (one helper), without outputs and
// with reward and done bits, 9,400 environments 26.9 / 26.0 and 30.8 / 27.8 us; 20,011 54.6 / 54.7 and 60.4 / 62.5.
// A batch of one pair per SM gets a helper on each of the three other schedulers: the one helper's 84 cycles per step
// were as many as the stepping warp's 88. 2,048 x 10,000: 450 -> 389 us, 75 cycles per step, of which 50 are the stepping warp's
// instructions; contracted 500 steps 24.7 -> 16.9, supplied actions 30.6 -> 23.2. (With two pairs per SM three helpers each
// are slower, 9,400 x 500 28.7 against 26.0; for a policy, which the stepping warp evaluates, they gain 1-3 %.
// The reciprocal of the denominator by a polynomial and a Newton step, which gives the same quotients and does not
// wait for the special-function unit: 389 -> 378, but 26.4 -> 26.9 with outputs; not kept.)
struct CartBehind {
    float xd, temp, thacc, c, fresh;  // of the step before: what its new velocity is made of, or is where its episode ended
    bool done;
    template <bool CONTRACT>
    __device__ __forceinline__ float velocity() const {
        float v;
        if (CONTRACT) {
            v = __fmaf_rn(kTau, __fmaf_rn(__fmul_rn(thacc, c), kXaccK, temp), xd);
        } else {
            const float p1 = __fmul_rn(__fmul_rn(kPML, thacc), c);
            v = __fadd_rn(xd, __fmul_rn(kTau, __fsub_rn(temp, div_mtot_core(p1))));
        }
        return done ? fresh : v;
    }
};
template <bool LIMIT, bool CONTRACT, int STREAMS, int CHUNK>
__device__ __forceinline__ void consume_step_behind(const RolloutParams &p, const PairBuffers<CHUNK> &buf, uint32_t b, int s,
                                                    uint32_t lane, uint32_t t1, StreamCursor &sc, State &z, CartBehind &cart,
                                                    uint32_t &cnt, uint32_t &begin) {
    const float4 fresh = buf.start[b][s][lane];
    const float force = buf.force[b][s][lane];
    const float xd = cart.velocity<CONTRACT>();
    const float sn = sin_small(z.th), c = cos_small(z.th);
    float nx, nth, nthd, temp, thacc;
    if (CONTRACT) {
        const float t1_ = __fmul_rn(__fmul_rn(z.thd, z.thd), kPML);
        temp = __fmul_rn(__fmaf_rn(t1_, sn, force), kRcpMTot);
        const float num = __fmaf_rn(-c, temp, __fmul_rn(kG, sn));
        const float den = __fmaf_rn(__fmul_rn(c, c), kDenK, kDenC);
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(den));
        thacc = __fmul_rn(num, r);
        nx = __fmaf_rn(kTau, xd, z.x);
        nth = __fmaf_rn(kTau, z.thd, z.th);
        nthd = __fmaf_rn(kTau, thacc, z.thd);
    } else {
        const float t2 = __fmul_rn(__fmul_rn(kPML, __fmul_rn(z.thd, z.thd)), sn);
        temp = div_mtot_core(__fadd_rn(force, t2));
        const float num = __fsub_rn(__fmul_rn(kG, sn), __fmul_rn(c, temp));
        const float den = __fsub_rn(0.5f * kFT, div_mtot_core(__fmul_rn(0.5f * kMPole, __fmul_rn(c, c))));
        thacc = div_tame(num, den);
        nx = __fadd_rn(z.x, __fmul_rn(kTau, xd));
        nth = __fadd_rn(z.th, __fmul_rn(kTau, z.thd));
        nthd = __fadd_rn(z.thd, __fmul_rn(kTau, thacc));
    }
    bool done = (fabsf(nx) > kXT) | (fabsf(nth) > kTT);
    if (LIMIT) done |= (t1 - begin) >= p.max_steps;
    cart = CartBehind{xd, temp, thacc, c, fresh.y, done};
    cnt += done ? 1u : 0u;
    begin = done ? t1 : begin;
    z.x = done ? fresh.x : nx;
    z.th = done ? fresh.z : nth;
    z.thd = done ? fresh.w : nthd;
    if (STREAMS == 1) {
        const uint32_t m = __ballot_sync(0xffffffffu, done && sc.valid);
        if (lane == 0u) *sc.done = m;
        sc.done += sc.words;
        if (sc.valid) *sc.rew = 1.0f;
        sc.rew += sc.n;
    }
}

// The step in the loops over a chunk: written out in both, or one lambda for both. The same operations, but the compiler
// gives other registers and another order, and no form is the quicker one everywhere. Time by a lambda over written out, 64 to
// 500 steps, 4,737 to 45,001 environments, without outputs, reward and done bits, all outputs: contracted, long hand-overs
// 0.98-1.01, 1.00-1.06, 0.98-1.01 (linear policies 14,001 x 500 with reward and done bits 39.4 / 38.0 us), short ones 1.00,
// hashed and supplied actions 1.00-1.02 and the others 0.99-1.00, hashed actions 1.02 (24,001 x 500 88 / 75 us) and one policy
// each 1.03 (27,001 x 500 97 / 79); canonical 0.97-1.00, 0.96-1.00, 0.98-1.01.
template <int POLICY, int CHUNK, bool LIMIT, bool CONTRACT, int STREAMS>
constexpr bool kWrittenOut = CONTRACT && (STREAMS == 1 ? CHUNK == kLongChunk || POLICY == 0
                                                      : STREAMS == 3 && CHUNK == kShortChunk && !LIMIT && POLICY != 1);

// START_IN: the start states are the caller's data and may hold any angle.
// HELPERS: warps that hash for the stepping one, every HELPERS-th step each; supplied start states have one. BEHIND: see CartBehind.
// kChunk: steps per hand-over.
template <int POLICY, bool START_IN, int PAIRS, int HELPERS, bool BEHIND, int kChunk, bool LIMIT, bool CONTRACT, int STREAMS>
__global__ void __launch_bounds__(32 * (1 + HELPERS) * PAIRS) rollout_assisted_kernel(const __grid_constant__ RolloutParams p) {
    __shared__ PairBuffers<kChunk> s_buf[PAIRS];
    __shared__ uint32_t s_stepping;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    bool producer;
    uint32_t pair = 0u, helper = 0u;
    if constexpr (PAIRS == 1) {
        const uint32_t steps = stepping_warp<HELPERS>(s_stepping);
        producer = warp != steps;
        if (HELPERS > 1) helper = warp > steps ? warp - 1u : warp;
        if constexpr (kUniformRole<POLICY, START_IN, CONTRACT, STREAMS>) producer = __shfl_sync(0xffffffffu, (int)producer, 0) != 0;
    } else {
        producer = warp >= (uint32_t)PAIRS;
        pair = producer ? warp - PAIRS : warp;  // (not warp % PAIRS: 9,401 x 400, step limit, start states given, 41.9 / 44.8 us)
    }
    const int64_t task = (int64_t)blockIdx.x * PAIRS + pair;
    // The warps of a pair leave here together, before their first barrier; no other pair uses
    // their barrier. Nothing that differs between the warps of a pair (or between lanes) may
    // decide an exit or a barrier from here on: each warp must execute exactly 1 + n_chunks
    // barriers, a count fixed by the launch parameters, or its partner waits for ever.
    if (task >= p.n_tasks) return;
    PairBuffers<kChunk> &buf = s_buf[pair];
    const uint32_t n_chunks = (p.T + kChunk - 1) / kChunk;

    int64_t idx = task * 32 + lane;
    const bool valid = idx < p.n;
    if (!valid) idx = p.n - 1;  // idle lanes shadow the last environment and store nothing
    const uint32_t env = p.env_offset + (uint32_t)idx;
    const FoldedKeys kr = fold_keys(make_keys(p.salt_r, env));

    if (producer) {
        const bool given = POLICY == 0 && p.action_bits_in;
        const FoldedKeys ka = fold_keys(make_keys(p.salt_a, env));
        const int64_t words = (p.n + 31) >> 5;
        for (uint32_t c = 0; c <= n_chunks; ++c) {
            // chunk c is written while the consumer works on chunk c - 1 (other buffer); the
            // buffer written here was last read in chunk c - 2, which the barrier before closed
            if (c < n_chunks) {
                const uint32_t b = c & 1u, tc = p.t0 + c * kChunk, row0 = c * kChunk;
                const int rows = (int)min((uint32_t)kChunk, p.T - row0);  // steps of this chunk
                // The caller's actions: row (t - t0) of [T][words], one word per warp task. Lane s
                // fetches the word of the chunk's step s, all in one load issued before the
                // hashing below and used after it, when it has long arrived.
                uint32_t my_word = 0u;
                if (given) {
                    const uint32_t row = row0 + lane;
                    if (lane < (uint32_t)kChunk && row < p.T)
                        my_word = __ldg(p.action_bits_in + (int64_t)row * words + task);
                }
                if (START_IN) {
                    // the chunk's rows of [T][4][n], all in flight at once
                    static_assert(!START_IN || HELPERS == 1, "one helper fetches all rows");
                    const float *src = p.start_in + (int64_t)row0 * 4 * p.n + idx;
#pragma unroll 4
                    for (int s = 0; s < rows; ++s) {
                        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&buf.start[b][s][lane]);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4u * q), "l"(src) : "memory");
                            src += p.n;
                        }
                    }
                }
                if (!START_IN || (POLICY == 0 && !given)) {
#pragma unroll 4
                    for (int s = helper; s < rows; s += HELPERS) {
                        const uint32_t t = tc + s;
                        if (!START_IN) {
                            const State f = start_state_folded(kr, fold16(4u * (t + 1u)));
                            buf.start[b][s][lane] = make_float4(f.x, f.xd, f.th, f.thd);
                        }
                        if (POLICY == 0 && !given)
                            buf.force[b][s][lane] = force_from_signbit(action_signbit_folded(ka, fold16(t)));
                    }
                }
                if (given) {
#pragma unroll 4
                    for (int s = helper; s < rows; s += HELPERS) {
                        const uint32_t word = __shfl_sync(0xffffffffu, my_word, s);
                        buf.force[b][s][lane] = force_from_signbit((word << (31u - lane)) & 0x80000000u);
                    }
                }
                // a lane's own copies have landed before it arrives at the barrier
                if (START_IN) asm volatile("cp.async.wait_all;" ::: "memory");
            }
            pair_barrier<PAIRS, HELPERS>(pair);
        }
        return;
    }

    State z;
    if (p.init_planes) {
        z.x = p.init_planes[idx];
        z.xd = p.init_planes[p.init_stride + idx];
        z.th = p.init_planes[2 * p.init_stride + idx];
        z.thd = p.init_planes[3 * p.init_stride + idx];
    } else {
        z = start_state_folded(kr, fold16(4u * p.t0));
    }
    LinearW own = {};
    if (POLICY == 6) {  // parameter q of env i at env_weights[q*n + i]
#pragma unroll
        for (int q = 0; q < 8; ++q) own.w[q / 4][q % 4] = p.env_weights[(int64_t)q * p.n + idx];
        own.b[0] = p.env_weights[8 * p.n + idx];
        own.b[1] = p.env_weights[9 * p.n + idx];
    }
    // as in the general kernel: the returns follow from the time of the last termination, and
    // only the step limit needs the carried-in episode length inside the loop
    uint32_t cnt = 0u, begin = p.t0 - ((LIMIT && p.ep_len_io) ? p.ep_len_io[idx] : 0u);
    const uint32_t t_end = p.t0 + p.T;
    StreamCursor sc;
    sc.n = p.n;
    sc.words = (p.n + 31) >> 5;
    sc.valid = valid;
    sc.rew = p.reward_stream ? p.reward_stream + idx : nullptr;
    sc.traj = p.trajectory ? p.trajectory + idx : nullptr;
    sc.done = p.done_bits ? p.done_bits + task : nullptr;  // one 32-env word per warp task
    sc.act = p.action_bits ? p.action_bits + task : nullptr;
    pair_barrier<PAIRS, HELPERS>(pair);  // chunk 0 is there
    static_assert(!BEHIND || (POLICY == 0 && !START_IN && STREAMS <= 1), "see CartBehind");
    constexpr int kUnroll = BEHIND ? kBehindUnroll : kStepUnroll;
    CartBehind cart;
    constexpr bool kOut = !BEHIND && !START_IN && kWrittenOut<POLICY, kChunk, LIMIT, CONTRACT, STREAMS>;
    for (uint32_t c = 0; c < n_chunks; ++c) {
        const uint32_t b = c & 1u, tc = p.t0 + c * kChunk;
        const int steps = (int)min((uint32_t)kChunk, t_end - tc);
        auto one = [&](int s) {
            if constexpr (BEHIND) consume_step_behind<LIMIT, CONTRACT, STREAMS>(p, buf, b, s, lane, tc + s + 1u, sc, z, cart, cnt, begin);
            else consume_step<POLICY, !START_IN, LIMIT, CONTRACT, STREAMS>(p, buf, b, s, lane, tc + s + 1u, own, sc, z, cnt, begin);
        };
        if (c != 0u && steps == kChunk) {
#pragma unroll kUnroll
            for (int s = 0; s < kChunk; ++s) {
                if constexpr (kOut) consume_step<POLICY, true, LIMIT, CONTRACT, STREAMS>(p, buf, b, s, lane, tc + s + 1u, own, sc, z, cnt, begin);
                else one(s);
            }
        } else {
            // The caller's initial state may hold any angle: the very first step tests it per
            // lane. From the second step on every angle is a survivor's (<= 0.2095) or a start
            // state's (<= 0.05).
            int s = 0;
            if (c == 0u) {
                consume_step<POLICY, false, LIMIT, CONTRACT, STREAMS>(p, buf, b, 0, lane, tc + 1u, own, sc, z, cnt, begin);
                cart = CartBehind{0.0f, 0.0f, 0.0f, 0.0f, z.xd, true};
                s = 1;
            }
#pragma unroll kUnroll
            for (; s < steps; ++s) {
                if constexpr (kOut) consume_step<POLICY, true, LIMIT, CONTRACT, STREAMS>(p, buf, b, s, lane, tc + s + 1u, own, sc, z, cnt, begin);
                else one(s);
            }
        }
        pair_barrier<PAIRS, HELPERS>(pair);
    }
    if (BEHIND && p.T) z.xd = cart.velocity<CONTRACT>();

    unsigned long long tot_ret = 0, tot_cnt = 0;
    if (valid) {
        const uint32_t carried = p.ep_len_io ? p.ep_len_io[idx] : 0u;
        const uint32_t first_begin = p.t0 - carried;
        const uint32_t ret = cnt ? begin - first_begin : 0u;
        const uint32_t running = t_end - begin + ((!LIMIT && cnt == 0u) ? carried : 0u);
        if (p.ep_return_sum) p.ep_return_sum[idx] = (float)ret;
        if (p.ep_count) p.ep_count[idx] = cnt;
        if (p.ep_len_io) p.ep_len_io[idx] = running;
        if (p.out_planes) {
            p.out_planes[idx] = z.x;
            p.out_planes[p.out_stride + idx] = z.xd;
            p.out_planes[2 * p.out_stride + idx] = z.th;
            p.out_planes[3 * p.out_stride + idx] = z.thd;
        }
        tot_ret = ret;
        tot_cnt = cnt;
    }
    if (p.totals) {
        for (int o = 16; o > 0; o >>= 1) {
            tot_ret += __shfl_down_sync(0xffffffffu, tot_ret, o);
            tot_cnt += __shfl_down_sync(0xffffffffu, tot_cnt, o);
        }
        if (lane == 0 && (tot_ret | tot_cnt)) {
            atomicAdd(p.totals, tot_ret);
            atomicAdd(p.totals + 1, tot_cnt);
        }
    }
}

template <int POLICY, bool START_IN, int PAIRS, int HELPERS, bool BEHIND, int CHUNK, bool CONTRACT, int STREAMS>
void launch_assisted_helpers(const RolloutParams &p, cudaStream_t s) {
    const unsigned grid = (unsigned)((p.n_tasks + PAIRS - 1) / PAIRS), block = 32 * (1 + HELPERS) * PAIRS;
    if (p.max_steps)
        rollout_assisted_kernel<POLICY, START_IN, PAIRS, HELPERS, BEHIND, CHUNK, true, CONTRACT, STREAMS><<<grid, block, 0, s>>>(p);
    else
        rollout_assisted_kernel<POLICY, START_IN, PAIRS, HELPERS, BEHIND, CHUNK, false, CONTRACT, STREAMS><<<grid, block, 0, s>>>(p);
}
template <int POLICY, bool START_IN, int PAIRS, int CHUNK, bool CONTRACT, int STREAMS>
void launch_assisted_pairs(const RolloutParams &p, cudaStream_t s) {
    if constexpr (POLICY == 0 && !START_IN && STREAMS <= 1) {
        // (from 8 and 32 steps on: shorter launches take 0.05 us longer with either; 2,048 x 1, 8, 16 steps, before / after 0.98,
        // 1.02, 1.09; 9,472 x 16, 32, 128 with reward and done bits 1.00, 1.02, 1.09)
        if (p.n_tasks <= sm_count() && p.T >= 8u) return launch_assisted_helpers<0, false, 1, 3, true, CHUNK, CONTRACT, STREAMS>(p, s);
        if (p.n_tasks <= sm_count() * 2 && p.T >= 32u) return launch_assisted_helpers<0, false, 1, 1, true, CHUNK, CONTRACT, STREAMS>(p, s);
    }
    launch_assisted_helpers<POLICY, START_IN, PAIRS, 1, false, CHUNK, CONTRACT, STREAMS>(p, s);
}
template <int POLICY, bool START_IN, int CHUNK, bool CONTRACT, int STREAMS>
void launch_assisted_limit(const RolloutParams &p, cudaStream_t s) {
    if constexpr (kMayPair<POLICY, START_IN, CONTRACT, STREAMS>) {
        if (two_pairs<STREAMS>(p)) return launch_assisted_pairs<POLICY, START_IN, 2, CHUNK, CONTRACT, STREAMS>(p, s);
    }
    launch_assisted_pairs<POLICY, START_IN, START_IN && STREAMS == 0 ? 2 : 1, CHUNK, CONTRACT, STREAMS>(p, s);
}
template <int POLICY, bool START_IN, int CHUNK, bool CONTRACT>
void launch_assisted_streams(const RolloutParams &p, cudaStream_t s) {
    const bool rd = p.reward_stream && p.done_bits;
    if (rd && !p.action_bits && !p.trajectory)
        launch_assisted_limit<POLICY, START_IN, CHUNK, CONTRACT, 1>(p, s);
    else if (rd && p.action_bits && p.trajectory)
        launch_assisted_limit<POLICY, START_IN, CHUNK, CONTRACT, 3>(p, s);
    else if (p.reward_stream || p.done_bits || p.action_bits || p.trajectory)
        launch_assisted_limit<POLICY, START_IN, CHUNK, CONTRACT, 2>(p, s);
    else
        launch_assisted_limit<POLICY, START_IN, CHUNK, CONTRACT, 0>(p, s);
}
// Supplied start states come in short chunks at all sizes (build time).
template <int POLICY, bool START_IN>
void launch_assisted_chunk(const RolloutParams &p, bool contracted, cudaStream_t s) {
    if (!START_IN && long_chunks(p, contracted)) {
        contracted ? launch_assisted_streams<POLICY, START_IN, START_IN ? kShortChunk : kLongChunk, true>(p, s)
                   : launch_assisted_streams<POLICY, START_IN, START_IN ? kShortChunk : kLongChunk, false>(p, s);
    } else {
        contracted ? launch_assisted_streams<POLICY, START_IN, kShortChunk, true>(p, s)
                   : launch_assisted_streams<POLICY, START_IN, kShortChunk, false>(p, s);
    }
}

}  // namespace

}  // namespace cp
