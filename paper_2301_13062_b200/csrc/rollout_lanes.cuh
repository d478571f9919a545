// Rollout under a shared tanh network with the network of an environment spread over G lanes
// (paper Sec. VI: fusing simulation with neural network inference), for batches too small to fill
// the chip.
//
// One lane per environment evaluates the hidden units one after another; with a few warps per
// scheduler nothing hides that. Here lane = g * E + e: the G lanes g of environment e (E = 32 / G
// environments per warp)
//   * all hold the state and all step it (the same instructions for every lane: no cost);
//   * evaluate H / G hidden units each, side by side, their weights in registers, and sum their part of the
//     estimate of l1 - l0 (policy_screen.cuh); a deep network's first activations go through a row of
//     shared memory per environment;
//   * add the parts pairwise by shuffles. Where a warp has a sum that does not decide, its lanes compute
//     the defined logits together (lanes_defined_action): one lane by itself takes several thousand cycles,
//     and one such environment after another lengthened launches by up to a fifth (4-64-2, 4,096 x 500, twelve
//     policies: 139 .. 162 us against 133 .. 143). The deep network's lanes go by themselves: together they
//     cost every launch 16 us for the few that gain (133 .. 154 against 148 .. 156).
// One lane per environment (G = 1) is this kernel for 4-16-2's weights in registers, where the general one loads every weight in
// every step, and for the larger networks, whose weights are loaded here too, for the shorter chain below and for per-step
// outputs without a test of each in every step.
//
// What a step waits for is its chain: network, action, acceleration, rates, network. All of the step that does not
// depend on the action is taken out of it (euler_both_ways: both candidates of the new rates, the termination test and
// the restart), so that it runs while the special-function unit works on the activations, and the chain is network,
// one selection, network. 4-64-2, 4,096 x 500: 510 -> 372 cycles per step (134 -> 97 us), of which 128 are that unit's sixteen
// results; 4-16-2 324 -> 243; with all outputs 168 -> 117 and 152 -> 80 us (these also by what follows). With one
// warp per scheduler issue is no bound (192 instructions); with three of 4-16-2's one-lane warps it is: 222
// instructions, the packed ones two slots each, of 370 cycles per warp and step.
// The start state an environment would continue from is hashed on every step ahead of the network, one
// component per lane where there are four: that work fills issue slots the network leaves empty, and a
// finished environment just takes it.
//
// One warp per scheduler also waits for its instructions: the loop holds nothing that most steps do not
// need. The first step from a caller's states and the steps of a warp that stands at a supplied start state, whose angles
// need the library's sine and cosine, are a copy of the step of their own (128 steps on 4,096 environments, in
// one loop / apart: 4-16-2 37 / 27 us, 4-32-2 49 / 35, 4-64-2 41 / 35, 4-16-16-2 49 / 39).
//
// Warps exchange nothing: a warp's E environments are whole bytes of the bit planes' words (handing 32 steps of bits over in
// shared memory and writing words, one branch and one barrier in every 32 steps, cost 30 .. 90 ns per step).
#pragma once
#include <type_traits>

#include "cartpole_device.cuh"
#include "cartpole_internal.h"
#include "policy_screen.cuh"

namespace cp {

// One step before its action is known. Only the accelerations depend on the action: the new position and angle,
// and with them the termination test and whatever replaces the state of a finished environment, follow from the
// rates the step began with, and the new rates have two candidates, one per direction of the force. Both are
// computed by packed operations (low half: pushed left, high half: right), about as many as one, while the policy
// is still deciding; what is left after it is one selection. Each half performs the operations of euler_step<true> / euler_step_contracted<true> in
// their order: the same bits. Domain: |theta| <= 0.22, as there.
struct BothWays {
    float x, th;
    bool done;
    f32x2 xd, thd;
};
template <bool CONTRACT>
__device__ __forceinline__ BothWays euler_both_ways(const State &z) {
    BothWays n;
    const float s = sin_small(z.th), c = cos_small(z.th);
    const f32x2 cc = splat2(c);
    if (CONTRACT) {
        const float t1 = __fmul_rn(__fmul_rn(z.thd, z.thd), kPML);
        const f32x2 temp = mul2(pack2(__fmaf_rn(t1, s, -kF), __fmaf_rn(t1, s, kF)), splat2(kRcpMTot));
        const f32x2 num = fma2(splat2(-c), temp, splat2(__fmul_rn(kG, s)));
        const float den = __fmaf_rn(__fmul_rn(c, c), kDenK, kDenC);
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(den));
        const f32x2 thacc = mul2(num, splat2(r));
        const f32x2 xacc = fma2(mul2(thacc, cc), splat2(kXaccK), temp);
        n.x = __fmaf_rn(kTau, z.xd, z.x);
        n.th = __fmaf_rn(kTau, z.thd, z.th);
        n.xd = fma2(splat2(kTau), xacc, splat2(z.xd));
        n.thd = fma2(splat2(kTau), thacc, splat2(z.thd));
    } else {
        const float t2 = __fmul_rn(__fmul_rn(kPML, __fmul_rn(z.thd, z.thd)), s);
        const f32x2 temp = div_mtot_core2(pack2(__fadd_rn(-kF, t2), __fadd_rn(kF, t2)));
        const f32x2 num = add_product2(splat2(__fmul_rn(kG, s)), mul2(cc, temp));  // n0 - n1
        const float den = __fsub_rn(0.5f * kFT, div_mtot_core(__fmul_rn(0.5f * kMPole, __fmul_rn(c, c))));
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(den));
        const f32x2 q = mul2(num, splat2(r));
        const f32x2 rem = fma2(splat2(-den), q, num);
        const f32x2 thacc = fma2(rem, splat2(r), q);
        const f32x2 np1 = mul2(mul2(splat2(-kPML), thacc), cc);
        const f32x2 xacc = add2(temp, div_mtot_core2(np1));  // temp - p2
        n.x = __fadd_rn(z.x, __fmul_rn(kTau, z.xd));
        n.th = __fadd_rn(z.th, __fmul_rn(kTau, z.thd));
        n.xd = add_product2(splat2(z.xd), mul2(splat2(-kTau), xacc));
        n.thd = add_product2(splat2(z.thd), mul2(splat2(-kTau), thacc));
    }
    n.done = (fabsf(n.x) > kXT) | (fabsf(n.th) > kTT);
    return n;
}

// Keeps the compiler from reading a lane's weight again in every step (the launch parameters are
// constant memory, which serves one address per warp and access).
__device__ __forceinline__ float in_register(float v) {
    asm volatile("" : "+f"(v));
    return v;
}

// U units of a layer with IN inputs, on one lane: unit g * U + u of the layer.
template <int U, int IN>
struct LaneLayer {
    float w[U][IN], b[U];
    // layer: w[units][IN] then b[units], as the caller gave them
    __device__ __forceinline__ void load(const float *layer, int units, uint32_t g) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int unit = (int)g * U + u;
#pragma unroll
            for (int i = 0; i < IN; ++i) w[u][i] = in_register(layer[unit * IN + i]);
            b[u] = in_register(layer[units * IN + unit]);
        }
    }
    // Sums of this lane's units, left to right from the bias; SPLIT: few long chains, each as two.
    template <bool SPLIT>
    __device__ __forceinline__ void sums(const float (&in)[IN], float (&h)[U]) const {
        constexpr int HALF = SPLIT ? IN / 2 : IN;
#pragma unroll
        for (int u = 0; u < U; ++u) h[u] = b[u];
#pragma unroll
        for (int i = 0; i < HALF; ++i) {
#pragma unroll
            for (int u = 0; u < U; ++u) h[u] = __fmaf_rn(w[u][i], in[i], h[u]);
        }
        if constexpr (SPLIT) {
            float rest[U] = {};
#pragma unroll
            for (int i = HALF; i < IN; ++i) {
#pragma unroll
                for (int u = 0; u < U; ++u) rest[u] = __fmaf_rn(w[u][i], in[i], rest[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) h[u] = __fadd_rn(h[u], rest[u]);
        }
    }
};
template <int NET, int G>
struct LaneNetwork {
    using S = NetShape<NET>;
    static constexpr int U = S::H / G;
    // Units 2q and 2q + 1 of the lane by one packed operation: half the instructions of a loop that waits for issue, with
    // one or two lanes per environment; alone on its scheduler a warp waits for latency, which they don't shorten.
    static constexpr bool kPaired = G <= 2;
    // One lane, and more weights than it has registers: they are read from the launch parameters in every step.
    static constexpr bool kReads = G == 1 && NET != 2;
    LaneLayer<kPaired ? 1 : U, 4> first;
    f32x2 paired[kPaired && !kReads ? U / 2 : 1][5], paired_step[kPaired && !kReads ? U / 2 : 1];
    LaneLayer<S::kDeep && !kPaired ? U : 1, S::kDeep && !kPaired ? S::H : 1> second;  // unused unless the network is deep
    float step[kPaired ? 1 : U];                             // w1[j] - w0[j] of this lane's last-layer units
    __device__ __forceinline__ void load(const RolloutParams &p, uint32_t g) {
        if constexpr (kReads) {
        } else if constexpr (kPaired) {
            static_assert(!S::kDeep, "one hidden layer");
            // (+ 0, which the compiler cannot know: from an address it knows it reads one lane's weights again in every step,
            // 60 to 72 registers instead of 142 to 160)
            const float *w = p.w + (p.n >> 62), *logits = w + S::kLogits;
#pragma unroll
            for (int q = 0; q < U / 2; ++q) {
                const int unit = (int)g * U + 2 * q;
#pragma unroll
                for (int i = 0; i < 4; ++i) paired[q][i] = pack2(in_register(w[unit * 4 + i]), in_register(w[unit * 4 + 4 + i]));
                paired[q][4] = pack2(in_register(w[4 * S::H + unit]), in_register(w[4 * S::H + unit + 1]));
                paired_step[q] = pack2(in_register(__fsub_rn(logits[S::H + unit], logits[unit])), in_register(__fsub_rn(logits[S::H + unit + 1], logits[unit + 1])));
            }
        } else {
            first.load(p.w, S::H, g);
            if constexpr (S::kDeep) second.load(p.w + S::kSecond, S::H, g);
            const float *logits = p.w + S::kLogits + g * U;
#pragma unroll
            for (int u = 0; u < U; ++u) step[u] = in_register(__fsub_rn(logits[S::H + u], logits[u]));
        }
    }
    // Arguments of the units 2q and 2q + 1, paired.
    __device__ __forceinline__ f32x2 arguments(int q, const State &z) const {
        f32x2 h = paired[q][4];
        h = fma2(paired[q][0], splat2(z.x), h);
        h = fma2(paired[q][1], splat2(z.xd), h);
        h = fma2(paired[q][2], splat2(z.th), h);
        return fma2(paired[q][3], splat2(z.thd), h);
    }
};

// Floats per environment's row of shared memory: 16 bytes more than the activations, so that the 16-byte
// reads of up to eight environments' rows fall into different banks.
template <int H>
constexpr int kRow = H + 4;

// The activations of all H units of an environment, from its lanes' U each.
template <int H, int U>
__device__ __forceinline__ void share_activations(float *row, uint32_t g, const float (&mine)[U], float (&all)[H]) {
#pragma unroll
    for (int u = 0; u < U; ++u) row[g * U + u] = mine[u];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < H; j += 4) {
        const float4 v = *reinterpret_cast<const float4 *>(row + j);
        all[j] = v.x;
        all[j + 1] = v.y;
        all[j + 2] = v.z;
        all[j + 3] = v.w;
    }
    __syncwarp();  // the row is read before it is written again
}

// The action by the defined logits of a network with one hidden layer, by all lanes of the environment
// together: their units' activations side by side, then one of the two logits each, left to right from its bias.
template <int NET, int G, bool CONTRACT>
__device__ __forceinline__ uint32_t lanes_defined_action(const RolloutParams &p, const LaneNetwork<NET, G> &net, const State &z, float *row, uint32_t g) {
    using S = NetShape<NET>;
    constexpr int H = S::H, U = LaneNetwork<NET, G>::U;
    float h[U];
    if constexpr (LaneNetwork<NET, G>::kPaired) {
#pragma unroll
        for (int q = 0; q < U / 2; ++q) unpack2(net.arguments(q, z), h[2 * q], h[2 * q + 1]);
    } else {
        const float obs[4] = {z.x, z.xd, z.th, z.thd};
        net.first.template sums<false>(obs, h);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) row[g * U + u] = CONTRACT ? tanh_contracted(h[u]) : tanh_canonical(h[u]);
    __syncwarp();
    const float *logits = p.w + S::kLogits, *w = logits + (g & 1u) * H;
    float mine = logits[2 * H + (g & 1u)];
#pragma unroll 4
    for (int j = 0; j < H; ++j) mine = __fmaf_rn(w[j], row[j], mine);
    __syncwarp();
    const float other = __shfl_xor_sync(0xffffffffu, mine, 32 / G);  // the neighbouring lane of the environment
    const bool right = (g & 1u) ? mine > other : other > mine;
    return right ? 0x80000000u : 0u;
}

// The first hidden layer's activations of this lane's units.
template <int NET, int G>
__device__ __forceinline__ void lanes_activations(const float *w, float base, const LaneNetwork<NET, G> &net, const State &z, float (&h)[LaneNetwork<NET, G>::U]) {
    constexpr int U = LaneNetwork<NET, G>::U;
    if constexpr (LaneNetwork<NET, G>::kReads) {
        h[0] = screen_estimate<NET>(w, base, z);
    } else if constexpr (LaneNetwork<NET, G>::kPaired) {
#pragma unroll
        for (int q = 0; q < U / 2; ++q) unpack2(tanh_screen2(net.arguments(q, z)), h[2 * q], h[2 * q + 1]);
    } else {
        const float obs[4] = {z.x, z.xd, z.th, z.thd};
        net.first.template sums<false>(obs, h);
#pragma unroll
        for (int u = 0; u < U; ++u) h[u] = tanh_screen(h[u]);
    }
}

// The action of this lane's environment, from them. Every lane sums its own units' part of the estimate; the
// parts are added pairwise over the environment's lanes, so that all of them hold the same sum.
template <int NET, int G, bool CONTRACT>
__device__ __forceinline__ uint32_t lanes_action(const RolloutParams &p, const LaneNetwork<NET, G> &net, const State &z,
                                                 float (&h)[LaneNetwork<NET, G>::U], float *row, uint32_t g) {
    using S = NetShape<NET>;
    constexpr int U = LaneNetwork<NET, G>::U;
    float part = 0.0f;
    if constexpr (LaneNetwork<NET, G>::kReads) {
        part = h[0];
    } else if constexpr (LaneNetwork<NET, G>::kPaired) {
        f32x2 sum = mul2(net.paired_step[0], pack2(h[0], h[1]));
#pragma unroll
        for (int q = 1; q < U / 2; ++q) sum = fma2(net.paired_step[q], pack2(h[2 * q], h[2 * q + 1]), sum);
        float lo, hi;
        unpack2(sum, lo, hi);
        part = __fadd_rn(lo, hi);
    } else {
        if constexpr (S::kDeep) {
            float all[S::H];
            share_activations(row, g, h, all);
            net.second.template sums<U <= 2>(all, h);
#pragma unroll
            for (int u = 0; u < U; ++u) h[u] = tanh_screen(h[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) part = __fmaf_rn(net.step[u], h[u], part);
    }
#pragma unroll
    for (int o = 32 / G; o < 32; o <<= 1) part = __fadd_rn(part, __shfl_xor_sync(0xffffffffu, part, o));
    const float estimate = LaneNetwork<NET, G>::kReads ? part : __fadd_rn(p.screen_base, part);
    uint32_t sb = screen_action(estimate);
    const bool open = !screen_decides(estimate, p.screen_bound);
    if constexpr (S::kDeep || G == 1) {
        if (open) sb = defined_action<NET, CONTRACT>(p.w, p.w + S::kLogits, z);
        __syncwarp();
    } else if (__any_sync(0xffffffffu, open)) {  // warp-uniform
        const uint32_t defined = lanes_defined_action<NET, G, CONTRACT>(p, net, z, row, g);
        if (open) sb = defined;
    }
    return sb;
}

// NET: 2 (4-16-2), 4 (4-32-2), 5 (4-64-2), 7 (4-16-16-2). G: lanes per environment. STREAMS: any
// combination of the per-step outputs. The step limit is a run-time option: next to a network's evaluation
// its test costs nothing.
template <int NET, int G, bool STREAMS, bool CONTRACT>
__global__ void __launch_bounds__(128, NET == 7 && !STREAMS ? 0 : 3) rollout_lanes_kernel(const __grid_constant__ RolloutParams p) {
    constexpr int E = 32 / G, W = 4;     // environments per warp; warps of a CTA, one per scheduler
    constexpr int C = G >= 4 ? 1 : 4 / G;  // state components that a lane hashes and stores
    static_assert(!STREAMS || E >= 8, "a warp writes whole bytes of the bit planes");
    constexpr int ROW = G == 1 ? 1 : kRow<NetShape<NET>::H>;  // one lane: not used
    __shared__ __align__(16) float s_rows[W * E * ROW];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t e = lane % E, g = lane / E, c = (g * C) & 3u;  // c: the first of the lane's components
    float *const row = s_rows + (warp * E + e) * ROW;
    const int64_t base = ((int64_t)blockIdx.x * W + warp) * E;
    int64_t idx = base + e;
    const bool valid = idx < p.n;
    if (!valid) idx = p.n - 1;  // idle lanes shadow the last environment and store nothing
    // A warp that lies wholly past the end must not read what the last environment's warp rewrites at its
    // end (a batch advanced in place, its episode lengths): nothing orders the two. Its lanes step
    // along from a hashed state instead. (Per lane without per-step outputs, per warp with them: the
    // order of the kernel's instructions hangs on it. 4-16-2, 128 steps: 1.00 of the time without the test
    // and 1.03 the other way round; contracted 4-32-2 with outputs 1.00 and 1.07.)
    const bool owned = STREAMS ? base < p.n : valid;
    const FoldedKeys kr = fold_keys(make_keys(p.salt_r, p.env_offset + (uint32_t)idx));
    State z;
    if (p.init_planes && owned) {
        z.x = p.init_planes[idx];
        z.xd = p.init_planes[p.init_stride + idx];
        z.th = p.init_planes[2 * p.init_stride + idx];
        z.thd = p.init_planes[3 * p.init_stride + idx];
    } else {
        z = start_state_folded(kr, fold16(4u * p.t0));
    }
    LaneNetwork<NET, G> net;
    net.load(p, g);
    const uint32_t carried = p.ep_len_io && owned ? p.ep_len_io[idx] : 0u;
    // begin: global time at which the running episode began (as in the general kernel)
    uint32_t cnt = 0u, begin = p.t0 - carried;
    const int64_t words = (p.n + 31) >> 5;
    const float *start = p.start_in ? p.start_in + (int64_t)c * p.n + idx : nullptr;
    // (Pointers of lanes that write nothing are null and advanced all the same, never followed.)
    // Per-step outputs, by the environment's own warp alone: a lane stores its components of the trajectory, and
    // lane 0 the done bits and lane 1 the action bits of the warp's E environments, which are whole bytes of the row's word.
    const bool keeps = STREAMS && p.trajectory && valid && g < 4u;
    float *tr = keeps ? p.trajectory + (int64_t)c * p.n + idx : nullptr;
    uint32_t *plane = lane == 0u ? p.done_bits : lane == 1u ? p.action_bits : nullptr;
    const bool writes = STREAMS && plane && base < words * 32;
    uint8_t *bits = reinterpret_cast<uint8_t *>(plane) + base / 8;

    // Supplied start states: a lane copies its components of a row into its own place of a ring in shared memory, three
    // steps before they are used (a step is shorter than the way to L2) and into the slot that the step before has used.
    constexpr uint32_t kSlots = 4u, kAhead = kSlots - 1u;
    __shared__ float s_ahead[kSlots][C][32 * W];
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(&s_ahead[0][0][threadIdx.x]);
    auto request = [&](uint32_t k) {
        if (k < p.T) {
#pragma unroll
            for (int q = 0; q < C; ++q)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(ring + (k % kSlots * C + q) * (128u * W)), "l"(start + q * p.n) : "memory");
            start += 4 * p.n;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // general: a state may hold any angle; given: supplied start states
    auto step = [&](auto general, auto given, uint32_t k) {
        const uint32_t t1 = p.t0 + k + 1u;
        float h[LaneNetwork<NET, G>::U];
        // (One lane per environment, canonical: ahead of the rest in program order too, or the compiler loads 4-16-2's weights
        // in every step: without outputs 0.59 to 0.84 of the time, with them 0.96 to 1.00; the larger networks with outputs 0.96
        // to 1.00, without 1.00 to 1.03; the other forms 0.94 to 1.23.)
        constexpr bool FIRST = G == 1 && !CONTRACT && (NET == 2 || STREAMS) && !decltype(general)::value;
        if (FIRST) lanes_activations<NET, G>(p.w, p.screen_base, net, z, h);
        // the start state that a finished environment continues from: this lane's components of it
        float mine[C];
        if constexpr (decltype(given)::value) asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
#pragma unroll
        for (int q = 0; q < C; ++q) {
            if constexpr (decltype(given)::value) mine[q] = *(volatile float *)&s_ahead[k % kSlots][q][threadIdx.x];
            else mine[q] = start_component_folded(kr, fold16(4u * t1), c + q);
        }
        if constexpr (decltype(given)::value) request(k + kAhead);
        auto component = [&](int q) { return G == 1 ? mine[q % C] : __shfl_sync(0xffffffffu, mine[q % C], e + q / C * E); };
        uint32_t sb;
        bool done;
        if constexpr (decltype(general)::value) {
            lanes_activations<NET, G>(p.w, p.screen_base, net, z, h);
            sb = lanes_action<NET, G, CONTRACT>(p, net, z, h, row, g);
            const float force = force_from_signbit(sb);
            done = CONTRACT ? euler_step_contracted<false>(z, force) : euler_step<false>(z, force);
            if (p.max_steps) done |= (t1 - begin) >= p.max_steps;
            const State f = {component(0), component(1), component(2), component(3)};
            z.x = done ? f.x : z.x;
            z.xd = done ? f.xd : z.xd;
            z.th = done ? f.th : z.th;
            z.thd = done ? f.thd : z.thd;
        } else {
            // everything that does not wait for the action, in the shadow of the network
            const State f = {component(0), component(1), component(2), component(3)};
            const BothWays n = euler_both_ways<CONTRACT>(z);
            done = n.done;
            if (p.max_steps) done |= (t1 - begin) >= p.max_steps;
            float xd0, xd1, thd0, thd1;
            unpack2(n.xd, xd0, xd1);
            unpack2(n.thd, thd0, thd1);
            float x = done ? f.x : n.x, th = done ? f.th : n.th;
            xd0 = done ? f.xd : xd0;
            xd1 = done ? f.xd : xd1;
            thd0 = done ? f.thd : thd0;
            thd1 = done ? f.thd : thd1;
            asm volatile("" : "+f"(x), "+f"(th), "+f"(xd0), "+f"(xd1), "+f"(thd0), "+f"(thd1));  // not after its branch
            if (!FIRST) lanes_activations<NET, G>(p.w, p.screen_base, net, z, h);
            sb = lanes_action<NET, G, CONTRACT>(p, net, z, h, row, g);
            z.x = x;
            z.xd = sb ? xd1 : xd0;
            z.th = th;
            z.thd = sb ? thd1 : thd0;
        }
        cnt += done ? 1u : 0u;
        begin = done ? t1 : begin;
        if (STREAMS) {
            const uint32_t dm = __ballot_sync(0xffffffffu, done && valid);
            const uint32_t am = __ballot_sync(0xffffffffu, sb != 0u && valid);
            const uint32_t mine = lane ? am : dm;
            if (writes) {
                if (E == 32) *reinterpret_cast<uint32_t *>(bits) = mine;
                else if (E == 16) *reinterpret_cast<uint16_t *>(bits) = (uint16_t)mine;
                else *bits = (uint8_t)mine;
            }
            bits += 4 * words;
            if (C == 1) {
                const float v = c < 2u ? (c ? z.xd : z.x) : (c == 2u ? z.th : z.thd);
                if (keeps) tr[0] = v;
            } else if (keeps) {
                tr[0] = C == 2 && c ? z.th : z.x;
                tr[p.n] = C == 2 && c ? z.thd : z.xd;
                if (C == 4) {
                    tr[2 * p.n] = z.th;
                    tr[3 * p.n] = z.thd;
                }
            }
            tr += 4 * p.n;
        }
    };
    // Rows [from, to) of the reward plane for the warp's own environments, after their steps: G rows at a time.
    auto rewards = [&](uint32_t from, uint32_t to) {
        if (!STREAMS || !p.reward_stream || !valid) return;
        float *out = p.reward_stream + (int64_t)(from + g) * p.n + idx;
        for (uint32_t r = from + g; r < to; r += G, out += (int64_t)G * p.n) *out = 1.0f;
    };
    uint32_t k = 0u;
    auto steps = [&](auto &&one) {
        while (k < p.T) {
            const uint32_t from = k, to = STREAMS ? min(p.T, (k | 31u) + 1u) : p.T;
#pragma unroll 1
            for (; k < to; ++k) one();
            rewards(from, to);
        }
    };
    const std::true_type yes{};
    const std::false_type no{};
    if (p.start_in) {
        for (uint32_t r = 0; r < kAhead; ++r) request(r);
        steps([&]() {
            if (__all_sync(0xffffffffu, fabsf(z.th) <= kSmallAngle)) step(no, yes, k);
            else step(yes, yes, k);
        });
    } else {
        if (p.init_planes && p.T) {
            step(yes, no, k++);
            rewards(0u, 1u);
        }
        steps([&]() { step(no, no, k); });
    }

    unsigned long long tot_ret = 0, tot_cnt = 0;
    if (valid && g == 0u) {
        const uint32_t ret = cnt ? begin - (p.t0 - carried) : 0u;
        if (p.ep_return_sum) p.ep_return_sum[idx] = (float)ret;
        if (p.ep_count) p.ep_count[idx] = cnt;
        if (p.ep_len_io) p.ep_len_io[idx] = p.t0 + p.T - begin;
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

namespace {

template <int NET, int G, bool STREAMS, bool CONTRACT>
cudaError_t launch_lanes_one(RolloutParams &p, cudaStream_t s) {
    constexpr int W = 4;
    const int64_t per_cta = W * (32 / G);
    const int64_t grid = (p.n + per_cta - 1) / per_cta;
    if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    rollout_lanes_kernel<NET, G, STREAMS, CONTRACT><<<(unsigned)grid, 32 * W, 0, s>>>(p);
    count_launch();
    return cudaGetLastError();
}

// The instances that rollout_lanes_for asks for.
template <int NET, bool STREAMS, bool CONTRACT>
cudaError_t launch_lanes_g(RolloutParams &p, int g, cudaStream_t s) {
    if constexpr (STREAMS || NET == 2 || NET == 5)
        if (g == 1) return launch_lanes_one<NET, 1, STREAMS, CONTRACT>(p, s);
    if constexpr (NET == 2 || NET == 4)
        if (g == 2) return launch_lanes_one<NET, 2, STREAMS, CONTRACT>(p, s);
    if constexpr (!STREAMS && (NET == 4 || NET == 5 || (NET == 7 && !CONTRACT)))
        if (g == 8) return launch_lanes_one<NET, 8, STREAMS, CONTRACT>(p, s);
    return launch_lanes_one<NET, 4, STREAMS, CONTRACT>(p, s);
}

template <int NET, bool CONTRACT>
cudaError_t launch_lanes_net(RolloutParams &p, int g, bool streams, cudaStream_t s) {
    return streams ? launch_lanes_g<NET, true, CONTRACT>(p, g, s) : launch_lanes_g<NET, false, CONTRACT>(p, g, s);
}

}  // namespace

}  // namespace cp
