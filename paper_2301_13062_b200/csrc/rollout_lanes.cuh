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
// With the defined logits in every step, whose order is a chain of one multiply-add per hidden unit, the 4-64-2
// network's step took 1,190 cycles on 4,096 environments; it takes 510 (500 steps: 303 -> 133 us).
// The start state an environment would continue from is hashed on every step ahead of the network,
// by four lanes, one component each: that work fills issue slots the network leaves empty, and a
// finished environment just takes it.
//
// One warp per scheduler also waits for its instructions: the loop holds nothing that most steps do not
// need. The first step from a caller's states and all steps from supplied start states, whose angles need the
// library's sine and cosine, are a copy of the step of their own (128 steps on 4,096 environments, in
// one loop / apart: 4-16-2 37 / 27 us, 4-32-2 49 / 35, 4-64-2 41 / 35, 4-16-16-2 49 / 39).
//
// Warps only exchange data when bit planes are written: the G warps of a CTA then hold the 32
// environments of one bit-plane word, leave their bits of 32 steps in shared memory and write the
// words together. All of a CTA's warps make the same T steps, so they meet the same barriers.
#pragma once
#include <type_traits>

#include "cartpole_device.cuh"
#include "cartpole_internal.h"
#include "policy_screen.cuh"

namespace cp {

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
    LaneLayer<U, 4> first;
    LaneLayer<S::kDeep ? U : 1, S::kDeep ? S::H : 1> second;  // unused unless the network is deep
    float step[U];                                           // w1[j] - w0[j] of this lane's last-layer units
    __device__ __forceinline__ void load(const RolloutParams &p, uint32_t g) {
        first.load(p.w, S::H, g);
        if constexpr (S::kDeep) second.load(p.w + S::kSecond, S::H, g);
        const float *logits = p.w + S::kLogits + g * U;
#pragma unroll
        for (int u = 0; u < U; ++u) step[u] = in_register(__fsub_rn(logits[S::H + u], logits[u]));
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
    const float obs[4] = {z.x, z.xd, z.th, z.thd};
    float h[U];
    net.first.template sums<false>(obs, h);
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

// The action of this lane's environment. Every lane sums its own units' part of the estimate; the
// parts are added pairwise over the environment's lanes, so that all of them hold the same sum.
template <int NET, int G, bool CONTRACT>
__device__ __forceinline__ uint32_t lanes_action(const RolloutParams &p, const LaneNetwork<NET, G> &net, const State &z, float *row, uint32_t g) {
    using S = NetShape<NET>;
    constexpr int U = LaneNetwork<NET, G>::U;
    const float obs[4] = {z.x, z.xd, z.th, z.thd};
    float h[U];
    net.first.template sums<false>(obs, h);
#pragma unroll
    for (int u = 0; u < U; ++u) h[u] = tanh_screen(h[u]);
    if constexpr (S::kDeep) {
        float all[S::H];
        share_activations(row, g, h, all);
        net.second.template sums<U <= 2>(all, h);
#pragma unroll
        for (int u = 0; u < U; ++u) h[u] = tanh_screen(h[u]);
    }
    float part = 0.0f;
#pragma unroll
    for (int u = 0; u < U; ++u) part = __fmaf_rn(net.step[u], h[u], part);
#pragma unroll
    for (int o = 32 / G; o < 32; o <<= 1) part = __fadd_rn(part, __shfl_xor_sync(0xffffffffu, part, o));
    const float estimate = __fadd_rn(p.screen_base, part);
    uint32_t sb = screen_action(estimate);
    const bool open = !screen_decides(estimate, p.screen_bound);
    if constexpr (S::kDeep) {
        if (open) sb = defined_action<NET, CONTRACT, 1>(p.w, p.w + S::kLogits, z);
        __syncwarp();
    } else if (__any_sync(0xffffffffu, open)) {  // warp-uniform
        const uint32_t defined = lanes_defined_action<NET, G, CONTRACT>(p, net, z, row, g);
        if (open) sb = defined;
    }
    return sb;
}

// Warps of a CTA: one per scheduler, and as many as hold the 32 environments of a bit-plane word
// where such words are written by several warps.
template <int G, bool STREAMS>
constexpr int kLaneWarps = STREAMS ? G : 4;

// NET: 2 (4-16-2), 4 (4-32-2), 5 (4-64-2), 7 (4-16-16-2). G: lanes per environment. STREAMS: any
// combination of the per-step outputs. The step limit is a run-time option: next to a network's evaluation
// its test costs nothing.
template <int NET, int G, bool STREAMS, bool CONTRACT>
__global__ void __launch_bounds__(32 * kLaneWarps<G, STREAMS>) rollout_lanes_kernel(const __grid_constant__ RolloutParams p) {
    static_assert(G >= 4, "four lanes of an environment hash the components of its start state");
    constexpr int E = 32 / G, W = kLaneWarps<G, STREAMS>;
    constexpr int ROW = kRow<NetShape<NET>::H>;
    __shared__ __align__(16) float s_rows[W * E * ROW];
    __shared__ uint32_t s_bits[STREAMS ? 2 : 1][32][W];  // done bits low, action bits high, of 32 steps
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t e = lane % E, g = lane / E, c = g & 3u;  // c: the state component this lane hashes and stores
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
    float *tr = STREAMS && p.trajectory ? p.trajectory + (int64_t)c * p.n + idx : nullptr;
    const float *start = p.start_in ? p.start_in + (int64_t)c * p.n + idx : nullptr;

    // general: a state may hold any angle
    auto step = [&](auto general, uint32_t k) {
        const uint32_t t1 = p.t0 + k + 1u;
        float fresh;
        if (decltype(general)::value && start) {
            fresh = __ldg(start);
            start += 4 * p.n;
        } else {
            fresh = start_component_folded(kr, fold16(4u * t1), c);
        }
        const uint32_t sb = lanes_action<NET, G, CONTRACT>(p, net, z, row, g);
        const float force = force_from_signbit(sb);
        constexpr bool SMALL = !decltype(general)::value;
        bool done = CONTRACT ? euler_step_contracted<SMALL>(z, force) : euler_step<SMALL>(z, force);
        if (p.max_steps) done |= (t1 - begin) >= p.max_steps;
        const float fx = __shfl_sync(0xffffffffu, fresh, e), fxd = __shfl_sync(0xffffffffu, fresh, e + E);
        const float fth = __shfl_sync(0xffffffffu, fresh, e + 2 * E), fthd = __shfl_sync(0xffffffffu, fresh, e + 3 * E);
        cnt += done ? 1u : 0u;
        begin = done ? t1 : begin;
        z.x = done ? fx : z.x;
        z.xd = done ? fxd : z.xd;
        z.th = done ? fth : z.th;
        z.thd = done ? fthd : z.thd;
        if (STREAMS) {
            const uint32_t dm = __ballot_sync(0xffffffffu, done && valid);
            const uint32_t am = __ballot_sync(0xffffffffu, sb != 0u && valid);
            if (tr) {
                if (valid && g < 4u) tr[0] = c < 2u ? (c ? z.xd : z.x) : (c == 2u ? z.th : z.thd);
                tr += 4 * p.n;
            }
            {
                constexpr uint32_t kMine = (1u << E) - 1u;
                const uint32_t half = (k >> 5) & 1u;
                if (lane == 0u) s_bits[half][k & 31u][warp] = (dm & kMine) | (am & kMine) << 16;
                if ((k & 31u) == 31u || k + 1u == p.T) {
                    // all warps of the CTA get here after the same step; the other half of s_bits is
                    // only written again once every warp has passed the next such barrier
                    __syncthreads();
                    const uint32_t row0 = k & ~31u, rows = (k & 31u) + 1u;
                    if (threadIdx.x < rows) {
                        uint32_t d = 0u, a = 0u;
#pragma unroll
                        for (int w = 0; w < W; ++w) {
                            const uint32_t b = s_bits[half][threadIdx.x][w];
                            d |= (b & 0xffffu) << (w * E);
                            a |= (b >> 16) << (w * E);
                        }
                        const int64_t word = (int64_t)(row0 + threadIdx.x) * words + blockIdx.x;
                        if (p.done_bits) p.done_bits[word] = d;
                        if (p.action_bits) p.action_bits[word] = a;
                    }
                    const int64_t env = (int64_t)blockIdx.x * 32 + lane;
                    if (p.reward_stream && env < p.n)
                        for (uint32_t r = warp; r < rows; r += W) p.reward_stream[(int64_t)(row0 + r) * p.n + env] = 1.0f;
                }
            }
        }
    };
    uint32_t k = 0u;
    if (p.start_in) {
        for (; k < p.T; ++k) step(std::true_type{}, k);
    } else if (p.init_planes && p.T) {
        step(std::true_type{}, k++);
    }
    for (; k < p.T; ++k) step(std::false_type{}, k);

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
    constexpr int W = kLaneWarps<G, STREAMS>;
    const int64_t per_cta = W * (32 / G);
    const int64_t grid = (p.n + per_cta - 1) / per_cta;
    if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    rollout_lanes_kernel<NET, G, STREAMS, CONTRACT><<<(unsigned)grid, 32 * W, 0, s>>>(p);
    count_launch();
    return cudaGetLastError();
}

template <int NET, bool STREAMS, bool CONTRACT>
cudaError_t launch_lanes_g(RolloutParams &p, int g, cudaStream_t s) {
    if constexpr (STREAMS)  // rollout_lanes_for: four lanes wherever per-step outputs are written
        return launch_lanes_one<NET, 4, true, CONTRACT>(p, s);
    else
        return g == 4 ? launch_lanes_one<NET, 4, false, CONTRACT>(p, s) : launch_lanes_one<NET, 8, false, CONTRACT>(p, s);
}

template <int NET, bool CONTRACT>
cudaError_t launch_lanes_net(RolloutParams &p, int g, bool streams, cudaStream_t s) {
    return streams ? launch_lanes_g<NET, true, CONTRACT>(p, g, s) : launch_lanes_g<NET, false, CONTRACT>(p, g, s);
}

}  // namespace

}  // namespace cp
