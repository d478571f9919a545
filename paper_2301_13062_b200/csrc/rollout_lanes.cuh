// Rollout under a shared tanh network with the network of an environment spread over G lanes
// (paper Sec. VI: fusing simulation with neural network inference), for batches too small to fill
// the chip.
//
// One lane per environment evaluates the hidden units one after another; with a few warps per
// scheduler nothing hides that, and a step of a 4-64-2 network takes 2,250 cycles although its
// longest dependency chain is a fifth of that. Here lane = g * E + e: the G lanes g of environment e
// (E = 32 / G environments per warp)
//   * all hold the state and all step it (the same instructions for every lane: no cost);
//   * evaluate H / G hidden units each, side by side, their weights in registers;
//   * exchange the activations through a row of shared memory per environment, and all run the two
//     logit chains (whose order is part of the definition; they are what bounds the step now).
// Every operation is the scalar one of mlp_action / mlp_deep_action on the same operands in the same
// order, so the action has the same bits. (Two units or both logits per packed operation halve the
// issue slots but measured slower: latency is what is paid here, and a packed operation's is longer.)
// The start state an environment would continue from is hashed on every step ahead of the network,
// by four lanes, one component each: that work fills issue slots the chains leave empty, and a
// finished environment just takes it.
//
// Warps only exchange data when bit planes are written: the G warps of a CTA then hold the 32
// environments of one bit-plane word, leave their bits of 32 steps in shared memory and write the
// words together. All of a CTA's warps make the same T steps, so they meet the same barriers.
#pragma once
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

// A layer's weights of one lane. The layer's units come in BLOCKS equal runs, each run shared out to
// the G lanes, U units each: unit (block * G + g) * U + u.
template <int U, int BLOCKS, int IN>
struct LaneLayer {
    float w[BLOCKS][U][IN], b[BLOCKS][U];
    // layer: w[units][IN] then b[units], as the caller gave them
    __device__ __forceinline__ void load(const float *layer, int units, int lanes, uint32_t g) {
#pragma unroll
        for (int k = 0; k < BLOCKS; ++k) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int unit = (k * lanes + (int)g) * U + u;
#pragma unroll
                for (int i = 0; i < IN; ++i) w[k][u][i] = in_register(layer[unit * IN + i]);
                b[k][u] = in_register(layer[units * IN + unit]);
            }
        }
    }
    // activations of this lane's units of one block from the inputs, left at `mine`
    template <bool CONTRACT>
    __device__ __forceinline__ void run(int k, const float (&in)[IN], float *mine) const {
        float h[U];
#pragma unroll
        for (int u = 0; u < U; ++u) h[u] = b[k][u];
#pragma unroll
        for (int i = 0; i < IN; ++i) {
#pragma unroll
            for (int u = 0; u < U; ++u) h[u] = __fmaf_rn(w[k][u][i], in[i], h[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) h[u] = CONTRACT ? tanh_contracted(h[u]) : tanh_canonical(h[u]);
        if constexpr (U % 4 == 0) {
#pragma unroll
            for (int u = 0; u < U; u += 4) *reinterpret_cast<float4 *>(mine + u) = make_float4(h[u], h[u + 1], h[u + 2], h[u + 3]);
        } else if constexpr (U == 2) {
            *reinterpret_cast<float2 *>(mine) = make_float2(h[0], h[1]);
        } else {
            mine[0] = h[0];
        }
    }
};
template <int NET, int G>
struct LaneNetwork {
    using S = NetShape<NET>;
    static constexpr int BLOCKS = S::H >= 64 ? 2 : 1;  // (measured slower with 32 units: the halves are too short)
    static constexpr int U = S::H / G / BLOCKS;
    LaneLayer<U, BLOCKS, 4> first;
    LaneLayer<S::kDeep ? U : 1, 1, S::kDeep ? S::H : 1> second;  // unused unless the network is deep
    float out[S::H], bias;                                       // this lane's logit: even lanes 0, odd lanes 1
    __device__ __forceinline__ void load(const RolloutParams &p, uint32_t g) {
        first.load(p.w, S::H, G, g);
        if constexpr (S::kDeep) second.load(p.w + S::kSecond, S::H, G, g);
        const float *logits = p.w + S::kLogits;
#pragma unroll
        for (int j = 0; j < S::H; ++j) out[j] = in_register(logits[(g & 1u) * S::H + j]);
        bias = in_register(logits[2 * S::H + (g & 1u)]);
    }
};

// Floats per environment's row: 16 bytes more than the activations, so that the 16-byte reads of
// up to eight environments' rows fall into different banks.
template <int H>
constexpr int kRow = H + 4;

template <int NET, int G, bool CONTRACT>
__device__ __forceinline__ uint32_t lanes_action(const LaneNetwork<NET, G> &net, const State &z, float *row, uint32_t g) {
    using S = NetShape<NET>;
    using N = LaneNetwork<NET, G>;
    constexpr int H = S::H, PER = H / N::BLOCKS;  // units per block
    const float obs[4] = {z.x, z.xd, z.th, z.thd};
    float h[PER];
    auto read_block = [&](int k) {
        __syncwarp();
#pragma unroll
        for (int j = 0; j < PER; j += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(row + k * PER + j);
            h[j] = v.x;
            h[j + 1] = v.y;
            h[j + 2] = v.z;
            h[j + 3] = v.w;
        }
    };
    net.first.template run<CONTRACT>(0, obs, row + (int)g * N::U);
    if constexpr (S::kDeep) {
        read_block(0);
        __syncwarp();  // the row is read before the next layer overwrites it
        net.second.template run<CONTRACT>(0, h, row + (int)g * N::U);
    }
    float mine = net.bias;
#pragma unroll
    for (int k = 0; k < N::BLOCKS; ++k) {
        read_block(k);
        // the next block's units do not depend on this block's part of the chain: they overlap
        if (k + 1 < N::BLOCKS) net.first.template run<CONTRACT>(k + 1, obs, row + (k + 1) * PER + (int)g * N::U);
#pragma unroll
        for (int j = 0; j < PER; ++j) mine = __fmaf_rn(net.out[k * PER + j], h[j], mine);
    }
    __syncwarp();  // the row is read before the next step overwrites it
    const float other = __shfl_xor_sync(0xffffffffu, mine, 32 / G);  // the neighbouring lane of the environment
    const bool right = (g & 1u) ? mine > other : other > mine;
    return right ? 0x80000000u : 0u;
}

// Warps of a CTA: one per scheduler, and as many as hold the 32 environments of a bit-plane word
// where such words are written by several warps.
template <int G, bool STREAMS>
constexpr int kLaneWarps = STREAMS ? G : 4;

// NET: 2 (4-16-2), 4 (4-32-2), 5 (4-64-2), 7 (4-16-16-2). G: lanes per environment. STREAMS: any
// combination of the per-step outputs. Step limit, supplied start states and caller's initial states
// are run-time options: next to a network's evaluation their tests cost nothing.
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

    for (uint32_t k = 0; k < p.T; ++k) {
        const uint32_t t1 = p.t0 + k + 1u;
        float fresh;
        if (start) {
            fresh = __ldg(start);
            start += 4 * p.n;
        } else {
            fresh = start_component_folded(kr, fold16(4u * t1), c);
        }
        const uint32_t sb = lanes_action<NET, G, CONTRACT>(net, z, row, g);
        const float force = force_from_signbit(sb);
        // a caller's states may hold any angle: its initial ones on the first step, supplied start states always
        bool done;
        if (p.start_in || (k == 0u && p.init_planes))
            done = CONTRACT ? euler_step_contracted<false>(z, force) : euler_step<false>(z, force);
        else
            done = CONTRACT ? euler_step_contracted<true>(z, force) : euler_step<true>(z, force);
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
    if constexpr (STREAMS) {  // rollout_lanes_for: four lanes wherever per-step outputs are written
        return launch_lanes_one<NET, 4, true, CONTRACT>(p, s);
    } else if constexpr (NetShape<NET>::H >= 32) {
        if (g == 16) return launch_lanes_one<NET, 16, STREAMS, CONTRACT>(p, s);
    }
    if constexpr (!STREAMS)
        return g == 4 ? launch_lanes_one<NET, 4, false, CONTRACT>(p, s) : launch_lanes_one<NET, 8, false, CONTRACT>(p, s);
}

template <int NET, bool CONTRACT>
cudaError_t launch_lanes_net(RolloutParams &p, int g, bool streams, cudaStream_t s) {
    return streams ? launch_lanes_g<NET, true, CONTRACT>(p, g, s) : launch_lanes_g<NET, false, CONTRACT>(p, g, s);
}

}  // namespace

}  // namespace cp
