// The shared network policies decide an action by the larger of two logits, and the logits
// themselves go nowhere. So every kernel first takes an estimate of l1 - l0 that is cheap and has
// a proven bound on its distance from the defined logits' difference: where it is larger than the
// bound, its sign is the action. Only where it is not are the defined logits computed, in their
// defined order, by the environment that needs them. The actions are those of the definition,
// always; what changes is how many operations most of them take.
//
//   estimate = (b1 - b0) + sum_j (w1[j] - w0[j]) * h~_j     h~_j: the special-function unit's tanh
//
// One result of that unit per hidden unit instead of two, no polynomial beside it, one
// multiply-add instead of two, and no order to keep. The bound (policy_bound, in policy_bound.h)
// grows with the weights and with kTanhScreenError; with the weight distributions of inputs.py it
// sends one to two environments in 10,000 steps to the defined logits, at most one in 1,000.
//
// NaN anywhere makes the comparison with the bound fail, which sends the environment to the defined
// logits; so do weights beyond the range the bound was derived for (its bound is infinite then).
#pragma once
#include "cartpole_device.cuh"
#include "cartpole_internal.h"

namespace cp {

// tanh by the special-function unit, one instruction. Its distance from either arithmetic's tanh is at
// most kTanhScreenError (policy_bound.h) over every float32 (measured: 7.987e-6 for both, cp_selftest_screen).
__device__ __forceinline__ float tanh_screen(float x) {
    float r;
    asm("tanh.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ f32x2 tanh_screen2(f32x2 x) {
    float a, b;
    unpack2(x, a, b);
    return pack2(tanh_screen(a), tanh_screen(b));
}

// The shared tanh networks: 2 (4-16-2), 4 (4-32-2), 5 (4-64-2), 7 (4-16-16-2).
__host__ __device__ constexpr bool is_network(int policy) { return policy == 2 || policy == 4 || policy == 5 || policy == 7; }

template <int NET>
struct NetShape {
    static constexpr int H = NET == 4 ? 32 : NET == 5 ? 64 : 16;
    static constexpr bool kDeep = NET == 7;
    // floats before the second hidden layer, and before the logits (W[2][H], b[2]), as the caller gives them
    static constexpr int kSecond = 5 * H;
    static constexpr int kLogits = kSecond + (kDeep ? H * (H + 1) : 0);
    static constexpr int kCount = kLogits + 2 * H + 2;
    // RolloutParams::w (screen_units): the caller's weights, the first layer again with the weights of units
    // 2q and 2q + 1 side by side (input 0, .., input 3, bias), then w1[j] - w0[j]
    static constexpr int kUnitFirst = kCount, kUnitSteps = kUnitFirst + 5 * H;
    static_assert(kUnitSteps + H <= kMaxPolicyFloats, "RolloutParams::w holds the layout");
    static_assert(kUnitFirst % 2 == 0 && kUnitSteps % 2 == 0, "pairs are read as such");
};

// The action by the defined logits: every sum left to right from its bias. w: the hidden layers' weights; logits:
// W[2][H], b[2]. Two units at a time, whose tanhs share their instructions;
// few environments come here, so the code is kept short: loops over the units, not unrolled.
template <int NET, bool CONTRACT>
__device__ __forceinline__ uint32_t defined_action(const float *w, const float *logits, const State &z) {
    using S = NetShape<NET>;
    constexpr int H = S::H;
    auto first = [&](int j) {
        float acc = w[4 * H + j];
        acc = __fmaf_rn(w[4 * j + 0], z.x, acc);
        acc = __fmaf_rn(w[4 * j + 1], z.xd, acc);
        acc = __fmaf_rn(w[4 * j + 2], z.th, acc);
        return __fmaf_rn(w[4 * j + 3], z.thd, acc);
    };
    auto tanh2 = [](float a, float b, float &ha, float &hb) {
        const f32x2 v = pack2(a, b);
        unpack2(CONTRACT ? tanh_contracted_pair(v) : tanh_pair(v), ha, hb);
    };
    float l0 = logits[2 * H], l1 = logits[2 * H + 1];
    auto logit_terms = [&](int j, float a, float b) {  // of units j and j + 1
        float ha, hb;
        tanh2(a, b, ha, hb);
        l0 = __fmaf_rn(logits[j], ha, l0);
        l1 = __fmaf_rn(logits[H + j], ha, l1);
        l0 = __fmaf_rn(logits[j + 1], hb, l0);
        l1 = __fmaf_rn(logits[H + j + 1], hb, l1);
    };
    if constexpr (S::kDeep) {
        const float *w2 = w + S::kSecond, *b2 = w2 + H * H;
        float h1[H];
#pragma unroll
        for (int j = 0; j < H; j += 2) tanh2(first(j), first(j + 1), h1[j], h1[j + 1]);
#pragma unroll 1
        for (int k = 0; k < H; k += 2) {
            float a = b2[k], b = b2[k + 1];
#pragma unroll
            for (int j = 0; j < H; ++j) {
                a = __fmaf_rn(w2[H * k + j], h1[j], a);
                b = __fmaf_rn(w2[H * (k + 1) + j], h1[j], b);
            }
            logit_terms(k, a, b);
        }
    } else {
#pragma unroll 2
        for (int j = 0; j < H; j += 2) logit_terms(j, first(j), first(j + 1));
    }
    return (l1 > l0) ? 0x80000000u : 0u;
}

// Estimate for one environment, two hidden units per packed operation, from the layout of screen_units.
template <int NET>
__device__ __forceinline__ float screen_estimate(const float *w, float base, const State &z) {
    using S = NetShape<NET>;
    constexpr int H = S::H;
    const f32x2 *first = reinterpret_cast<const f32x2 *>(w + S::kUnitFirst);
    const f32x2 x = splat2(z.x), xd = splat2(z.xd), th = splat2(z.th), thd = splat2(z.thd);
    auto units = [&](int q) {  // 2q and 2q + 1
        f32x2 acc = first[5 * q + 4];
        acc = fma2(first[5 * q + 0], x, acc);
        acc = fma2(first[5 * q + 1], xd, acc);
        acc = fma2(first[5 * q + 2], th, acc);
        acc = fma2(first[5 * q + 3], thd, acc);
        return tanh_screen2(acc);
    };
    float lo, hi;
    if constexpr (S::kDeep) {
        const f32x2 *w2 = reinterpret_cast<const f32x2 *>(w + S::kSecond);
        const float *b2 = w + S::kSecond + H * H, *steps = w + S::kUnitSteps;
        f32x2 h1[H / 2];
#pragma unroll
        for (int q = 0; q < H / 2; ++q) h1[q] = units(q);
        float est = base;
#pragma unroll
        for (int k = 0; k < H; ++k) {
            f32x2 acc = pack2(b2[k], 0.0f);
#pragma unroll
            for (int q = 0; q < H / 2; ++q) acc = fma2(w2[H / 2 * k + q], h1[q], acc);
            unpack2(acc, lo, hi);
            est = __fmaf_rn(steps[k], tanh_screen(__fadd_rn(lo, hi)), est);
        }
        return est;
    } else {
        const f32x2 *steps = reinterpret_cast<const f32x2 *>(w + S::kUnitSteps);
        f32x2 est = pack2(base, 0.0f);
#pragma unroll
        for (int q = 0; q < H / 2; ++q) est = fma2(steps[q], units(q), est);
        unpack2(est, lo, hi);
        return __fadd_rn(lo, hi);
    }
}

// Estimates for the two environments of a thread, from the same layout: every pair of weights is loaded once for both.
template <int NET>
__device__ __forceinline__ void screen_estimate_two(const float *w, float base, const State &a, const State &b, float (&e)[2]) {
    using S = NetShape<NET>;
    constexpr int H = S::H;
    static_assert(!S::kDeep, "one hidden layer");
    const f32x2 *first = reinterpret_cast<const f32x2 *>(w + S::kUnitFirst), *steps = reinterpret_cast<const f32x2 *>(w + S::kUnitSteps);
    const f32x2 za[4] = {splat2(a.x), splat2(a.xd), splat2(a.th), splat2(a.thd)};
    const f32x2 zb[4] = {splat2(b.x), splat2(b.xd), splat2(b.th), splat2(b.thd)};
    f32x2 ea = pack2(base, 0.0f), eb = ea;
#pragma unroll
    for (int q = 0; q < H / 2; ++q) {
        f32x2 ha = first[5 * q + 4], hb = ha;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const f32x2 v = first[5 * q + i];
            ha = fma2(v, za[i], ha);
            hb = fma2(v, zb[i], hb);
        }
        const f32x2 v = steps[q];
        ea = fma2(v, tanh_screen2(ha), ea);
        eb = fma2(v, tanh_screen2(hb), eb);
    }
    float lo, hi;
    unpack2(ea, lo, hi);
    e[0] = __fadd_rn(lo, hi);
    unpack2(eb, lo, hi);
    e[1] = __fadd_rn(lo, hi);
}

// Does the estimate decide? (false for NaN, and for every estimate where the bound is infinite)
__device__ __forceinline__ bool screen_decides(float estimate, float bound) { return fabsf(estimate) > bound; }
__device__ __forceinline__ uint32_t screen_action(float estimate) { return estimate > 0.0f ? 0x80000000u : 0u; }

}  // namespace cp
