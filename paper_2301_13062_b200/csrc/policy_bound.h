// The bound of the network policies' estimate (policy_screen.cuh). Host arithmetic only, so that it is
// checked without a GPU.
#pragma once
#include <cmath>

namespace cp {

// Distance of the special-function unit's tanh (tanh_screen) from either arithmetic's tanh, at most, over every
// float32 (measured: 7.987e-6 for both, cp_selftest_screen).
constexpr double kTanhScreenError = 8.0e-6;

// Roundings that a term of the estimate goes through at most, in the kernels' orders.
// Units 2q and 2q + 1 of one lane side by side, a multiply-add per pair onto the base, then both halves' sum; a second
// hidden layer's units one after another (screen_estimate, screen_estimate_two).
constexpr int units_rounds(int units, bool deep) { return deep ? units : units / 2 + 1; }
// An environment's units spread over `lanes` lanes (rollout_lanes.cuh): with one or two lanes a pair of units per
// product or multiply-add and both halves' sum, with more one unit each; then a sum per doubling of the lanes and the base.
constexpr int lanes_rounds(int units, int lanes) {
    int rounds = (lanes <= 2 ? units / lanes / 2 + 1 : units / lanes) + 1;
    for (; lanes > 1; lanes /= 2) ++rounds;
    return rounds;
}

struct PolicyBound {
    float base;   // the estimate's constant term, b1 - b0
    float bound;  // largest distance of an estimate from l1 - l0; negative: every estimate that is not NaN decides
};

// w: the policy as the caller gave it: W1[units][4], b1[units], with a second hidden layer W2[units][units], b2[units],
// then the logits' W[2][units], b[2]. rounds: roundings that a term of the estimate goes through at most.
// steps[units] becomes w1[j] - w0[j].
//
// Let u = 2^-24 (half an ulp), h_j the activations of the definition (|h_j| <= 1), and v_j = w1[j] - w0[j].
//  * First layer: the estimate's arguments have the bits of the definition's (same operands, same
//    order), so |h~_j - h_j| <= E1 = kTanhScreenError, which covers both arithmetics' tanh
//    (cp_selftest_screen compares over every float32).
//  * A second hidden layer of n units sums in another order: both sums miss the exact one by at most
//    (n + 1) u (|b| + sum |w|), the operands differ by E1, and tanh does not stretch distances. The estimate's
//    tanh is within E1 of the definition's at the same argument, and the definition's at the two arguments within
//    their distance and twice its own miss of the real tanh, which is at most 2.4e-7 in either arithmetic
//    (cp_selftest_tanh), so that twice it is far below another E1: E2_k =
//    E1 sum_j |w2[k][j]| + 2 (n + 2) u (|b2[k]| + sum_j |w2[k][j]|) + 2 E1.
//  * A sum over h_j rounds each of its partial sums once. Those of a defined logit, left to right, are at
//    most |b_i| + |w_i[0]| + .. + |w_i[k]|, so the logit misses its exact sum by u times the sum of these over k.
//  * The estimate's order depends on the kernel; `rounds` says how many roundings a term goes through at
//    most, each of a partial sum of at most |b1 - b0| + sum |v_j|, two more for v_j and b1 - b0 themselves.
// Estimate and l1 - l0 then differ by at most the sum of all that and sum_j E_j |v_j|; 1/16 more for
// the second-order terms and this computation itself, and 1e-37 for results too small
// to be normal numbers. Weights of 1e30 and more in sum (or not finite) could overflow in the estimate where
// they do not in the logits: their bound is infinite.
// Logits of the same weights (a network whose last layer starts at zero) are the same sums of the same
// activations, so l1 > l0 never holds: the estimate, zero for all finite activations, decides without a bound. With
// the bound above it never did, and every step took the defined logits after it.
inline PolicyBound policy_bound(const float *w, int units, bool deep, int rounds, float *steps) {
    const double u = std::ldexp(1.0, -24), e1 = kTanhScreenError;
    const float *second = w + 5 * units, *logits = second + (deep ? units * (units + 1) : 0);
    double moved = 0.0, total = std::fabs((double)logits[2 * units]) + std::fabs((double)logits[2 * units + 1]), partial = 0.0;
    const double base = (double)logits[2 * units + 1] - (double)logits[2 * units];
    double span = std::fabs(base);
    bool same = base == 0.0;
    for (int j = 0; j < units; ++j) {
        double e = e1;
        if (deep) {
            double row = 0.0;
            for (int i = 0; i < units; ++i) row += std::fabs((double)second[units * j + i]);
            e = e1 * (row + 2.0) + 2.0 * (units + 2) * u * (row + std::fabs((double)second[units * units + j]));
        }
        const double v = (double)logits[units + j] - (double)logits[j];
        steps[j] = (float)v;
        same = same && v == 0.0;
        moved += e * std::fabs(v);
        span += std::fabs(v);
        total += std::fabs((double)logits[j]) + std::fabs((double)logits[units + j]);
        partial += total;
    }
    if (same && total < 1e30) return {0.0f, -1.0f};
    const double bound = 1.0625 * (moved + (rounds + 2) * u * span + u * partial) + 1e-37;
    return {(float)base, bound < 1e30 && total < 1e30 ? std::nextafterf((float)bound, INFINITY) : INFINITY};
}

}  // namespace cp
