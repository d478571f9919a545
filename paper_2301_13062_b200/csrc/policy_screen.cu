// Host side of the network policies' screen (policy_screen.cuh): the bound of a policy's estimate,
// the layouts the kernels read, and the self-test of the special-function unit's tanh.
#include "policy_screen.cuh"

#include <cmath>
#include <cstring>

namespace cp {

namespace {

// The bound. Let u = 2^-24 (half an ulp), h_j the activations of the definition (|h_j| <= 1), and
// v_j = w1[j] - w0[j].
//  * First layer: the estimate's arguments have the bits of the definition's (same operands, same
//    order), so |h~_j - h_j| <= E1 = kTanhScreenError, which covers both arithmetics' tanh
//    (cp_selftest_screen compares over every float32).
//  * A second hidden layer of n units sums in another order: both sums miss the exact one by at most
//    (n + 1) u (|b| + sum |w|), the operands differ by E1, tanh does not stretch distances, and the
//    definition's own tanh misses the real one by less than E1: E2_k = E1 sum_j |w2[k][j]| +
//    2 (n + 2) u (|b2[k]| + sum_j |w2[k][j]|) + 2 E1.
//  * A sum over h_j rounds each of its partial sums once. Those of a defined logit, left to right, are at
//    most |b_i| + |w_i[0]| + .. + |w_i[k]|, so the logit misses its exact sum by u times the sum of these over k.
//  * The estimate's order depends on the kernel; `rounds` says how many roundings a term goes through at
//    most, each of a partial sum of at most |b1 - b0| + sum |v_j|, two more for v_j and b1 - b0 themselves.
// Estimate and l1 - l0 then differ by at most the sum of all that and sum_j E_j |v_j|; 1/16 more for
// the second-order terms and this computation itself, and 1e-37 for results too small
// to be normal numbers. Weights of 1e30 and more in sum (or not finite) could overflow in the estimate where
// they do not in the logits: their bound is infinite.
template <int NET>
void screen(RolloutParams &p, float *steps, int rounds) {
    using S = NetShape<NET>;
    constexpr int H = S::H;
    const double u = std::ldexp(1.0, -24), e1 = kTanhScreenError;
    const float *logits = p.w + S::kLogits;
    double moved = 0.0, total = std::fabs((double)logits[2 * H]) + std::fabs((double)logits[2 * H + 1]), partial = 0.0;
    const double base = (double)logits[2 * H + 1] - (double)logits[2 * H];
    double span = std::fabs(base);
    for (int j = 0; j < H; ++j) {
        double e = e1;
        if (S::kDeep) {
            double row = 0.0;
            for (int i = 0; i < H; ++i) row += std::fabs((double)p.w[S::kSecond + H * j + i]);
            e = e1 * (row + 2.0) + 2.0 * (H + 2) * u * (row + std::fabs((double)p.w[S::kSecond + H * H + j]));
        }
        const double v = (double)logits[H + j] - (double)logits[j];
        steps[j] = (float)v;
        moved += e * std::fabs(v);
        span += std::fabs(v);
        total += std::fabs((double)logits[j]) + std::fabs((double)logits[H + j]);
        partial += total;
    }
    const double bound = 1.0625 * (moved + (rounds + 2) * u * span + u * partial) + 1e-37;
    p.screen_base = (float)base;
    p.screen_bound = bound < 1e30 && total < 1e30 ? std::nextafter((float)bound, INFINITY) : INFINITY;
}

template <int NET>
void pairs(RolloutParams &p) {
    using S = NetShape<NET>;
    constexpr int H = S::H;
    float steps[H];
    screen<NET>(p, steps, H);
    std::memmove(p.w + S::kPairLogits, p.w + S::kLogits, (2 * H + 2) * sizeof(float));
    for (int i = S::kLogits - 1; i >= 0; --i) p.w[2 * i] = p.w[2 * i + 1] = p.w[i];
    for (int j = 0; j < H; ++j) p.w[S::kPairSteps + 2 * j] = p.w[S::kPairSteps + 2 * j + 1] = steps[j];
}

template <int NET>
void units(RolloutParams &p) {
    using S = NetShape<NET>;
    constexpr int H = S::H;
    screen<NET>(p, p.w + S::kUnitSteps, S::kDeep ? H : H / 2 + 1);
    for (int j = 0; j < H; ++j)
        for (int i = 0; i < 5; ++i) p.w[S::kUnitFirst + 10 * (j / 2) + 2 * i + j % 2] = p.w[i < 4 ? 4 * j + i : 4 * H + j];
}

template <int NET>
void bound_alone(RolloutParams &p) {  // four or eight lanes: H / 4 or H / 8 terms, two or three shuffles, the base
    float steps[NetShape<NET>::H];
    screen<NET>(p, steps, NetShape<NET>::H / 4 + 3);
}

}  // namespace

void screen_pairs(RolloutParams &p, int policy) {
    switch (policy) {
        case 2: return pairs<2>(p);
        case 4: return pairs<4>(p);
        case 5: return pairs<5>(p);
        default: return pairs<7>(p);
    }
}

void screen_units(RolloutParams &p, int policy) {
    switch (policy) {
        case 2: return units<2>(p);
        case 4: return units<4>(p);
        case 5: return units<5>(p);
        default: return units<7>(p);
    }
}

void screen_bound(RolloutParams &p, int policy) {
    switch (policy) {
        case 2: return bound_alone<2>(p);
        case 4: return bound_alone<4>(p);
        case 5: return bound_alone<5>(p);
        default: return bound_alone<7>(p);
    }
}

// ---- self-test: tanh of the special-function unit against the tanhs of the definition ----
// Over every float32: out[0] largest |tanh_screen - tanh_canonical| and out[1] largest
// |tanh_screen - tanh_contracted|, in units of 1e-12; out[2] += values for which one of the three is
// NaN and another is not.
__global__ void screen_selftest_kernel(unsigned long long *out) {
    double worst[2] = {0.0, 0.0};
    unsigned long long odd = 0;
    for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < (1ull << 32); k += (uint64_t)gridDim.x * blockDim.x) {
        const float x = __uint_as_float((uint32_t)k);
        const float a = tanh_screen(x), b[2] = {tanh_canonical(x), tanh_contracted(x)};
        for (int i = 0; i < 2; ++i) {
            if (isnan(a) != isnan(b[i])) ++odd;
            else if (!isnan(a)) worst[i] = fmax(worst[i], fabs((double)a - (double)b[i]));
        }
    }
    unsigned long long m[2] = {(unsigned long long)(worst[0] * 1e12), (unsigned long long)(worst[1] * 1e12)};
    for (int o = 16; o > 0; o >>= 1) {
        for (int i = 0; i < 2; ++i) {
            const unsigned long long other = __shfl_down_sync(0xffffffffu, m[i], o);
            m[i] = other > m[i] ? other : m[i];
        }
        odd += __shfl_down_sync(0xffffffffu, odd, o);
    }
    if ((threadIdx.x & 31) == 0) {
        for (int i = 0; i < 2; ++i) atomicMax(out + i, m[i]);
        if (odd) atomicAdd(out + 2, odd);
    }
}

cudaError_t launch_screen_selftest(unsigned long long *out, cudaStream_t s) {
    screen_selftest_kernel<<<sm_count() * 8, 256, 0, s>>>(out);
    count_launch();
    return cudaGetLastError();
}

}  // namespace cp
