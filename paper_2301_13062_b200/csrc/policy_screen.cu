// Host side of the network policies' screen (policy_screen.cuh): the layouts the kernels read, with the bound
// of a policy's estimate (policy_bound.h), and the self-test of the special-function unit's tanh.
#include "policy_bound.h"
#include "policy_screen.cuh"

namespace cp {

namespace {

template <int NET>
void screen(RolloutParams &p, float *steps, int rounds) {
    const PolicyBound b = policy_bound(p.w, NetShape<NET>::H, NetShape<NET>::kDeep, rounds, steps);
    p.screen_base = b.base;
    p.screen_bound = b.bound;
}

template <int NET>
void units(RolloutParams &p) {
    using S = NetShape<NET>;
    constexpr int H = S::H;
    screen<NET>(p, p.w + S::kUnitSteps, units_rounds(H, S::kDeep));
    for (int j = 0; j < H; ++j)
        for (int i = 0; i < 5; ++i) p.w[S::kUnitFirst + 10 * (j / 2) + 2 * i + j % 2] = p.w[i < 4 ? 4 * j + i : 4 * H + j];
}

template <int NET>
void bound_alone(RolloutParams &p, int lanes) {
    constexpr int H = NetShape<NET>::H;
    float steps[H];
    screen<NET>(p, steps, lanes_rounds(H, lanes));
}

}  // namespace

void screen_units(RolloutParams &p, int policy) {
    switch (policy) {
        case 2: return units<2>(p);
        case 4: return units<4>(p);
        case 5: return units<5>(p);
        default: return units<7>(p);
    }
}

void screen_bound(RolloutParams &p, int policy, int lanes) {
    switch (policy) {
        case 2: return bound_alone<2>(p, lanes);
        case 4: return bound_alone<4>(p, lanes);
        case 5: return bound_alone<5>(p, lanes);
        default: return bound_alone<7>(p, lanes);
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
