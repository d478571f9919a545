#include "cartpole_device.cuh"
#include "cartpole_internal.h"

namespace cp {

// The fused step (step_kernel.cu) for large batches whose planes cannot be accessed as float4 (a
// plain [4, n] array with n not a multiple of 4: every plane starts at another offset from 16
// bytes). A warp owns
// kStrided * 32 consecutive environments, lane l those at l, l + 32, ..., so that every access is one
// contiguous run of the warp, wherever the plane starts, and a thread has kStrided loads per plane
// in flight.
//
// Bound: HBM, as the float4 form (37 bytes per environment and step, 38 with supplied actions). The
// one-environment-per-thread form that used to serve these batches had a quarter of the bytes in
// flight and four times the CTAs: 5,000,011 environments in a [4, n] tensor 82.0 -> 33.0 us per launch
// (5.8 TB/s; float4 form on aligned planes 31.0), 16,777,217 280 -> 101 us, 1,048,577 18.3 -> 8.8 us.
constexpr int kStrided = 4;
__global__ void __launch_bounds__(256, 1) step_strided_kernel(const __grid_constant__ StepParams p) {
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t i0 = warp * (32 * kStrided) + (threadIdx.x & 31u);
    if (i0 >= p.n) return;
    const bool has_action = p.action != nullptr;
    int64_t idx[kStrided];
    uint32_t sb[kStrided];
#pragma unroll
    for (int j = 0; j < kStrided; ++j) {
        idx[j] = i0 + 32 * j < p.n ? i0 + 32 * j : i0;  // past the end: repeat the thread's first one, store nothing
        sb[j] = has_action ? 0u : action_signbit(make_keys(p.salt_a, p.env_offset + (uint32_t)idx[j]), p.t);
    }
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
    State z[kStrided];
#pragma unroll
    for (int j = 0; j < kStrided; ++j)
        z[j] = {p.in[idx[j]], p.in[p.in_stride + idx[j]], p.in[2 * p.in_stride + idx[j]], p.in[3 * p.in_stride + idx[j]]};
    if (has_action) {
#pragma unroll
        for (int j = 0; j < kStrided; ++j) sb[j] = p.action[idx[j]] ? 0x80000000u : 0u;
    }
    uint32_t len[kStrided] = {};
    if (p.ep_len) {
#pragma unroll
        for (int j = 0; j < kStrided; ++j) len[j] = p.ep_len[idx[j]] + 1u;
    }
    uint32_t dmask = 0u;
#pragma unroll
    for (int j = 0; j < kStrided; ++j) {
        const bool d = euler_step(z[j], force_from_signbit(sb[j])) || (p.max_steps && len[j] >= p.max_steps);
        dmask |= (d ? 1u : 0u) << j;
    }
    // one restart per pass, as in the vector form
    uint32_t pending = dmask;
    while (pending) {
        const int j = __ffs(pending) - 1;
        pending &= pending - 1;
        const State r = start_state(make_keys(p.salt_r, p.env_offset + (uint32_t)(i0 + 32 * j)), p.t + 1u);
#pragma unroll
        for (int q = 0; q < kStrided; ++q)
            if (q == j) z[q] = r;
    }
#pragma unroll
    for (int j = 0; j < kStrided; ++j) {
        const int64_t i = i0 + 32 * j;
        if (i >= p.n) break;
        const bool d = (dmask >> j) & 1u;
        p.out[i] = z[j].x;
        p.out[p.out_stride + i] = z[j].xd;
        p.out[2 * p.out_stride + i] = z[j].th;
        p.out[3 * p.out_stride + i] = z[j].thd;
        if (p.ep_len) p.ep_len[i] = d ? 0u : len[j];
        if (p.reward) p.reward[i] = 1.0f;
        if (p.done) p.done[i] = d ? 1 : 0;
    }
}

cudaError_t launch_step_strided(const StepParams &p, cudaStream_t s) {
    const int block = g_tuning.step_block;
    const int64_t threads = (p.n + 32 * kStrided - 1) / (32 * kStrided) * 32;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((threads + block - 1) / block));
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = g_tuning.step_pdl;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, step_strided_kernel, p);
    count_launch();
    return e;
}

}  // namespace cp
