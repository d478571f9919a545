// One step whose outputs lie in page-locked HOST memory (cp_step_host on batches beyond the ones that a kernel reads
// from there too): a CTA computes kEnvs environments from device memory, leaves their new states and
// done flags in shared memory and stores each plane's stretch by whole 128-byte lines.
//
// What bounds it is the way to host memory: every 128-byte store of a warp that does not start on a line crosses the bus as
// two, and rows of an odd number of environments start anywhere. By lines only the ends of a CTA's stretches do.
#include "cartpole_device.cuh"
#include "cartpole_internal.h"

namespace cp {

namespace {

constexpr int kThreads = 256, kPer = 4, kEnvs = kThreads * kPer;

}  // namespace

__global__ void __launch_bounds__(kThreads) step_host_kernel(const __grid_constant__ StepParams p) {
    __shared__ float s_state[4][kEnvs];
    __shared__ uint8_t s_done[kEnvs];
    const int64_t first = (int64_t)blockIdx.x * kEnvs;
    const int count = (int)min((int64_t)kEnvs, p.n - first);
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int at = k * kThreads + threadIdx.x;
        if (at >= count) break;
        const int64_t i = first + at;
        const uint32_t env = p.env_offset + (uint32_t)i;
        State z = {p.in[i], p.in[p.in_stride + i], p.in[2 * p.in_stride + i], p.in[3 * p.in_stride + i]};
        const uint32_t sb = p.action ? (p.action[i] ? 0x80000000u : 0u) : action_signbit(make_keys(p.salt_a, env), p.t);
        const bool d = euler_step(z, force_from_signbit(sb));
        if (d) z = start_state(make_keys(p.salt_r, env), p.t + 1u);
        s_state[0][at] = z.x;
        s_state[1][at] = z.xd;
        s_state[2][at] = z.th;
        s_state[3][at] = z.thd;
        s_done[at] = d ? 1 : 0;
    }
    __syncthreads();
    // thread k's element of a plane: the one that lies k places (mod kThreads) after the line the stretch begins in
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        float *out = q < 4 ? p.out + q * p.out_stride + first : p.reward + first;
        const int into = (int)(reinterpret_cast<uintptr_t>(out) >> 2 & 31u);
        for (int at = (int)threadIdx.x - into; at < count; at += kThreads)
            if (at >= 0) out[at] = q < 4 ? s_state[q < 4 ? q : 0][at] : 1.0f;
    }
    uint8_t *out = p.done + first;
    const int into = (int)(reinterpret_cast<uintptr_t>(out) & 127u);
    for (int at = (int)threadIdx.x * 4 - into; at < count; at += kThreads * 4) {
        if (at >= 0 && at + 4 <= count) {
            *reinterpret_cast<uint32_t *>(out + at) =
                (uint32_t)s_done[at] | (uint32_t)s_done[at + 1] << 8 | (uint32_t)s_done[at + 2] << 16 | (uint32_t)s_done[at + 3] << 24;
        } else {
            for (int b = 0; b < 4; ++b)
                if (at + b >= 0 && at + b < count) out[at + b] = s_done[at + b];
        }
    }
}

// reward and done must not be null; ep_len is not looked at.
cudaError_t launch_step_host(const StepParams &p, cudaStream_t s) {
    const int64_t grid = (p.n + kEnvs - 1) / kEnvs;
    if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    step_host_kernel<<<(unsigned)grid, kThreads, 0, s>>>(p);
    count_launch();
    return cudaGetLastError();
}

}  // namespace cp
