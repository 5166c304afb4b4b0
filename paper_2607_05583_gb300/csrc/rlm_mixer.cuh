// rlm_mixer.cuh -- device helpers of the mixer wrapper (Sec. 3.4) shared by its
// kernels.
#pragma once

#include <cuda_runtime.h>

namespace rlm {

// The gate sigma(v) = 1 / (1 + e^-v).
__device__ __forceinline__ float gatef(float v) { return __fdividef(1.0f, 1.0f + __expf(-v)); }

// Head coupling: C = I + (lambda_c / sqrt(H)) tanh(c_raw), H x H row-major, built
// by the calling block's threads (the caller synchronises before reading it).
__device__ __forceinline__ void build_coupling(float *C, const float *c_raw, float lam, int H) {
    const float k = lam * rsqrtf((float)H);
    for (int i = threadIdx.x; i < H * H; i += blockDim.x)
        C[i] = (i / H == i % H ? 1.0f : 0.0f) + k * tanhf(c_raw[i]);
}

// The same in two parts, for a kernel that issues other loads between them: a matrix of more
// entries than the block has threads is requested whole, without registers, and each
// entry then turned in place by the thread that requested it; a smaller one is read in
// the second part: straight, or in the same loop (kLoop), which is smaller and faster in the
// 512-thread instance of the decode step only (B = 128, D = 256, M = 16, H = 8 3.08 us a step against
// 3.27; B = 1 2.12 against 2.05, B = 4, H = 32 3.5 against 3.4, H = 64 7.0 against 6.6).  (With one
// load after the other / entries kept in registers / this: H = 64 8.3 / 6.3 / 6.6, H = 32 3.9 / 3.3 / 3.4,
// H = 8 at B = 64 2.82 / 2.94 / 2.68.)
__device__ __forceinline__ void request_coupling(float *C, const float *c_raw, int H) {
    if (H * H <= blockDim.x) return;
    for (int i = threadIdx.x; i < H * H; i += blockDim.x)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(C + i)),
                     "l"(c_raw + i)
                     : "memory");
}
template <bool kLoop>
__device__ __forceinline__ void finish_coupling(float *C, const float *c_raw, float lam, int H) {
    const bool small = H * H <= blockDim.x;
    const float k = lam * rsqrtf((float)H);
    auto entry = [&](int i, float raw) { C[i] = (i / H == i % H ? 1.0f : 0.0f) + k * tanhf(raw); };
    if (kLoop) {
        if (!small) asm volatile("cp.async.wait_all;" ::: "memory");
        const float *src = small ? c_raw : C;
        for (int i = threadIdx.x; i < H * H; i += blockDim.x) entry(i, src[i]);
    } else if (small) {
        if (threadIdx.x < H * H) entry(threadIdx.x, c_raw[threadIdx.x]);
    } else {
        asm volatile("cp.async.wait_all;" ::: "memory");
        for (int i = threadIdx.x; i < H * H; i += blockDim.x) entry(i, C[i]);
    }
}

}  // namespace rlm
