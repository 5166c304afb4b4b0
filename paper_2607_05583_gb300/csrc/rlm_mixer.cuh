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
// the second part.  (Decode steps, us, with one load after the other / entries kept in registers /
// this: H = 64 8.3 / 6.3 / 7.0, H = 32 3.9 / 3.3 / 3.6, H = 8 at B = 64 2.82 / 2.94 / 2.70.)
__device__ __forceinline__ void request_coupling(float *C, const float *c_raw, int H) {
    if (H * H <= blockDim.x) return;
    for (int i = threadIdx.x; i < H * H; i += blockDim.x)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(C + i)),
                     "l"(c_raw + i)
                     : "memory");
}
__device__ __forceinline__ void finish_coupling(float *C, const float *c_raw, float lam, int H) {
    const bool small = H * H <= blockDim.x;
    if (!small) asm volatile("cp.async.wait_all;" ::: "memory");
    const float *src = small ? c_raw : C;
    const float k = lam * rsqrtf((float)H);
    for (int i = threadIdx.x; i < H * H; i += blockDim.x) C[i] = (i / H == i % H ? 1.0f : 0.0f) + k * tanhf(src[i]);
}

}  // namespace rlm
