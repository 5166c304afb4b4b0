// rlm_short.cu -- sequences of at most 8 tokens on the CUDA cores (fp32 arithmetic): the
// recurrence itself (Eq. 4), a few lanes per (batch row, channel) that share its modes.
//
// A call is bound by the parameters' sines and exponentials, one set per (b, d, m), and by
// reading and writing states; the chunked scan (rlm_simt.cu) would fill one of its chunks of
// 64 positions to an eighth and build a table of powers besides.  Up to 8 tokens the
// recurrence is as exact (its lambda is applied 7 times at most; from 33 tokens on the scan's
// error is half of it).  GB300, us a call in fp32, three launches of chunked recurrences / the
// scan's wide tiles / this: forward from a state B = 8, L = 8, D = 256, M = 16 21 / 13 / 4.0, B = 64, L = 1,
// D = 2048, M = 1 23 / 147 / 3.8; backward (with its reduction) 21 / 17 / 5.6 and 31 / 271 / 12.7,
// B = 1, L = 1, D = 768, M = 33 17 / 53 / 5.0.
#include <type_traits>

#include "rlm_device.cuh"
#include "rlm_internal.h"

namespace rlm {
namespace {

constexpr int kLen = 8;
constexpr int kBlock = 128;

// A thread's place: channel d of batch row blockIdx.y, modes grp, grp + tpc, ...
struct Place {
    int d, grp, tpc;
    bool on;
};
__device__ __forceinline__ Place place(int D, int log2_tpc) {
    const int i = blockIdx.x * kBlock + threadIdx.x;
    return {i >> log2_tpc, i & ((1 << log2_tpc) - 1), 1 << log2_tpc, (i >> log2_tpc) < D};
}

// The sums over the modes' lanes, stored by the first one.
template <typename T>
__device__ __forceinline__ void store_sums(float (&acc)[kLen], const Place &p, T *out, int L, int D) {
#pragma unroll
    for (int t = 0; t < kLen; ++t) {
        if (t >= L) break;
        for (int o = p.tpc >> 1; o > 0; o >>= 1) acc[t] += __shfl_xor_sync(0xffffffffu, acc[t], o);
        if (p.on && p.grp == 0) st_elem(out + (int64_t)t * D, acc[t]);
    }
}

template <typename T>
__global__ void __launch_bounds__(kBlock) k_short_forward(
    const T *__restrict__ x, T *__restrict__ y, int L, int D, int M, int log2_tpc, const float *__restrict__ decay,
    const float *__restrict__ freq, const float *__restrict__ amp, const float *__restrict__ phase,
    const float2 *state_in, float2 *state_out, float4 *coef_out) {
    const Place p = place(D, log2_tpc);
    const int64_t b = blockIdx.y, at = b * L * D + p.d;
    float xv[kLen], acc[kLen];
#pragma unroll
    for (int t = 0; t < kLen; ++t) {
        xv[t] = p.on && t < L ? ld_elem(x + at + (int64_t)t * D) : 0.0f;
        acc[t] = 0.0f;
    }
    for (int m = p.grp; m < M && p.on; m += p.tpc) {
        const int pm = p.d * M + m;
        const int64_t sm = b * D * M + pm;
        const float ga = decay[pm], om = freq[pm];
        const float2 S0 = state_in ? state_in[sm] : make_float2(0.0f, 0.0f);
        const float2 lam = lambda_pow(ga, om, 1.0f), c = mode_coef(amp[pm], phase[pm]);
        float2 s = S0, l = make_float2(0.0f, 0.0f);   // from the entering state, and from zero
#pragma unroll
        for (int t = 0; t < kLen; ++t) {
            if (t >= L) break;
            s = cfma(lam, s, make_float2(xv[t], 0.0f));
            l = cfma(lam, l, make_float2(xv[t], 0.0f));
            acc[t] = fmaf(c.x, s.x, fmaf(-c.y, s.y, acc[t]));
        }
        if (state_out) state_out[sm] = state_in ? cfma(lambda_pow(ga, om, (float)L), S0, l) : l;
        if (coef_out && b == 0) coef_out[pm] = make_float4(lam.x, lam.y, c.x, c.y);
    }
    store_sums(acc, p, y + at, L, D);
}

// Reverse time: the adjoint S and its Jordan partner R, G = sum x S and P = sum x R of this
// row; with kG (a terminal-state gradient g) its second adjoint conj(g) lambda^(L-1-t) joins dx,
// and J = sum x_t (L-1-t) lambda^(L-1-t).  At token 0 the initial state's terms, as in the scan.
template <typename T, bool kG>
__global__ void __launch_bounds__(kBlock) k_short_backward(
    const T *__restrict__ dy, const T *__restrict__ x, T *__restrict__ dx, int L, int D, int M, int log2_tpc,
    const float *__restrict__ decay, const float *__restrict__ freq, const float *__restrict__ amp,
    const float *__restrict__ phase, const float2 *state_in, const float2 *g, float2 *d_state_in, float2 *part_g,
    float2 *part_p, float2 *part_j) {
    const Place p = place(D, log2_tpc);
    const int64_t b = blockIdx.y, at = b * L * D + p.d;
    const float2 z = make_float2(0.0f, 0.0f);
    float uv[kLen], xv[kLen], acc[kLen];
#pragma unroll
    for (int t = 0; t < kLen; ++t) {
        const bool in = p.on && t < L;
        uv[t] = in ? ld_elem(dy + at + (int64_t)t * D) : 0.0f;
        xv[t] = in ? ld_elem(x + at + (int64_t)t * D) : 0.0f;
        acc[t] = 0.0f;
    }
    for (int m = p.grp; m < M && p.on; m += p.tpc) {
        const int pm = p.d * M + m;
        const int64_t sm = b * D * M + pm;
        const float ga = decay[pm], om = freq[pm];
        const float2 gg = kG ? g[sm] : z, si = state_in ? state_in[sm] : z;
        const float2 lam = lambda_pow(ga, om, 1.0f), c = mode_coef(amp[pm], phase[pm]);
        float2 s = z, r = z, G = z, P = z;
        float2 phi = conj2(gg), U = make_float2(1.0f, 0.0f), Q = z, J = z;
#pragma unroll
        for (int t = kLen - 1; t >= 0; --t) {
            if (t >= L) continue;
            r = cmul(lam, make_float2(r.x + s.x, r.y + s.y));
            s = cfma(lam, s, make_float2(uv[t], 0.0f));
            acc[t] = fmaf(c.x, s.x, fmaf(-c.y, s.y, acc[t]));
            G = make_float2(fmaf(xv[t], s.x, G.x), fmaf(xv[t], s.y, G.y));
            P = make_float2(fmaf(xv[t], r.x, P.x), fmaf(xv[t], r.y, P.y));
            if (kG) {
                acc[t] += phi.x;
                J = make_float2(fmaf(xv[t], Q.x, J.x), fmaf(xv[t], Q.y, J.y));
                phi = cmul(lam, phi);
                Q = cmul(lam, make_float2(Q.x + U.x, Q.y + U.y));
                U = cmul(lam, U);
            }
        }
        const float2 ls = cmul(lam, s);   // lambda S_0
        const float2 lL = kG ? lambda_pow(ga, om, (float)L) : z;
        if (kG) J = cmul(conj2(gg), J);
        if (state_in) {
            G = cfma(si, ls, G);
            P = cfma(si, cmul(lam, make_float2(r.x + s.x, r.y + s.y)), P);
            if (kG) {
                const float2 ji = cmul(si, lL);
                J = cfma(conj2(gg), make_float2((float)L * ji.x, (float)L * ji.y), J);
            }
        }
        if (d_state_in) {
            float2 ds = conj2(cmul(c, ls));
            if (kG) ds = cfma(gg, conj2(lL), ds);
            d_state_in[sm] = ds;
        }
        part_g[sm] = G;
        part_p[sm] = P;
        if (kG) part_j[sm] = J;
    }
    store_sums(acc, p, dx + at, L, D);
}

// Lanes per (b, d): up to 8, more while the grid is short of four warps a scheduler, but no
// more than there are modes.
int log2_lanes(int64_t B, int D, int M) {
    int l = 0;
    while ((1 << l) < M && (l < 3 || (l < 5 && ((B * D) << l) < (int64_t)sm_count() * 512))) ++l;
    return l;
}

dim3 grid_of(int64_t B, int D, int l) { return dim3((unsigned)((((int64_t)D << l) + kBlock - 1) / kBlock), (unsigned)B); }

}  // namespace

bool short_supported(int64_t L) { return L <= kLen; }

cudaError_t short_prefill(const void *x, void *y, rlm_dtype dt, int64_t B, int64_t L, int D, int M, const float *decay,
                          const float *freq, const float *amp, const float *phase, const float *state_in, float *state_out,
                          float *coef_out, cudaStream_t st) {
    const int l = log2_lanes(B, D, M);
    auto go = [&](auto t) {
        using T = decltype(t);
        k_short_forward<T><<<grid_of(B, D, l), kBlock, 0, st>>>(
            static_cast<const T *>(x), static_cast<T *>(y), (int)L, D, M, l, decay, freq, amp, phase,
            reinterpret_cast<const float2 *>(state_in), reinterpret_cast<float2 *>(state_out),
            reinterpret_cast<float4 *>(coef_out));
    };
    if (dt == RLM_BF16) go(__nv_bfloat16());
    else go(float());
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t short_backward(const void *dy, const void *x, void *dx, rlm_dtype dt, int64_t B, int64_t L, int D, int M,
                           const float *decay, const float *freq, const float *amp, const float *phase,
                           const float *state_in, const float *d_state_out, float *d_state_in, float2 *part_g,
                           float2 *part_p, float2 *part_j, cudaStream_t st) {
    const int l = log2_lanes(B, D, M);
    auto go = [&](auto t, auto with_g) {
        using T = decltype(t);
        k_short_backward<T, decltype(with_g)::value><<<grid_of(B, D, l), kBlock, 0, st>>>(
            static_cast<const T *>(dy), static_cast<const T *>(x), static_cast<T *>(dx), (int)L, D, M, l, decay, freq, amp,
            phase, reinterpret_cast<const float2 *>(state_in), reinterpret_cast<const float2 *>(d_state_out),
            reinterpret_cast<float2 *>(d_state_in), part_g, part_p, part_j);
    };
    auto with = [&](auto g) { dt == RLM_BF16 ? go(__nv_bfloat16(), g) : go(float(), g); };
    if (d_state_out) with(std::true_type{});
    else with(std::false_type{});
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace rlm
