// rlm_simt.cu -- chunked complex-diagonal scan on the CUDA cores (fp32).
//
// Runs what the tensor-core paths do not cover: the fp32-I/O prefill with more
// than 16 modes, an initial state with a length that is not a multiple of 64, the
// scratch-array prefill, and the backward pass for fp32 I/O and M > 32.  All
// arithmetic is fp32.
//
// Chunked form, C = 64 tokens, chunks from token 0 (the last may be partial and is
// padded with zero drives).  With S_k the state entering chunk k and W_k = c lambda S_k:
//
//   L_k       = sum_p lambda^(63-p) x_{k,p}                     chunk-local end state
//   S_{k+1}   = lambda^64 S_k + L_k                             carry
//   y_{k,p}   = sum_{p'<=p} K[p-p'] x_{k,p'} + sum_m Re(lambda^p W_k)
//
// The backward is the same scan of dy in reverse time: processing time
// tau = 64 nch - 1 - t puts the padding first, and position p of a chunk is then
// 63 minus its position in time, so L_k is the adjoint's Dp, the output formula gives
// dx, and only the Jordan partner (weights 63 - p), the x-side projections and the
// lag correlation are added:
//
//   Dq_k = sum_p (63-p) lambda^(63-p) dy_p,   R_{k+1} = lambda^64 (R_k + 64 S_k) + Dq_k
//   Xp_k = sum_p lambda^p x_p,                Xq_k = sum_p (p+1) lambda^p x_p
//   G += lambda Xp_k S_k,                     P += lambda (Xp_k R_k + Xq_k S_k)
//   rho[n] = sum_k sum_u dy_u x_{u+n},        G += sum_n lambda^n rho[n], P += sum_n n lambda^n rho[n]
//
// Every sum over positions or modes is a small matrix product, which costs 2 FMA per
// token and mode (4 with the Jordan partner) where the token-by-token recurrence
// costs 4 (8) plus 2 for the readout: at M = 32 about 170 FMA per token-channel
// forward and 410 backward, against 320 and 830.
//
// One warp owns one channel and a tile of 16 chunks (1024 tokens); its products are
// register tiles (lane = 8 row groups x 4 column groups, columns = chunks) over
// tables and drives in shared memory, issued as packed two-lane FMAs
// (fma.rn.f32x2: 63 against 52 TFLOP/s with three distinct register operands at the
// two warps a scheduler has here, and half the issue slots).  A block is 4 channels
// (a 16-byte fp32 slice of each token row) and walks the tiles of a segment of the
// sequence with the state in registers, so that chunk states never touch memory.  Few
// (batch row, channel group) pairs are split into segments of whole tiles: a first
// launch forms each segment's end state from zero, and the second enters segment s
// with the combination of the states before it.
//
// What bounds it: shared-load wavefronts (four a 16-byte load of a warp: at M = 32 about 1900 a
// warp and tile forward, against 1350 cycles of FMA) at 40-50 % of their rate, since two
// warps a scheduler (tables and accumulators allow no more at M = 32) do not hide the loads'
// latency.  GB300, us per call, against the three launches of token-by-token recurrences with
// chunk states in memory that this replaces:
//
//   fp32, B = 2, L = 4096, D = 512, M = 32: forward 247 -> 56, backward 303 -> 117
//   fp32, B = 4, L = 2048, D = 256, M = 48: forward and backward 162 (with the power table of
//     a whole chunk, one block a SM, 305)
//   bf16 from a state, B = 8, L = 1000, D = 256, M = 16: 75 -> 27
//
// and the error against 64 bits is a half to a third of the recurrences' (3e-6 -> 1e-6 for
// the gradients of the first line).
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "rlm_device.cuh"
#include "rlm_internal.h"

namespace rlm {
namespace {

typedef unsigned long long u64;

constexpr int kC = 64;               // chunk length
constexpr int kCols = 16;            // chunks per tile
constexpr int kTile = kC * kCols;    // 1024 tokens
constexpr int kCh = 4;               // channels (warps) per block
constexpr int kThreads = 32 * kCh;
constexpr int kHalf = kC / 2;
// The power table holds lambda^n for n < 32 only (it is what limits the blocks a SM holds):
// products over a chunk run as two halves, joined by lambda^32.
constexpr int kPwStride = kHalf + 2;   // float2 per mode row: n < 32, then lambda^32 and lambda^64; rows 4 banks apart
// One channel's tile: [p / 2][column][p % 2] in rows of 32 words and 4 of padding, see slot().
constexpr int kRowWords = 2 * kCols + 4, kFieldWords = kHalf * kRowWords;
constexpr int kKernCopy = kC + 16;        // K reversed, then zeros (negative lags)
constexpr int kKernWords = 2 * kKernCopy; // that, and the same shifted by one

// Shared memory of a block, in floats: per channel the power table and c of every mode
// (complex), the reversed lag kernel, and for output passes two field tiles, the drive's
// and x's (forward: the second half's W).
constexpr int chan_words(int modes, bool out) {
    return 2 * modes * (kPwStride + 1) + kKernWords + (out ? 2 : 1) * kFieldWords;
}
// Resident blocks a SM, for registers and shared memory alike.  (A third block at 17 to 32
// modes, with 168 registers a thread, made the forward of B = 2, L = 4096, D = 512, M = 32 fp32 70
// us against 62 and its backward 159 against 133.)
__host__ __device__ constexpr int blocks_per_sm(int modes, bool bwd) {
    return modes > 16 ? 2 : bwd ? 3 : 4;
}
constexpr int smem_bytes(int modes, bool out) { return kCh * chan_words(modes, out) * 4; }

__device__ __forceinline__ u64 pack2(float a, float b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ u64 dup2(float a) { return pack2(a, a); }
__device__ __forceinline__ float2 unpack2(u64 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ void fma2(u64 &d, u64 a, u64 b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ void add2(u64 &d, u64 a) { asm("add.rn.f32x2 %0, %0, %1;" : "+l"(d) : "l"(a)); }
// Word of columns 2 h, 2 h + 1 in row r of a field tile (rows are position pairs, or modes
// of W).  The padding puts the 16-byte words that eight lanes write into eight rows in
// different banks, and leaves every address of the product loops a constant from the lane's.
// (Permuted 16-byte words of unpadded rows cost an XOR, a shift and an add a load: forward and
// backward of B = 2, L = 4096, D = 512, M = 32 fp32 60.1 and 135 us against 57.7 and 127.)
__device__ __forceinline__ int slot(int r, int h) { return r * kRowWords + 4 * h; }
__device__ __forceinline__ float2 shfl2(float2 v, int src) {
    return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

struct ScanArgs {
    const void *u;            // the scanned drive: x (forward), dy (backward)
    const void *x;            // backward: x
    void *out;                // y, or dx
    int bf16;                 // element type of the fields (0: fp32)
    int rev;                  // reverse time (backward)
    int64_t L;
    int B, D, M;
    int nch, ntiles;          // chunks and tiles of the sequence
    int gpr;                  // column groups (of 4) of a tile that one batch row takes: 4, or 1 / 2 (packed)
    int nseg, tps;            // segments, tiles per segment
    const float *decay, *freq, *amp, *phase;
    float2 *seg_s, *seg_r;    // [nseg][B][D][M] segment end states (pair) from zero
    const float2 *enter;      // nullable (forward): the state before token 0, as segment 0 reads it
    const float2 *state_in;   // nullable (backward)
    float2 *state_out;        // nullable (forward)
    float4 *coef_out;         // nullable (forward)
    float2 *part_g, *part_p;  // backward: [tiles of rows][nseg][D][M]
    float2 *part_j;           // with g
    const float2 *g;          // nullable: gradient of the terminal state
    float2 *d_state_in;       // nullable
};

// The 4 channels d .. d + 3 of token t.
__device__ __forceinline__ float4 load4(const void *f, int bf16, int64_t e) {
    if (bf16) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(static_cast<const __nv_bfloat16 *>(f) + e));
        return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u),
                           __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
    }
    return __ldg(reinterpret_cast<const float4 *>(static_cast<const float *>(f) + e));
}
__device__ __forceinline__ void store4(void *f, int bf16, int64_t e, float4 v) {
    if (bf16) {
        __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
        *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(f) + e) =
            make_uint2(*reinterpret_cast<uint32_t *>(&a), *reinterpret_cast<uint32_t *>(&b));
    } else {
        *reinterpret_cast<float4 *>(static_cast<float *>(f) + e) = v;
    }
}

// Projection of the drive tile on the power table: for the lane's modes g + 8 j and
// columns 4 cg + c, acc = sum_p lambda^e(p) x_p and (JORDAN) accq = sum_p w(p) lambda^e(p) x_p,
// with e = 63 - p, w = 63 - p (TO_END) or e = p, w = p + 1.  The half with the larger
// exponents runs first, on the table of the other, and is then carried by lambda^32.  The
// weights are never formed: accq adds up acc before every position (TO_END; after every
// position), which counts position p 63 - p (p + 1) times.  pw points at the row of
// mode g.  Per pair of positions: J + 2 16-byte shared loads, the drives duplicated into both
// halves, 8 J packed FMAs (and as many adds) on (Re, Im).
// Weighted products instead of the sums: backward of B = 4, L = 8000, D = 256, M = 16 fp32 166 us
// against 147, of B = 2, L = 4096, D = 512, M = 32 125 against 117.  (Four pairs unrolled against
// two: the 32-mode forward 57.7 -> 56.4 us, the 16-mode backward 147 -> 145, but the backward of
// M = 48 118 -> 120.)
template <int J, bool JORDAN, bool TO_END>
__device__ __forceinline__ void project(const float2 *pw, const float *xs, int cg, u64 (&acc)[J][4],
                                        u64 (&accq)[JORDAN ? J : 1][4]) {
#pragma unroll
    for (int j = 0; j < J; ++j)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            acc[j][c] = 0ull;
            if (JORDAN) accq[j][c] = 0ull;
        }
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        if (h) {
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const float2 l32 = pw[8 * j * kPwStride + kHalf];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float2 a = cmul(l32, unpack2(acc[j][c]));
                    acc[j][c] = pack2(a.x, a.y);
                    if (JORDAN) {
                        const float2 q = cmul(l32, unpack2(accq[j][c]));
                        accq[j][c] = pack2(q.x, q.y);
                    }
                }
            }
        }
        const int p0 = TO_END == (h == 0) ? 0 : kHalf;   // the half's first position
#pragma unroll (J == 4 && JORDAN ? 2 : 4)
        for (int u = 0; u < kHalf / 2; ++u) {
            const int v0 = TO_END ? u : kHalf / 2 - 1 - u, pp = p0 / 2 + v0;
            const float4 xa = *reinterpret_cast<const float4 *>(xs + slot(pp, 2 * cg));
            const float4 xb = *reinterpret_cast<const float4 *>(xs + slot(pp, 2 * cg + 1));
            ulonglong2 a[J];
            const int n = TO_END ? kHalf - 2 - 2 * v0 : 2 * v0;
#pragma unroll
            for (int j = 0; j < J; ++j) a[j] = *reinterpret_cast<const ulonglong2 *>(pw + 8 * j * kPwStride + n);
            const float v[2][4] = {{xa.x, xa.z, xb.x, xb.z}, {xa.y, xa.w, xb.y, xb.w}};
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int e = TO_END ? i : 1 - i;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const u64 d = dup2(v[e][c]);
#pragma unroll
                    for (int j = 0; j < J; ++j) {
                        const u64 aj = (e == 0) == TO_END ? a[j].y : a[j].x;
                        if (JORDAN && TO_END) add2(accq[j][c], acc[j][c]);
                        fma2(acc[j][c], aj, d);
                        if (JORDAN && !TO_END) add2(accq[j][c], acc[j][c]);
                    }
                }
            }
        }
    }
}

// acc[2 j + e][c] += the causal product of row p = 16 j + 2 g + e: sum_{p' <= p} K[p-p'] x_{p'}
// (the two halves of an accumulator take even and odd p' and are added at the end), on
// packed pairs (K[p-p'], K[p-p'-1]) of the reversed kernel kq (kq[q] = K[63 - q], zeros
// after; the copy behind it, shifted by one, keeps the pairs of even rows aligned).
// In the diagonal 16-row blocks the zeros stand for the later drives.  kGuard: a tile
// with an infinite or NaN drive skips them instead, so that earlier outputs stay clean.
// A pair of K serves every (row block, position block) with the same distance l, so SG
// position blocks are held at once: shared-load wavefronts bound these products, 576 with
// one at a time, 448 with two and 384 with four.  (One against two in the forward: 57.7 ->
// 55.6 us at B = 2, L = 4096, D = 512, M = 32 fp32; against four in its backward: 127.7 -> 125.)
template <bool kGuard, int SG>
__device__ __forceinline__ void causal(const float *kq, const float *xs, int g, int cg, u64 (&acc)[8][4]) {
#pragma unroll
    for (int s0 = 0; s0 < 4; s0 += SG) {
#pragma unroll (SG == 4 ? 2 : 1)
        for (int u = 0; u < 8; ++u) {
            u64 x[SG][4];   // positions 16 (s0 + i) + 2 u and the next
#pragma unroll
            for (int i = 0; i < SG; ++i) {
                const float *row = xs + slot(8 * (s0 + i) + u, 2 * cg);
                const ulonglong2 xa = *reinterpret_cast<const ulonglong2 *>(row);
                const ulonglong2 xb = *reinterpret_cast<const ulonglong2 *>(row + 4);
                x[i][0] = xa.x;
                x[i][1] = xa.y;
                x[i][2] = xb.x;
                x[i][3] = xb.y;
            }
#pragma unroll
            for (int l = 0; l < 4 - s0; ++l) {
                const int q1 = kC - 1 - (16 * l + 2 * g + 1) + 2 * u;   // row e = 1: even
                const u64 k1 = *reinterpret_cast<const u64 *>(kq + q1);
                const u64 k0 = *reinterpret_cast<const u64 *>(kq + kKernCopy + q1);   // row e = 0: kq[q1 + 1], kq[q1 + 2]
#pragma unroll
                for (int i = 0; i < SG; ++i) {
                    const int j = s0 + i + l;
                    if (j >= 4) continue;
                    if (kGuard && l == 0) {
                        // Rows 2 g, 2 g + 1 of the block against its positions 2 u, 2 u + 1.
                        const float2 f0 = unpack2(k0), f1 = unpack2(k1);
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const float2 v = unpack2(x[i][c]);
                            float2 a0 = unpack2(acc[2 * j][c]), a1 = unpack2(acc[2 * j + 1][c]);
                            if (u <= g) {
                                a0.x = fmaf(f0.x, v.x, a0.x);
                                a1.x = fmaf(f1.x, v.x, a1.x);
                                a1.y = fmaf(f1.y, v.y, a1.y);
                            }
                            if (u < g) a0.y = fmaf(f0.y, v.y, a0.y);
                            acc[2 * j][c] = pack2(a0.x, a0.y);
                            acc[2 * j + 1][c] = pack2(a1.x, a1.y);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            fma2(acc[2 * j][c], k0, x[i][c]);
                            fma2(acc[2 * j + 1][c], k1, x[i][c]);
                        }
                    }
                }
            }
        }
    }
}

// acc += Re(sum_m lambda^p W) over `modes` modes: W is staged as (Re, -Im) per column, so
// a packed FMA on (Re lambda^p, Im lambda^p) accumulates both halves of the real part.  Rows
// p >= 32 take lambda^(p-32) and lambda^32 W (w2).
__device__ __forceinline__ void up_project(const float2 *pw, const float *w1, const float *w2, int modes, int g, int cg,
                                           u64 (&acc)[8][4]) {
#pragma unroll 2
    for (int m = 0; m < modes; ++m) {
        ulonglong2 a[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) a[j] = *reinterpret_cast<const ulonglong2 *>(pw + m * kPwStride + 16 * j + 2 * g);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float *ws = h ? w2 : w1;
            const ulonglong2 wa = *reinterpret_cast<const ulonglong2 *>(ws + slot(m, 2 * cg));
            const ulonglong2 wb = *reinterpret_cast<const ulonglong2 *>(ws + slot(m, 2 * cg + 1));
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int r = 2 * (2 * h + j);
                fma2(acc[r][0], a[j].x, wa.x);
                fma2(acc[r][1], a[j].x, wa.y);
                fma2(acc[r][2], a[j].x, wb.x);
                fma2(acc[r][3], a[j].x, wb.y);
                fma2(acc[r + 1][0], a[j].y, wa.x);
                fma2(acc[r + 1][1], a[j].y, wa.y);
                fma2(acc[r + 1][2], a[j].y, wb.x);
                fma2(acc[r + 1][3], a[j].y, wb.y);
            }
        }
    }
}

// lambda^n, n < 64, from a mode's table row.
__device__ __forceinline__ float2 power(const float2 *row, int n) {
    return n < kHalf ? row[n] : cmul(row[kHalf], row[n - kHalf]);
}

// sum_{p < tail} lambda^(tail-1-p) x_p of one column, in every lane: the four lanes of a mode
// take every fourth power, and lambda^(n+32) shares the table entry of lambda^n.  (A single
// lane walking the positions took up to 10 us of a call: B = 2, L = 4095, D = 512, M = 32 fp32
// 76.4 us against 66.2 at L = 4096.)
__device__ __forceinline__ float2 partial_end(const float2 *row, const float *xs, int col, int tail, int cg) {
    float2 lo = make_float2(0.0f, 0.0f), hi = lo;
    auto x = [&](int p) {
        return p >= 0 ? xs[slot(p >> 1, col >> 1) + 2 * (col & 1) + (p & 1)] : 0.0f;
    };
#pragma unroll 4
    for (int n = cg; n < kHalf; n += 4) {
        const float2 z = row[n];
        const float v = x(tail - 1 - n), w = x(tail - 1 - n - kHalf);
        lo.x = fmaf(z.x, v, lo.x);
        lo.y = fmaf(z.y, v, lo.y);
        hi.x = fmaf(z.x, w, hi.x);
        hi.y = fmaf(z.y, w, hi.y);
    }
    lo = cfma(row[kHalf], hi, lo);
#pragma unroll
    for (int o = 8; o <= 16; o <<= 1) {
        lo.x += __shfl_xor_sync(0xffffffffu, lo.x, o);
        lo.y += __shfl_xor_sync(0xffffffffu, lo.y, o);
    }
    return lo;
}

// acc[n] += sum_u dy_u x_{u + 16 l + n} over the 16 positions u of block a, one column
// (the lane's); positions past the chunk count as zero.
__device__ __forceinline__ void correlate(const float *dys, const float *xs, int col, int a, int l, float (&acc)[16]) {
    float dv[16], xv[32];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const float2 v = *reinterpret_cast<const float2 *>(dys + slot(8 * a + u, col >> 1) + 2 * (col & 1));
        dv[2 * u] = v.x;
        dv[2 * u + 1] = v.y;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float2 v = a + l + h < 4
                                 ? *reinterpret_cast<const float2 *>(xs + slot(8 * (a + l + h) + u, col >> 1) + 2 * (col & 1))
                                 : make_float2(0.0f, 0.0f);
            xv[16 * h + 2 * u] = v.x;
            xv[16 * h + 2 * u + 1] = v.y;
        }
#pragma unroll
    for (int u = 0; u < 16; ++u)
#pragma unroll
        for (int n = 0; n < 16; ++n) acc[n] = fmaf(dv[u], xv[u + n], acc[n]);
}

// v[n] summed over the 16 columns (lanes of one half); lane `col` receives lag n = col.
__device__ __forceinline__ float sum_columns(float (&v)[16], int col) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
        const bool up = col & o;
#pragma unroll
        for (int n = 0; n < o; ++n) {
            const float keep = up ? v[n + o] : v[n], send = up ? v[n] : v[n + o];
            v[n] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return v[0];
}

// One block: channels 4 blockIdx.x .. + 3 of batch row blockIdx.z, segment blockIdx.y.
// Sequences of at most 4 (8) chunks leave most of a tile's 16 columns empty, so there a
// tile holds 4 (2) batch rows, one (two) column groups each, and blockIdx.z counts
// tiles: b below is then the lane's own row, clamped; `mine` says whether it exists.
// kOut: write outputs (else only the segment's end state, from zero).
template <int J, int NP, bool BWD, bool kOut>
__global__ void __launch_bounds__(kThreads, blocks_per_sm(8 * J * NP, BWD)) k_scan(const ScanArgs A) {
    constexpr int kModes = 8 * J * NP;
    constexpr bool kX = BWD && kOut;   // the x tile is needed
    constexpr int kSG = BWD && J == 4 ? 4 : 2;   // (see causal(); the forward with four: 55.6 -> 57.7 us)
    constexpr bool kAhead = !BWD && J == 4;   // the next tile's drive is loaded a tile ahead
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int g = lane & 7, cg = lane >> 3;
    const int seg = blockIdx.y;
    const int rpt = 4 / A.gpr, gbase = cg & ~(A.gpr - 1);   // batch rows of a tile; the row's first column group
    const bool mine = (int)blockIdx.z * rpt + cg / A.gpr < A.B;
    const int64_t b = min((int)blockIdx.z * rpt + cg / A.gpr, A.B - 1);
    const int d0 = kCh * blockIdx.x, d = d0 + w, M = A.M, D = A.D;
    constexpr int kWords = chan_words(kModes, kOut);
    constexpr int kTableWords = 2 * kModes * (kPwStride + 1) + kKernWords;   // before the field tiles
    float2 *pw = reinterpret_cast<float2 *>(smem + w * kWords);
    float2 *cs = pw + kModes * kPwStride;        // c of every mode
    float *kq = smem + w * kWords + 2 * kModes * (kPwStride + 1);
    float *us = kq + kKernWords;                 // drive tile, then W, then the output tile
    float *xs = us + (kOut ? kFieldWords : 0);   // x tile (backward), then lambda^32 W
    pdl_launch_dependents();

    const int tail = (int)(A.L & (kC - 1));                 // tokens of the partial last chunk
    const int tile_end = min(A.ntiles, (seg + 1) * A.tps);
    // The thread's 8 tokens of a tile, 4 channels each (zeros outside the sequence).
    const int Li = (int)A.L, t_last = A.nch * kC - 1;
    // The thread's column: its batch row, and its first token's tau in tile 0.
    const int fcol = tid & (kCols - 1), frow = (int)blockIdx.z * rpt + fcol / (4 * A.gpr);
    const int ftau = (fcol & (4 * A.gpr - 1)) * kC + (tid >> 4);
    const int64_t fbase = (int64_t)frow * A.L;
    auto fetch = [&](const void *f, int tile, float4 (&v)[8]) {
        const int tau = tile * kTile + ftau;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int t = A.rev ? t_last - tau - 8 * i : tau + 8 * i;
            v[i] = t >= 0 && t < Li && frow < A.B ? load4(f, A.bf16, (fbase + t) * D + d0)
                                                  : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
    };
    // The 32-mode forward loads the next tile's drive ahead of this tile's outputs (67 -> 62
    // us at B = 2, L = 4096, D = 512, M = 32 fp32).  The backward has no registers for it
    // (132 -> 143 us), the smaller forward needs them for its fourth block a SM.  There the
    // first tile's lines move to L2 while the tables are built (later tiles' made the M = 16 fp32
    // backward of B = 4, L = 8000, D = 256 189 us against 183).
    if (!kAhead && frow < A.B) {
        const int tau = seg * A.tps * kTile + ftau, e = A.bf16 ? 2 : 4;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int t = A.rev ? t_last - tau - 8 * i : tau + 8 * i;
            if (t < 0 || t >= Li) continue;
            const int64_t at = ((fbase + t) * D + d0) * e;
            prefetch_l2(static_cast<const char *>(A.u) + at);
            if (kX) prefetch_l2(static_cast<const char *>(A.x) + at);
        }
    }
    float4 nextu[8], nextx[kX ? 8 : 1];

    // ---- tables: lambda^n, n < 32 (an exact power every 8, products between), 32 and 64
    {
        constexpr int kLpm = kModes >= 32 ? 1 : 32 / kModes;   // lanes per mode
#pragma unroll 1
        for (int m = lane / kLpm; m < kModes; m += 32) {
            float2 *row = pw + m * kPwStride;
            const bool on = m < M;
            const float ga = on ? A.decay[d * M + m] : 0.0f, om = on ? A.freq[d * M + m] : 0.0f;
            const float am = kOut && on ? A.amp[d * M + m] : 0.0f, ph = kOut && on ? A.phase[d * M + m] : 0.0f;
            if (!BWD && A.enter && on)   // used after the tables
                prefetch_l2(A.enter + ((int64_t)min((int)blockIdx.z * rpt, A.B - 1) * D + d) * M + m);
            const float2 l1 = lambda_pow(ga, om, 1.0f);
#pragma unroll 1
            for (int n0 = 8 * (lane % kLpm); n0 < kHalf; n0 += 8 * kLpm) {
                float2 z = lambda_pow(ga, om, (float)n0);
                if (!on) z = make_float2(0.0f, 0.0f);
                row[n0] = z;
#pragma unroll
                for (int e = 1; e < 8; ++e) row[n0 + e] = z = cmul(z, l1);
            }
            if (lane % kLpm == 0) {
                const float2 z = make_float2(0.0f, 0.0f);
                row[kHalf] = on ? lambda_pow(ga, om, (float)kHalf) : z;
                row[kHalf + 1] = on ? lambda_pow(ga, om, (float)kC) : z;
                if (kOut) cs[m] = on ? mode_coef(am, ph) : z;
            }
        }
    }
    if (kOut) pdl_wait();   // the segments' end states (the tables needed parameters only)
    __syncwarp();
    // ---- the state (pair) entering the segment, of the lane's modes
    float2 S0[NP][J], R0[BWD ? NP : 1][J];
#pragma unroll
    for (int q = 0; q < NP; ++q)
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int m = 8 * J * q + 8 * j + g;
            const bool on = m < M;
            const float ga = on ? A.decay[d * M + m] : 0.0f, om = on ? A.freq[d * M + m] : 0.0f;
            const float2 z = make_float2(0.0f, 0.0f);
            const int64_t sm = (b * D + d) * M + m;
            S0[q][j] = !BWD && A.enter && on && mine && seg == 0 ? A.enter[sm] : z;
            if (BWD) R0[q][j] = z;
            if (kOut && seg > 0 && on) {
                // The earlier segments' end states, each carried over the segments between.
                const float nf = (float)(A.tps * kTile);
                const float2 lN = lambda_pow(ga, om, nf);
                const int64_t st = (int64_t)A.B * D * M;
                float2 S = z, R = z;
#pragma unroll 4
                for (int r = 0; r < seg; ++r) {
                    if (BWD)
                        R = cfma(lN, make_float2(fmaf(nf, S.x, R.x), fmaf(nf, S.y, R.y)), A.seg_r[sm + r * st]);
                    S = cfma(lN, S, A.seg_s[sm + r * st]);
                }
                S0[q][j] = S;
                if (BWD) R0[q][j] = R;
            }
            if (!BWD && kOut && A.coef_out && blockIdx.z == 0 && seg == A.nseg - 1 && cg == 0 && on) {
                const float2 l1 = pw[m * kPwStride + 1];   // the exact lambda times lambda^0 = 1
                A.coef_out[d * M + m] = make_float4(l1.x, l1.y, cs[m].x, cs[m].y);
            }
            // The output launch's segment 0 starts from this copy: by then a state_out that
            // is state_in's buffer may be written by the last segment's block.
            if (!kOut && !BWD && seg == 0 && A.enter && cg == 0 && on)
                A.seg_s[sm + (int64_t)(A.nseg - 1) * A.B * D * M] = S0[q][j];
        }
    __syncwarp();
    if (kOut) {
        // K[n] = sum_m Re(c lambda^n), stored reversed (and once more shifted by one).
        float k0 = 0.0f, k1 = 0.0f;
        for (int m = 0; m < M; ++m) {
            const float2 c = cs[m], p = pw[m * kPwStride + lane], c2 = cmul(c, pw[m * kPwStride + kHalf]);
            k0 = fmaf(c.x, p.x, fmaf(-c.y, p.y, k0));
            k1 = fmaf(c2.x, p.x, fmaf(-c2.y, p.y, k1));
        }
        kq[63 - lane] = k0;
        kq[31 - lane] = k1;
        kq[kKernCopy + 62 - lane] = k0;
        if (lane < 31) kq[kKernCopy + 30 - lane] = k1;
        if (lane < 16) kq[kC + lane] = kq[kKernCopy + kC + lane] = 0.0f;
        if (lane == 0) kq[kKernCopy + kC - 1] = 0.0f;
    }
    __syncwarp();

    float2 G[kX ? NP : 1][J], P[kX ? NP : 1][J], Jg[kX ? NP : 1][J];
    float rho_a = 0.0f, rho_b = 0.0f;   // lane (h, n): lags 16 h + n and 16 (3 - h) + n
    if (kX) {
#pragma unroll
        for (int q = 0; q < NP; ++q)
#pragma unroll
            for (int j = 0; j < J; ++j) G[q][j] = P[q][j] = Jg[q][j] = make_float2(0.0f, 0.0f);
    }
    if (kAhead) fetch(A.u, seg * A.tps, nextu);
    for (int tile = seg * A.tps; tile < tile_end; ++tile) {
        // ---- stage the tile: thread (column, position), 4 channels each
        const int t0 = tile * kTile + ftau;   // tau of the thread's first token
        bool odd = false;   // an infinite or NaN drive
        auto stage = [&](const float4 (&v)[8], float *base) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int p = (tid >> 4) + 8 * i, col = tid & (kCols - 1);
                float *o = base + slot(p >> 1, col >> 1) + 2 * (col & 1) + (p & 1);
                o[0] = v[i].x;
                o[kWords] = v[i].y;
                o[2 * kWords] = v[i].z;
                o[3 * kWords] = v[i].w;
            }
        };
        float *base = smem + kTableWords;
        if (!kAhead) fetch(A.u, tile, nextu);
        if constexpr (kX) fetch(A.x, tile, nextx);
        stage(nextu, base);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            // x - x is zero for a finite x.
            const float z = (nextu[i].x - nextu[i].x) + (nextu[i].y - nextu[i].y) + (nextu[i].z - nextu[i].z) +
                            (nextu[i].w - nextu[i].w);
            odd |= !(z == 0.0f);
        }
        if constexpr (kX) stage(nextx, base + kFieldWords);
        const bool guard = __syncthreads_or(kOut && odd);

        // ---- chunk-local states, carry over the 16 columns (and G, P)
        const int chunk0 = tile * kCols + 4 * (cg - gbase);   // the lane's first chunk
        u64 ls[NP][J][4];   // lambda S of the state entering each of the lane's columns
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            u64 acc[J][4], accq[BWD ? J : 1][4];
            project<J, BWD, true>(pw + (8 * J * q + g) * kPwStride, us, cg, acc, accq);
            float2 Rn[BWD ? J : 1][4];
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const float2 *row = pw + (8 * J * q + 8 * j + g) * kPwStride;
                const float2 a = row[kHalf + 1], a2 = cmul(a, a), a4 = cmul(a2, a2);
                const float2 lam = row[1];
                // The lane's four columns from zero ...
                float2 es = make_float2(0.0f, 0.0f), er = es;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (BWD)
                        er = cfma(a, make_float2(fmaf((float)kC, es.x, er.x), fmaf((float)kC, es.y, er.y)),
                                  unpack2(accq[j][c]));
                    es = cfma(a, es, unpack2(acc[j][c]));
                }
                // ... the state entering them (over the mode's lanes in this row) ...
                float2 T = S0[q][j], U = BWD ? R0[q][j] : T, S = T, R = U, send = T;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (i >= A.gpr) break;   // the same for every lane
                    if (gbase + i == cg) {
                        S = T;
                        R = U;
                    }
                    const float2 ei = shfl2(es, g + 8 * (gbase + i));
                    if (BWD)
                        U = cfma(a4, make_float2(fmaf(4.0f * kC, T.x, U.x), fmaf(4.0f * kC, T.y, U.y)),
                                 shfl2(er, g + 8 * (gbase + i)));
                    T = cfma(a4, T, ei);
                }
                S0[q][j] = T;
                if (BWD) R0[q][j] = U;
                // ... and entering each of them.
                const int m = 8 * J * q + 8 * j + g;
                const bool on = m < M;
#pragma unroll
                for (int c = 0; c < (kOut ? 4 : 0); ++c) {
                    const float2 lsv = cmul(lam, S);
                    ls[q][j][c] = pack2(lsv.x, lsv.y);
                    if (kX) {
                        Rn[j][c] = cmul(lam, R);
                        R = cfma(a, make_float2(fmaf((float)kC, S.x, R.x), fmaf((float)kC, S.y, R.y)),
                                 unpack2(accq[j][c]));
                        S = cfma(a, S, unpack2(acc[j][c]));
                        if (chunk0 + c == A.nch - 1 && on && mine) {
                            // The chunk of token 0: (S, R) is the adjoint pair there.
                            const int64_t sm = (b * D + d) * M + m;
                            const float2 l0 = cmul(lam, S);
                            const float2 gg = A.g ? A.g[sm] : make_float2(0.0f, 0.0f);
                            const float2 lL =
                                A.g ? lambda_pow(A.decay[d * M + m], A.freq[d * M + m], (float)A.L) : gg;
                            if (A.state_in) {
                                const float2 si = A.state_in[sm];
                                G[q][j] = cfma(si, l0, G[q][j]);
                                P[q][j] = cfma(si, cmul(lam, make_float2(R.x + S.x, R.y + S.y)), P[q][j]);
                                const float2 ji = cmul(si, lL);
                                Jg[q][j].x = fmaf((float)A.L, ji.x, Jg[q][j].x);
                                Jg[q][j].y = fmaf((float)A.L, ji.y, Jg[q][j].y);
                            }
                            if (A.d_state_in) {
                                const float2 v = cmul(cs[m], l0);
                                A.d_state_in[sm] = cfma(gg, make_float2(lL.x, -lL.y), make_float2(v.x, -v.y));
                            }
                        }
                    } else {
                        const float2 next = cfma(a, S, unpack2(acc[j][c]));
                        if (chunk0 + c == A.nch - 1) {
                            if (tail)
                                send = S;
                            else if (on && mine && A.state_out)
                                A.state_out[(b * D + d) * M + m] = next;
                        }
                        S = next;
                    }
                }
                if (!BWD && kOut && tail && tile == A.ntiles - 1 && A.state_out)
                    for (int r = 0; r < rpt; ++r) {
                        const int col = r * 4 * A.gpr + (A.nch - 1 - tile * kCols);   // row r's last chunk
                        const float2 f = partial_end(row, us, col, tail, cg);
                        if (cg == col >> 2 && on && mine)
                            A.state_out[(b * D + d) * M + m] = cfma(power(row, tail), send, f);
                    }
            }
            if (kX) {
                u64 xp[J][4], xq[J][4];
                project<J, true, false>(pw + (8 * J * q + g) * kPwStride, xs, cg, xp, xq);
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    const int m = 8 * J * q + 8 * j + g;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float2 s = unpack2(ls[q][j][c]), p = unpack2(xp[j][c]), v = unpack2(xq[j][c]);
                        G[q][j] = cfma(p, s, G[q][j]);
                        P[q][j] = cfma(p, Rn[j][c], cfma(v, s, P[q][j]));
                    }
                    if (A.g && m < M) {
                        // J over the whole chunks: L - 1 - t = E + p with E = L minus the chunk's end.
                        const float ga = A.decay[d * M + m], om = A.freq[d * M + m];
                        float2 z = make_float2(0.0f, 0.0f);
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const int64_t E = A.L - (int64_t)(A.nch - chunk0 - c) * kC;
                            if (E >= 0 && chunk0 + c < A.nch) {
                                z = c == 0 || E < kC ? lambda_pow(ga, om, (float)E) : cmul(z, pw[m * kPwStride + kHalf + 1]);
                                const float2 p = unpack2(xp[j][c]), v = unpack2(xq[j][c]);
                                const float Ef = (float)(E - 1);
                                Jg[q][j] = cfma(z, make_float2(fmaf(Ef, p.x, v.x), fmaf(Ef, p.y, v.y)), Jg[q][j]);
                            }
                        }
                        if (tail && tile == 0) {
                            // The partial last chunk (the row's first column): its tokens are
                            // positions p >= 64 - tail, L - 1 - t = p - (64 - tail), shared out
                            // among the row's lanes.
                            const float2 *row = pw + m * kPwStride;
                            for (int n = cg - gbase; n < tail; n += A.gpr) {
                                const int p = n + kC - tail;
                                const float v = (float)n * xs[slot(p >> 1, 2 * gbase) + (p & 1)];
                                const float2 z = power(row, n);
                                Jg[q][j].x = fmaf(z.x, v, Jg[q][j].x);
                                Jg[q][j].y = fmaf(z.y, v, Jg[q][j].y);
                            }
                        }
                    }
                }
            }
        }
        if (!kOut) {
            if (kAhead && tile + 1 < tile_end) fetch(A.u, tile + 1, nextu);
            __syncthreads();   // every warp is done with the tile
            continue;
        }
        if (kX) {
            // Lag correlation: lane = (column, half); the half takes lag blocks {0, 3} or
            // {1, 2}, whose 10 non-empty (u block, lag block) pairs fall in 4 + 2 steps.
            const int col = lane & 15, h = lane >> 4;
            float r0[16], r1[16];
#pragma unroll
            for (int n = 0; n < 16; ++n) r0[n] = r1[n] = 0.0f;
#pragma unroll 1
            for (int a = 0; a < 4; ++a) correlate(us, xs, col, a, h, r0);
#pragma unroll 1
            for (int a = 0; a < 2; ++a) correlate(us, xs, col, a, 3 - h, r1);
            rho_a += sum_columns(r0, col);
            rho_b += sum_columns(r1, col);
        }

        // ---- outputs
        u64 acc[8][4];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[r][c] = 0ull;
        if (guard)
            causal<true, kSG>(kq, us, g, cg, acc);
        else
            causal<false, kSG>(kq, us, g, cg, acc);
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            __syncwarp();   // the warp is done reading the tile (or the previous W)
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int m = 8 * J * q + 8 * j + g;
                float2 W[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float2 v = cmul(cs[m], unpack2(ls[q][j][c]));
                    W[c] = m < M ? make_float2(v.x, -v.y) : make_float2(0.0f, 0.0f);
                }
                if (kX && A.g && m < M) {
                    // Terminal-state gradient: its adjoint conj(g) lambda^(L-1-t) enters a
                    // whole chunk as conj(g) lambda^E with E = L minus the chunk's end.
                    const float ga = A.decay[d * M + m], om = A.freq[d * M + m];
                    const float2 gg = A.g[(b * D + d) * M + m];
                    float2 z = make_float2(0.0f, 0.0f);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int64_t E = A.L - (int64_t)(A.nch - chunk0 - c) * kC;
                        if (E >= 0 && chunk0 + c < A.nch) {
                            z = c == 0 || E < kC ? lambda_pow(ga, om, (float)E) : cmul(z, pw[m * kPwStride + kHalf + 1]);
                            const float2 v = cmul(make_float2(gg.x, -gg.y), z);
                            W[c].x += v.x;
                            W[c].y -= v.y;
                        }
                    }
                }
                *reinterpret_cast<float4 *>(us + slot(8 * j + g, 2 * cg)) = make_float4(W[0].x, W[0].y, W[1].x, W[1].y);
                *reinterpret_cast<float4 *>(us + slot(8 * j + g, 2 * cg + 1)) =
                    make_float4(W[2].x, W[2].y, W[3].x, W[3].y);
                const float2 l32 = conj2(pw[m * kPwStride + kHalf]);   // (W is kept conjugated)
#pragma unroll
                for (int c = 0; c < 4; ++c) W[c] = cmul(l32, W[c]);
                *reinterpret_cast<float4 *>(xs + slot(8 * j + g, 2 * cg)) = make_float4(W[0].x, W[0].y, W[1].x, W[1].y);
                *reinterpret_cast<float4 *>(xs + slot(8 * j + g, 2 * cg + 1)) =
                    make_float4(W[2].x, W[2].y, W[3].x, W[3].y);
            }
            __syncwarp();
            if (kAhead && q == NP - 1 && tile + 1 < tile_end) fetch(A.u, tile + 1, nextu);
            up_project(pw + 8 * J * q * kPwStride, us, xs, min(8 * J, M - 8 * J * q), g, cg, acc);
        }
        float y[8][4];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float2 v = unpack2(acc[r][c]);
                y[r][c] = v.x + v.y;
            }
        if (kX && A.g && tail && chunk0 == 0) {
            // The terminal-state term of the partial last chunk.
            for (int m = 0; m < M; ++m) {
                const float2 gg = A.g[(b * D + d) * M + m];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const int n = 16 * (r >> 1) + 2 * g + (r & 1) - (kC - tail);
                    if (n >= 0) {
                        const float2 z = power(pw + m * kPwStride, n);
                        y[r][0] = fmaf(gg.x, z.x, fmaf(gg.y, z.y, y[r][0]));
                    }
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            *reinterpret_cast<float4 *>(us + slot(8 * j + g, 2 * cg)) =
                make_float4(y[2 * j][0], y[2 * j + 1][0], y[2 * j][1], y[2 * j + 1][1]);
            *reinterpret_cast<float4 *>(us + slot(8 * j + g, 2 * cg + 1)) =
                make_float4(y[2 * j][2], y[2 * j + 1][2], y[2 * j][3], y[2 * j + 1][3]);
        }
        __syncthreads();
        // A thread reads here the words it wrote when staging, and writes them again for
        // the next tile: no barrier is needed between.
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int p = (tid >> 4) + 8 * i, col = tid & (kCols - 1);
            const float *o = base + slot(p >> 1, col >> 1) + 2 * (col & 1) + (p & 1);
            const int t = A.rev ? t_last - t0 - 8 * i : t0 + 8 * i;
            if (t >= 0 && t < Li && frow < A.B)
                store4(A.out, A.bf16, (fbase + t) * D + d0, make_float4(o[0], o[kWords], o[2 * kWords], o[3 * kWords]));
        }
    }

    if (!kOut) {
        if (cg == 0) {
#pragma unroll
            for (int q = 0; q < NP; ++q)
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    const int m = 8 * J * q + 8 * j + g;
                    const int64_t o = (((int64_t)seg * A.B + b) * D + d) * M + m;
                    if (m < M) {
                        A.seg_s[o] = S0[q][j];
                        if (BWD) A.seg_r[o] = R0[q][j];
                    }
                }
        }
        return;
    }
    if (kX) {
        // The within-chunk terms: lane cg takes lags 16 cg .. 16 cg + 15 of its modes; the
        // sums over cg complete G, P and J.
        const int h = lane >> 4;
        __syncwarp();
        kq[16 * h + (lane & 15)] = rho_a;
        kq[16 * (3 - h) + (lane & 15)] = rho_b;
        __syncwarp();
#pragma unroll
        for (int q = 0; q < NP; ++q)
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int m = 8 * J * q + 8 * j + g;
                float2 gs = G[q][j], ps = P[q][j], js = Jg[q][j];
                if (A.g && m < M) {
                    // conj(g) J, g the lane's row's (Jg of a row that does not exist is zero).
                    const float2 gg = A.g[(b * D + d) * M + m];
                    js = cmul(make_float2(gg.x, -gg.y), js);
                }
                float2 gw = make_float2(0.0f, 0.0f), pn = gw;
                for (int n = 16 * cg; n < 16 * cg + 16; ++n) {
                    const float2 z = pw[m * kPwStride + (n & (kHalf - 1))];
                    const float r = kq[n], nr = (float)n * r;
                    gw.x = fmaf(z.x, r, gw.x);
                    gw.y = fmaf(z.y, r, gw.y);
                    pn.x = fmaf(z.x, nr, pn.x);
                    pn.y = fmaf(z.y, nr, pn.y);
                }
                const float2 up = cg < 2 ? make_float2(1.0f, 0.0f) : pw[m * kPwStride + kHalf];
                gs = cfma(up, gw, gs);
                ps = cfma(up, pn, ps);
#pragma unroll
                for (int o = 8; o <= 16; o <<= 1) {
                    gs.x += __shfl_xor_sync(0xffffffffu, gs.x, o);
                    gs.y += __shfl_xor_sync(0xffffffffu, gs.y, o);
                    ps.x += __shfl_xor_sync(0xffffffffu, ps.x, o);
                    ps.y += __shfl_xor_sync(0xffffffffu, ps.y, o);
                    js.x += __shfl_xor_sync(0xffffffffu, js.x, o);
                    js.y += __shfl_xor_sync(0xffffffffu, js.y, o);
                }
                if (cg == 0 && m < M) {
                    const int64_t o = (((int64_t)blockIdx.z * A.nseg + seg) * D + d) * M + m;
                    A.part_g[o] = gs;
                    A.part_p[o] = ps;
                    if (A.g) A.part_j[o] = js;
                }
            }
    }
}

// One thread per (d, m): fixed-order sum of the partials
// over (b, k), then the four gradients.  The sums are compensated (Kahan) fp32
// sums, so the result is reproducible and its error stays near one rounding
// however many partials are added; the combination with
// c = A e^{i phi} (formed as the forward forms it, fp32 sincosf) uses fmaf for
// the differences.  Double precision made this launch 3-4x slower on this part
// (low FP64 rate): 4.8 against 1.4 us at D = 512, M = 32, four partials.
// ws_j (nullable): partials of conj(g) J from a terminal-state gradient, which
// add -Re and -Im of their sum to dgamma and domega.
struct KahanSum {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float v) {
        const float y = v - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
};
__global__ void __launch_bounds__(256) k_grad_reduce(
    int64_t B, int D, int M, int nch, const float *__restrict__ amp,
    const float *__restrict__ phase, const float2 *ws_s, const float2 *ws_r, const float2 *ws_j, float *__restrict__ g_decay,
    float *__restrict__ g_freq, float *__restrict__ g_amp, float *__restrict__ g_phase) {
    const int pm = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();
    if (pm >= D * M) return;
    const float am = amp[pm], ph = phase[pm];
    KahanSum gr, gi, pr, pi, jr, ji;
    const int64_t n = B * nch, stride = (int64_t)D * M;
    // Four partials' loads in flight before their adds (the sum order is fixed).
    for (int64_t bk0 = 0; bk0 < n; bk0 += 4) {
        float2 g[4], p[4], j[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t off = (bk0 + u) * stride + pm;
            const bool in = bk0 + u < n;
            g[u] = in ? ws_s[off] : make_float2(0.0f, 0.0f);
            p[u] = in ? ws_r[off] : make_float2(0.0f, 0.0f);
            j[u] = in && ws_j ? ws_j[off] : make_float2(0.0f, 0.0f);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (bk0 + u >= n) break;
            gr.add(g[u].x);
            gi.add(g[u].y);
            pr.add(p[u].x);
            pi.add(p[u].y);
            if (ws_j) {
                jr.add(j[u].x);
                ji.add(j[u].y);
            }
        }
    }
    float sph, cph;
    sincosf(ph, &sph, &cph);
    const float cr = am * cph, ci = am * sph;
    g_amp[pm] = fmaf(cph, gr.s, -sph * gi.s);            // Re(e^{i phi} G)
    g_phase[pm] = -fmaf(cr, gi.s, ci * gr.s);            // -Im(c G)
    g_decay[pm] = -fmaf(cr, pr.s, -ci * pi.s) - jr.s;    // -Re(c P) - Re(conj(g) J)
    g_freq[pm] = -fmaf(cr, pi.s, ci * pr.s) - ji.s;      // -Im(c P) - Im(conj(g) J)
}


// Launch shape.  A block is a 4-channel group of a batch row; where these blocks
// would leave SMs idle the sequence is cut into as many segments of whole tiles as fill
// the resident blocks once.  The segments cost one more launch and a second projection
// of the drive (38 % of the forward's FMA at M = 32, 31 % of the backward's), so they
// are only taken when at least two of them fit.
struct Geometry {
    int nch, ntiles, nseg, tps, gpr;
    int zdim;   // blocks along the batch
};

Geometry geometry(int64_t B, int64_t L, int D, int M, bool bwd, int max_seg) {
    Geometry q;
    q.nch = (int)((L + kC - 1) / kC);
    q.ntiles = (q.nch + kCols - 1) / kCols;
    const int64_t slots = (int64_t)sm_count() * blocks_per_sm(M, bwd);
    const int64_t groups = B * (D / kCh);
    q.nseg = (int)std::max<int64_t>(1, std::min<int64_t>({slots / groups, (int64_t)q.ntiles, (int64_t)max_seg}));
    q.tps = (q.ntiles + q.nseg - 1) / q.nseg;
    q.nseg = (q.ntiles + q.tps - 1) / q.tps;
    // Packed rows cost a block nothing and divide their number by up to four: at B = 22,
    // L = 74, D = 88, M = 16 (fp32 backward with state terms) 484 blocks, just over one
    // wave, become 132: 63.6 -> 32.8 us.
    q.gpr = q.nch <= 4 ? 1 : q.nch <= 8 ? 2 : 4;
    q.zdim = (int)((B * q.gpr + 3) / 4);
    return q;
}

template <int J, int NP, bool BWD, bool kOut>
cudaError_t launch_scan(const ScanArgs &a, int nseg, int zdim, cudaStream_t st) {
    constexpr int bytes = smem_bytes(8 * J * NP, kOut);
    auto *k = k_scan<J, NP, BWD, kOut>;
    if (bytes > 48 * 1024) {
        // Once per device (a bit each; devices past 64 set it on every call).
        static std::atomic<unsigned long long> done{0};
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const unsigned long long bit = dev < 64 ? 1ull << dev : 0;
        if (!(done.load(std::memory_order_acquire) & bit)) {
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
            if (e != cudaSuccess) return e;
            done.fetch_or(bit, std::memory_order_release);
        }
    }
    const dim3 grid((unsigned)(a.D / kCh), (unsigned)nseg, (unsigned)zdim);
    count_launches(1);
    if (kOut && a.nseg > 1) return launch_dependent(k, grid, kThreads, bytes, st, a);
    k<<<grid, kThreads, bytes, st>>>(a);
    return cudaGetLastError();
}

template <bool BWD>
cudaError_t run_scan(ScanArgs &a, int zdim, cudaStream_t st) {
    auto pass = [&](auto out, int nseg) {
        constexpr bool kOut = decltype(out)::value;
        if (a.M <= 8) return launch_scan<1, 1, BWD, kOut>(a, nseg, zdim, st);
        if (a.M <= 16) return launch_scan<2, 1, BWD, kOut>(a, nseg, zdim, st);
        if (a.M <= 32) return launch_scan<4, 1, BWD, kOut>(a, nseg, zdim, st);
        return launch_scan<4, 2, BWD, kOut>(a, nseg, zdim, st);
    };
    if (a.nseg > 1) {
        const cudaError_t e = pass(std::false_type{}, a.nseg - 1);
        if (e != cudaSuccess) return e;
        if (!BWD && a.enter) a.enter = a.seg_s + (int64_t)(a.nseg - 1) * a.B * a.D * a.M;
    }
    return pass(std::true_type{}, a.nseg);
}

}  // namespace

// The workspace contract.  Sizes are stated in chunks of simt_chunk_len() tokens (8
// bytes per chunk, channel and mode; the backward in chunks of its own length, 24
// bytes); the segments above never need more (at most one state per 1024 tokens).
int simt_chunk_len(int64_t B, int64_t L, int D) {
    const int64_t target = (int64_t)sm_count() * 2048;
    const int64_t per_chunk = std::max<int64_t>(1, B * (int64_t)D);
    int64_t nch = (target + per_chunk - 1) / per_chunk;
    nch = std::max<int64_t>(1, nch);
    int64_t C = (L + nch - 1) / nch;
    C = std::max<int64_t>(16, std::min<int64_t>(1024, C));
    return (int)C;
}

namespace {
int bwd_ws_chunks(int64_t B, int64_t L, int D) {
    const int64_t target = (int64_t)sm_count() * 512;
    const int64_t per_chunk = std::max<int64_t>(1, B * (int64_t)D);
    const int64_t nch = std::max<int64_t>(1, (target + per_chunk - 1) / per_chunk);
    const int64_t C = std::max<int64_t>(16, std::min<int64_t>(4096, (L + nch - 1) / nch));
    return (int)((L + C - 1) / C);
}
}  // namespace

size_t simt_prefill_ws_bytes(int64_t B, int64_t L, int D, int M) {
    const int C = simt_chunk_len(B, L, D);
    return (size_t)B * ((L + C - 1) / C) * D * M * sizeof(float2);
}

size_t simt_backward_ws_bytes(int64_t B, int64_t L, int D, int M) {
    return 3 * (size_t)B * bwd_ws_chunks(B, L, D) * D * M * sizeof(float2);
}

cudaError_t simt_prefill(const void *x, void *y, rlm_dtype dt, int64_t B, int64_t L, int D,
                         int M, const float *decay, const float *freq, const float *amp,
                         const float *phase, const float *state_in, float *state_out, float *coef_out,
                         void *ws, cudaStream_t st) {
    const Geometry q = geometry(B, L, D, M, false, 1 << 15);
    ScanArgs a = {};
    a.u = x;
    a.out = y;
    a.bf16 = dt == RLM_BF16;
    a.L = L;
    a.B = (int)B;
    a.gpr = q.gpr;
    a.D = D;
    a.M = M;
    a.nch = q.nch;
    a.ntiles = q.ntiles;
    a.nseg = q.nseg;
    a.tps = q.tps;
    a.decay = decay;
    a.freq = freq;
    a.amp = amp;
    a.phase = phase;
    a.seg_s = static_cast<float2 *>(ws);   // nseg <= ceil(L / 1024) <= the contract's chunks
    a.enter = reinterpret_cast<const float2 *>(state_in);
    a.state_out = reinterpret_cast<float2 *>(state_out);
    a.coef_out = reinterpret_cast<float4 *>(coef_out);
    return run_scan<false>(a, q.zdim, st);
}

cudaError_t grad_reduce(int64_t nparts, int D, int M, const float *amp, const float *phase,
                        const float2 *G, const float2 *P, const float2 *J, float *g_decay, float *g_freq,
                        float *g_amp, float *g_phase, cudaStream_t st) {
    count_launches(1);
    return launch_dependent(k_grad_reduce, dim3((unsigned)((D * M + 255) / 256)), 256, 0, st, nparts, D, M, 1, amp, phase,
                            G, P, J, g_decay, g_freq, g_amp, g_phase);
}

cudaError_t simt_backward(const void *dy, const void *x, void *dx, rlm_dtype dt, int64_t B,
                          int64_t L, int D, int M, const float *decay, const float *freq,
                          const float *amp, const float *phase, const float *state_in,
                          const float *d_state_out, float *d_state_in, float *g_decay,
                          float *g_freq, float *g_amp, float *g_phase, void *ws, cudaStream_t st) {
    // A segment needs five workspace units (its pair, and its G, P and J partials)
    // where the contract states three a chunk; one segment keeps no pair.
    const Geometry q = geometry(B, L, D, M, true, std::max(1, 3 * bwd_ws_chunks(B, L, D) / 5));
    const int64_t unit = (int64_t)q.nseg * B * D * M;
    ScanArgs a = {};
    a.u = dy;
    a.x = x;
    a.out = dx;
    a.bf16 = dt == RLM_BF16;
    a.rev = 1;
    a.L = L;
    a.B = (int)B;
    a.gpr = q.gpr;
    a.D = D;
    a.M = M;
    a.nch = q.nch;
    a.ntiles = q.ntiles;
    a.nseg = q.nseg;
    a.tps = q.tps;
    a.decay = decay;
    a.freq = freq;
    a.amp = amp;
    a.phase = phase;
    a.part_g = static_cast<float2 *>(ws);
    a.part_p = a.part_g + unit;
    a.part_j = a.part_p + unit;
    a.seg_s = a.part_j + unit;
    a.seg_r = a.seg_s + unit;
    a.state_in = reinterpret_cast<const float2 *>(state_in);
    a.g = reinterpret_cast<const float2 *>(d_state_out);
    a.d_state_in = reinterpret_cast<float2 *>(d_state_in);
    const cudaError_t e = run_scan<true>(a, q.zdim, st);
    if (e != cudaSuccess) return e;
    return grad_reduce((int64_t)q.zdim * q.nseg, D, M, amp, phase, a.part_g, a.part_p, d_state_out ? a.part_j : nullptr, g_decay,
                       g_freq, g_amp, g_phase, st);
}

}  // namespace rlm
