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
// Sequences of at most 8 tokens take rlm_short.cu.  Up to 20 chunks, a wide tile's positions and
// columns would be mostly padding: there the narrow tile (4 chunks, one column a lane) is
// taken where use_narrow() says so.  In it a partial chunk alone leaves out the
// position blocks and chunk sums that it does not need, and above 32 modes two warps share
// a channel, 32 modes each.
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
// latency.  The wide backward above 32 modes also spills: 255 registers, 0.4 KB a thread.  GB300, us per call, against the three launches of token-by-token recurrences with
// chunk states in memory that this replaces:
//
//   fp32, B = 2, L = 4096, D = 512, M = 32: forward 247 -> 56, backward 303 -> 117
//   fp32, B = 4, L = 2048, D = 256, M = 48: forward and backward 162 (with the power table of
//     a whole chunk, one block a SM, 305)
//   bf16 from a state, B = 8, L = 1000, D = 256, M = 16: 75 -> 27
//   short or few: fp32 backward B = 8, L = 24, D = 768, M = 32 44 -> 13 (wide tiles 64); from a
//     state B = 64, L = 33, D = 768, M = 16 103 -> 52 (109).  Still slower than those: M > 32 in the
//     backward of one row of 64 channels at L = 500 to 1025 (1.2 to 1.9 x), M = 1 at B = 64, D = 2048,
//     L = 9 to 17 (1.2 to 1.5 x).
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
constexpr int kCh = 4;               // channels (warps) per block
constexpr int kThreads = 32 * kCh;
constexpr int kHalf = kC / 2;
// The power table holds lambda^n for n < 32 only (it is what limits the blocks a SM holds):
// products over a chunk run as two halves, joined by lambda^32.
constexpr int kPwStride = kHalf + 2;   // float2 per mode row: n < 32, then lambda^32 and lambda^64; rows 4 banks apart
// A tile of one channel, NC columns (chunks) a lane: 16 chunks (1024 tokens), or 4 (256) where
// the sequences are short or few, see geometry(): [p / 2][column][p % 2].  Row r holds
// positions 2 r and 2 r + 1, or mode r of W.  The padding puts the words that eight lanes
// write into eight rows in different banks, and leaves every address of the product loops a
// constant from the lane's.  (Permuted 16-byte words of unpadded rows cost an XOR, a shift
// and an add a load: forward and backward of B = 2, L = 4096, D = 512, M = 32 fp32 60.1 and 135
// us against 57.7 and 127.)
template <int NC>
struct Tile {
    static constexpr int kCols = 4 * NC, kTokens = kC * kCols;
    static constexpr int kRowWords = 2 * kCols + 4, kFieldWords = kHalf * kRowWords;
    static __device__ __forceinline__ constexpr int at(int r, int col) { return r * kRowWords + 2 * col; }
};
constexpr int kKernCopy = kC + 16;        // K reversed, then zeros (negative lags)
constexpr int kKernWords = 2 * kKernCopy; // that, and the same shifted by one

// Shared memory of a block, in floats: per channel the power table and c of every mode
// (complex), the reversed lag kernel, and for output passes two field tiles, the drive's
// and x's (forward: the second half's W).
// With the modes of a channel shared between two warps (hw = 2) each warp has tiles of its own
// for W as well.
constexpr int chan_words(int modes, int nc, int hw, bool out) {
    return 2 * modes * (kPwStride + 1) + kKernWords + (hw == 2 ? 6 : out ? 2 : 1) * (kHalf * (8 * nc + 4));
}
// Resident blocks a SM, for registers and shared memory alike.  (A third block at 17 to 32
// modes, with 168 registers a thread, made the forward of B = 2, L = 4096, D = 512, M = 32 fp32 70
// us against 62 and its backward 159 against 133.)  Narrow tiles (nc = 1) need fewer registers; at
// more than 32 modes their blocks have 256 threads.
__host__ __device__ constexpr int blocks_per_sm(int modes, int nc, bool bwd) {
    return nc == 1 ? (modes > 32 ? 2 : modes > 16 ? 4 : modes > 8 ? 5 : 6) : modes > 16 ? 2 : bwd ? 3 : 4;
}
constexpr int smem_bytes(int modes, int nc, int hw, bool out) { return kCh * chan_words(modes, nc, hw, out) * 4; }

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
// The (even, odd) position pairs of a lane's NC columns, cg its column group; and back.
template <int NC>
__device__ __forceinline__ void load_columns(const float *xs, int r, int cg, u64 (&v)[NC]) {
    const float *row = xs + Tile<NC>::at(r, NC * cg);
    if constexpr (NC == 4) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(row), b = *reinterpret_cast<const ulonglong2 *>(row + 4);
        v[0] = a.x;
        v[1] = a.y;
        v[2] = b.x;
        v[3] = b.y;
    } else {
        v[0] = *reinterpret_cast<const u64 *>(row);
    }
}
template <int NC>
__device__ __forceinline__ void store_columns(float *xs, int r, int cg, const float2 (&v)[NC]) {
    float *row = xs + Tile<NC>::at(r, NC * cg);
    if constexpr (NC == 4) {
        *reinterpret_cast<float4 *>(row) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
        *reinterpret_cast<float4 *>(row + 4) = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
    } else {
        *reinterpret_cast<float2 *>(row) = v[0];
    }
}
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
template <int NC, int J, bool JORDAN, bool TO_END>
__device__ __forceinline__ void project(const float2 *pw, const float *xs, int cg, u64 (&acc)[J][NC],
                                        u64 (&accq)[JORDAN ? J : 1][NC]) {
#pragma unroll
    for (int j = 0; j < J; ++j)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
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
                for (int c = 0; c < NC; ++c) {
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
            u64 x[NC];
            load_columns<NC>(xs, pp, cg, x);
            ulonglong2 a[J];
            const int n = TO_END ? kHalf - 2 - 2 * v0 : 2 * v0;
#pragma unroll
            for (int j = 0; j < J; ++j) a[j] = *reinterpret_cast<const ulonglong2 *>(pw + 8 * j * kPwStride + n);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int e = TO_END ? i : 1 - i;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const float2 v = unpack2(x[c]);
                    const u64 d = dup2(e ? v.y : v.x);
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
// Only blocks lo .. hi - 1 of 16 positions hold drives (NC = 1; else all four).
template <int NC, bool kGuard, int SG>
__device__ __forceinline__ void causal(const float *kq, const float *xs, int g, int cg, int lo, int hi, u64 (&acc)[8][NC]) {
#pragma unroll
    for (int s0 = 0; s0 < 4; s0 += SG) {
        if (NC == 1 && (s0 + SG <= lo || s0 >= hi)) continue;
#pragma unroll (SG == 4 ? 2 : 1)
        for (int u = 0; u < 8; ++u) {
            u64 x[SG][NC];   // positions 16 (s0 + i) + 2 u and the next
#pragma unroll
            for (int i = 0; i < SG; ++i) load_columns<NC>(xs, 8 * (s0 + i) + u, cg, x[i]);
#pragma unroll
            for (int l = 0; l < 4 - s0; ++l) {
                if (NC == 1 && s0 + l >= hi) break;
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
                        for (int c = 0; c < NC; ++c) {
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
                        for (int c = 0; c < NC; ++c) {
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
// p >= 32 take lambda^(p-32) and lambda^32 W (w2).  Rows of blocks hi and up are left out (NC = 1).
template <int NC>
__device__ __forceinline__ void up_project(const float2 *pw, const float *w1, const float *w2, int modes, int g, int cg,
                                           int hi, u64 (&acc)[8][NC]) {
#pragma unroll 2
    for (int m = 0; m < modes; ++m) {
        ulonglong2 a[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) a[j] = *reinterpret_cast<const ulonglong2 *>(pw + m * kPwStride + 16 * j + 2 * g);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (NC == 1 && 2 * h >= hi) break;
            u64 w[NC];
            load_columns<NC>(h ? w2 : w1, m, cg, w);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int r = 2 * (2 * h + j);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    fma2(acc[r][c], a[j].x, w[c]);
                    fma2(acc[r + 1][c], a[j].y, w[c]);
                }
            }
        }
    }
}

// lambda^n, n < 64, from a mode's table row.
__device__ __forceinline__ float2 power(const float2 *row, int n) {
    return n < kHalf ? row[n] : cmul(row[kHalf], row[n - kHalf]);
}

// Sums over the partial chunk in one column, for the lane's J modes of a group, in every
// lane: sum_{p < tail} lambda^(tail-1-p) x_p, or (JT) sum_{n < tail} n lambda^n x_{n + 64 - tail}.
// The four lanes of a mode take every fourth power, and lambda^(n+32) shares the table entry
// of lambda^n.  (A single lane walking the positions took up to 10 us of a call: B = 2, L = 4095,
// D = 512, M = 32 fp32 76.4 us against 66.2 at L = 4096.)
template <int NC, int J, bool JT>
__device__ __forceinline__ void partial_sums(const float2 *pw, const float *xs, int col, int tail, int cg, float2 (&f)[J]) {
    float2 hi[J];
#pragma unroll
    for (int j = 0; j < J; ++j) f[j] = hi[j] = make_float2(0.0f, 0.0f);
    auto x = [&](int n) {
        const int p = JT ? n + kC - tail : tail - 1 - n;
        return (JT ? p < kC : p >= 0) ? xs[Tile<NC>::at(p >> 1, col) + (p & 1)] : 0.0f;
    };
#pragma unroll (J == 1 ? 4 : 2)
    for (int n = cg; n < kHalf && n < tail; n += 4) {
        float v = x(n), w = x(n + kHalf);
        if (JT) {
            v *= (float)n;
            w *= (float)(n + kHalf);
        }
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const float2 z = pw[8 * j * kPwStride + n];
            f[j].x = fmaf(z.x, v, f[j].x);
            f[j].y = fmaf(z.y, v, f[j].y);
            hi[j].x = fmaf(z.x, w, hi[j].x);
            hi[j].y = fmaf(z.y, w, hi[j].y);
        }
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
        f[j] = cfma(pw[8 * j * kPwStride + kHalf], hi[j], f[j]);
#pragma unroll
        for (int o = 8; o <= 16; o <<= 1) {
            f[j].x += __shfl_xor_sync(0xffffffffu, f[j].x, o);
            f[j].y += __shfl_xor_sync(0xffffffffu, f[j].y, o);
        }
    }
}

// acc[n] += sum_u dy_u x_{u + 16 l + n} over the 16 positions u of block a, one column
// (the lane's); positions past the chunk count as zero.
template <int NC>
__device__ __forceinline__ void correlate(const float *dys, const float *xs, int col, int a, int l, float (&acc)[16]) {
    float dv[16], xv[32];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const float2 v = *reinterpret_cast<const float2 *>(dys + Tile<NC>::at(8 * a + u, col));
        dv[2 * u] = v.x;
        dv[2 * u + 1] = v.y;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float2 v = a + l + h < 4
                                 ? *reinterpret_cast<const float2 *>(xs + Tile<NC>::at(8 * (a + l + h) + u, col))
                                 : make_float2(0.0f, 0.0f);
            xv[16 * h + 2 * u] = v.x;
            xv[16 * h + 2 * u + 1] = v.y;
        }
#pragma unroll
    for (int u = 0; u < 16; ++u)
#pragma unroll
        for (int n = 0; n < 16; ++n) acc[n] = fmaf(dv[u], xv[u + n], acc[n]);
}

// v[n] summed over the tile's columns (4 NC consecutive lanes); lane `col` of them receives the
// lags n = 4 col / NC .. of the first 4 / NC entries.
template <int NC>
__device__ __forceinline__ void sum_columns(float (&v)[16], int col) {
#pragma unroll
    for (int o = 2 * NC, k = 8; o > 0; o >>= 1, k >>= 1) {
        const bool up = col & o;
#pragma unroll
        for (int n = 0; n < k; ++n) {
            const float keep = up ? v[n + k] : v[n], send = up ? v[n] : v[n + k];
            v[n] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
}

// One block: channels 4 blockIdx.x .. + 3 of batch row blockIdx.z, segment blockIdx.y.
// Sequences of at most NC (2 NC) chunks leave most of a tile's columns empty, so there a
// tile holds 4 (2) batch rows, one (two) column groups each, and blockIdx.z counts
// tiles: b below is then the lane's own row, clamped; `mine` says whether it exists.
// kOut: write outputs (else only the segment's end state, from zero).  HW = 2: the warp of
// modes 0 .. 31 forms the causal products, that of the others the lag correlation; both parts of K
// and of the outputs are added in shared memory.
template <int NC, int J, int NP, int HW, bool BWD, bool kOut>
__global__ void __launch_bounds__(HW * kThreads, blocks_per_sm(8 * J * NP * HW, NC, BWD)) k_scan(const ScanArgs A) {
    static_assert(HW == 1 || (NC == 1 && kOut), "two warps a channel: narrow tiles only");
    constexpr int kModes = 8 * J * NP;   // of a warp
    using T = Tile<NC>;
    constexpr int kCols = T::kCols, kTile = T::kTokens, kFieldWords = T::kFieldWords;
    constexpr int kPass = HW * kThreads / kCols, kPasses = kC / kPass;   // positions the threads stage at once
    constexpr bool kX = BWD && kOut;   // the x tile is needed
    constexpr int kSG = BWD && J == 4 ? 4 : 2;   // (see causal(); the forward with four: 55.6 -> 57.7 us)
    constexpr bool kAhead = NC == 4 && !BWD && J == 4;   // the next tile's drive is loaded a tile ahead
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, lane = tid & 31, w = (tid >> 5) & (kCh - 1);
    const int hm = HW == 2 ? tid >> 7 : 0;   // which of the channel's warps, modes 32 hm ..
    const int g = lane & 7, cg = lane >> 3;
    const int seg = blockIdx.y;
    const int rpt = 4 / A.gpr, gbase = cg & ~(A.gpr - 1);   // batch rows of a tile; the row's first column group
    const bool mine = (int)blockIdx.z * rpt + cg / A.gpr < A.B;
    const int64_t b = min((int)blockIdx.z * rpt + cg / A.gpr, A.B - 1);
    const int nrows = min(rpt, A.B - (int)blockIdx.z * rpt);   // rows that exist
    const int d0 = kCh * blockIdx.x, d = d0 + w, D = A.D;
    const int M = HW == 2 ? min(kModes, A.M - kModes * hm) : A.M;   // the warp's modes, its m-th at pm(m), bm(m)
    // (Formed where they are used: kept in registers they cost the fp32 training step at B = 2,
    // L = 4096, D = 512, M = 32 four of 175 us.)
    auto pm = [&](int m) { return d * A.M + kModes * hm + m; };
    auto bm = [&](int m) { return (b * D + d) * A.M + kModes * hm + m; };
    constexpr int kWords = chan_words(HW * kModes, NC, HW, kOut), kTable = 2 * kModes * (kPwStride + 1);
    constexpr int kTableWords = HW * kTable + kKernWords;   // before the field tiles
    float2 *pw = reinterpret_cast<float2 *>(smem + w * kWords + hm * kTable);
    float2 *cs = pw + kModes * kPwStride;        // c of every mode
    float *kq = smem + w * kWords + HW * kTable;
    float *us = kq + kKernWords;                 // drive tile; HW = 1: then W, then the output tile
    float *xs = us + (kOut ? kFieldWords : 0);   // x tile (backward); HW = 1: then lambda^32 W
    float *w1 = HW == 2 ? xs + (1 + 2 * hm) * kFieldWords : us, *w2 = HW == 2 ? w1 + kFieldWords : xs;
    pdl_launch_dependents();

    const int tail = (int)(A.L & (kC - 1));                 // tokens of the partial last chunk
    // A sequence of one partial chunk (on the narrow tile): drives in blocks lo .. hi - 1 of 16
    // positions only, no chunk before or after, so the chunk sums serve the state terms alone.
    const bool single = NC == 1 && A.nch == 1 && tail != 0;
    const bool ends = !single || (BWD && (A.state_in || A.d_state_in)), enters = !single || (!BWD && A.enter);
    const int lo = single && BWD ? (kC - tail) >> 4 : 0, hi = single && !BWD ? (tail + 15) >> 4 : 4;
    const int tile_end = min(A.ntiles, (seg + 1) * A.tps);
    // The thread's tokens of a tile, 4 channels each (zeros outside the sequence).
    const int Li = (int)A.L, t_last = A.nch * kC - 1;
    // The thread's column: its batch row, and its first token's tau in tile 0.
    const int fcol = tid & (kCols - 1), frow = (int)blockIdx.z * rpt + fcol / (NC * A.gpr);
    const int ftau = (fcol & (NC * A.gpr - 1)) * kC + tid / kCols;
    const int64_t fbase = (int64_t)frow * A.L;
    auto fetch = [&](const void *f, int tile, float4 (&v)[kPasses]) {
        const int tau = tile * kTile + ftau;
#pragma unroll
        for (int i = 0; i < kPasses; ++i) {
            const int t = A.rev ? t_last - tau - kPass * i : tau + kPass * i;
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
        for (int i = 0; i < kPasses; ++i) {
            const int t = A.rev ? t_last - tau - kPass * i : tau + kPass * i;
            if (t < 0 || t >= Li) continue;
            const int64_t at = ((fbase + t) * D + d0) * e;
            prefetch_l2(static_cast<const char *>(A.u) + at);
            if (kX) prefetch_l2(static_cast<const char *>(A.x) + at);
        }
    }
    float4 nextu[kPasses], nextx[kX ? kPasses : 1];

    // ---- tables: lambda^n, n < 32 (an exact power every 8, products between), 32 and 64
    {
        constexpr int kLpm = kModes >= 32 ? 1 : 32 / kModes;   // lanes per mode
#pragma unroll 1
        for (int m = lane / kLpm; m < kModes; m += 32) {
            float2 *row = pw + m * kPwStride;
            const bool on = m < M;
            const float ga = on ? A.decay[pm(m)] : 0.0f, om = on ? A.freq[pm(m)] : 0.0f;
            const float am = kOut && on ? A.amp[pm(m)] : 0.0f, ph = kOut && on ? A.phase[pm(m)] : 0.0f;
            if (!BWD && A.enter && on)   // used after the tables
                prefetch_l2(A.enter + ((int64_t)min((int)blockIdx.z * rpt, A.B - 1) * D + d) * A.M + kModes * hm + m);
            const float2 l1 = lambda_pow(ga, om, 1.0f);
#pragma unroll 1
            for (int n0 = 8 * (lane % kLpm); n0 < kHalf; n0 += 8 * kLpm) {
                float2 z = make_float2(0.0f, 0.0f);
                if (on && !(single && n0 > tail)) z = lambda_pow(ga, om, (float)n0);   // (zeros past a short sequence)
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
            const float ga = on ? A.decay[pm(m)] : 0.0f, om = on ? A.freq[pm(m)] : 0.0f;
            const float2 z = make_float2(0.0f, 0.0f);
            const int64_t sm = bm(m);
            S0[q][j] = !BWD && A.enter && on && mine && seg == 0 ? A.enter[sm] : z;
            if (BWD) R0[q][j] = z;
            if (kOut && seg > 0 && on) {
                // The earlier segments' end states, each carried over the segments between.
                const float nf = (float)(A.tps * kTile);
                const float2 lN = lambda_pow(ga, om, nf);
                const int64_t st = (int64_t)A.B * D * A.M;
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
                A.coef_out[pm(m)] = make_float4(l1.x, l1.y, cs[m].x, cs[m].y);
            }
            // The output launch's segment 0 starts from this copy: by then a state_out that
            // is state_in's buffer may be written by the last segment's block.
            if (!kOut && !BWD && seg == 0 && A.enter && cg == 0 && on)
                A.seg_s[sm + (int64_t)(A.nseg - 1) * A.B * D * A.M] = S0[q][j];
        }
    __syncwarp();
    if (kOut) {
        // K[n] = sum_m Re(c lambda^n), stored reversed (and once more shifted by one).
        float k0 = 0.0f, k1 = 0.0f;
        auto add = [&](int m) {
            const float2 c = cs[m], p = pw[m * kPwStride + lane], c2 = cmul(c, pw[m * kPwStride + kHalf]);
            k0 = fmaf(c.x, p.x, fmaf(-c.y, p.y, k0));
            k1 = fmaf(c2.x, p.x, fmaf(-c2.y, p.y, k1));
        };
        if constexpr (NC == 4) {   // (unrolled, the 16-mode backward of L = 8000 took 148 us against 144)
            for (int m = 0; m < M; ++m) add(m);
        } else {
#pragma unroll 4
            for (int m = 0; m < M; ++m) add(m);
        }
        if constexpr (HW == 2) {   // the first warp adds the second's part
            if (hm) {
                w1[lane] = k0;
                w1[32 + lane] = k1;
            }
            __syncthreads();
            if (!hm) {
                const float *o = w1 + 2 * kFieldWords;
                k0 += o[lane];
                k1 += o[32 + lane];
            }
        }
        if (!hm) {
            kq[63 - lane] = k0;
            kq[31 - lane] = k1;
            kq[kKernCopy + 62 - lane] = k0;
            if (lane < 31) kq[kKernCopy + 30 - lane] = k1;
            if (lane < 16) kq[kC + lane] = kq[kKernCopy + kC + lane] = 0.0f;
            if (lane == 0) kq[kKernCopy + kC - 1] = 0.0f;
        }
    }
    __syncwarp();

    float2 G[kX ? NP : 1][J], P[kX ? NP : 1][J], Jg[kX ? NP : 1][J];
    // NC = 4: lane (h, n): lags 16 h + n and 16 (3 - h) + n.  NC = 1: lane (h, col): lags
    // 4 col + i of the lag blocks that group h correlates.
    float rho_a[4 / NC] = {}, rho_b[4 / NC] = {};
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
        auto stage = [&](const float4 (&v)[kPasses], float *base) {
#pragma unroll
            for (int i = 0; i < kPasses; ++i) {
                const int p = tid / kCols + kPass * i, col = tid & (kCols - 1);
                float *o = base + T::at(p >> 1, col) + (p & 1);
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
        for (int i = 0; i < kPasses; ++i) {
            // x - x is zero for a finite x.
            const float z = (nextu[i].x - nextu[i].x) + (nextu[i].y - nextu[i].y) + (nextu[i].z - nextu[i].z) +
                            (nextu[i].w - nextu[i].w);
            odd |= !(z == 0.0f);
        }
        if constexpr (kX) stage(nextx, base + kFieldWords);
        const bool guard = __syncthreads_or(kOut && odd);

        // ---- chunk-local states, carry over the 16 columns (and G, P)
        const int chunk0 = tile * kCols + NC * (cg - gbase);   // the lane's first chunk
        u64 ls[NP][J][NC];   // lambda S of the state entering each of the lane's columns
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            u64 acc[J][NC], accq[BWD ? J : 1][NC];
            if (ends) {
                project<NC, J, BWD, true>(pw + (8 * J * q + g) * kPwStride, us, cg, acc, accq);
            } else {
#pragma unroll
                for (int j = 0; j < J; ++j)
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        acc[j][c] = 0ull;
                        if (BWD) accq[j][c] = 0ull;
                    }
            }
            float2 Rn[BWD ? J : 1][NC], send[BWD ? 1 : J];   // send: the state entering the partial last chunk
#pragma unroll
            for (int j = 0; j < J; ++j) {
                if (!ends) {   // nothing but the state entering the sequence
                    const float2 v = BWD ? make_float2(0.0f, 0.0f) : cmul(pw[(8 * J * q + 8 * j + g) * kPwStride + 1], S0[q][j]);
                    ls[q][j][0] = pack2(v.x, v.y);
                    if (!BWD) send[j] = S0[q][j];
                    continue;
                }
                const float2 *row = pw + (8 * J * q + 8 * j + g) * kPwStride;
                const float2 a = row[kHalf + 1], a2 = cmul(a, a), a4 = NC == 4 ? cmul(a2, a2) : a;   // a^NC
                const float2 lam = row[1];
                // The lane's columns from zero ...
                float2 es = make_float2(0.0f, 0.0f), er = es;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    if (BWD)
                        er = cfma(a, make_float2(fmaf((float)kC, es.x, er.x), fmaf((float)kC, es.y, er.y)),
                                  unpack2(accq[j][c]));
                    es = cfma(a, es, unpack2(acc[j][c]));
                }
                // ... the state entering them (over the mode's lanes in this row) ...
                float2 V = S0[q][j], U = BWD ? R0[q][j] : V, S = V, R = U;
                if (!BWD) send[j] = V;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (i >= A.gpr) break;   // the same for every lane
                    if (gbase + i == cg) {
                        S = V;
                        R = U;
                    }
                    const float2 ei = shfl2(es, g + 8 * (gbase + i));
                    if (BWD)
                        U = cfma(a4, make_float2(fmaf((float)(NC * kC), V.x, U.x), fmaf((float)(NC * kC), V.y, U.y)),
                                 shfl2(er, g + 8 * (gbase + i)));
                    V = cfma(a4, V, ei);
                }
                S0[q][j] = V;
                if (BWD) R0[q][j] = U;
                // ... and entering each of them.
                const int m = 8 * J * q + 8 * j + g;
                const bool on = m < M;
#pragma unroll
                for (int c = 0; c < (kOut ? NC : 0); ++c) {
                    const float2 lsv = cmul(lam, S);
                    ls[q][j][c] = pack2(lsv.x, lsv.y);
                    if (kX) {
                        Rn[j][c] = cmul(lam, R);
                        R = cfma(a, make_float2(fmaf((float)kC, S.x, R.x), fmaf((float)kC, S.y, R.y)),
                                 unpack2(accq[j][c]));
                        S = cfma(a, S, unpack2(acc[j][c]));
                        if (chunk0 + c == A.nch - 1 && on && mine) {
                            // The chunk of token 0: (S, R) is the adjoint pair there.
                            const int64_t sm = bm(m);
                            const float2 l0 = cmul(lam, S);
                            const float2 gg = A.g ? A.g[sm] : make_float2(0.0f, 0.0f);
                            const float2 lL =
                                A.g ? lambda_pow(A.decay[pm(m)], A.freq[pm(m)], (float)A.L) : gg;
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
                                send[j] = S;
                            else if (on && mine && A.state_out)
                                A.state_out[bm(m)] = next;
                        }
                        S = next;
                    }
                }
            }
            if (!BWD && kOut && tail && tile == A.ntiles - 1 && A.state_out)
                for (int r = 0; r < nrows; ++r) {
                    const int col = r * NC * A.gpr + (A.nch - 1 - tile * kCols);   // row r's last chunk
                    float2 f[J];
                    partial_sums<NC, J, false>(pw + (8 * J * q + g) * kPwStride, us, col, tail, cg, f);
#pragma unroll
                    for (int j = 0; j < J; ++j) {
                        const int m = 8 * J * q + 8 * j + g;
                        if (cg == col / NC && m < M)
                            A.state_out[bm(m)] = cfma(power(pw + m * kPwStride, tail), send[j], f[j]);
                    }
                }
            if (kX && !single) {
                u64 xp[J][NC], xq[J][NC];
                project<NC, J, true, false>(pw + (8 * J * q + g) * kPwStride, xs, cg, xp, xq);
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    const int m = 8 * J * q + 8 * j + g;
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const float2 s = unpack2(ls[q][j][c]), p = unpack2(xp[j][c]), v = unpack2(xq[j][c]);
                        G[q][j] = cfma(p, s, G[q][j]);
                        P[q][j] = cfma(p, Rn[j][c], cfma(v, s, P[q][j]));
                    }
                    if (A.g && m < M) {
                        // J over the whole chunks: L - 1 - t = E + p with E = L minus the chunk's end.
                        const float ga = A.decay[pm(m)], om = A.freq[pm(m)];
                        float2 z = make_float2(0.0f, 0.0f);
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            const int64_t E = A.L - (int64_t)(A.nch - chunk0 - c) * kC;
                            if (E >= 0 && chunk0 + c < A.nch) {
                                z = c == 0 || E < kC ? lambda_pow(ga, om, (float)E) : cmul(z, pw[m * kPwStride + kHalf + 1]);
                                const float2 p = unpack2(xp[j][c]), v = unpack2(xq[j][c]);
                                const float Ef = (float)(E - 1);
                                Jg[q][j] = cfma(z, make_float2(fmaf(Ef, p.x, v.x), fmaf(Ef, p.y, v.y)), Jg[q][j]);
                            }
                        }
                    }
                }
            }
            if (kX && A.g && tail && tile == 0) {
                // The partial last chunk (each row's first column): its tokens are
                // positions p >= 64 - tail, with L - 1 - t = p - (64 - tail).
                if constexpr (NC == 4) {   // (most rows of a wide tile exist: shared out among a row's lanes)
#pragma unroll
                    for (int j = 0; j < J; ++j) {
                        const float2 *row = pw + (8 * J * q + 8 * j + g) * kPwStride;
                        for (int n = cg - gbase; n < tail; n += A.gpr) {
                            const int p = n + kC - tail;
                            const float v = (float)n * xs[T::at(p >> 1, NC * gbase) + (p & 1)];
                            const float2 z = power(row, n);
                            Jg[q][j].x = fmaf(z.x, v, Jg[q][j].x);
                            Jg[q][j].y = fmaf(z.y, v, Jg[q][j].y);
                        }
                    }
                } else {
                    for (int r = 0; r < nrows; ++r) {
                        float2 f[J];
                        partial_sums<NC, J, true>(pw + (8 * J * q + g) * kPwStride, xs, r * NC * A.gpr, tail, cg, f);
#pragma unroll
                        for (int j = 0; j < J; ++j)
                            if (cg == r * A.gpr) Jg[q][j] = make_float2(Jg[q][j].x + f[j].x, Jg[q][j].y + f[j].y);
                    }
                }
            }
        }
        if (!kOut) {
            if (kAhead && tile + 1 < tile_end) fetch(A.u, tile + 1, nextu);
            __syncthreads();   // every warp is done with the tile
            continue;
        }
        if (kX && hm == HW - 1) {
            float r0[16], r1[16];
#pragma unroll
            for (int n = 0; n < 16; ++n) r0[n] = r1[n] = 0.0f;
            const int col = lane & (kCols - 1), h = lane / kCols;
            if constexpr (NC == 4) {
                // Lag correlation: lane = (column, half); the half takes lag blocks {0, 3} or
                // {1, 2}, whose 10 non-empty (u block, lag block) pairs fall in 4 + 2 steps.
#pragma unroll 1
                for (int a = 0; a < 4; ++a) correlate<NC>(us, xs, col, a, h, r0);
#pragma unroll 1
                for (int a = 0; a < 2; ++a) correlate<NC>(us, xs, col, a, 3 - h, r1);
            } else {
                // Eight lane groups h take one pair each, then two of them the rest (lag block 2):
                // (h, 0), h < 4; (h - 4, 1), h < 7; (0, 3); (h, 2), h < 2.
                correlate<NC>(us, xs, col, h == 7 ? 0 : h & 3, h < 4 ? 0 : h < 7 ? 1 : 3, r0);
                if (hi - lo > 2 && h < 2) correlate<NC>(us, xs, col, h, 2, r1);
            }
            sum_columns<NC>(r0, col);
            sum_columns<NC>(r1, col);
#pragma unroll
            for (int i = 0; i < 4 / NC; ++i) {
                rho_a[i] += r0[i];
                rho_b[i] += r1[i];
            }
        }

        // ---- outputs
        u64 acc[8][NC];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[r][c] = 0ull;
        if (hm == 0) {
            if (guard)
                causal<NC, true, kSG>(kq, us, g, cg, lo, hi, acc);
            else
                causal<NC, false, kSG>(kq, us, g, cg, lo, hi, acc);
        }
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            if (!enters) break;
            __syncwarp();   // the warp is done reading the tile (or the previous W)
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int m = 8 * J * q + 8 * j + g;
                float2 W[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const float2 v = cmul(cs[m], unpack2(ls[q][j][c]));
                    W[c] = m < M ? make_float2(v.x, -v.y) : make_float2(0.0f, 0.0f);
                }
                if (kX && A.g && m < M) {
                    // Terminal-state gradient: its adjoint conj(g) lambda^(L-1-t) enters a
                    // whole chunk as conj(g) lambda^E with E = L minus the chunk's end.
                    const float ga = A.decay[pm(m)], om = A.freq[pm(m)];
                    const float2 gg = A.g[bm(m)];
                    float2 z = make_float2(0.0f, 0.0f);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const int64_t E = A.L - (int64_t)(A.nch - chunk0 - c) * kC;
                        if (E >= 0 && chunk0 + c < A.nch) {
                            z = c == 0 || E < kC ? lambda_pow(ga, om, (float)E) : cmul(z, pw[m * kPwStride + kHalf + 1]);
                            const float2 v = cmul(make_float2(gg.x, -gg.y), z);
                            W[c].x += v.x;
                            W[c].y -= v.y;
                        }
                    }
                }
                store_columns<NC>(w1, 8 * j + g, cg, W);
                const float2 l32 = conj2(pw[m * kPwStride + kHalf]);   // (W is kept conjugated)
#pragma unroll
                for (int c = 0; c < NC; ++c) W[c] = cmul(l32, W[c]);
                store_columns<NC>(w2, 8 * j + g, cg, W);
            }
            __syncwarp();
            if (kAhead && q == NP - 1 && tile + 1 < tile_end) fetch(A.u, tile + 1, nextu);
            up_project<NC>(pw + 8 * J * q * kPwStride, w1, w2, min(8 * J, M - 8 * J * q), g, cg, hi, acc);
        }
        float y[8][NC];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const float2 v = unpack2(acc[r][c]);
                y[r][c] = v.x + v.y;
            }
        if (kX && A.g && tail && tile == 0) {
            // The terminal-state term of the partial last chunk.  Narrow tiles, whose blocks are few
            // and wait for nothing else here, take g through the tiles' memory (free by now) so
            // that its loads are in flight together: one after the other
            // they took 50k cycles of a block at M = 64, L = 48.
            float2 *gs = reinterpret_cast<float2 *>(w1);   // [mode][row]
            if constexpr (NC == 1) {
                __syncwarp();
                for (int m = g; m < M && chunk0 == 0; m += 8) gs[m * 4 + cg] = A.g[bm(m)];
                __syncwarp();
            }
            for (int m = 0; m < M && chunk0 == 0; ++m) {
                const float2 gg = NC == 1 ? gs[m * 4 + cg] : A.g[bm(m)];
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
        auto store_y = [&] {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float2 v[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) v[c] = make_float2(y[2 * j][c], y[2 * j + 1][c]);
                store_columns<NC>(w1, 8 * j + g, cg, v);
            }
        };
        if constexpr (HW == 2) {   // the first warp adds the second's part
            if (hm) store_y();
            __syncthreads();
            if (!hm) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    u64 o[NC];
                    load_columns<NC>(w1 + 2 * kFieldWords, 8 * j + g, cg, o);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const float2 v = unpack2(o[c]);
                        y[2 * j][c] += v.x;
                        y[2 * j + 1][c] += v.y;
                    }
                }
            }
        }
        if (hm == 0) store_y();
        __syncthreads();
        // HW = 1: a thread reads here the words it wrote when staging, and writes them again for
        // the next tile: no barrier is needed between.  HW = 2: staging writes other words.
#pragma unroll
        for (int i = 0; i < kPasses; ++i) {
            const int p = tid / kCols + kPass * i, col = tid & (kCols - 1);
            const float *o = base + (HW == 2 ? 2 * kFieldWords : 0) + T::at(p >> 1, col) + (p & 1);
            const int t = A.rev ? t_last - t0 - kPass * i : t0 + kPass * i;
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
                    const int64_t o = (((int64_t)seg * A.B + b) * D + d) * A.M + m;
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
        const int h = lane / kCols, col = lane & (kCols - 1);
        __syncwarp();
        if (hm != HW - 1) {
        } else if constexpr (NC == 4) {
            kq[16 * h + col] = rho_a[0];
            kq[16 * (3 - h) + col] = rho_b[0];
        } else {
            kq[lane] = kq[32 + lane] = 0.0f;
#pragma unroll 1
            for (int k = 0; k < 8; ++k) {   // the groups of a lag block one after the other
                __syncwarp();
                if (k != h) continue;
                float *o = kq + 16 * (h < 4 ? 0 : h < 7 ? 1 : 3) + 4 * col, *o2 = kq + 32 + 4 * col;
#pragma unroll
                for (int i = 0; i < 4 / NC; ++i) {
                    o[i] += rho_a[i];
                    if (h < 2) o2[i] += rho_b[i];
                }
            }
        }
        if (HW == 2) __syncthreads();
        __syncwarp();
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            float2 gw[J], pn[J];
#pragma unroll
            for (int j = 0; j < J; ++j) gw[j] = pn[j] = make_float2(0.0f, 0.0f);
#pragma unroll 2
            for (int n = 16 * cg; n < 16 * cg + 16; ++n) {
                const float r = kq[n], nr = (float)n * r;
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    const float2 z = pw[(8 * J * q + 8 * j + g) * kPwStride + (n & (kHalf - 1))];
                    gw[j].x = fmaf(z.x, r, gw[j].x);
                    gw[j].y = fmaf(z.y, r, gw[j].y);
                    pn[j].x = fmaf(z.x, nr, pn[j].x);
                    pn[j].y = fmaf(z.y, nr, pn[j].y);
                }
            }
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int m = 8 * J * q + 8 * j + g;
                float2 js = Jg[q][j];
                if (A.g && m < M && mine) {
                    // conj(g) J, g the lane's row's.
                    const float2 gg = A.g[bm(m)];
                    js = cmul(make_float2(gg.x, -gg.y), js);
                }
                const float2 up = cg < 2 ? make_float2(1.0f, 0.0f) : pw[m * kPwStride + kHalf];
                float2 gs = cfma(up, gw[j], G[q][j]), ps = cfma(up, pn[j], P[q][j]);
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
                    const int64_t o = (((int64_t)blockIdx.z * A.nseg + seg) * D + d) * A.M + kModes * hm + m;
                    A.part_g[o] = gs;
                    A.part_p[o] = ps;
                    if (A.g) A.part_j[o] = js;
                }
            }
        }
    }
}

// One thread per (d, m): fixed-order sum of its n partials, then the four gradients.  The
// sums are compensated (Kahan) fp32 sums, so the result is reproducible and its error stays
// near one rounding however many partials are added; the combination with
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
    int64_t n, int D, int M, const float *__restrict__ amp,
    const float *__restrict__ phase, const float2 *ws_s, const float2 *ws_r, const float2 *ws_j, float *__restrict__ g_decay,
    float *__restrict__ g_freq, float *__restrict__ g_amp, float *__restrict__ g_phase) {
    const int pm = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();
    if (pm >= D * M) return;
    const float am = amp[pm], ph = phase[pm];
    KahanSum gr, gi, pr, pi, jr, ji;
    const int64_t stride = (int64_t)D * M;
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
    int zdim;      // blocks along the batch
    bool narrow;   // tiles of 4 chunks
};

// Whether narrow tiles (4 chunks) are faster than wide ones (16): estimated walks, in wide
// tiles.  A narrow tile takes `tile` of a wide one's time, and from `share` blocks a SM on
// blocks share the SM's time; fitted to 73 to 438 shapes a line (B = 1 to 64, L = 65 to 1025,
// D = 64 to 2048).  Beyond 20 chunks wide tiles win, by their segments too.  Us a call in fp32,
// wide and narrow: backward B = 1, L = 65, D = 64, M = 64 55 and 19; B = 1, L = 193, D = 256, M = 17
// 28 and 16; forward from a state B = 1, L = 65, D = 256, M = 64 20 and 12; wide is taken for the
// backward of B = 64, L = 193, D = 64, M = 16, 26 and 42.
bool use_narrow(int64_t B, int nch, int D, int M, bool bwd) {
    struct Cost {
        double tile, share1, share4;
    };
    static const Cost kCost[2][4] = {{{0.55, 1.5, 1.25}, {0.5, 1.0, 1.0}, {0.6, 1.5, 1.25}, {0.5, 1.0, 1.0}},
                                     {{0.6, 1.5, 1.25}, {0.65, 1.5, 1.25}, {0.4, 2.0, 1.5}, {0.3, 1.25, 1.25}}};
    const Cost &c = kCost[bwd][M <= 8 ? 0 : M <= 16 ? 1 : M <= 32 ? 2 : 3];
    auto walk = [&](int nc, double share) {
        const int gpr = nch <= nc ? 1 : nch <= 2 * nc ? 2 : 4;
        const double blocks = (double)((B * gpr + 3) / 4 * (D / kCh));
        return ((nch + 4 * nc - 1) / (4 * nc)) * std::max(1.0, blocks / (share * sm_count()));
    };
    return nch == 1 || (nch <= 20 && c.tile * walk(1, c.share1) < walk(4, c.share4));
}

Geometry geometry(int64_t B, int64_t L, int D, int M, bool bwd, int max_seg) {
    Geometry q;
    q.nch = (int)((L + kC - 1) / kC);
    q.narrow = use_narrow(B, q.nch, D, M, bwd);
    const int nc = q.narrow ? 1 : 4;
    q.ntiles = (q.nch + 4 * nc - 1) / (4 * nc);
    const int64_t slots = (int64_t)sm_count() * blocks_per_sm(M, nc, bwd);
    const int64_t groups = B * (D / kCh);
    q.nseg = q.narrow ? 1 : (int)std::max<int64_t>(1, std::min<int64_t>({slots / groups, (int64_t)q.ntiles, (int64_t)max_seg}));
    q.tps = (q.ntiles + q.nseg - 1) / q.nseg;
    q.nseg = (q.ntiles + q.tps - 1) / q.tps;
    // Packed rows cost a block nothing and divide their number by up to four: at B = 22,
    // L = 74, D = 88, M = 16 (fp32 backward with state terms) 484 blocks, just over one
    // wave, become 132: 63.6 -> 32.8 us.
    q.gpr = q.nch <= nc ? 1 : q.nch <= 2 * nc ? 2 : 4;
    q.zdim = (int)((B * q.gpr + 3) / 4);
    return q;
}

template <int NC, int J, int NP, int HW, bool BWD, bool kOut>
cudaError_t launch_scan(const ScanArgs &a, int nseg, int zdim, cudaStream_t st) {
    constexpr int bytes = smem_bytes(8 * J * NP * HW, NC, HW, kOut);
    auto *k = k_scan<NC, J, NP, HW, BWD, kOut>;
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
    if (kOut && a.nseg > 1) return launch_dependent(k, grid, HW * kThreads, bytes, st, a);
    k<<<grid, HW * kThreads, bytes, st>>>(a);
    return cudaGetLastError();
}

template <int NC, bool BWD, bool kOut>
cudaError_t pass_scan(const ScanArgs &a, int nseg, int zdim, cudaStream_t st) {
    if (a.M <= 8) return launch_scan<NC, 1, 1, 1, BWD, kOut>(a, nseg, zdim, st);
    if (a.M <= 16) return launch_scan<NC, 2, 1, 1, BWD, kOut>(a, nseg, zdim, st);
    if (a.M <= 32) return launch_scan<NC, 4, 1, 1, BWD, kOut>(a, nseg, zdim, st);
    if constexpr (NC == 1) return launch_scan<1, 4, 1, 2, BWD, kOut>(a, nseg, zdim, st);
    else return launch_scan<NC, 4, 2, 1, BWD, kOut>(a, nseg, zdim, st);
}

template <bool BWD>
cudaError_t run_scan(ScanArgs &a, const Geometry &q, cudaStream_t st) {
    if (q.narrow) return pass_scan<1, BWD, true>(a, 1, q.zdim, st);
    if (a.nseg > 1) {
        const cudaError_t e = pass_scan<4, BWD, false>(a, a.nseg - 1, q.zdim, st);
        if (e != cudaSuccess) return e;
        if (!BWD && a.enter) a.enter = a.seg_s + (int64_t)(a.nseg - 1) * a.B * a.D * a.M;
    }
    return pass_scan<4, BWD, true>(a, a.nseg, q.zdim, st);
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
    if (short_supported(L))
        return short_prefill(x, y, dt, B, L, D, M, decay, freq, amp, phase, state_in, state_out, coef_out, st);
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
    return run_scan<false>(a, q, st);
}

cudaError_t grad_reduce(int64_t nparts, int D, int M, const float *amp, const float *phase,
                        const float2 *G, const float2 *P, const float2 *J, float *g_decay, float *g_freq,
                        float *g_amp, float *g_phase, cudaStream_t st) {
    count_launches(1);
    return launch_dependent(k_grad_reduce, dim3((unsigned)((D * M + 255) / 256)), 256, 0, st, nparts, D, M, amp, phase,
                            G, P, J, g_decay, g_freq, g_amp, g_phase);
}

cudaError_t simt_backward(const void *dy, const void *x, void *dx, rlm_dtype dt, int64_t B,
                          int64_t L, int D, int M, const float *decay, const float *freq,
                          const float *amp, const float *phase, const float *state_in,
                          const float *d_state_out, float *d_state_in, float *g_decay,
                          float *g_freq, float *g_amp, float *g_phase, void *ws, cudaStream_t st) {
    if (short_supported(L)) {
        const int64_t n = B * D * M;   // the contract holds three units a row
        float2 *pg = static_cast<float2 *>(ws), *pp = pg + n, *pj = pp + n;
        const cudaError_t e = short_backward(dy, x, dx, dt, B, L, D, M, decay, freq, amp, phase, state_in, d_state_out,
                                             d_state_in, pg, pp, pj, st);
        if (e != cudaSuccess) return e;
        return grad_reduce(B, D, M, amp, phase, pg, pp, d_state_out ? pj : nullptr, g_decay, g_freq, g_amp, g_phase, st);
    }
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
    const cudaError_t e = run_scan<true>(a, q, st);
    if (e != cudaSuccess) return e;
    return grad_reduce((int64_t)q.zdim * q.nseg, D, M, amp, phase, a.part_g, a.part_p, d_state_out ? a.part_j : nullptr, g_decay,
                       g_freq, g_amp, g_phase, st);
}

}  // namespace rlm
