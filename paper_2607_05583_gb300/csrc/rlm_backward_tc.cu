// rlm_backward_tc.cu -- tcgen05 tensor-core backward pass for bf16 I/O, M <= 32.
//
// The loss depends on y = K * x (Eq. 2, K[n] = sum_m Re(c_m lambda_m^n)), so with
// the adjoint drive dy:
//
//   dx[t]  = sum_{s>=t} K[s-t] dy[s]                       anti-causal mixing
//   G_m    = sum_t x[t] S^_m[t],  S^_m[t] = sum_{s>=t} lambda^(s-t) dy[s]
//   P_m    = sum_t x[t] R^_m[t],  R^_m[t] = sum_{s>=t} (s-t) lambda^(s-t) dy[s]
//
// and the four parameter gradients follow from G and P and c = A e^{i phi}
// (dA = Re(e^{i phi} G), dphi = -Im(c G), dgamma = -Re(c P), domega = -Im(c P)).
//
// Chunked form.  With chunks of C = 64 tokens, position i of chunk k, the pair
// entering chunk k from the right (S^n_k = S^(kC + C), R^n_k likewise) and
// a = lambda^C:
//
//   Dp_k = sum_i lambda^i dy_{k,i}        Dq_k = sum_i i lambda^i dy_{k,i}
//   S^ at chunk start:  S^_k = a S^n_k + Dp_k
//   R^ at chunk start:  R^_k = a (R^n_k + C S^n_k) + Dq_k
//   cross-chunk terms:  G += sum_i lambda^(C-i) E_S[i],
//                       P += sum_i lambda^(C-i) (E_R[i] + (C-i) E_S[i]),
//                       E_S[i] = sum_k S^n_k x_{k,i},  E_R[i] = sum_k R^n_k x_{k,i}
//   within-chunk terms: G += sum_n lambda^n rho[n],  P += sum_n n lambda^n rho[n],
//                       rho[n] = sum_k sum_i dy_{k,i+n} x_{k,i}   (0 <= n < C)
//   dx_{k,i} = sum_{j>=i} K[j-i] dy_{k,j} + sum_m Re(c lambda^(C-i) S^n_k)
//
// Every sum over the positions or the chunks of a tile is a dense product and
// runs on the tensor cores (tcgen05.mma, kind::f16, bf16 operands, fp32
// accumulators in TMEM), 32 chunks (a 2048-token tile) at a time:
//
//   accP  = [Vp ; Vq] (128 x 64) DY   the lambda^i rows as bf16 high parts plus
//           low parts (an extra M = 64 product): dgamma = -Re(c P) can be a
//           near-orthogonal projection of a large P, so single-bf16 powers cost
//           up to 2 % there
//   accD  = T' (64 x 64) DY + U' (64 x 64) S^n      (T'[i][j] = K[j-i], j >= i)
//   accQ += [DY^T ; X^T] X   over all tiles: Q[i][j] = sum_k dy_{k,i} x_{k,j},
//           whose sub-diagonals i - j = n are rho[n]
//   accE += [S^n ; R^n] X    over all tiles (K = chunks; the pair as bf16 high
//           plus low parts): E_S and E_R, weighted by lambda^(C-i) once at the end
//
// The chunk scan of (S^, R^) runs in reverse time in fp32 registers: the warp
// of TMEM quarter q carries modes 8q .. 8q+7 with four lanes per mode, lane l
// reading accumulator row 32q + l (the Re / Im rows of Dp and of Dq); all four
// carry the mode's complex pair (no shuffle on the recurrence), and each records
// its own component for row 32q + l of the [S^n ; R^n] operand.
//
// Data layout.  The per-channel tables (40 KB) leave room for one channel per
// CTA, so the backward works on a channel-major copy of x and dy ([B*D][Lp] bf16,
// Lp = L rounded up to whole tiles, zero past L), written by a transpose kernel:
// every tile of one channel is then 4 KB of contiguous memory, which TMA loads
// with the 128-byte swizzle straight into the K-major operand layout.  dx is
// written channel-major (64-byte runs per warp store) and a second transpose
// writes the [B][L][D] field.
//
// One CTA = one channel of one or more batch rows (RowPlan below; the tables are the
// channel's, the carry and the sums Q and E restart at each row), two CTAs per SM (256
// TMEM columns each):
//   warps 0-3  reverse scan; at a row's end they read E, form the cross-chunk (G, P), add
//              rho and write the row's partials.
//   warps 4-5  dx epilogue (quarters 0, 1: positions 0-63); at a row's end the diagonal
//              sums rho of Q.
//   warp 6     TMA producer, which loads while the others build the tables.
//   warp 7     TMEM allocation (and the tables, with warps 0-5 and 8-9).
//   warp 8     MMA issue: projections and Q; warp 9: T', U' and E.
//   The kernel may start while the input transposes drain (pdl_wait): only the producer
//   waits for them, so the tables are built meanwhile.
// Several rows a CTA (kRows): TMEM additions truncate, so Q and E are summed over one row
// only, as with one row a CTA, and the rows' (G, P) are added in compensated fp32 by
// k_grad_reduce.  Both leave TMEM while the next row's first tile is projected and
// scanned; Q moves to warp 9, whose next products overwrite them.  (Summed over up to 16
// tiles in TMEM the error of dA against 64 bits at B = 8, L = 4096, D = 256, M = 16 was 2.68e-6
// against 2.59e-6, mean of 8 seeds; now 2.59e-6.  That took 51 us a call where this takes 68 and one
// row a CTA 90; 85, 105 and 145 with both state terms.  Q and E issued by warp 7 instead:
// as fast for several rows, 20 us slower for one of 16 tiles.)
//
// Every wait is bounded: after kWaitLimitCycles the waiting thread sets a shared
// abort flag and the device status word (RLM_ERR_TIMEOUT); all roles then leave
// their loops, drain what they issued, and the CTA frees its TMEM and returns.
#include <cuda.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "rlm_device.cuh"
#include "rlm_internal.h"

namespace rlm {

// Device status word of this translation unit (RLM_OK or RLM_ERR_TIMEOUT).
__device__ int g_bwd_status = 0;

namespace {

constexpr int kC = 64;                 // chunk length
constexpr int kNT = 32;                // chunks per tile
constexpr int kTile = kC * kNT;        // 2048 tokens
constexpr int kMaxModes = 32;          // one scan lane per mode
constexpr int kWarps = 10;
constexpr int kThreads = kWarps * 32;
constexpr int kSlots = 4;              // tile ring depth (dy + x per slot)
constexpr int kTmemCols = 256;
constexpr long long kWaitLimitCycles = 4000000000ll;  // about 2 s at 2 GHz

// TMEM columns.
constexpr int kColP = 0;     // [2] x 32: [Vp ; Vq] DY
constexpr int kColD = 64;    // [2] x 32: dx
constexpr int kColQ = 128;   // 64: DY^T X over the sequence
constexpr int kColE = 192;   // 64: [S^n ; R^n] X over the sequence

// Shared memory map (bytes from a 1024-aligned base).
// Tables, K-major without swizzle (8-row x 16-byte core matrices, LBO 128 between
// K groups, SBO 1024 between row groups):
//   U'    (64 rows, K = 64 state rows 2m + ri)  at 0
//   T'    (64 rows, K = 64 positions)           at 8192
//   A_P   (128 rows, K = 64 positions)          at 16384
//   A_Plo (64 rows: low parts of the Vp rows)   at 32768
// A_P row 32 q + l: l < 16 the (Re, Im) row l % 2 of the Vp part of mode
// 8 q + l / 2, l >= 16 that of the Vq part of mode 8 q + (l - 16) / 2.
// Low-part row 16 q + l (l < 16) lands, through the M = 64 accumulator layout
// (lanes 0-15 of each quarter), on lane 32 q + l: the same Vp row.
// A 128-row operand starting at U' reads T' as its rows 64-127, one starting at
// T' reads the first half of A_P: those accumulator rows are never read.
constexpr int kOffU = 0;
constexpr int kOffT = 8192;
constexpr int kOffAP = 16384;
constexpr int kOffAPlo = 32768;
constexpr int kOffRing = 40960;                 // [kSlots] x (dy 4 KB, x 4 KB)
constexpr int kSlotBytes = 8192;
// The carried pair [S^n ; R^n] (128 rows x 32 chunks, bf16), high parts then
// low parts, double-buffered.  Row 32 q + l follows the A_P row layout (S^n for
// l < 16, R^n for l >= 16).  Element (row r, chunk k) at
// (r / 8) * 512 + (k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2: the K-major A
// operand of the E product (LBO 128, SBO 512), and, restricted to the S^n rows of
// one quarter, the MN-major B operand of the up-projection (N = chunks, SBO 128;
// K = the 16 S^n rows, LBO 512).
constexpr int kOffBs = kOffRing + kSlots * kSlotBytes;   // [2] x (hi 8 KB, lo 8 KB)
constexpr int kBsBuf = 16384;
// rho[n] of a row, double-buffered: the part of each epilogue warp's 32 rows of Q.
constexpr int kOffRho = kOffBs + 2 * kBsBuf;             // [2][2][64] fp32
// 16 columns of an epilogue warp's 32 rows of Q, row i - c of element (i, c): every row is a
// diagonal.  Cells that no element meets stay zero.
constexpr int kQsRows = 47, kQsStride = 18;
constexpr int kOffQs = kOffRho + 2 * 2 * 64 * 4;         // [2 warps][47][18] fp32
constexpr int kOffBar = kOffQs + 2 * kQsRows * kQsStride * 4;
constexpr int kNumBars = 32;
constexpr int kOffMisc = kOffBar + kNumBars * 8;
constexpr int kSmemBytes = kOffMisc + 64 + 1024;         // + alignment slack
static_assert(kOffRing % 1024 == 0 && kSlotBytes % 1024 == 0, "swizzled tiles need 1024-byte alignment");
static_assert(2 * (kSmemBytes + 1024) <= 233472, "two CTAs per SM");
// Prologue scratch (lambda^n for n = 0..64, c, K), in the carried-pair buffers,
// which nobody touches before the prologue ends.
constexpr int kPwStride = 65;
constexpr int kOffPw = kOffBs;                                  // [32][65] float2
constexpr int kOffCf = kOffPw + kMaxModes * kPwStride * 8;      // [32] float2
constexpr int kOffK = kOffCf + kMaxModes * 8;                   // [64] float
static_assert(kOffK + 64 * 4 <= kOffRho, "prologue scratch does not fit");

// Barrier indices.
constexpr int kBarSlotFull = 0;                  // [kSlots]
constexpr int kBarSlotEmpty = kSlots;            // [kSlots]: scan warp 0 + epilogue warp 4
constexpr int kBarPFull = 2 * kSlots;            // [2]: projections (one row a block: and Q) committed
constexpr int kBarPEmpty = kBarPFull + 2;        // [2]: 4 scan warps read them
constexpr int kBarSFull = kBarPEmpty + 2;        // [2]: 4 scan warps wrote [S^n ; R^n]
constexpr int kBarBsEmpty = kBarSFull + 2;       // [2]: U' and E products done with it
constexpr int kBarDFull = kBarBsEmpty + 2;       // [2]: dx accumulator (and E) complete
constexpr int kBarDEmpty = kBarDFull + 2;        // [2]: 2 epilogue warps read it
constexpr int kBarRowFull = kBarDEmpty + 2;      // a row's Q and E complete
constexpr int kBarRowFree = kBarRowFull + 1;     // ... and read: 4 scan + 2 epilogue warps
constexpr int kBarRhoFull = kBarRowFree + 1;     // [2]: 2 epilogue warps wrote rho of a row
constexpr int kBarRhoEmpty = kBarRhoFull + 2;    // [2]: 4 scan warps read it
static_assert(kBarRhoEmpty + 2 <= kNumBars, "too many barriers");

// ------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
// A waiting thread is suspended until the phase completes or about 0.2 ms pass,
// so idle roles do not take issue slots from the scan.
__device__ __forceinline__ bool bar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(200000u)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void bar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}
// Bounded wait on an mbarrier phase; false once this CTA has aborted.
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
    if (bar_try(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
        if (bar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > kWaitLimitCycles) {
            *abort_flag = 1;
            atomicExch(&g_bwd_status, (int)RLM_ERR_TIMEOUT);
            return false;
        }
    }
}
// The same for a whole warp: one answer for all its lanes, which then stay together.
__device__ __forceinline__ bool wait_bar_warp(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
    return __all_sync(0xffffffffu, wait_bar(bar, parity, abort_flag));
}
// Drain wait (teardown): bounded, no abort check.
__device__ __forceinline__ void drain_bar(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!bar_try(bar, parity))
        if (clock64() - t0 > kWaitLimitCycles) break;
}
__device__ __forceinline__ void fence_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int c0, int c1,
                                            int c2, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}

// UMMA shared-memory descriptors (bit 46: descriptor version; bits 61-63: layout).
// No swizzle, K-major: LBO = byte distance of core matrices adjacent along K,
// SBO = along M/N.
__device__ __forceinline__ uint64_t desc_plain(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}
// 128-byte swizzle (rows of 128 bytes, 8-row atoms of 1024 bytes).  K-major: SBO =
// distance of 8-row groups.  MN-major: LBO = distance of 64-element groups along
// M/N, SBO = distance of 8-row groups along K.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                        uint32_t accum) {
    asm volatile(
        "{ .reg .pred p; setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; }" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accum)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
          "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&v)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
                 : "memory");
}

// Instruction descriptors, kind::f16: fp32 accumulate, bf16 A and B (bit 15: A
// MN-major, bit 16: B MN-major).
//   kIdescN32    M = 128, N = 32, both K-major          (projections, T')
//   kIdescN32M64 M = 64,  N = 32, both K-major          (low parts of Vp)
//   kIdescU      M = 128, N = 32, B MN-major            (up-projection of S^n)
//   kIdescQ      M = 128, N = 64, both MN-major         (Q)
//   kIdescE      M = 128, N = 64, B MN-major            (E)
constexpr uint32_t kIdescBase = (1u << 4) | (1u << 7) | (1u << 10);
constexpr uint32_t kIdescN32 = kIdescBase | ((uint32_t)(32 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
constexpr uint32_t kIdescN32M64 = kIdescBase | ((uint32_t)(32 >> 3) << 17) | ((uint32_t)(64 >> 4) << 24);
constexpr uint32_t kIdescU = kIdescN32 | (1u << 16);
constexpr uint32_t kIdescQ =
    kIdescBase | (1u << 15) | (1u << 16) | ((uint32_t)(64 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
constexpr uint32_t kIdescE = kIdescBase | (1u << 16) | ((uint32_t)(64 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);

// Byte offset of element (row r, k) in a K-major no-swizzle table with K = 64.
__host__ __device__ constexpr int kmaj(int r, int k) {
    return (r >> 3) * 1024 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2;
}
// Byte offset of row r, chunk group g (chunks 8g .. 8g+7) in a carried-pair buffer.
__host__ __device__ constexpr int pairoff(int r, int g) { return (r >> 3) * 512 + g * 128 + (r & 7) * 16; }

// Row r of one carried-pair chunk group (chunks 8g .. 8g+7): bf16 high parts
// into the first 8 KB of the buffer, low parts into the second.
__device__ __forceinline__ void store_pair_row(uint32_t buf, int r, int g, const float (&v)[8]) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        h[e] = pack_bf16x2(v[2 * e], v[2 * e + 1]);
        l[e] = pack_bf16x2(v[2 * e] - __uint_as_float(h[e] << 16), v[2 * e + 1] - __uint_as_float(h[e] & 0xffff0000u));
    }
    const uint32_t a = buf + pairoff(r, g);
    st_shared_v4(a, h[0], h[1], h[2], h[3]);
    st_shared_v4(a + 8192, l[0], l[1], l[2], l[3]);
}

// Which rows a CTA takes.  A CTA spends about 6 tiles' time on its tables, the pipeline's
// fill and drain, so short sequences of many rows run several rows of a channel per CTA;
// the grid then shrinks, and a last wave that is nearly empty costs more than the
// prologues saved.  Up to three levels: blocks below end[0] take r[0] rows each, of
// channels from 0 on, the next ones r[1] rows of channels from ch[1] on, and so on, fewer
// rows each, so that the large units start first and small ones fill the tail.  Same box,
// one row per block and now, us: B = 8, L = 4096, D = 256, M = 16 with both state terms (this
// kernel and k_terminal_tc) 145 -> 105; B = 7, L = 465, D = 160, M = 32 45 -> 36; B = 64, L = 200,
// D = 512, M = 16 1012 -> 470.
struct RowPlan {
    int r[3];       // rows per block of the level
    int end[3];     // one past the level's last block
    int ch[3];      // the level's first channel
    int B, D;
};
__host__ __device__ __forceinline__ int level_of(const RowPlan &p, int blk) {
    return blk < p.end[0] ? 0 : blk < p.end[1] ? 1 : 2;
}
__host__ __device__ __forceinline__ void rows_of(const RowPlan &p, int blk, int &d, int &b0, int &nrows) {
    const int l = level_of(p, blk);
    const int r = p.r[l], u = (p.B + r - 1) / r, at = blk - (l ? p.end[l - 1] : 0);
    d = p.ch[l] + at / u;
    b0 = at % u * r;
    nrows = r < p.B - b0 ? r : p.B - b0;
}

// Q += [DY^T ; X^T] X over a tile's 32 chunks (K = chunks): MN-major views of the swizzled
// dy and x tiles at sdy; rows 64-127 (X^T X) are not read.
__device__ __forceinline__ void add_q(uint32_t tmem, uint32_t sdy, bool accum) {
    const uint64_t dqa = desc_sw128(sdy, 4096, 1024), dqb = desc_sw128(sdy + 4096, 16, 1024);
#pragma unroll
    for (int ks = 0; ks < 2; ++ks)
        umma_ss(tmem + kColQ, dqa + ks * (2048 >> 4), dqb + ks * (2048 >> 4), kIdescQ, (accum || ks > 0) ? 1u : 0u);
}

struct BwdArgs {
    const float *decay, *freq, *amp, *phase;
    float2 *part_g, *part_p;  // [B*D][M] (backward)
    const float2 *state_in;   // nullable, [B*D][M] (time-reversed prefill: state before token 0)
    float2 *state_out;        // nullable, [B*D][M] (time-reversed prefill)
    int64_t L;
    RowPlan plan;
    float4 *coef_out;         // nullable, [D][M]   (time-reversed prefill)
    float2 *d_state_in;       // nullable, [B*D][M] (backward: gradient of the forward's state_in)
    __nv_bfloat16 *dxT;       // [B*D][Lp]
    int64_t Lp;
    int D, M;
    int ntiles;               // Lp / kTile
};

// kGrad: the backward pass.  !kGrad: the causal prefill of a time-reversed drive
// (dy = x reversed within [0, L)), which is the same reverse-time scan without the
// parameter gradients: its output is y reversed, and the adjoint state it ends
// with, sum_s lambda^s x_{L-1-s}, is the prompt's terminal state (Sec. 3.2).
// A state s_in before token 0 acts from reversed position L on: lambda^(L-L')
// s_in joins the pair entering the chunk that ends at L' = L rounded up to a
// chunk (|lambda^(L-L')| <= exp(63 gamma)), which gives lambda^(t+1) s_in at
// token t and lambda^L s_in in the end state; positions >= L are never stored.
template <bool kGrad, bool kRows>
__global__ void __launch_bounds__(kThreads, 2)
    k_backward_tc(const __grid_constant__ CUtensorMap tmap_dy, const __grid_constant__ CUtensorMap tmap_x,
                  const BwdArgs args) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // The time-reversed prefill keeps one row per CTA: it serves few rows, and the row
    // bookkeeping cost it 3 %.
    int d = blockIdx.x % args.D, b0 = blockIdx.x / args.D, nrows = 1;
    if (kRows) rows_of(args.plan, blockIdx.x, d, b0, nrows);
    const int row0 = b0 * args.D + d;           // b * D + d of the first row; the next ones D apart
    const int M = args.M, ntiles = args.ntiles;
    const int nv = kRows ? nrows * ntiles : ntiles;   // tiles of the walk: each row's in reverse, row after row
    constexpr int w_prod = 6, w_alloc = 7, w_mma_p = 8, w_mma_d = 9;
    // Threads that build the tables: all but the producer's.
    constexpr int kBuilders = kThreads - 32;
    const int bt = warp < w_prod ? tid : tid - 32;
    auto sync_builders = [] { asm volatile("bar.sync 2, %0;" ::"n"(kBuilders) : "memory"); };
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kOffBar);
    auto bar = [&](int i) { return smem_u32(bars + i); };
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + kOffMisc);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kOffMisc + 16);

    if (tid == 0) {
        *abort_flag = 0;
        for (int i = 0; i < kSlots; ++i) {
            bar_init(bar(kBarSlotFull + i), 1);
            bar_init(bar(kBarSlotEmpty + i), 2);
        }
        for (int i = 0; i < 2; ++i) {
            bar_init(bar(kBarPFull + i), 1);
            bar_init(bar(kBarPEmpty + i), 4);
            bar_init(bar(kBarSFull + i), 4);
            bar_init(bar(kBarBsEmpty + i), 1);
            bar_init(bar(kBarDFull + i), 1);
            bar_init(bar(kBarDEmpty + i), 2);
            bar_init(bar(kBarRhoFull + i), 2);
            bar_init(bar(kBarRhoEmpty + i), 4);
        }
        bar_init(bar(kBarRowFull), 1);
        bar_init(bar(kBarRowFree), 6);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == w_alloc) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // Tile v of the walk is tile ntiles - 1 - v % ntiles of row v / ntiles.
    auto load_tile = [&](int v) {
        const int slot = v % kSlots, rr = kRows ? v / ntiles : 0;
        const int chunk0 = (ntiles - 1 - (v - rr * ntiles)) * kNT, row = row0 + rr * args.D;
        const uint32_t dst = sbase + kOffRing + slot * kSlotBytes;
        bar_expect_tx(bar(kBarSlotFull + slot), kGrad ? 8192u : 4096u);
        tma_load_3d(dst, &tmap_dy, 0, chunk0, row, bar(kBarSlotFull + slot));
        if (kGrad) tma_load_3d(dst + 4096, &tmap_x, 0, chunk0, row, bar(kBarSlotFull + slot));
    };
    // (No pdl_launch_dependents() here: blocks of the output transpose beside the last wave
    // cost 5 us at B = 4, L = 32768, D = 512.)
    if (warp != w_prod) {
    // ------------------------------------------------------------ constants
    // Stage 1: lambda^n (n = 0..64) and c for every mode slot (zero past M):
    // thread (m, g) runs n = 8g .. 8g+7 as one exact power and seven products
    // (relative error below 1e-6, far inside the low parts' 2^-17).
    float2 *pw = reinterpret_cast<float2 *>(smem + kOffPw);
    float2 *cf = reinterpret_cast<float2 *>(smem + kOffCf);
    float *kt = reinterpret_cast<float *>(smem + kOffK);
    if (kGrad)
        for (int i = bt; i < 2 * kQsRows * kQsStride; i += kBuilders) reinterpret_cast<float *>(smem + kOffQs)[i] = 0.0f;
    static_assert(kMaxModes * 9 == kBuilders, "one builder per mode and group of powers");
    {
        const int m = bt / 9, g = bt % 9;
        float2 *o = pw + m * kPwStride + 8 * g;
        if (m < M) {
            const float ga = args.decay[d * M + m], om = args.freq[d * M + m];
            const float2 l1 = lambda_pow(ga, om, 1.0f);
            float2 z = lambda_pow(ga, om, (float)(8 * g));
            o[0] = z;
            if (g < 8) {
#pragma unroll
                for (int e = 1; e < 8; ++e) {
                    z = cmul(z, l1);
                    o[e] = z;
                }
            }
        } else {
            for (int e = 0; e < (g < 8 ? 8 : 1); ++e) o[e] = make_float2(0.0f, 0.0f);
        }
    }
    if (bt >= kBuilders - kMaxModes) {
        const int m = bt - (kBuilders - kMaxModes);
        cf[m] = m >= M ? make_float2(0.0f, 0.0f)
                             : mode_coef(args.amp[d * M + m], args.phase[d * M + m]);
    }
    sync_builders();
    // Stage 2: K[n] (Eq. 1 at integer lags, modes summed in a fixed order), the
    // projection table and the up-projection U', one 16-byte core-matrix row
    // (8 consecutive K elements of one row) per task; consecutive tasks take
    // consecutive rows, so each quarter-warp's stores fill 128 contiguous bytes.
    if (bt < 4 * kC) {   // whole warps: four lanes a lag, eight modes each
        const int n = bt >> 2, m0 = 8 * (bt & 3);
        float acc = 0.0f;
#pragma unroll
        for (int m = m0; m < m0 + 8; ++m) {
            const float2 p = pw[m * kPwStride + n], c = cf[m];
            acc = fmaf(c.x, p.x, fmaf(-c.y, p.y, acc));
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if ((bt & 3) == 0) kt[n] = acc;
    }
    for (int t = bt; t < 1024 + 512; t += kBuilders) {
        if (t < 1024) {
            // A_P row r, k = 8 kg .. 8 kg + 7: lambda^k (Vp rows, with low parts) or
            // k lambda^k (Vq rows).
            const int kg = t >> 7, r = t & 127;
            const int l = r & 31, m = 8 * (r >> 5) + ((l & 15) >> 1), ri = l & 1;
            const bool jordan = l >= 16;
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float v[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int n = 8 * kg + 2 * e + u;
                    const float2 p = pw[m * kPwStride + n];
                    const float w = ri ? p.y : p.x;
                    v[u] = jordan ? (float)n * w : w;
                }
                hi[e] = pack_bf16x2(v[0], v[1]);
                lo[e] = pack_bf16x2(v[0] - __uint_as_float(hi[e] << 16), v[1] - __uint_as_float(hi[e] & 0xffff0000u));
            }
            st_shared_v4(sbase + kOffAP + kmaj(r, 8 * kg), hi[0], hi[1], hi[2], hi[3]);
            if (!jordan) st_shared_v4(sbase + kOffAPlo + kmaj(16 * (r >> 5) + l, 8 * kg), lo[0], lo[1], lo[2], lo[3]);
        } else {
            // U'[i][2m + ri] = Re(c lambda^(C-i)), -Im(c lambda^(C-i)) for modes 4 kg .. 4 kg + 3.
            const int u = t - 1024, kg = u >> 6, i = u & 63;
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int m = 4 * kg + e;
                const float2 z = cmul(cf[m], pw[m * kPwStride + (kC - i)]);
                w[e] = pack_bf16x2(z.x, -z.y);
            }
            st_shared_v4(sbase + kOffU + kmaj(i, 8 * kg), w[0], w[1], w[2], w[3]);
        }
    }
    sync_builders();
    // Stage 3: the transposed Toeplitz block T'[i][j] = K[j - i] (j >= i).
    for (int t = bt; t < 512; t += kBuilders) {
        const int kg = t >> 6, i = t & 63;
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int j = 8 * kg + 2 * e;
            w[e] = pack_bf16x2(j >= i ? kt[j - i] : 0.0f, j + 1 >= i ? kt[j + 1 - i] : 0.0f);
        }
        st_shared_v4(sbase + kOffT + kmaj(i, 8 * kg), w[0], w[1], w[2], w[3]);
    }
    fence_async_smem();
    tc_fence_before();
    sync_builders();
    tc_fence_after();
    }

    const int last = nv - 1;
    // Scan lanes: lane l of quarter q owns row 32 q + l of the projections and of
    // [S^n ; R^n] (mode mE = 8 q + (l % 16) / 2; role s = 2 (l >= 16) + l % 2:
    // Re / Im of Dp and S^n, of Dq and R^n).
    if (warp < 4) {
        // ---------------------------------------------------- reverse chunk scan
        const int s = ((lane >> 4) << 1) | (lane & 1), mE = 8 * warp + ((lane & 15) >> 1);
        const bool onE = mE < M;
        const float gamE = onE ? args.decay[d * M + mE] : 0.0f, omgE = onE ? args.freq[d * M + mE] : 0.0f;
        // The adjoint pair; after a row's last tile it is (S_0, R_0).
        float2 S = make_float2(0.0f, 0.0f), R = make_float2(0.0f, 0.0f);
        const int q = warp, base = lane & 14;   // the mode's rows: base, base + 1, base + 16, base + 17
        const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16);
        const float2 a = lambda_pow(gamE, omgE, (float)kC);
        const int prow = 32 * q + lane;         // this lane's [S^n ; R^n] row
        // State before token 0 (reversed-time prefill): chunk kinj of the walk.
        float2 inj = make_float2(0.0f, 0.0f);
        int kinj = -1;
        if (!kGrad && args.state_in) {
            const int64_t Lr = (args.L + kC - 1) / kC * kC;
            kinj = (int)(Lr / kC) - 1;
            if (onE)
                inj = cmul(lambda_pow(gamE, omgE, (float)(args.L - Lr)), args.state_in[(int64_t)row0 * M + mE]);
        }
        bool ok = true;
        // Row r of the walk: E = [S^n ; R^n] X over the row and the within-chunk rho leave TMEM
        // for fp32 and become the row's (G, P); the next row's first products then overwrite
        // both accumulators.
        const float2 l1 = lambda_pow(gamE, omgE, 1.0f);
        const float2 l4 = lambda_pow(gamE, omgE, 4.0f), l32 = lambda_pow(gamE, omgE, 32.0f),
                     ls0 = lambda_pow(gamE, omgE, (float)s);
        float gin = 0.0f, gii = 0.0f, pin = 0.0f, pii = 0.0f;   // the initial state's share of (G, P), role 0
        auto finish_row = [&](int r) {
            if (!wait_bar_warp(bar(kBarRowFull), r & 1, abort_flag)) return false;
            tc_fence_after();
            // Weights lambda^(C-i), C - i = 16 (3 - h) + k with k = 1 .. 16: the four blocks h of 16
            // columns share the powers lambda^k, and Horner steps of lambda^16 join them.
            float2 w = l1, z = l1;
            float2 A[4], J[4];   // sum lambda^k x, sum k lambda^k x
#pragma unroll
            for (int h = 0; h < 4; ++h) A[h] = J[h] = make_float2(0.0f, 0.0f);
#pragma unroll 1
            for (int eg = 3; eg >= 0; --eg) {
                uint32_t ev[4][4];
#pragma unroll
                for (int h = 0; h < 4; ++h) tmem_ld4(tl + kColE + 16 * h + 4 * eg, ev[h]);
                tmem_wait_ld();
                if (kRows && eg == 0) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) bar_arrive(bar(kBarRowFree));
                }
#pragma unroll
                for (int e = 3; e >= 0; --e) {
                    const float k = (float)(16 - 4 * eg - e);
                    const float2 kw = make_float2(k * w.x, k * w.y);
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const float x = __uint_as_float(ev[h][e]);
                        A[h].x = fmaf(w.x, x, A[h].x);
                        A[h].y = fmaf(w.y, x, A[h].y);
                        J[h].x = fmaf(kw.x, x, J[h].x);
                        J[h].y = fmaf(kw.y, x, J[h].y);
                    }
                    z = w;
                    w = cmul(w, l1);
                }
            }
            float2 a = A[0], j = J[0];   // z = lambda^16
#pragma unroll
            for (int h = 1; h < 4; ++h) {
                j = cfma(z, make_float2(fmaf(16.0f, a.x, j.x), fmaf(16.0f, a.y, j.y)), J[h]);
                a = cfma(z, a, A[h]);
            }
            // G = sum w (E_S.re + i E_S.im), P = sum w E_R + sum (C - i) w E_S.
            float gr = 0.0f, gi = 0.0f, pr, pi;
            if (s == 0) { gr = a.x; gi = a.y; pr = j.x; pi = j.y; }
            else if (s == 1) { gr = -a.y; gi = a.x; pr = -j.y; pi = j.x; }
            else if (s == 2) { pr = a.x; pi = a.y; }
            else { pr = -a.y; pi = a.x; }
            // Within-chunk terms: lags n = s, s + 4, ... < 32 from rho, and n + 32, which share
            // lambda^n (steps of lambda^4 from the exact lambda^s) and take lambda^32 at the end.
            if (!wait_bar_warp(bar(kBarRhoFull + (r & 1)), (r >> 1) & 1, abort_flag)) return false;
            const float *rho = reinterpret_cast<const float *>(smem + kOffRho) + (r & 1) * 128;
            float2 ln = ls0;
            float2 gh = make_float2(0.0f, 0.0f), ph = gh;
#pragma unroll 4
            for (int e = 0; e < kC / 8; ++e) {
                const int n = 4 * e + s;
                const float v = rho[n] + rho[64 + n], u = rho[96 + n], nv = v * (float)n, nu = u * (float)n;
                gr = fmaf(v, ln.x, gr);
                gi = fmaf(v, ln.y, gi);
                pr = fmaf(nv, ln.x, pr);
                pi = fmaf(nv, ln.y, pi);
                gh.x = fmaf(u, ln.x, gh.x);
                gh.y = fmaf(u, ln.y, gh.y);
                ph.x = fmaf(nu, ln.x, ph.x);
                ph.y = fmaf(nu, ln.y, ph.y);
                ln = cmul(ln, l4);
            }
            const float2 g2 = cfma(l32, gh, make_float2(gr, gi));
            const float2 p2 = cfma(l32, make_float2(fmaf(32.0f, gh.x, ph.x), fmaf(32.0f, gh.y, ph.y)), make_float2(pr, pi));
            gr = g2.x;
            gi = g2.y;
            pr = p2.x;
            pi = p2.y;
            __syncwarp();
            if (kRows && lane == 0) bar_arrive(bar(kBarRhoEmpty + (r & 1)));
            gr += gin;
            gi += gii;
            pr += pin;
            pi += pii;
            // The sum over the mode's four lanes; role 0 writes the row's partials.
#pragma unroll
            for (int o = 1; o <= 16; o <<= 4) {
                gr += __shfl_xor_sync(0xffffffffu, gr, o);
                gi += __shfl_xor_sync(0xffffffffu, gi, o);
                pr += __shfl_xor_sync(0xffffffffu, pr, o);
                pi += __shfl_xor_sync(0xffffffffu, pi, o);
            }
            if (s == 0 && onE) {
                const int64_t at = (int64_t)(row0 + r * args.D) * M + mE;
                args.part_g[at] = make_float2(gr, gi);
                args.part_p[at] = make_float2(pr, pi);
            }
            return true;
        };
        int row = row0, tv = 0;   // the current row and its tile
        int ended = 0;            // rows whose last tile has been scanned
        bool pending = false;     // the last of them waits for finish_row
        // (Several rows: one pass more than there are tiles, so that finish_row is inlined once.)
        for (int v = 0; v < nv + (kRows ? 1 : 0); ++v) {
            if (!kRows || v < nv) {
                const int bb = v & 1;
                if (kRows && tv == 0) S = R = make_float2(0.0f, 0.0f);
                if (!wait_bar(bar(kBarPFull + bb), (v >> 1) & 1, abort_flag)) break;
                tc_fence_after();
                if (warp == 0 && lane == 0) bar_arrive(bar(kBarSlotEmpty + v % kSlots));
                const uint32_t pb = sbase + kOffBs + bb * kBsBuf;
                const int cinj = kinj - (last - v) * kNT;   // chunk of this tile that takes s_in, if any
#pragma unroll
                for (int h = 1; h >= 0; --h) {   // chunks 31 .. 0
                    uint32_t pv[16];
                    tmem_ld16(tl + kColP + 32 * bb + 16 * h, pv);
                    tmem_wait_ld();
                    if (h == 1) {
                        if (!wait_bar(bar(kBarBsEmpty + bb), ((v >> 1) & 1) ^ 1, abort_flag)) {
                            ok = false;
                            break;
                        }
                    } else {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) bar_arrive(bar(kBarPEmpty + bb));
                    }
#pragma unroll
                    for (int g = 1; g >= 0; --g) {
                        float own[8];
#pragma unroll
                        for (int n = 7; n >= 0; --n) {
                            const float p = __uint_as_float(pv[8 * g + n]);
                            const float dpr = __shfl_sync(0xffffffffu, p, base);
                            const float dpi = __shfl_sync(0xffffffffu, p, base + 1);
                            const float dqr = __shfl_sync(0xffffffffu, p, base + 16);
                            const float dqi = __shfl_sync(0xffffffffu, p, base + 17);
                            // The pair entering chunk 16 h + 8 g + n from the right.
                            if (!kGrad && 16 * h + 8 * g + n == cinj) S = make_float2(S.x + inj.x, S.y + inj.y);
                            own[n] = (s & 2) ? ((s & 1) ? R.y : R.x) : ((s & 1) ? S.y : S.x);
                            const float2 w = make_float2(fmaf((float)kC, S.x, R.x), fmaf((float)kC, S.y, R.y));
                            R = cfma(a, w, make_float2(dqr, dqi));
                            S = cfma(a, S, make_float2(dpr, dpi));
                        }
                        store_pair_row(pb, prow, 2 * h + g, own);
                    }
                }
                if (!ok) break;
                fence_async_smem();
                __syncwarp();
                if (lane == 0) bar_arrive(bar(kBarSFull + bb));
            }
            if (!kGrad) continue;
            // A row is finished after the next one's first tile, whose scan hides the last products.
            if (kRows && pending) {
                pending = false;
                if (!finish_row(ended - 1)) break;
            }
            if ((kRows && v == nv) || ++tv < ntiles) continue;
            // The row's end: (S, R) is the adjoint pair at token 0.  The forward's initial
            // state s_in (Sec. 3.2-3.3): G += s_in lambda S_0, P += s_in lambda (R_0 + S_0),
            // once per mode; the gradient of s_in is conj(c lambda S_0).
            if (s == 0 && onE && (args.state_in || args.d_state_in)) {
                const int64_t at = (int64_t)row * M + mE;
                const float2 ls = cmul(l1, S);
                if (args.state_in) {
                    const float2 si = args.state_in[at];
                    const float2 g0 = cmul(si, ls), p0 = cmul(si, cmul(l1, make_float2(R.x + S.x, R.y + S.y)));
                    gin = g0.x;
                    gii = g0.y;
                    pin = p0.x;
                    pii = p0.y;
                }
                if (args.d_state_in) {
                    const float2 c = mode_coef(args.amp[d * M + mE], args.phase[d * M + mE]);
                    const float2 cls = cmul(c, ls);
                    args.d_state_in[at] = make_float2(cls.x, -cls.y);
                }
            }
            __syncwarp();   // the next tile's tensor-memory loads are warp-wide
            ++ended;
            pending = true;
            tv = 0;
            row += args.D;
        }
        if (kGrad && !kRows && pending) finish_row(0);
        if (!kGrad && ok && s == 0 && onE) {
            // The adjoint state after the first chunk is the prompt's terminal state.
            if (args.state_out) args.state_out[(int64_t)row0 * M + mE] = S;
            if (args.coef_out && row0 < args.D) {
                const float2 c = mode_coef(args.amp[d * M + mE], args.phase[d * M + mE]);
                args.coef_out[d * M + mE] = make_float4(l1.x, l1.y, c.x, c.y);
            }
        }
    } else if (warp < 6) {
        // ---------------------------------------------------- dx epilogue
        const int q = warp & 3;   // 0 or 1: positions 32 q + lane
        const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16);
        // The tile's positions in dxT: rows D apart, tiles from the end of each.
        __nv_bfloat16 *rowp = args.dxT + (int64_t)row0 * args.Lp + 32 * q + lane;
        int tile = ntiles - 1, r = 0;   // r: row of the walk
        for (int v = 0; v < nv; ++v) {
            const int bb = v & 1;
            if (!wait_bar(bar(kBarDFull + bb), (v >> 1) & 1, abort_flag)) break;
            tc_fence_after();
            uint32_t r0[16], r1[16];
            tmem_ld16(tl + kColD + 32 * bb, r0);
            tmem_ld16(tl + kColD + 32 * bb + 16, r1);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                bar_arrive(bar(kBarDEmpty + bb));
                if (warp == 4) {
                    bar_arrive(bar(kBarBsEmpty + bb));
                    bar_arrive(bar(kBarSlotEmpty + v % kSlots));
                }
            }
            // Channel-major dx: each store instruction writes 64 contiguous bytes.
            __nv_bfloat16 *out = rowp + (int64_t)tile * kTile;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                out[k * kC] = __float2bfloat16_rn(__uint_as_float(r0[k]));
                out[(k + 16) * kC] = __float2bfloat16_rn(__uint_as_float(r1[k]));
            }
            if (--tile >= 0 || !kGrad) continue;
            // The row's end: diagonal sums of Q over the row, rho[n] = sum_k Q[n+k][k].  Each warp
            // takes its 32 rows, 16 columns at a time, through its own staging buffer, where a row
            // holds a diagonal's cells (row stride 18 words: the 8-byte reads hit 32 banks), and
            // adds them into its part of rho; the readers add the two warps' parts.  (Rows kept as
            // rows, with a range check a cell: B = 8, L = 4096, D = 256, M = 16 69.7 us against 68.1.)
            float *qs = reinterpret_cast<float *>(smem + kOffQs) + q * kQsRows * kQsStride;
            float *rho = reinterpret_cast<float *>(smem + kOffRho) + (r & 1) * 128 + q * 64;
            if (!wait_bar_warp(bar(kBarRowFull), r & 1, abort_flag)) break;
            tc_fence_after();
            if (kRows && !wait_bar_warp(bar(kBarRhoEmpty + (r & 1)), ((r >> 1) & 1) ^ 1, abort_flag)) break;
            rho[lane] = rho[lane + 32] = 0.0f;
#pragma unroll 1
            for (int h = 0; h < 2 + 2 * q; ++h) {
                uint32_t qv[16];
                tmem_ld16(tl + kColQ + 16 * h, qv);
                tmem_wait_ld();
                if (kRows && h == 1 + 2 * q) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) bar_arrive(bar(kBarRowFree));
                }
#pragma unroll
                for (int e = 0; e < 16; ++e) qs[(lane - e + 15) * kQsStride + e] = __uint_as_float(qv[e]);
                __syncwarp();
                // Element (32 q + i, 16 h + e) went to row i - e + 15: row k is diagonal k + at.
                const int at = 32 * q - 16 * h - 15;
                auto add = [&](int k) {
                    if (k >= kQsRows || k + at < 0) return;
                    float a = 0.0f, b = 0.0f;
#pragma unroll
                    for (int e = 0; e < 16; e += 2) {
                        const float2 v = *reinterpret_cast<const float2 *>(qs + k * kQsStride + e);
                        a += v.x;
                        b += v.y;
                    }
                    rho[k + at] += a + b;
                };
                add(lane);
                add(lane + 32);
                __syncwarp();
            }
            __syncwarp();
            if (lane == 0) bar_arrive(bar(kBarRhoFull + (r & 1)));
            ++r;
            tile = ntiles - 1;
            rowp += (int64_t)args.D * args.Lp;
        }
    } else if (warp == w_prod) {
        // ---------------------------------------------------- TMA producer
        if (lane == 0) {
            pdl_wait();
            int issued = 0;
            for (; issued < nv; ++issued) {
                const int slot = issued % kSlots;
                if (!wait_bar(bar(kBarSlotEmpty + slot), ((issued / kSlots) & 1) ^ 1, abort_flag)) break;
                load_tile(issued);
            }
            // Drain: every issued load lands before the CTA may exit.
            for (int k = issued > kSlots ? issued - kSlots : 0; k < issued; ++k)
                drain_bar(bar(kBarSlotFull + k % kSlots), (k / kSlots) & 1);
        }
        __syncwarp();
    } else if (warp == w_mma_p) {
        // ---------------------------------------------------- MMA: projections (and Q)
        if (lane == 0) {
            const uint64_t dap = desc_plain(sbase + kOffAP, 128, 1024);
            const uint64_t dapl = desc_plain(sbase + kOffAPlo, 128, 1024);
            int v = 0;
            for (; v < nv; ++v) {
                const int slot = v % kSlots, bb = v & 1;
                if (!wait_bar(bar(kBarSlotFull + slot), (v / kSlots) & 1, abort_flag)) break;
                if (!wait_bar(bar(kBarPEmpty + bb), ((v >> 1) & 1) ^ 1, abort_flag)) break;
                tc_fence_after();
                const uint32_t sdy = sbase + kOffRing + slot * kSlotBytes;
                const uint64_t ddy = desc_sw128(sdy, 16, 1024);
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    umma_ss(tmem + kColP + 32 * bb, dap + ks * 16, ddy + ks * 2, kIdescN32, ks > 0);
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    umma_ss(tmem + kColP + 32 * bb, dapl + ks * 16, ddy + ks * 2, kIdescN32M64, 1u);
                if (kGrad && !kRows) add_q(tmem, sdy, v > 0);
                umma_commit(bar(kBarPFull + bb));
            }
            // Drain: the last group's completion implies all earlier ones.
            if (v > 0) drain_bar(bar(kBarPFull + ((v - 1) & 1)), ((v - 1) >> 1) & 1);
        }
        __syncwarp();
    } else if (warp == w_mma_d) {
        // ---------------------------------------------------- MMA: T', U', E (and Q)
        if (lane == 0) {
            const uint64_t dt = desc_plain(sbase + kOffT, 128, 1024);
            const uint64_t du = desc_plain(sbase + kOffU, 128, 1024);
            int v = 0;
            for (; v < nv; ++v) {
                const int slot = v % kSlots, bb = v & 1;
                if (!wait_bar(bar(kBarSlotFull + slot), (v / kSlots) & 1, abort_flag)) break;
                if (!wait_bar(bar(kBarDEmpty + bb), ((v >> 1) & 1) ^ 1, abort_flag)) break;
                tc_fence_after();
                const uint32_t sdy = sbase + kOffRing + slot * kSlotBytes;
                const uint64_t ddy = desc_sw128(sdy, 16, 1024);
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    umma_ss(tmem + kColD + 32 * bb, dt + ks * 16, ddy + ks * 2, kIdescN32, ks > 0);
                // Several rows a block: Q is issued here, so that a row's first products, which
                // overwrite Q and E, hold up dx alone until the row before has left both.
                const int tv = kRows ? v % ntiles : v;
                const bool fresh = kRows && tv == 0 && v > 0;
                if (kRows && !fresh) add_q(tmem, sdy, tv > 0);
                if (!wait_bar(bar(kBarSFull + bb), (v >> 1) & 1, abort_flag)) {
                    umma_commit(bar(kBarDFull + bb));   // so that the drain below tracks T'
                    ++v;
                    break;
                }
                tc_fence_after();
                const uint32_t pb = sbase + kOffBs + bb * kBsBuf;
                auto add_u = [&](int part) {
                    // dx += U' S^n: B = the S^n rows of quarter ks (MN-major).
                    const uint64_t dbu = desc_plain(pb + part * 8192, 512, 128);
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        umma_ss(tmem + kColD + 32 * bb, du + ks * 16, dbu + ks * (2048 >> 4), kIdescU, 1u);
                };
                auto add_e = [&](int part) {
                    // E += [S^n ; R^n] X (K = chunks).
                    const uint64_t dea = desc_plain(pb + part * 8192, 128, 512), dxm = desc_sw128(sdy + 4096, 16, 1024);
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks)
                        umma_ss(tmem + kColE, dea + ks * (256 >> 4), dxm + ks * (2048 >> 4), kIdescE,
                                (tv > 0 || part > 0 || ks > 0) ? 1u : 0u);
                };
                if (kRows && fresh) {
                    add_u(0);
                    add_u(1);
                    if (!wait_bar(bar(kBarRowFree), (v / ntiles - 1) & 1, abort_flag)) {
                        umma_commit(bar(kBarDFull + bb));
                        ++v;
                        break;
                    }
                    tc_fence_after();
                    add_q(tmem, sdy, false);
                    add_e(0);
                    add_e(1);
                } else {
#pragma unroll
                    for (int part = 0; part < 2; ++part) {   // high parts, then low parts
                        add_u(part);
                        if (kGrad) add_e(part);
                    }
                }
                if (kGrad && (kRows ? tv == ntiles - 1 : v == nv - 1)) umma_commit(bar(kBarRowFull));
                umma_commit(bar(kBarDFull + bb));
            }
            if (v > 0) drain_bar(bar(kBarDFull + ((v - 1) & 1)), ((v - 1) >> 1) & 1);
        }
        __syncwarp();
    }

    tc_fence_before();
    __syncthreads();   // every role has left its loop
    tc_fence_after();
    if (warp == w_alloc)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kTmemCols));
}

// ------------------------------------------------------------ terminal-state gradient
// The loss term Re(conj(g) s_L) of a terminal-state gradient g = d_state_out
// (Sec. 3.2-3.3) adds, per (b, d) row and mode, with s = L - 1 - j:
//   dx_j     += Re(sum_m conj(g_m) lambda_m^s),
//   J_m       = sum_j x_j s lambda_m^s (+ L lambda^L s_in),  written as conj(g) J
//               (the reduction subtracts its Re and Im from dgamma and domega),
//   d_state_in += g conj(lambda^L).
// Its adjoint state is the closed form conj(g) lambda^s, so no scan is needed.
// Chunk n (tokens 64 n + i) lies fully before L when E_n = L - 64 - 64 n >= 0;
// then lambda^s = lambda^E_n lambda^(63-i) with both exponents >= 0, and
//   J += lambda^E_n (E_n p_n + q_n),  p_n = sum_i lambda^(63-i) x,  q_n = sum_i (63-i) lambda^(63-i) x
//   dx[i][n] = Re(W_n lambda^(63-i)),  W_n = conj(g) lambda^E_n,
// both on the tensor cores (p, q: the projections of the main pass with the
// table reversed in i; dx: an up-projection of W).  The one chunk that holds
// token L - 1 without ending there (L % 64 != 0) is evaluated directly in fp32,
// so no negative power of lambda is ever formed.  One CTA per row or run of rows of
// one channel (RowPlan), walking each row's tiles from the end of the sequence:
//   warps 0-3  per tile: the chunk weights W_n = conj(g) lambda^E_n (steps of
//              lambda^64 in four chains; each tile's first weight carried from
//              the previous tile by lambda^2048), the W rows, and conj(g) J from
//              the projections (each lane weights its own TMEM row, the mode's
//              four rows are added at the end);
//   warps 4-5  dx epilogue: dxT += dx (positions 0-63; the old values come
//              with the x tile, so no global read waits in the loop);
//   warp 6     TMA producer (per slot: the x tile, swizzled for the product, and
//              the dxT tile, plain), TMEM allocation;
//   warp 7     MMA issue: projections into P, then the W up-projection into D.
constexpr int kTmWarps = 8;
constexpr int kTmThreads = kTmWarps * 32;
constexpr int kTmSlots = 4;
constexpr int kTmCols = 128;
constexpr int kTmColP = 0;    // [2] x 32: projections (rows as in A_P)
constexpr int kTmColD = 64;   // [2] x 32: dx (lanes 0-63)
constexpr int kTmOffU = 0;                                  // U_g: 64 rows x K 64 (rows 64-127 of its M=128 product read kTmOffA)
constexpr int kTmOffA = 8192;                               // reversed projection table, 128 rows
constexpr int kTmOffAlo = 24576;                            // its low parts, 64 rows
constexpr int kTmOffRing = 32768;                           // [kTmSlots] x (4 KB) + dxT (4 KB) tiles
constexpr int kTmSlotBytes = 8192;
constexpr int kTmOffW = kTmOffRing + kTmSlots * kTmSlotBytes;   // [2] W buffers, 8 KB each (pair layout)
constexpr int kTmOffPw = kTmOffW + 2 * 8192;                // [32][65] float2: lambda^s, s = 0..64
constexpr int kTmOffBar = kTmOffPw + kMaxModes * kPwStride * 8;
constexpr int kTmNumBars = 24;
constexpr int kTmOffMisc = kTmOffBar + kTmNumBars * 8;
constexpr int kTmSmemBytes = kTmOffMisc + 64 + 1024;        // + alignment slack
static_assert(kTmOffRing % 1024 == 0, "swizzled tiles need 1024-byte alignment");
static_assert(2 * (kTmSmemBytes + 1024) <= 233472, "two CTAs per SM");
constexpr int kTmSlotFull = 0, kTmSlotEmpty = kTmSlots, kTmPFull = 2 * kTmSlots, kTmPEmpty = kTmPFull + 2,
              kTmWFull = kTmPEmpty + 2, kTmWEmpty = kTmWFull + 2, kTmDFull = kTmWEmpty + 2,
              kTmDEmpty = kTmDFull + 2;
static_assert(kTmDEmpty + 2 <= kTmNumBars, "too many barriers");

// SlotEmpty counts the projection commit and the two epilogue warps.
struct TermArgs {
    const float *decay, *freq;     // [D][M]
    const float2 *g;               // d_state_out, [B*D][M]
    const float2 *state_in;        // nullable, [B*D][M]
    float2 *d_state_in;            // nullable, [B*D][M]: += g conj(lambda^L)
    float2 *part_j;                // [B*D][M]: conj(g) J
    const __nv_bfloat16 *xT;       // [B*D][Lp] channel-major x (the partial chunk's direct sum)
    __nv_bfloat16 *dxT;            // [B*D][Lp]: += the g term of dx
    int64_t L, Lp;
    int D, M, ntiles;
    RowPlan plan;
};

__global__ void __launch_bounds__(kTmThreads, 2)
    k_terminal_tc(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_dx,
                  const TermArgs args) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int d, b0, nrows;
    rows_of(args.plan, blockIdx.x, d, b0, nrows);
    const int row0 = b0 * args.D + d;   // b * D + d of the first row; the next ones D apart
    const int M = args.M, ntiles = args.ntiles, nv = nrows * ntiles;
    const int64_t L = args.L;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kTmOffBar);
    auto bar = [&](int i) { return smem_u32(bars + i); };
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + kTmOffMisc);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kTmOffMisc + 16);
    float2 *pw = reinterpret_cast<float2 *>(smem + kTmOffPw);

    if (tid == 0) {
        *abort_flag = 0;
        for (int i = 0; i < kTmSlots; ++i) {
            bar_init(bar(kTmSlotFull + i), 1);
            bar_init(bar(kTmSlotEmpty + i), 3);
        }
        for (int i = 0; i < 2; ++i) {
            bar_init(bar(kTmPFull + i), 1);
            bar_init(bar(kTmPEmpty + i), 4);
            bar_init(bar(kTmWFull + i), 4);
            bar_init(bar(kTmWEmpty + i), 1);
            bar_init(bar(kTmDFull + i), 1);
            bar_init(bar(kTmDEmpty + i), 2);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 6) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(kTmCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // lambda^s for s = 0..64 per mode slot (zero past M): thread (m, e) forms
    // s = 8 e .. 8 e + 7 (and s = 64 for e = 7) as one exact power and products.
    {
        const int m = tid >> 3, e = tid & 7;
        float2 *o = pw + m * kPwStride + 8 * e;
        if (m < M) {
            const float ga = args.decay[d * M + m], om = args.freq[d * M + m];
            const float2 l1 = lambda_pow(ga, om, 1.0f);
            float2 z = lambda_pow(ga, om, (float)(8 * e));
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                o[k] = z;
                z = cmul(z, l1);
            }
            if (e == 7) o[8] = z;
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) o[k] = make_float2(0.0f, 0.0f);
            if (e == 7) o[8] = make_float2(0.0f, 0.0f);
        }
    }
    __syncthreads();
    // The tables (K index k = position i within the chunk; value at lambda^(63-k)):
    //   A rows as A_P (row r: mode 8 (r / 32) + (r % 16) / 2, Re/Im by r % 2;
    //   r % 32 < 16: lambda^(63-k), else (63-k) lambda^(63-k)), low parts of the
    //   first kind into the M = 64 table;
    //   U_g[k][2m + ri] = Re lambda_m^(63-k), -Im lambda_m^(63-k).
    for (int t = tid; t < 1024 + 512; t += kTmThreads) {
        if (t < 1024) {
            const int kg = t >> 7, r = t & 127;
            const int l = r & 31, m = 8 * (r >> 5) + ((l & 15) >> 1), ri = l & 1;
            const bool jordan = l >= 16;
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float v[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int k = 8 * kg + 2 * e + u;
                    const float2 p = pw[m * kPwStride + (kC - 1 - k)];
                    const float w = ri ? p.y : p.x;
                    v[u] = jordan ? (float)(kC - 1 - k) * w : w;
                }
                hi[e] = pack_bf16x2(v[0], v[1]);
                lo[e] = pack_bf16x2(v[0] - __uint_as_float(hi[e] << 16), v[1] - __uint_as_float(hi[e] & 0xffff0000u));
            }
            st_shared_v4(sbase + kTmOffA + kmaj(r, 8 * kg), hi[0], hi[1], hi[2], hi[3]);
            if (!jordan) st_shared_v4(sbase + kTmOffAlo + kmaj(16 * (r >> 5) + l, 8 * kg), lo[0], lo[1], lo[2], lo[3]);
        } else {
            const int u = t - 1024, kg = u >> 6, k = u & 63;
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 z = pw[(4 * kg + e) * kPwStride + (kC - 1 - k)];
                w[e] = pack_bf16x2(z.x, -z.y);
            }
            st_shared_v4(sbase + kTmOffU + kmaj(k, 8 * kg), w[0], w[1], w[2], w[3]);
        }
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (tid == 0) pdl_launch_dependents();
    pdl_wait();   // the tables needed parameters only; what follows reads the main pass's results
    // The chunk holding token L - 1 when it does not end there (-1: none).
    const int64_t n_part = (L % kC) ? (L - 1) / kC : -1;

    if (warp < 4) {
        // ---------------------------------------------------- weights, W, J
        const int q = warp, l = lane;
        const int m = 8 * q + ((l & 15) >> 1), ri = l & 1;
        const bool jordan = l >= 16, on = m < M;
        const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16);
        const float gam = on ? args.decay[d * M + m] : 0.0f, omg = on ? args.freq[d * M + m] : 0.0f;
        const float2 l64 = lambda_pow(gam, omg, (float)kC), l2048 = lambda_pow(gam, omg, (float)kTile);
        const float2 l512 = lambda_pow(gam, omg, 512.0f), l1024 = lambda_pow(gam, omg, 1024.0f),
                     l1536 = lambda_pow(gam, omg, 1536.0f);
        const int prow = 32 * q + (l & 15);   // this lane's W row
        // The last chunk that ends at or before token L - 1 (-1: none).
        const int64_t nfull = L >= kC ? (L - kC) / kC : -1;
        float jr[4] = {0.0f, 0.0f, 0.0f, 0.0f}, ji[4] = {0.0f, 0.0f, 0.0f, 0.0f};   // this lane's share of conj(g) J
        float2 T = make_float2(0.0f, 0.0f);   // lambda^E of the next tile's chunk 31, once known
        bool haveT = false;
        bool ok = true;
        int row = row0, tv = 0;   // the current row and its tile
        float2 gc = make_float2(0.0f, 0.0f);   // conj(g) of the row
        for (int v = 0; v < nv && ok; ++v) {
            const int bb = v & 1;
            if (tv == 0) {
                haveT = false;
                if (on) gc = conj2(args.g[(int64_t)row * M + m]);
            }
            const int64_t n0 = (int64_t)(ntiles - 1 - tv) * kNT;   // the tile's first chunk
            // Weights W_n = conj(g) lambda^E_n of the tile's chunks, E_n = L - 64 - 64 n
            // (zero where E_n < 0), from the tile's last full chunk ctop down by steps
            // of lambda^64.  lambda^E at ctop is an exact power in the first one or
            // two tiles (E < 4200); after that chunk 31's comes from the previous
            // tile's by one step of lambda^2048.
            const int64_t ctop64 = nfull - n0;
            const int ctop = ctop64 < 0 ? -1 : (ctop64 > kNT - 1 ? kNT - 1 : (int)ctop64);
            float2 z = make_float2(0.0f, 0.0f);
            if (ctop >= 0) {
                const float2 a = (ctop == kNT - 1 && haveT) ? T : lambda_pow(gam, omg, (float)(L - kC - kC * (n0 + ctop)));
                if (ctop == kNT - 1) {
                    T = cmul(a, l2048);
                    haveT = true;
                }
                z = cmul(gc, a);
            }
            float2 w[kNT];
            if (ctop == kNT - 1) {
                // A full tile: four independent chains of eight steps.
                float2 z1 = cmul(z, l512), z2 = cmul(z, l1024), z3 = cmul(z, l1536);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    w[31 - k] = z;
                    w[23 - k] = z1;
                    w[15 - k] = z2;
                    w[7 - k] = z3;
                    z = cmul(z, l64);
                    z1 = cmul(z1, l64);
                    z2 = cmul(z2, l64);
                    z3 = cmul(z3, l64);
                }
            } else {
#pragma unroll
                for (int c = kNT - 1; c >= 0; --c) {
                    if (c > ctop) {
                        w[c] = make_float2(0.0f, 0.0f);
                    } else {
                        w[c] = z;
                        z = cmul(z, l64);
                    }
                }
            }
            // W rows (Re / Im of W_n) for the dx product.
            if (!wait_bar(bar(kTmWEmpty + bb), ((v >> 1) & 1) ^ 1, abort_flag)) break;
            {
                // Lane l < 16 stores chunk groups 0-1 of its row, lane l + 16 (the same
                // mode and component, so the same weights) groups 2-3.
                const uint32_t wb = sbase + kTmOffW + bb * 8192;
#pragma unroll
                for (int gg = 0; gg < 2; ++gg) {
                    uint32_t h[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 a0 = jordan ? w[16 + 8 * gg + 2 * e] : w[8 * gg + 2 * e];
                        const float2 a1 = jordan ? w[16 + 8 * gg + 2 * e + 1] : w[8 * gg + 2 * e + 1];
                        h[e] = ri ? pack_bf16x2(a0.y, a1.y) : pack_bf16x2(a0.x, a1.x);
                    }
                    st_shared_v4(wb + pairoff(prow, gg + (jordan ? 2 : 0)), h[0], h[1], h[2], h[3]);
                }
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) bar_arrive(bar(kTmWFull + bb));
            // conj(g) J from this lane's projection row: value v_n (Re or Im of p_n or
            // q_n) enters as W_n f_n v_n (times i for an Im row), f_n = E_n for p, 1 for q.
            if (!wait_bar(bar(kTmPFull + bb), (v >> 1) & 1, abort_flag)) {
                ok = false;
                break;
            }
            tc_fence_after();
            uint32_t pa[16], pb[16];
            tmem_ld16(tl + kTmColP + 32 * bb, pa);
            tmem_ld16(tl + kTmColP + 32 * bb + 16, pb);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive(bar(kTmPEmpty + bb));
            // E_n as fp32 (exact below 2^24): one 64-bit conversion per tile.
            const float e0 = (float)(L - kC - kC * n0);
#pragma unroll
            for (int c = 0; c < kNT; ++c) {
                const float f = jordan ? 1.0f : fmaf(-(float)kC, (float)c, e0);
                const float val = __uint_as_float(c < 16 ? pa[c] : pb[c - 16]) * f;
                // (ri ? i : 1) * w * val, four accumulators
                jr[c & 3] = fmaf(ri ? -w[c].y : w[c].x, val, jr[c & 3]);
                ji[c & 3] = fmaf(ri ? w[c].x : w[c].y, val, ji[c & 3]);
            }
            if (++tv < ntiles) continue;
            // The row's end: conj(g) J of the row, over the mode's four lanes; one of them adds the
            // part of the chunk that holds token L - 1 (L % 64 != 0) directly, and the state terms.
            const bool lead = on && !jordan && ri == 0;
            if (lead && n_part >= 0) {
                const __nv_bfloat16 *xp = args.xT + (int64_t)row * args.Lp + n_part * kC;
                const int cnt = (int)(L - n_part * kC);   // tokens of the chunk before L
                float pr = 0.0f, pi = 0.0f;
                for (int i = 0; i < cnt; ++i) {
                    const int e = cnt - 1 - i;
                    const float xv = __bfloat162float(xp[i]) * (float)e;
                    const float2 p = pw[m * kPwStride + e];
                    pr = fmaf(p.x, xv, pr);
                    pi = fmaf(p.y, xv, pi);
                }
                const float2 t = cmul(gc, make_float2(pr, pi));
                jr[0] += t.x;
                ji[0] += t.y;
            }
            float jsr = (jr[0] + jr[1]) + (jr[2] + jr[3]), jsi = (ji[0] + ji[1]) + (ji[2] + ji[3]);
            jsr += __shfl_xor_sync(0xffffffffu, jsr, 1);
            jsi += __shfl_xor_sync(0xffffffffu, jsi, 1);
            jsr += __shfl_xor_sync(0xffffffffu, jsr, 16);
            jsi += __shfl_xor_sync(0xffffffffu, jsi, 16);
            if (lead) {
                const float2 lL = lambda_pow(gam, omg, (float)L);
                const int64_t at = (int64_t)row * M + m;
                if (args.state_in) {
                    const float2 t = cmul(gc, cmul(args.state_in[at], lL));
                    jsr = fmaf((float)L, t.x, jsr);
                    jsi = fmaf((float)L, t.y, jsi);
                }
                args.part_j[at] = make_float2(jsr, jsi);
                if (args.d_state_in) {
                    const float2 prev = args.d_state_in[at];
                    args.d_state_in[at] = cfma(conj2(gc), conj2(lL), prev);
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) jr[k] = ji[k] = 0.0f;
            __syncwarp();   // the next tile's tensor-memory loads are warp-wide
            tv = 0;
            row += args.D;
        }
    } else if (warp < 6) {
        // ---------------------------------------------------- dx epilogue
        const int q = warp & 3;   // positions 32 q + lane
        const int i = 32 * q + lane;
        const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16);
        int row = row0, tile = ntiles - 1;
        for (int v = 0; v < nv; ++v) {
            const int bb = v & 1, slot = v % kTmSlots;
            // The old dx values of this tile (plain [chunk][position] layout).
            if (!wait_bar(bar(kTmSlotFull + slot), (v / kTmSlots) & 1, abort_flag)) break;
            const __nv_bfloat16 *sdx =
                reinterpret_cast<const __nv_bfloat16 *>(smem + kTmOffRing + slot * kTmSlotBytes + 4096) + i;
            float prev[kNT];
#pragma unroll
            for (int c = 0; c < kNT; ++c) prev[c] = __bfloat162float(sdx[c * kC]);
            __syncwarp();
            if (lane == 0) bar_arrive(bar(kTmSlotEmpty + slot));
            if (!wait_bar(bar(kTmDFull + bb), (v >> 1) & 1, abort_flag)) break;
            tc_fence_after();
            uint32_t r0[16], r1[16];
            tmem_ld16(tl + kTmColD + 32 * bb, r0);
            tmem_ld16(tl + kTmColD + 32 * bb + 16, r1);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive(bar(kTmDEmpty + bb));
            const int64_t n0 = (int64_t)tile * kNT;
            float add[kNT];
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                add[c] = __uint_as_float(r0[c]);
                add[c + 16] = __uint_as_float(r1[c]);
            }
            // The chunk holding token L - 1 (weight zero in the product): direct sum.
            if (n_part >= n0 && n_part < n0 + kNT) {
                const int64_t j = n_part * kC + i;
                float fx = 0.0f;
                if (j < L) {
                    const int s = (int)(L - 1 - j);
                    for (int mm = 0; mm < M; ++mm) {
                        const float2 p = pw[mm * kPwStride + s], gg = args.g[(int64_t)row * M + mm];
                        fx = fmaf(gg.x, p.x, fmaf(gg.y, p.y, fx));   // Re(conj(g) lambda^s)
                    }
                }
                const int cp = (int)(n_part - n0);
#pragma unroll
                for (int c = 0; c < kNT; ++c)
                    if (c == cp) add[c] += fx;
            }
            // dxT += add (one more bf16 rounding of the main pass's dx, well
            // inside the bf16 tolerance).
            __nv_bfloat16 *out = args.dxT + (int64_t)row * args.Lp + n0 * kC + i;
#pragma unroll
            for (int c = 0; c < kNT; ++c) out[c * kC] = __float2bfloat16_rn(prev[c] + add[c]);
            if (--tile < 0) {
                tile = ntiles - 1;
                row += args.D;
            }
        }
    } else if (warp == 6) {
        // ---------------------------------------------------- TMA producer
        if (lane == 0) {
            int issued = 0;
            int row = row0, tile = ntiles - 1;
            for (; issued < nv; ++issued) {
                const int slot = issued % kTmSlots;
                if (!wait_bar(bar(kTmSlotEmpty + slot), ((issued / kTmSlots) & 1) ^ 1, abort_flag)) break;
                bar_expect_tx(bar(kTmSlotFull + slot), 8192u);
                tma_load_3d(sbase + kTmOffRing + slot * kTmSlotBytes, &tmap_x, 0, tile * kNT, row,
                            bar(kTmSlotFull + slot));
                tma_load_3d(sbase + kTmOffRing + slot * kTmSlotBytes + 4096, &tmap_dx, 0, tile * kNT, row,
                            bar(kTmSlotFull + slot));
                if (--tile < 0) {
                    tile = ntiles - 1;
                    row += args.D;
                }
            }
            for (int k = issued > kTmSlots ? issued - kTmSlots : 0; k < issued; ++k)
                drain_bar(bar(kTmSlotFull + k % kTmSlots), (k / kTmSlots) & 1);
        }
        __syncwarp();
    } else {
        // ---------------------------------------------------- MMA issue
        if (lane == 0) {
            const uint64_t da = desc_plain(sbase + kTmOffA, 128, 1024);
            const uint64_t dal = desc_plain(sbase + kTmOffAlo, 128, 1024);
            const uint64_t du = desc_plain(sbase + kTmOffU, 128, 1024);
            int last_bar = -1;
            uint32_t last_par = 0;
            for (int v = 0; v < nv; ++v) {
                const int slot = v % kTmSlots, bb = v & 1;
                if (!wait_bar(bar(kTmSlotFull + slot), (v / kTmSlots) & 1, abort_flag)) break;
                if (!wait_bar(bar(kTmPEmpty + bb), ((v >> 1) & 1) ^ 1, abort_flag)) break;
                tc_fence_after();
                const uint64_t dx = desc_sw128(sbase + kTmOffRing + slot * kTmSlotBytes, 16, 1024);
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    umma_ss(tmem + kTmColP + 32 * bb, da + ks * 16, dx + ks * 2, kIdescN32, ks > 0);
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    umma_ss(tmem + kTmColP + 32 * bb, dal + ks * 16, dx + ks * 2, kIdescN32M64, 1u);
                umma_commit(bar(kTmPFull + bb));
                umma_commit(bar(kTmSlotEmpty + slot));
                last_bar = kTmSlotEmpty + slot;
                last_par = (v / kTmSlots) & 1;
                if (!wait_bar(bar(kTmWFull + bb), (v >> 1) & 1, abort_flag)) break;
                if (!wait_bar(bar(kTmDEmpty + bb), ((v >> 1) & 1) ^ 1, abort_flag)) break;
                tc_fence_after();
                const uint64_t dw = desc_plain(sbase + kTmOffW + bb * 8192, 512, 128);
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    umma_ss(tmem + kTmColD + 32 * bb, du + ks * 16, dw + ks * (2048 >> 4), kIdescU, ks > 0);
                umma_commit(bar(kTmDFull + bb));
                umma_commit(bar(kTmWEmpty + bb));
                last_bar = kTmWEmpty + bb;
                last_par = (v >> 1) & 1;
            }
            // Drain: the last commit's completion implies every earlier product's.
            if (last_bar >= 0) drain_bar(bar(last_bar), last_par);
        }
        __syncwarp();
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 6)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmCols));
}

// ------------------------------------------------------------ layout transposes
// [B][L][D] -> [B*D][Lp], zero for positions >= L.  Grid z = rows * nf: field f of
// batch row z / nf is (src0, dst0) or (src1, dst1).  rev: position s holds token
// L - 1 - s (time reversed within [0, L)).
__global__ void __launch_bounds__(128) k_to_channel_major(const __nv_bfloat16 *__restrict__ src0,
                                                          const __nv_bfloat16 *__restrict__ src1,
                                                          __nv_bfloat16 *__restrict__ dst0,
                                                          __nv_bfloat16 *__restrict__ dst1, int64_t L, int D,
                                                          int64_t Lp, int nf, int rev) {
    pdl_launch_dependents();
    __shared__ uint32_t tile[64][33];   // [position][channel pair]
    const int64_t t0 = (int64_t)blockIdx.x * 64;
    const int c0 = blockIdx.y * 64;
    const int b = blockIdx.z / nf, f = blockIdx.z % nf;
    const __nv_bfloat16 *src = f ? src1 : src0;
    __nv_bfloat16 *dst = f ? dst1 : dst0;
    // Four 16-byte loads per thread, all issued before the tile is written.
    uint4 val[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int it = threadIdx.x + 128 * k;
        const int r = it >> 3, vq = it & 7;
        const int64_t sp = t0 + r;
        const int c = c0 + 8 * vq;
        val[k] = make_uint4(0, 0, 0, 0);
        if (sp < L && c < D) {
            const int64_t t = rev ? L - 1 - sp : sp;
            val[k] = __ldg(reinterpret_cast<const uint4 *>(src + ((int64_t)b * L + t) * D + c));
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int it = threadIdx.x + 128 * k;
        const int r = it >> 3, vq = it & 7;
        tile[r][4 * vq] = val[k].x;
        tile[r][4 * vq + 1] = val[k].y;
        tile[r][4 * vq + 2] = val[k].z;
        tile[r][4 * vq + 3] = val[k].w;
    }
    __syncthreads();
    for (int it = threadIdx.x; it < 512; it += 128) {
        const int cr = it >> 3, vq = it & 7;
        const int c = c0 + cr;
        if (c >= D) continue;
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t a = tile[8 * vq + 2 * e][cr >> 1], bw = tile[8 * vq + 2 * e + 1][cr >> 1];
            const uint32_t lo = (cr & 1) ? (a >> 16) : (a & 0xffffu);
            const uint32_t hi = (cr & 1) ? (bw >> 16) : (bw & 0xffffu);
            w[e] = lo | (hi << 16);
        }
        *reinterpret_cast<uint4 *>(dst + ((int64_t)b * D + c) * Lp + t0 + 8 * vq) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// [B*D][Lp] -> [B][L][D] for tokens t < L, token t read from position t, or from
// L - 1 - t when rev.  A tile covers 64 tokens x 64 channels; it loads the
// 8-aligned window of 72 positions that holds its (reversed) positions.
__global__ void __launch_bounds__(128) k_to_row_major(const __nv_bfloat16 *srcT,
                                                      __nv_bfloat16 *__restrict__ dst, int64_t L, int D,
                                                      int64_t Lp, int rev) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ uint32_t tile[64][37];   // [channel][position pair]
    const int64_t t0 = (int64_t)blockIdx.x * 64;
    const int c0 = blockIdx.y * 64;
    const int b = blockIdx.z;
    // First position of the window: t0 itself, or the last 64 tokens' mirror rounded down.
    const int64_t s_lo = rev ? ((L - t0 - 64) >= 0 ? (L - t0 - 64) & ~(int64_t)7 : -((t0 + 64 - L + 7) & ~(int64_t)7)) : t0;
    // A reversed window can straddle nine 8-position groups, a forward one is
    // eight; a thread issues its (at most five) 16-byte loads before writing the
    // tile.
    const int nv = rev ? 9 : 8, nload = 64 * nv;
    uint4 val[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const int it = threadIdx.x + 128 * k;
        const int cr = it / nv, vq = it % nv;
        const int c = c0 + cr;
        const int64_t sp = s_lo + 8 * vq;
        val[k] = make_uint4(0, 0, 0, 0);
        if (it < nload && c < D && sp >= 0 && sp < Lp)
            val[k] = *reinterpret_cast<const uint4 *>(srcT + ((int64_t)b * D + c) * Lp + sp);
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const int it = threadIdx.x + 128 * k;
        if (it >= nload) break;
        const int cr = it / nv, vq = it % nv;
        tile[cr][4 * vq] = val[k].x;
        tile[cr][4 * vq + 1] = val[k].y;
        tile[cr][4 * vq + 2] = val[k].z;
        tile[cr][4 * vq + 3] = val[k].w;
    }
    __syncthreads();
    for (int it = threadIdx.x; it < 512; it += 128) {
        const int r = it >> 3, vq = it & 7;
        const int64_t t = t0 + r;
        const int c = c0 + 8 * vq;
        if (t >= L || c >= D) continue;
        const int i = (int)((rev ? L - 1 - t : t) - s_lo);   // 0 <= i < 72
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t a = tile[8 * vq + 2 * e][i >> 1], bw = tile[8 * vq + 2 * e + 1][i >> 1];
            const uint32_t lo = (i & 1) ? (a >> 16) : (a & 0xffffu);
            const uint32_t hi = (i & 1) ? (bw >> 16) : (bw & 0xffffu);
            w[e] = lo | (hi << 16);
        }
        *reinterpret_cast<uint4 *>(dst + ((int64_t)b * L + t) * D + c) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// [B*D][Lp] -> [B][L][D] without reversal: a 256-thread block covers 128 tokens x
// 64 channels, so it reads 256 contiguous bytes of each channel row (the 64-token
// tile above reads 128).  Measured on the backward at B = 4, L = 32768, D = 512:
// the dx transpose 14 us shorter (0.380 -> 0.365 ms per call).  The same widening
// of the channel-major transpose made it slower.
constexpr int kRmTokens = 128, kRmChannels = 64;
__global__ void __launch_bounds__(256) k_to_row_major_wide(const __nv_bfloat16 *srcT,
                                                           __nv_bfloat16 *__restrict__ dst, int64_t L, int D,
                                                           int64_t Lp) {
    pdl_launch_dependents();
    pdl_wait();
    constexpr int kStride = kRmTokens / 2 + 1, kGroups = kRmTokens / 8;
    constexpr int kLoads = kRmChannels * kGroups / 256, kStores = kRmTokens * (kRmChannels / 8) / 256;
    __shared__ uint32_t tile[kRmChannels][kStride];   // [channel][position pair]
    const int64_t t0 = (int64_t)blockIdx.x * kRmTokens;
    const int c0 = blockIdx.y * kRmChannels;
    const int b = blockIdx.z;
    uint4 val[kLoads];
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
        const int it = threadIdx.x + 256 * k;
        const int cr = it / kGroups, vq = it % kGroups;
        const int c = c0 + cr;
        const int64_t sp = t0 + 8 * vq;
        val[k] = make_uint4(0, 0, 0, 0);
        if (c < D && sp < Lp) val[k] = *reinterpret_cast<const uint4 *>(srcT + ((int64_t)b * D + c) * Lp + sp);
    }
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
        const int it = threadIdx.x + 256 * k;
        const int cr = it / kGroups, vq = it % kGroups;
        tile[cr][4 * vq] = val[k].x;
        tile[cr][4 * vq + 1] = val[k].y;
        tile[cr][4 * vq + 2] = val[k].z;
        tile[cr][4 * vq + 3] = val[k].w;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kStores; ++k) {
        const int it = threadIdx.x + 256 * k;
        const int r = it / (kRmChannels / 8), vq = it % (kRmChannels / 8);
        const int64_t t = t0 + r;
        const int c = c0 + 8 * vq;
        if (t >= L || c >= D) continue;
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t a = tile[8 * vq + 2 * e][r >> 1], bw = tile[8 * vq + 2 * e + 1][r >> 1];
            const uint32_t lo = (r & 1) ? (a >> 16) : (a & 0xffffu);
            const uint32_t hi = (r & 1) ? (bw >> 16) : (bw & 0xffffu);
            w[e] = lo | (hi << 16);
        }
        *reinterpret_cast<uint4 *>(dst + ((int64_t)b * L + t) * D + c) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}
// Its launch (D % 8 == 0, which every tcgen05 backward shape has).
cudaError_t row_major_wide(const __nv_bfloat16 *srcT, __nv_bfloat16 *dst, int64_t B, int64_t L, int D, int64_t Lp,
                           cudaStream_t st) {
    return launch_dependent(k_to_row_major_wide,
                            dim3((unsigned)((L + kRmTokens - 1) / kRmTokens),
                                 (unsigned)((D + kRmChannels - 1) / kRmChannels), (unsigned)B),
                            256, 0, st, srcT, dst, L, D, Lp);
}

// ------------------------------------------------------------ host side
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                   const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                   const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// 3-D map over a channel-major [rows][Lp] bf16 field viewed as (64 positions,
// Lp / 64 chunks, rows); box = one tile of one row (64 x 32 x 1), loaded with the
// 128-byte swizzle of the UMMA operand layout, or plain ([chunk][position]).
bool make_chunk_map(CUtensorMap *map, const void *ptr, int64_t rows, int64_t Lp, bool swizzle = true) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)kC, (cuuint64_t)(Lp / kC), (cuuint64_t)rows};
    cuuint64_t strides[2] = {(cuuint64_t)kC * 2, (cuuint64_t)Lp * 2};
    cuuint32_t box[3] = {(cuuint32_t)kC, (cuuint32_t)kNT, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int64_t padded_len(int64_t L) { return (L + kTile - 1) / kTile * kTile; }

size_t field_bytes(int64_t B, int64_t L, int D) {
    return ((size_t)B * D * padded_len(L) * 2 + 1023) / 1024 * 1024;
}
size_t part_bytes(int64_t B, int D, int M) {
    return ((size_t)B * D * M * sizeof(float2) + 255) / 256 * 256;
}

}  // namespace

bool tc_backward_supported(int64_t B, int64_t L, int D, int M, rlm_dtype dt) {
    return dt == RLM_BF16 && M >= 1 && M <= kMaxModes && D >= 8 && D % 8 == 0 && B >= 1 && L >= 1 &&
           L <= ((int64_t)1 << 31) - kTile && B * (int64_t)D <= ((int64_t)1 << 31) - 1 &&
           2 * B <= 65535;
}

size_t tc_backward_ws_bytes(int64_t B, int64_t L, int D, int M) {
    return 3 * field_bytes(B, L, D) + 3 * part_bytes(B, D, M);   // G, P and conj(g) J partials
}

namespace {

// Longest walk of a block over several rows, in tiles; rows of more than 8 tiles stay alone.
// At 16 the fill (6 tiles) is about a quarter of a block's time; longer walks have not been
// measured with the rows handed over one by one.
constexpr int kMaxWalk = 16;

cudaError_t configure_once() {
    static std::mutex mu;
    static std::vector<int> configured;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    if ((int)configured.size() <= dev) configured.resize(dev + 1, 0);
    if (!configured[dev]) {
        cudaError_t e = cudaSuccess;
        for (auto *k : {k_backward_tc<true, true>, k_backward_tc<true, false>, k_backward_tc<false, false>})
            if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_terminal_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kTmSmemBytes);
        if (e != cudaSuccess) return e;
        configured[dev] = 1;
    }
    return cudaSuccess;
}

BwdArgs base_args(const float *decay, const float *freq, const float *amp, const float *phase, __nv_bfloat16 *outT,
                  int64_t Lp, int D, int M) {
    BwdArgs a;
    a.decay = decay;
    a.freq = freq;
    a.amp = amp;
    a.phase = phase;
    a.part_g = nullptr;
    a.part_p = nullptr;
    a.state_in = nullptr;
    a.state_out = nullptr;
    a.coef_out = nullptr;
    a.d_state_in = nullptr;
    a.dxT = outT;
    a.Lp = Lp;
    a.D = D;
    a.M = M;
    a.ntiles = (int)(Lp / kTile);
    a.L = 0;
    return a;
}

// The row plan with the shortest estimated walk, in units of one tile: the plain waves of
// every number of blocks per channel, and the descending levels r, r / 2, 1 that each
// fill whole waves of the resident blocks.  kFill: tables, fill and drain of a block.
RowPlan row_plan(int64_t B, int D, int ntiles) {
    constexpr int64_t kFill = 6;
    const int64_t slots = 2 * sm_count();
    RowPlan best = {{1, 1, 1}, {(int)(B * D), (int)(B * D), (int)(B * D)}, {0, 0, 0}, (int)B, D};
    int64_t cost = (B * D + slots - 1) / slots * (kFill + ntiles);
    if (ntiles > kMaxWalk / 2) return best;
    for (int64_t r = B; r > 1; r = (r + 1) / 2) {
        if (r * ntiles > kMaxWalk) continue;
        RowPlan p = {{1, 1, 1}, {0, 0, 0}, {0, 0, 0}, (int)B, D};
        int64_t left = D, blocks = 0, c = 0, rl = r;
        for (int l = 0; l < 3; ++l, rl = l == 2 ? 1 : (rl + 1) / 2) {
            const int64_t u = (B + rl - 1) / rl, per = kFill + rl * ntiles;
            // Whole waves of this level (the last one takes what is left).
            const int64_t waves = l < 2 && rl > 1 ? left * u / slots : (left * u + slots - 1) / slots;
            const int64_t chans = l < 2 && rl > 1 ? std::min(left, waves * slots / u) : left;
            p.r[l] = (int)rl;
            p.ch[l] = (int)(D - left);
            left -= chans;
            blocks += chans * u;
            p.end[l] = (int)blocks;
            c += (chans > 0 ? waves : 0) * per;
        }
        if (c < cost) {
            cost = c;
            best = p;
        }
        const int64_t u = (B + r - 1) / r, cs = (D * u + slots - 1) / slots * (kFill + r * ntiles);
        if (cs < cost) {
            cost = cs;
            const int n = (int)(D * u);
            best = RowPlan{{(int)r, (int)r, (int)r}, {n, n, n}, {0, 0, 0}, (int)B, D};
        }
    }
    return best;
}

}  // namespace

int backward_plan_block(int64_t B, int D, int ntiles, int blk, int out[4]) {
    const RowPlan p = row_plan(B, D, ntiles);
    if (blk >= 0 && blk < p.end[2]) {
        rows_of(p, blk, out[0], out[1], out[2]);
        out[3] = level_of(p, blk);
    }
    return p.end[2];
}

namespace {

// The backward kernel for the call's plan.  Blocks of one row each keep the instance without
// the hand-over between rows (340 us a call at B = 4, L = 32768, D = 512, M = 32, against 365 on the other).
cudaError_t launch_backward(const CUtensorMap &mdy, const CUtensorMap &mx, const BwdArgs &a, cudaStream_t st) {
    const dim3 grid((unsigned)a.plan.end[2]);
    if (a.plan.r[0] > 1) return launch_dependent(k_backward_tc<true, true>, grid, kThreads, kSmemBytes, st, mdy, mx, a);
    return launch_dependent(k_backward_tc<true, false>, grid, kThreads, kSmemBytes, st, mdy, mx, a);
}

// One call: transpose in (nf fields: x, or x and dy), the tcgen05 kernel, transpose
// out, in stream order.  (Running the transposes of one part of the problem beside
// the tcgen05 kernel of another gained nothing: beside two tcgen05 CTAs an SM has
// room for one 128-thread transpose block, too few loads in flight to use the
// DRAM bandwidth the tcgen05 kernel leaves.)
template <bool kGrad>
cudaError_t run_layout_and_scan(const CUtensorMap &mdy, const CUtensorMap &mx, BwdArgs a, int64_t B, int64_t L,
                                int D, int64_t Lp, const __nv_bfloat16 *src0, const __nv_bfloat16 *src1,
                                __nv_bfloat16 *dst0, __nv_bfloat16 *dst1, int nf, int rev,
                                const __nv_bfloat16 *outT, __nv_bfloat16 *out, cudaStream_t st) {
    const unsigned cg = (unsigned)((D + 63) / 64);
    k_to_channel_major<<<dim3((unsigned)(Lp / 64), cg, (unsigned)(B * nf)), 128, 0, st>>>(
        src0, src1, dst0, dst1, L, D, Lp, nf, rev);
    if (kGrad) a.plan = row_plan(B, D, a.ntiles);
    cudaError_t e = cudaSuccess;
    if constexpr (kGrad) e = launch_backward(mdy, mx, a, st);
    else e = launch_dependent(k_backward_tc<false, false>, dim3((unsigned)(B * D)), kThreads, kSmemBytes, st, mdy, mx, a);
    if (e != cudaSuccess) return e;
    if (rev)
        e = launch_dependent(k_to_row_major, dim3((unsigned)((L + 63) / 64), cg, (unsigned)B), 128, 0, st, outT, out, L,
                             D, Lp, rev);
    else
        e = row_major_wide(outT, out, B, L, D, Lp, st);
    count_launches(3);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace


cudaError_t tc_backward(const void *dy, const void *x, void *dx, int64_t B, int64_t L, int D, int M,
                        const float *decay, const float *freq, const float *amp, const float *phase,
                        const float *state_in, const float *d_state_out, float *d_state_in, float *g_decay,
                        float *g_freq, float *g_amp, float *g_phase, void *ws, cudaStream_t st) {
    if (!ws) return cudaErrorInvalidValue;
    const int64_t Lp = padded_len(L);
    char *w = static_cast<char *>(ws);
    auto *xT = reinterpret_cast<__nv_bfloat16 *>(w);
    auto *dyT = reinterpret_cast<__nv_bfloat16 *>(w + field_bytes(B, L, D));
    auto *dxT = reinterpret_cast<__nv_bfloat16 *>(w + 2 * field_bytes(B, L, D));
    auto *pg = reinterpret_cast<float2 *>(w + 3 * field_bytes(B, L, D));
    auto *pp = reinterpret_cast<float2 *>(w + 3 * field_bytes(B, L, D) + part_bytes(B, D, M));
    auto *pj = reinterpret_cast<float2 *>(w + 3 * field_bytes(B, L, D) + 2 * part_bytes(B, D, M));
    const int64_t rows = B * (int64_t)D;
    CUtensorMap mdy, mx;
    if (!make_chunk_map(&mdy, dyT, rows, Lp) || !make_chunk_map(&mx, xT, rows, Lp)) return cudaErrorInvalidValue;
    cudaError_t e = configure_once();
    if (e != cudaSuccess) return e;
    BwdArgs a = base_args(decay, freq, amp, phase, dxT, Lp, D, M);
    a.part_g = pg;
    a.part_p = pp;
    a.state_in = reinterpret_cast<const float2 *>(state_in);
    a.d_state_in = reinterpret_cast<float2 *>(d_state_in);
    if (!d_state_out) {
        e = run_layout_and_scan<true>(mdy, mx, a, B, L, D, Lp, static_cast<const __nv_bfloat16 *>(x),
                                      static_cast<const __nv_bfloat16 *>(dy), xT, dyT, 2, 0, dxT,
                                      static_cast<__nv_bfloat16 *>(dx), st);
        if (e != cudaSuccess) return e;
    } else {
        // A terminal-state gradient g adds Re(conj(g) lambda^(L-1-t)) to dx_t,
        // conj(g) J to the decay / frequency products and g conj(lambda^L) to the
        // gradient of s_in (Sec. 3.2-3.3).  After the main pass, k_terminal_tc
        // forms them in closed form (no scan) from the channel-major x and adds
        // its dx to the main pass's in the channel-major buffer; one transpose
        // then writes the sum.
        const unsigned cg = (unsigned)((D + 63) / 64);
        k_to_channel_major<<<dim3((unsigned)(Lp / 64), cg, (unsigned)(B * 2)), 128, 0, st>>>(
            static_cast<const __nv_bfloat16 *>(x), static_cast<const __nv_bfloat16 *>(dy), xT, dyT, L, D, Lp, 2, 0);
        a.plan = row_plan(B, D, a.ntiles);
        if ((e = launch_backward(mdy, mx, a, st)) != cudaSuccess) return e;
        TermArgs ta;
        ta.plan = a.plan;
        ta.decay = decay;
        ta.freq = freq;
        ta.g = reinterpret_cast<const float2 *>(d_state_out);
        ta.state_in = reinterpret_cast<const float2 *>(state_in);
        ta.d_state_in = reinterpret_cast<float2 *>(d_state_in);
        ta.part_j = pj;
        ta.xT = xT;
        ta.dxT = dxT;
        ta.L = L;
        ta.Lp = Lp;
        ta.D = D;
        ta.M = M;
        ta.ntiles = (int)(Lp / kTile);
        CUtensorMap mdx;
        if (!make_chunk_map(&mdx, dxT, rows, Lp, false)) return cudaErrorInvalidValue;
        if ((e = launch_dependent(k_terminal_tc, dim3((unsigned)ta.plan.end[2]), kTmThreads, kTmSmemBytes, st, mx, mdx,
                                  ta)) != cudaSuccess ||
            (e = row_major_wide(dxT, static_cast<__nv_bfloat16 *>(dx), B, L, D, Lp, st)) != cudaSuccess)
            return e;
        count_launches(4);   // transpose, pass, terminal-state terms, transpose
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return grad_reduce(rows / D, D, M, amp, phase, pg, pp, d_state_out ? pj : nullptr, g_decay, g_freq, g_amp,
                       g_phase, st);
}

bool tc_prefill_rev_supported(int64_t B, int64_t L, int D, int M, rlm_dtype dt) {
    return tc_backward_supported(B, L, D, M, dt);
}

size_t tc_prefill_rev_ws_bytes(int64_t B, int64_t L, int D, int) { return 2 * field_bytes(B, L, D); }

cudaError_t tc_prefill_rev(const void *x, void *y, int64_t B, int64_t L, int D, int M, const float *decay,
                           const float *freq, const float *amp, const float *phase, const float *state_in,
                           float *state_out, float *coef_out, void *ws, cudaStream_t st) {
    if (!ws) return cudaErrorInvalidValue;
    const int64_t Lp = padded_len(L);
    char *w = static_cast<char *>(ws);
    auto *xr = reinterpret_cast<__nv_bfloat16 *>(w);
    auto *yr = reinterpret_cast<__nv_bfloat16 *>(w + field_bytes(B, L, D));
    const int64_t rows = B * (int64_t)D;
    CUtensorMap mx;
    if (!make_chunk_map(&mx, xr, rows, Lp)) return cudaErrorInvalidValue;
    cudaError_t e = configure_once();
    if (e != cudaSuccess) return e;
    BwdArgs a = base_args(decay, freq, amp, phase, yr, Lp, D, M);
    a.state_in = reinterpret_cast<const float2 *>(state_in);
    a.state_out = reinterpret_cast<float2 *>(state_out);
    a.coef_out = reinterpret_cast<float4 *>(coef_out);
    a.L = L;
    return run_layout_and_scan<false>(mx, mx, a, B, L, D, Lp, static_cast<const __nv_bfloat16 *>(x), nullptr, xr, nullptr,
                             1, 1, yr, static_cast<__nv_bfloat16 *>(y), st);
}

cudaError_t read_and_clear_bwd_status(int *status, cudaStream_t st) {
    cudaError_t e = cudaMemcpyFromSymbolAsync(status, g_bwd_status, sizeof(int), 0,
                                              cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
    const int zero = 0;
    if ((e = cudaMemcpyToSymbolAsync(g_bwd_status, &zero, sizeof(int), 0, cudaMemcpyHostToDevice,
                                     st)) != cudaSuccess)
        return e;
    return cudaStreamSynchronize(st);
}

}  // namespace rlm
