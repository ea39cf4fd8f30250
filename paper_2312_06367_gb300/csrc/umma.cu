// Split-precision history sum, T_0 solve and projector apply on the 5th-generation tensor cores
// (tcgen05 + TMEM + TMA), sm_103a.
//
// Every matrix-times-block-of-vectors product of a step has the form
//     out[r][i] = sum_q sum_j A_q[i][j] x_q[r][j]            (r < 64 right-hand sides)
// with the matrix split into two 16-bit slices, A = A_hi + A_lo, and the vectors into XS slices,
// x = x_hi + x_mid (+ x_lo), each slice the rounded remainder of the previous ones.
//   FP16X3: fp16 slices of power-of-two scaled values; blocks in two slices (one scale per row of
//           every block), vectors in three (one scale per 64-element tile of each slot and
//           right-hand side), about 2^-22 relative per stored matrix entry and 2^-33 per vector
//           entry.  Five products: A_hi x_hi, A_hi x_mid, A_lo x_hi, A_hi x_lo, A_lo x_mid.
//   BF16X3: bf16 slices, blocks and vectors in two; three products (hi hi, hi lo, lo hi).
// Stored matrix errors are fixed perturbations of the operator.  The MOT post-processing
// differences consecutive y (Eq. post_processing), which magnifies errors that change from step
// to step (vector rounding, accumulation) by about |y| / |y_n - y_{n-1}|, so those are kept near
// or below FP32 level: the leading product A_hi x_hi has its own tensor-memory accumulator (D0),
// separate from the four smaller ones (D1), and each accumulator covers one 64-wide k tile only;
// the epilogue adds the tiles error-free (TwoSum pairs in registers), partial sums are reduced as such
// pairs, and y_n, dy_n and the projector's u are kept in FP64; b_n goes from its pair to its slices.
//
// Kernel layout (one CTA per SM, persistent, 320 threads):
//   warp 0   TMA producer: A tiles (128 x 64, 128B swizzle) with L2 evict-first, x tiles
//            (64 x 64 per slice) with L2 evict-last, into a 4-deep ring of shared-memory stages;
//   warp 1   one elected thread issues tcgen05.mma (M = 128, N = 64, K = 16) and commits each
//            stage back to the producer and each finished pair of accumulators to the epilogue;
//   warps 2-9 epilogue (one row and 32 right-hand sides per thread): per k tile, tcgen05.ld of D0
//            and D1 (four TMEM buffers, so the next tiles' MMAs overlap), exact power-of-two
//            rescaling, error-free accumulation, and at the end of the CTA's part of a row tile a
//            coalesced store of the (hi, lo) partial sums.
// Work split: stream-K over (row tile, q, k tile) iterations in row-tile-major order; of several products
// with the same matrix (the projector's steps) each has blocks of its own, so that a step's sums do not
// depend on how many are taken together.  A second kernel,
// k_tc_fix, sums every tile's partials in a fixed order as FP32 pairs and applies the consumer's
// epilogue: store (u, out), or split into slices for the next product (b_n), or both (y_n: FP64 for the
// post-processing and the slices of the history ring).  (Left to the CTA that finished a tile last, the
// sums of some ten partials ran in one SM per tile: 45 us of the 57 us solve at 1920 edges.)
// Every mbarrier wait is bounded (%globaltimer, 2 s) and reports a timeout.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "plan.h"
#include "simt.h"
#include "umma.h"

namespace tdc {

constexpr int BM = 128;      // rows per tile (UMMA M)
constexpr int BK = 64;       // 16-bit elements per 128-byte row of a tile
constexpr int NR = 64;       // right-hand sides (UMMA N)
constexpr int STAGES = 4;
#ifndef TDC_NEPI
#define TDC_NEPI 8
#endif
constexpr int NEPI = TDC_NEPI;              // epilogue warps: 4 TMEM lane quarters x NEPI / 4 column groups
constexpr int NTHREADS = 64 + 32 * NEPI;    // producer warp, MMA warp, epilogue warps
constexpr int EC = NR / (NEPI / 4);         // columns (right-hand sides) per epilogue warp
#ifndef TDC_LDC
#define TDC_LDC 16
#endif
constexpr int LDC = TDC_LDC < EC ? TDC_LDC : EC;   // TMEM columns per tcgen05.ld of the epilogue
#ifndef TDC_D0S
#define TDC_D0S 1
#endif
constexpr int D0S = TDC_D0S;  // accumulators of the leading product per k tile (each 64 / D0S wide in K)
static_assert(D0S == 1 || D0S == 2 || D0S == 4, "D0S divides the four K = 16 steps of a k tile");
constexpr int BUFC = (D0S + 1) * NR;                           // TMEM columns of one buffer (D0 parts, D1)
constexpr int NBUF = BUFC <= 128 ? 4 : (BUFC <= 256 ? 2 : 1);  // accumulator buffers in tensor memory
constexpr int TC_C = 4;      // steps per chunk: tests and post-processing of so many steps share their kernels

template <int XS>
struct Cfg {
    static constexpr int A_BYTES = BM * BK * 2;
    static constexpr int X_BYTES = NR * BK * 2;
    static constexpr int STAGE = 2 * A_BYTES + XS * X_BYTES;
    static constexpr int MISC = 1536;      // barriers, flags, reduction scratch, tile scales
    static constexpr int SMEM = STAGES * STAGE + 1024 /*align*/ + MISC;
    static_assert(SMEM <= 232448, "shared memory per CTA");
    static constexpr int TMEM_COLS = 512;   // NBUF buffers x (D0 parts, D1)
};

enum { FIX_PLAIN = 0, FIX_SPLIT = 1, FIX_SOLVE = 2 };

// what k_tc_fix does with a row tile's sums s[r][row]
struct FixOut {
    int mode;
    double* out;          // PLAIN: out[(rep NR + r) * ld_out + row]; SOLVE: per column c of the chunk [y_n | dy_n],
                          // y_n = y_{n-1} + dy_n with y_{n-1} in the column before (cyclic)
    int ld_out;
    uint16_t* xs[3];      // SPLIT/SOLVE: destination slices, each [slots][NR][ld_x]
    float* sx;            // inverse scales [slots][ld_x / 64][NR]
    int ld_x;             // multiple of 64
    int slot_ring;        // 0: slot 0; > 0: slot n % slot_ring
};

struct GemmArgs {
    int rows, cols;       // M extent, K extent of one block
    int nblk, ktiles, rtiles;
    int reps;             // independent products with the same matrix (vector slot and output by product)
    int64_t total;        // iterations of one product: rtiles * nblk * ktiles
    int maxseg;
    int slot_mode;        // 0: history (q = 0, 1 -> ring + 2 col + q, q >= 2 -> (n - (q - 1)) mod ring);
                          // 1: slot rep; 2: slot q
    int ring;
    int off;              // step = ctl->n + off, column of the chunk ctl->col + off
    int mark;             // device time of the history: 1 starts it, 2 adds it up
    int grid;             // blocks of one product
    float* partial;       // [reps grid][maxseg][2][NR][BM]  (hi, lo)
    const int* seg_ptr;   // [rtiles + 1]
    const int* seg_slot;  // partial slots of every row tile (of the first product), in a fixed order
    Ctl* ctl;
    uint32_t idesc;       // instruction descriptor (operand format)
    const float* sA;      // [rows] inverse row scales of A (one per row, common to all blocks)
    const float* sX;      // [slots][ktiles][NR] inverse scales of x
    FixOut fx;
};

// ---------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t gtimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

// test for the phase; a thread whose phase is open is suspended for up to 20 us (the hint) instead
// of spinning, so waiting warps leave the issue slots to the working ones
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity), "r"(20000u)
        : "memory");
    return ok != 0;
}

// bounded wait: false (and the step's timeout flag set) if the phase did not complete in WAIT_NS
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, Ctl* ctl) {
    if (mbar_try(b, parity)) return true;
    const uint64_t t0 = gtimer();
    while (!mbar_try(b, parity)) {
        if (gtimer() - t0 > WAIT_NS) {
            atomicExch(&ctl->timeout, 1);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}

__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, uint64_t* bar,
                                            uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}

// untiled bulk copy global -> shared (16-byte aligned, size a multiple of 16), counted on bar
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t sdesc(const void* tile) {
    const uint64_t addr = smem_u32(tile);
    uint64_t d = 0;
    d |= (addr & 0x3FFFFull) >> 4;          // start address
    d |= (uint64_t)1 << 16;                 // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;       // stride byte offset
    d |= (uint64_t)1 << 46;                 // descriptor version
    d |= (uint64_t)2 << 61;                 // 128-byte swizzle
    return d;
}

// instruction descriptor: kind::f16, (bf16 or fp16) x same -> f32, K-major A and B, M = 128, N
static uint32_t make_idesc(int n, bool bf16) {
    const uint32_t f = bf16 ? 1u : 0u;
    return (1u << 4) | (f << 7) | (f << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

// vector slot of block q; base: n mod ring
__device__ __forceinline__ int slot_of(const GemmArgs& g, int q, int rep, int base, int col) {
    if (g.slot_mode == 1) return rep;
    if (g.slot_mode == 2) return q;
    if (q < 2) return g.ring + 2 * col + q;
    const int sl = base - (q - 1);      // q - 1 <= ring
    return sl < 0 ? sl + g.ring : sl;
}

__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(id), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

// 32 lanes x 32 columns of 32-bit values per warp (one lane = one row per thread)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* v) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
}
// 32 lanes x 16 columns
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* v) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
}
template <int W>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t* v) {
    if constexpr (W == 32) tmem_ld32(taddr, v);
    else tmem_ld16(taddr, v);
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// TwoSum on packed pairs (two FP32 lanes per instruction, sm_100+): hi + lo += v with the rounding
// error of each addition carried into lo.  x - y is written fma(y, -1, x): one rounding, exact
// like the subtraction.
__device__ __forceinline__ void two_sum_acc2(float2& hi, float2& lo, float2 v) {
    const float2 m1 = make_float2(-1.f, -1.f);
    const float2 t = __fadd2_rn(hi, v);
    const float2 bp = __ffma2_rn(hi, m1, t);   // t - hi
    const float2 a = __ffma2_rn(bp, m1, t);    // t - bp
    const float2 e1 = __ffma2_rn(a, m1, hi);   // hi - (t - bp)
    const float2 e2 = __ffma2_rn(bp, m1, v);   // v - bp
    lo = __fadd2_rn(lo, __fadd2_rn(e1, e2));
    hi = t;
}

// the same for the product a b, unrounded
__device__ __forceinline__ void two_sum_fma2(float2& hi, float2& lo, float2 a, float2 b) {
    const float2 m1 = make_float2(-1.f, -1.f);
    const float2 t = __ffma2_rn(a, b, hi);
    const float2 bp = __ffma2_rn(hi, m1, t);                                    // t - hi
    const float2 e1 = __ffma2_rn(__ffma2_rn(bp, m1, t), m1, hi);                // hi - (t - bp)
    const float2 e2 = __ffma2_rn(a, b, make_float2(-bp.x, -bp.y));              // a b - bp
    lo = __fadd2_rn(lo, __fadd2_rn(e1, e2));
    hi = t;
}

__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float v) {
    const float t = hi + v;
    const float bp = t - hi;
    lo += (hi - (t - bp)) + (v - bp);
    hi = t;
}

template <bool F16>
__device__ __forceinline__ uint16_t to16(float v) {
    if constexpr (F16) return __half_as_ushort(__float2half_rn(v));
    else return __bfloat16_as_ushort(__float2bfloat16_rn(v));
}
template <bool F16>
__device__ __forceinline__ float from16(uint16_t b) {
    if constexpr (F16) return __half2float(__ushort_as_half(b));
    else return __bfloat162float(__ushort_as_bfloat16(b));
}

// power of two p with m * p in [2^13, 2^14) (1 for m == 0 or not finite): values scaled by p fill
// fp16 without overflow.  The exponent is clamped to +-100 so that tiny tiles (an incident pulse
// that has not arrived, FP32 subnormals) cannot produce an infinite scale.
__device__ __forceinline__ float fill_scale(float m) {
    if (!(m > 0.f) || !(m < INFINITY)) return 1.f;
    int e;
    frexpf(m, &e);             // m = f 2^e, f in [0.5, 1)
    int k = 14 - e;
    k = k > 100 ? 100 : (k < -100 ? -100 : k);
    return ldexpf(1.f, k);
}

// v (FP64, already scaled) -> XS 16-bit slices, each the rounded remainder of the previous ones
template <bool F16, int XS>
__device__ __forceinline__ void split_value(double v, uint16_t* out) {
#pragma unroll
    for (int i = 0; i < XS; ++i) {
        const uint16_t b = to16<F16>((float)v);
        out[i] = b;
        v -= (double)from16<F16>(b);
    }
}

// (H + L) (a float pair, already scaled) -> XS 16-bit slices: H's leading slice, then the
// remainder (H - s0) + L (exact subtraction, one rounding of the small remainder)
template <bool F16, int XS>
__device__ __forceinline__ void split_pair(float H, float L, uint16_t* out) {
    const uint16_t b0 = to16<F16>(H);
    out[0] = b0;
    float r = (H - from16<F16>(b0)) + L;
#pragma unroll
    for (int i = 1; i < XS; ++i) {
        const uint16_t b = to16<F16>(r);
        out[i] = b;
        r -= from16<F16>(b);
    }
}

// the slices that the FP64 value of H + L has: the sum is normalised first and the rounding error of the
// first remainder is carried to the next slice
template <bool F16, int XS>
__device__ __forceinline__ void split_sum(float H, float L, uint16_t* out) {
    const float h = H + L, l = L - (h - H);
    const uint16_t b0 = to16<F16>(h);
    out[0] = b0;
    float r = h - from16<F16>(b0), e = 0.f;
    two_sum_acc(r, e, l);
#pragma unroll
    for (int i = 1; i < XS; ++i) {
        const uint16_t b = to16<F16>(r);
        out[i] = b;
        r = (r - from16<F16>(b)) + e;
    }
}

#ifndef TDC_XHI_BITS
#define TDC_XHI_BITS 11
#endif
#ifndef TDC_FP16_XS
#define TDC_FP16_XS 3
#endif
constexpr int FP16_XS = TDC_FP16_XS;   // fp16 slices per vector entry on the FP16X3 path

// Vector slices: the leading slice keeps XHI significant bits (rounded to nearest), the others
// carry the remainder.  Fewer leading bits shorten the products A_hi x_hi that share the leading
// accumulator, so fewer of their bits fall below the tensor core's alignment window.
constexpr int XHI = TDC_XHI_BITS;
template <bool F16, int XS>
__device__ __forceinline__ void split_vector(double v, uint16_t* out) {
    if constexpr (XHI < 11 && F16 && XS == 3) {
        int e;
        const double m = frexp(v, &e);                        // v = m 2^e, |m| in [0.5, 1)
        const double h = ldexp(rint(ldexp(m, XHI)), e - XHI);  // v to XHI significant bits
        out[0] = to16<F16>((float)h);
        split_value<F16, 2>(v - h, out + 1);
    } else {
        split_value<F16, XS>(v, out);
    }
}

// ---------------------------------------------------------------- the GEMM kernel
template <int XS, bool F16>
__global__ void __launch_bounds__(NTHREADS, 1)
    k_tc_gemm(const __grid_constant__ CUtensorMap tAh, const __grid_constant__ CUtensorMap tAl,
              const __grid_constant__ CUtensorMap tX0, const __grid_constant__ CUtensorMap tX1,
              const __grid_constant__ CUtensorMap tX2, GemmArgs g) {
    using C = Cfg<XS>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* misc = smem + STAGES * C::STAGE;
    uint64_t* full = reinterpret_cast<uint64_t*>(misc);
    uint64_t* empty = full + STAGES;
    uint64_t* acc_full = empty + STAGES;     // [NBUF]
    uint64_t* acc_empty = acc_full + NBUF;   // [NBUF]
    uint64_t* sx_full = acc_empty + NBUF;    // [NBUF] the tile scales of a buffer have landed
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sx_full + NBUF);
    float* sx_buf = reinterpret_cast<float*>(misc + 512);   // [NBUF][NR] x scales of an accumulator's tile
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    const int64_t ipt = (int64_t)g.nblk * g.ktiles;     // iterations per row tile
    const int rep = (int)blockIdx.x / g.grid, cta = (int)blockIdx.x - rep * g.grid;
    const int64_t begin = (int64_t)cta * g.total / g.grid;
    const int64_t end = (int64_t)(cta + 1) * g.total / g.grid;
    Ctl* ctl = g.ctl;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(full + s, 1); mbar_init(empty + s, 1); }
        // acc_full: the MMA commit and the MMA thread's copy of the tile's x scales
        for (int b = 0; b < NBUF; ++b) { mbar_init(acc_full + b, 1); mbar_init(acc_empty + b, NEPI); mbar_init(sx_full + b, 1); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"((uint32_t)C::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    wait_prior();       // what was set up above does not depend on the kernel before
    const int64_t n = ctl->n + g.off;
    const int col = ctl->col + g.off;
    const int base = g.ring > 0 ? (int)(n % g.ring) : 0;
    if (g.mark && blockIdx.x == 0 && threadIdx.x == 0) {
        if (g.mark == 1) ctl->t_mark = device_ns();
        else ctl->hist_ns += device_ns() - ctl->t_mark;
    }

    if (warp == 0) {
        if (lane == 0) {
            const uint64_t pa = policy_evict_first(), pb = policy_evict_last();
            int stage = 0, buf = 0;
            uint32_t phase = 0, ephase = 0;   // ephase bit b: phase parity of accumulator buffer b
            // (row tile, block, k tile) of the iteration, advanced without divisions
            int rt = (int)(begin / ipt);
            int q = (int)((begin - rt * ipt) / g.ktiles);
            int kt = (int)(begin - rt * ipt - (int64_t)q * g.ktiles);
            for (int64_t it = begin; it < end; ++it) {
                const int slot = slot_of(g, q, rep, base, col);
                if (!mbar_wait(empty + stage, phase ^ 1u, ctl)) break;
                // the tile's 64 x scales go to its accumulator buffer's slot, free once the epilogue
                // has released that buffer (the tile NBUF earlier)
                if (!mbar_wait(acc_empty + buf, ((ephase >> buf) & 1u) ^ 1u, ctl)) break;
                ephase ^= 1u << buf;
                uint8_t* st = smem + stage * C::STAGE;
                mbar_expect_tx(sx_full + buf, NR * 4);
                bulk_load(sx_buf + buf * NR, g.sX + ((int64_t)slot * g.ktiles + kt) * NR, NR * 4, sx_full + buf);
                mbar_expect_tx(full + stage, C::STAGE);
                tma_load_3d(st, &tAh, kt * BK, rt * BM, q, full + stage, pa);
                tma_load_3d(st + C::A_BYTES, &tAl, kt * BK, rt * BM, q, full + stage, pa);
                uint8_t* xt = st + 2 * C::A_BYTES;
                tma_load_3d(xt, &tX0, kt * BK, 0, slot, full + stage, pb);
                tma_load_3d(xt + C::X_BYTES, &tX1, kt * BK, 0, slot, full + stage, pb);
                if constexpr (XS == 3) tma_load_3d(xt + 2 * C::X_BYTES, &tX2, kt * BK, 0, slot, full + stage, pb);
                if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                buf = buf + 1 == NBUF ? 0 : buf + 1;
                if (++kt == g.ktiles) {
                    kt = 0;
                    if (++q == g.nblk) {
                        q = 0;
                        ++rt;
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t id = g.idesc;
            int stage = 0;
            uint32_t phase = 0;
            uint32_t ephase = 0;   // bit b: phase parity of accumulator buffer b
            int buf = 0;
            // one accumulator pair per k tile: D0 = A_hi x_hi, D1 = the smaller products
            for (int64_t it = begin; it < end; ++it) {
                if (!mbar_wait(acc_empty + buf, ((ephase >> buf) & 1u) ^ 1u, ctl)) break;
                ephase ^= 1u << buf;
                tc_fence_after();
                const uint32_t d0 = tmem + (uint32_t)(buf * BUFC), d1 = d0 + D0S * NR;
                if (!mbar_wait(full + stage, phase, ctl)) break;
                tc_fence_after();
                uint8_t* st = smem + stage * C::STAGE;
                const uint64_t ah = sdesc(st), al = sdesc(st + C::A_BYTES);
                const uint64_t x0 = sdesc(st + 2 * C::A_BYTES), x1 = sdesc(st + 2 * C::A_BYTES + C::X_BYTES);
                const uint64_t x2 = sdesc(st + 2 * C::A_BYTES + 2 * C::X_BYTES);
#pragma unroll
                for (int k = 0; k < BK / 16; ++k) {
                    const uint64_t adv = (uint64_t)(k * 32) >> 4;   // 16 elements = 32 bytes along K
                    const uint32_t acc = k > 0 ? 1u : 0u;
                    constexpr int KPER = (BK / 16) / D0S;     // K = 16 steps per leading accumulator
                    umma(d0 + (uint32_t)((k / KPER) * NR), ah + adv, x0 + adv, id, (k % KPER) ? 1u : 0u);
                    umma(d1, ah + adv, x1 + adv, id, acc);
                    umma(d1, al + adv, x0 + adv, id, 1);
                    if constexpr (XS == 3) {
                        umma(d1, ah + adv, x2 + adv, id, 1);
                        umma(d1, al + adv, x1 + adv, id, 1);
                    }
                }
                umma_commit(empty + stage);
                if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                umma_commit(acc_full + buf);
                buf = buf + 1 == NBUF ? 0 : buf + 1;
            }
        }
    } else {
        // epilogue: NEPI warps; warp w reads TMEM lanes 32 (w % 4) .. + 31 (one row per thread) and
        // the EC columns (right-hand sides) of its group ch = (w - 2) / 4
        const int quad = warp & 3, ch = (warp - 2) >> 2;
        const int row = quad * 32 + lane, cbase = ch * EC;
        uint32_t fphase = 0;   // bit b: phase parity of accumulator buffer b
        float2 acc_hi[EC / 2], acc_lo[EC / 2];   // columns (2c, 2c + 1) packed
#pragma unroll
        for (int c = 0; c < EC / 2; ++c) acc_hi[c] = acc_lo[c] = make_float2(0.f, 0.f);
        int seg = 0, buf = 0;
        bool ok = true;
        int64_t tile = begin / ipt, pos = begin - tile * ipt;   // row tile and iteration within it
        for (int64_t it = begin; it < end; ++it) {
            if (ok && !mbar_wait(acc_full + buf, (fphase >> buf) & 1u, ctl)) ok = false;
            if (ok && !mbar_wait(sx_full + buf, (fphase >> buf) & 1u, ctl)) ok = false;
            fphase ^= 1u << buf;
            if (ok) {
                tc_fence_after();
                const float* sx = sx_buf + buf * NR + cbase;
                const uint32_t d0 = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * BUFC + cbase);
                float seal = 0.f;
#pragma unroll
                for (int c0 = 0; c0 < EC; c0 += LDC) {
                    uint32_t v0[D0S][LDC], v1[LDC];
#pragma unroll
                    for (int part = 0; part < D0S; ++part) tmem_ld<LDC>(d0 + part * NR + c0, v0[part]);
                    tmem_ld<LDC>(d0 + D0S * NR + c0, v1);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < LDC; c += 4) {
                        const float4 s4 = *reinterpret_cast<const float4*>(sx + c0 + c);
                        const float2 sc[2] = {make_float2(s4.x, s4.y), make_float2(s4.z, s4.w)};
                        seal = s4.w;
#pragma unroll
                        for (int u = 0; u < 4; u += 2) {   // power-of-two scales: the products are exact
                            const int k = (c0 + c + u) >> 1;
#pragma unroll
                            for (int part = 0; part < D0S; ++part)
                                two_sum_acc2(acc_hi[k], acc_lo[k],
                                             __fmul2_rn(make_float2(__uint_as_float(v0[part][c + u]),
                                                                    __uint_as_float(v0[part][c + u + 1])), sc[u >> 1]));
                            acc_lo[k] = __ffma2_rn(make_float2(__uint_as_float(v1[c + u]), __uint_as_float(v1[c + u + 1])),
                                                   sc[u >> 1], acc_lo[k]);
                        }
                    }
                }
                tc_fence_before();
                // The arrival lets the producer overwrite the tile's scales, and it does not wait for
                // shared-memory loads still in flight: the vote on the last one read does (without it
                // about one march in twenty took one tile's last scales from a later tile).
                const bool seen = __all_sync(0xffffffffu, seal == seal);
                if (lane == 0 && seen) mbar_arrive(acc_empty + buf);   // the warp's reads are complete
            }
            buf = buf + 1 == NBUF ? 0 : buf + 1;
            const bool tile_end = ++pos == ipt;
            if (it + 1 == end || tile_end) {   // end of this CTA's part of the row tile
                float* dst = g.partial + ((int64_t)blockIdx.x * g.maxseg + seg) * (int64_t)2 * NR * BM;
                // one power-of-two row scale for all blocks: applied once here (exact)
                const int grow = (int)tile * BM + row;
                const float sa = grow < g.rows ? g.sA[grow] : 1.f;
#pragma unroll
                for (int c = 0; c < EC / 2; ++c) {
                    dst[(int64_t)(cbase + 2 * c) * BM + row] = acc_hi[c].x * sa;
                    dst[(int64_t)(cbase + 2 * c + 1) * BM + row] = acc_hi[c].y * sa;
                    dst[(int64_t)(NR + cbase + 2 * c) * BM + row] = acc_lo[c].x * sa;
                    dst[(int64_t)(NR + cbase + 2 * c + 1) * BM + row] = acc_lo[c].y * sa;
                    acc_hi[c] = acc_lo[c] = make_float2(0.f, 0.f);
                }
                ++seg;
            }
            if (tile_end) { ++tile; pos = 0; }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)C::TMEM_COLS)
                     : "memory");
    }
}

// ---------------------------------------------------------------- sums of the partials, consumer epilogue
// One block per (64-row half of a tile, 8 right-hand sides): thread (row, two right-hand sides).  The
// tile's partials are added in a fixed order (TwoSum pairs); 64 rows are one k tile of the consumer.
constexpr int FIX_RB = 8;
template <int XS, bool F16>
__global__ void __launch_bounds__(256) k_tc_fix(GemmArgs g) {
    __shared__ float red[2][FIX_RB];
    wait_prior();
    const FixOut& fx = g.fx;
    const int tile = blockIdx.x >> 1, half = blockIdx.x & 1;
    const int rep = tile / g.rtiles, rt = tile - rep * g.rtiles;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = half * 64 + (warp & 1) * 32 + lane, r0 = blockIdx.y * FIX_RB + (warp >> 1) * 2;
    const int grow = rt * BM + row;
    float sh[2] = {0.f, 0.f}, sl_[2] = {0.f, 0.f};
    const int p1 = g.seg_ptr[rt + 1];
    const float* part = g.partial + ((int64_t)rep * g.grid * g.maxseg * 2 * NR + r0) * BM + row;
#pragma unroll 4
    for (int k = g.seg_ptr[rt]; k < p1; ++k) {
        const float* P = part + (int64_t)g.seg_slot[k] * 2 * NR * BM;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            two_sum_acc(sh[j], sl_[j], __ldcg(P + (int64_t)j * BM));
            sl_[j] += __ldcg(P + (int64_t)(NR + j) * BM);
        }
    }
    const int64_t n = g.ctl->n + g.off;
    const int col = g.ctl->col + g.off;
    if (fx.mode != FIX_SPLIT && grow < g.rows) {
        const int prev = col == 0 ? TC_C - 1 : col - 1;      // column of y_{n-1}
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const double v = (double)sh[j] + (double)sl_[j];
            if (fx.mode == FIX_SOLVE) {     // increment dy_n, and y_n = y_{n-1} + dy_n
                fx.out[(int64_t)((2 * col + 1) * NR + r0 + j) * fx.ld_out + grow] = v;
                fx.out[(int64_t)(2 * col * NR + r0 + j) * fx.ld_out + grow] =
                    fx.out[(int64_t)(2 * prev * NR + r0 + j) * fx.ld_out + grow] + v;
            } else {
                fx.out[(int64_t)(rep * NR + r0 + j) * fx.ld_out + grow] = v;
            }
        }
    }
    if (fx.mode == FIX_PLAIN || rt * BM + half * 64 >= fx.ld_x) return;
    const int slot = fx.slot_ring > 0 ? (int)(n % fx.slot_ring) : 0;
#pragma unroll
    for (int j = 0; j < 2; ++j) {       // tile maxima over the 64 rows: two warps
        float m = fabsf(sh[j] + sl_[j]);
        if (!(m == m)) m = INFINITY;
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) red[warp & 1][(warp >> 1) * 2 + j] = m;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float sc = fill_scale(fmaxf(red[0][(warp >> 1) * 2 + j], red[1][(warp >> 1) * 2 + j]));
        uint16_t sl[3];
        split_pair<F16, XS>(sh[j] * sc, sl_[j] * sc, sl);
        const int64_t off = ((int64_t)slot * NR + r0 + j) * fx.ld_x + grow;
#pragma unroll
        for (int i = 0; i < XS; ++i) fx.xs[i][off] = sl[i];
        if ((row & 63) == 0) fx.sx[((int64_t)slot * (fx.ld_x / 64) + (rt * 2 + half)) * NR + r0 + j] = 1.f / sc;
    }
}

// ---------------------------------------------------------------- operand preparation
// rowmax[r] = max(rowmax[r], max_c |scale A[r][c]|) (non-negative floats order as their bits).
// One block per row.
__global__ void k_row_absmax(const double* __restrict__ A, int rows, int cols, double scale, float* __restrict__ rowmax) {
    __shared__ double red[256];
    const int r = blockIdx.x;
    const double* a = A + (int64_t)r * cols;
    double m = 0.0;
    for (int c = threadIdx.x; c < cols; c += blockDim.x) m = fmax(m, fabs(scale * a[c]));
    red[threadIdx.x] = m;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + w]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        float mf = (float)red[0];
        if (!(mf == mf)) mf = INFINITY;
        atomicMax(reinterpret_cast<unsigned int*>(rowmax) + r, __float_as_uint(mf));
    }
}

// FP64 matrix block (rows x cols, times `scale`) -> 16-bit hi/lo [rows][ld] with zero padding; row r
// scaled by the power of two of rowmax[r] (the maximum over every block that shares the row
// scale; its inverse goes to inv_row).  One block per row.
template <bool F16>
__global__ void k_split_mat(const double* __restrict__ A, int rows, int cols, int ld, double scale,
                            const float* __restrict__ rowmax, uint16_t* __restrict__ hi, uint16_t* __restrict__ lo,
                            float* __restrict__ inv_row) {
    const int r = blockIdx.x;
    const double* a = A + (int64_t)r * cols;
    const float sc = fill_scale(rowmax[r]);
    for (int c = threadIdx.x; c < ld; c += blockDim.x) {
        const double v = c < cols ? scale * a[c] * (double)sc : 0.0;
        uint16_t sl[2];
        split_value<F16, 2>(v, sl);
        hi[(int64_t)r * ld + c] = sl[0];
        lo[(int64_t)r * ld + c] = sl[1];
    }
    if (threadIdx.x == 0) inv_row[r] = 1.f / sc;
}

// FP64 vectors x[q][r][cols] -> XS slices [q][NR][ld] and inverse scales [q][ld/64][NR], one
// scale per 64-element tile of every vector.  Grid (ld/64, nblk), 256 threads.
template <bool F16, int XS>
__global__ void __launch_bounds__(256) k_split_x(const double* __restrict__ x, int cols, int ld, uint16_t* __restrict__ X0,
                                                 uint16_t* __restrict__ X1, uint16_t* __restrict__ X2,
                                                 float* __restrict__ sX) {
    __shared__ double v[NR][65];
    __shared__ float scl[NR];
    const int kt = blockIdx.x, q = blockIdx.y, t = threadIdx.x;
    for (int i = t; i < NR * 64; i += 256) {
        const int r = i >> 6, c = i & 63, col = kt * 64 + c;
        v[r][c] = col < cols ? x[((int64_t)q * NR + r) * cols + col] : 0.0;
    }
    __syncthreads();
    if (t < NR) {
        float m = 0.f;
        for (int c = 0; c < 64; ++c) m = fmaxf(m, fabsf((float)v[t][c]));
        scl[t] = fill_scale(m);
        sX[((int64_t)q * (ld / 64) + kt) * NR + t] = 1.f / scl[t];
    }
    __syncthreads();
    uint16_t* dst[3] = {X0, X1, X2};
    for (int i = t; i < NR * 64; i += 256) {
        const int r = i >> 6, c = i & 63;
        uint16_t sl[3];
        split_vector<F16, XS>(v[r][c] * (double)scl[r], sl);
        const int64_t off = ((int64_t)q * NR + r) * ld + kt * 64 + c;
#pragma unroll
        for (int k = 0; k < XS; ++k) dst[k][off] = sl[k];
    }
}

// ---------------------------------------------------------------- plane-wave tests, split
// The tensor-core step marches the increments dy_n = y_n - y_{n-1} (y_i = 0 for i <= 0): subtracting
// the MOT recurrence at step n - 1 from that at step n (Sec. IV-B) gives
//     sum_{k >= 0} T_k dy_{n-k} = r_n - r_{n-1},      r_0 = 0,
// the same recurrence for the increments, and the post-processing (Eq. post_processing) uses dy_n
// itself: j_n = P^LH y_n + P^S dy_n / dtt, y_n = y_{n-1} + dy_n in FP64.  The per-step rounding of
// the split arithmetic then scales with |dy_n| instead of |y_n|; the time difference of y, which
// is what the post-processing magnifies, is never formed by subtraction.
//
// Increments of the plane-wave tests (Sec. II-C): e_m(t_n) - e_m(t_{n-1}) = sum_x c(x).p
// [env_r(x, t_n) - env_r(x, t_{n-1})] with env_r(x, t) = amp_r exp(-a^2), a = (t - k_r.x - t0_r) /
// width_r, and the difference written as -amp_r exp(-a_n^2) expm1(d (2 a_n - d)), d = dt / width_r,
// so that it keeps its relative precision (-amp_r exp(-(a_n - d)^2) where the argument is above 64: the
// factor would overflow); at n = 1 the test itself (r_0 = 0).  Same for h.  t - t0 is
// carried as an FP32 pair so that late times lose no digits of the pulse's argument.
// The tests of a chunk's TC_C steps are formed when it starts (in the march's first chunk: of the steps that
// the calls make, new_cols), in two kernels: the envelope increments
// once per quadrature point, step and wave (a point belongs to three RWG or about twelve BC functions:
// with one exponential pair per edge and point this took 106 us per step at 1920 edges, now 28 + 93 us per
// four steps), then one block
// per (64-edge tile, step) gathers them, compensated FP32 sums over the points, and splits the tile into
// the e and h slices of the step's slots with one scale per (slot, tile, wave).
constexpr int ENV_PB = 32;       // points per block (the waves' FP64 parameters are formed once per block)
__global__ void __launch_bounds__(NR * TC_C) k_env_tc(int npts, const double* __restrict__ exc, double dt, const Ctl* ctl, int most,
                                                      const float* __restrict__ pts, float* __restrict__ env) {
    wait_prior();
    const int r = threadIdx.x % NR, i = threadIdx.x / NR;      // wave, step of the chunk
    const int col = ctl->col;
    const Cols cs = new_cols(ctl, TC_C, ctl->n, col, most);
    if (i < cs.lo || i >= cs.hi) return;
    const double* P = exc + 11 * r;
    const float kx = (float)P[0], ky = (float)P[1], kz = (float)P[2], amp = (float)P[6], inv_w = (float)(1.0 / P[8]);
    const int64_t n = ctl->n - col + i;
    const double tt = (double)n * dt - P[7];
    const float tt_hi = (float)tt, tt_lo = (float)(tt - (double)tt_hi), d = (float)(dt / P[8]);
    const int p1 = min(npts, (int)(blockIdx.x + 1) * ENV_PB);
#pragma unroll 4
    for (int pt = blockIdx.x * ENV_PB; pt < p1; ++pt) {
        const float arg = ((tt_hi - fmaf(kx, pts[3 * pt], fmaf(ky, pts[3 * pt + 1], kz * pts[3 * pt + 2]))) + tt_lo) * inv_w;
        float v = amp * expf(-arg * arg);
        if (n != 1) {       // env(t_n) - env(t_{n-1})
            const float x = d * (2.f * arg - d), b = arg - d;
            // e^x would overflow behind the pulse, where v underflows; there e^-x is nothing beside 1
            v = x > 64.f ? -amp * expf(-b * b) : -v * expm1f(x);
        }
        env[((int64_t)pt * TC_C + i) * NR + r] = v;
    }
}

// Block (64-edge tile, step): 16 warps of 4 edges, two waves per lane in packed FP32x2 arithmetic;
// entries {c, point index} as one 16-byte load
constexpr int RHS_NW = 16;
constexpr int RHS_LD = 65;
constexpr int RHS_SMEM = 2 * 64 * RHS_LD * 8;
template <bool F16, int XS>
__global__ void __launch_bounds__(32 * RHS_NW) k_rhs_tc(int ne, const double* __restrict__ exc, const Ctl* ctl, int most,
                                                const int* __restrict__ eptr, const float* env,
                                                const float4* __restrict__ ent, const int* __restrict__ nE,
                                                uint16_t* __restrict__ X0, uint16_t* __restrict__ X1,
                                                uint16_t* __restrict__ X2, float* __restrict__ sX, int ring, int ld) {
    extern __shared__ float2 ev[];      // [e, h][edge][wave], row length RHS_LD: sums as FP32 pairs
    __shared__ float mred[2][RHS_NW][NR];
    __shared__ float scl[2][NR];
    wait_prior();
    const int tile = blockIdx.x, step = blockIdx.y;
    const Cols cs = new_cols(ctl, TC_C, ctl->n, ctl->col, most);
    if (step < cs.lo || step >= cs.hi) return;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    float2 pol[2][3];       // p and k x p of the lane's two waves
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        const double* P = exc + 11 * (2 * lane + w);
        const float k[3] = {(float)P[0], (float)P[1], (float)P[2]}, q[3] = {(float)P[3], (float)P[4], (float)P[5]};
        const float h[3] = {k[1] * q[2] - k[2] * q[1], k[2] * q[0] - k[0] * q[2], k[0] * q[1] - k[1] * q[0]};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (w == 0) { pol[0][c].x = q[c]; pol[1][c].x = h[c]; }
            else { pol[0][c].y = q[c]; pol[1][c].y = h[c]; }
        }
    }
    const float2* en = reinterpret_cast<const float2*>(env) + step * (NR / 2) + lane;
    float mx[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
    for (int el = warp; el < 64; el += RHS_NW) {
        const int mm = tile * 64 + el;
        int q = 0, end = 0;
        if (mm < ne) q = eptr[mm];
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            float2 hi = make_float2(0.f, 0.f), lo = hi;
            if (mm < ne) end = f == 0 ? q + nE[mm] : eptr[mm + 1];
#pragma unroll 4
            for (; q < end; ++q) {
                const float4 c = ent[q];
                const float2 v = en[(int64_t)__float_as_int(c.w) * (TC_C * NR / 2)];
                const float2 cp = __ffma2_rn(make_float2(c.x, c.x), pol[f][0],
                                             __ffma2_rn(make_float2(c.y, c.y), pol[f][1], __fmul2_rn(make_float2(c.z, c.z), pol[f][2])));
                two_sum_fma2(hi, lo, v, cp);
            }
            float2* dst = ev + (f * 64 + el) * RHS_LD + 2 * lane;
            dst[0] = make_float2(hi.x, lo.x);
            dst[1] = make_float2(hi.y, lo.y);
            mx[f][0] = fmaxf(mx[f][0], fabsf(hi.x + lo.x));
            mx[f][1] = fmaxf(mx[f][1], fabsf(hi.y + lo.y));
        }
    }
#pragma unroll
    for (int f = 0; f < 2; ++f) {
        mred[f][warp][2 * lane] = mx[f][0];
        mred[f][warp][2 * lane + 1] = mx[f][1];
    }
    __syncthreads();
    const int slot0 = ring + 2 * step;
    if (t < 2 * NR) {
        const int w = t / NR, j = t % NR;
        float m = 0.f;
        for (int k = 0; k < RHS_NW; ++k) {
            const float v = mred[w][k][j];
            m = v == v ? fmaxf(m, v) : INFINITY;
        }
        scl[w][j] = fill_scale(m);
        sX[((int64_t)(slot0 + w) * (ld / 64) + tile) * NR + j] = 1.f / scl[w][j];
    }
    __syncthreads();
    uint16_t* dst[3] = {X0, X1, X2};
    for (int i = t; i < 2 * NR * 32; i += 32 * RHS_NW) {      // two edges per thread and turn
        const int w = i / (NR * 32), j = i / 32 % NR, el = 2 * (i & 31);
        uint16_t sl[2][3];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float2 v = ev[(w * 64 + el + u) * RHS_LD + j];
            split_sum<F16, XS>(v.x * scl[w][j], v.y * scl[w][j], sl[u]);
        }
        const int64_t off = ((int64_t)(slot0 + w) * NR + j) * ld + tile * 64 + el;
#pragma unroll
        for (int k = 0; k < XS; ++k)
            *reinterpret_cast<uint32_t*>(dst[k] + off) = (uint32_t)sl[0][k] | ((uint32_t)sl[1][k] << 16);
    }
}

// ---------------------------------------------------------------- projector in / out
// z[r][c] = sum_j tsign[c][j] w[r][tedge[c][j]], w = dy_n / dtt - y_n (= (1/dtt - 1) y_n - y_{n-1}/dtt)
// from the FP64 y_n and dy_n; split into the z slices with one scale per (64-triangle tile, wave).  Grid
// z: the steps p0 .. ctl->n + adv - 1 still to post-process (at most TC_C), slot by slot.  (A march of one
// step, 7680 edges, K = 4, with the products of four steps: 666 us, 617 us with one.)
constexpr int PIN_RB = 16;      // waves per block
__device__ __forceinline__ int post_count(const Ctl* ctl, int adv) { return (int)(ctl->n + adv - ctl->p0); }
// column of the chunk of step p0 + k (ctl->col belongs to ctl->n)
__device__ __forceinline__ int post_col(const Ctl* ctl, int k) {
    const int c = ctl->col + (int)(ctl->p0 - ctl->n) + k;
    return c < 0 ? c + TC_C : c;
}
template <bool F16, int XS>
__global__ void __launch_bounds__(256) k_project_in_tc(DevMesh m, const Ctl* ctl, int adv, const double* y2,
                                                       double inv_dtt, uint16_t* __restrict__ Z0, uint16_t* __restrict__ Z1,
                                                       uint16_t* __restrict__ Z2, float* __restrict__ sZ, int ldc) {
    __shared__ double zv[PIN_RB][65];
    __shared__ float scl[PIN_RB];
    const int tile = blockIdx.x, rb = blockIdx.y * PIN_RB;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    wait_prior();
    const int k = blockIdx.z;
    if (k >= post_count(ctl, adv)) return;
    const double* yn = y2 + (int64_t)post_col(ctl, k) * 2 * NR * m.ne;      // y_n
    const double* dy = yn + (int64_t)NR * m.ne;                             // dy_n
    float mx = 0.f;
    // thread -> (wave rb + (t >> 4) ... ): 16 waves x 64 triangles, 4 per thread, triangles fastest
    for (int i = t; i < PIN_RB * 64; i += 256) {
        const int j = i >> 6, cl = i & 63, c = tile * 64 + cl, r = rb + j;
        double s = 0.0;
        if (c < m.nc) {
            for (int l = 0; l < 3; ++l) {
                const int e = m.tedge[3 * c + l];
                s = fma(m.tsign[3 * c + l], fma(dy[(int64_t)r * m.ne + e], inv_dtt, -yn[(int64_t)r * m.ne + e]), s);
            }
        }
        zv[j][cl] = s;
    }
    __syncthreads();
    // maxima: warp w covers waves 2w, 2w+1 (lanes 0-15 / 16-31), 4 triangles per lane
    {
        const int j = 2 * warp + (lane >> 4), c4 = (lane & 15) * 4;
        for (int l = 0; l < 4; ++l) mx = fmaxf(mx, fabsf((float)zv[j][c4 + l]));
        for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if ((lane & 15) == 0) {
            if (!(mx == mx)) mx = INFINITY;
            scl[j] = fill_scale(mx);
            sZ[((int64_t)k * (ldc / 64) + tile) * NR + rb + j] = 1.f / scl[j];
        }
    }
    __syncthreads();
    uint16_t* dst[3] = {Z0, Z1, Z2};
    for (int i = t; i < PIN_RB * 64; i += 256) {
        const int j = i >> 6, cl = i & 63;
        uint16_t sl[3];
        split_vector<F16, XS>(zv[j][cl] * (double)scl[j], sl);
        const int64_t off = ((int64_t)k * NR + rb + j) * ldc + tile * 64 + cl;
#pragma unroll
        for (int l = 0; l < XS; ++l) dst[l][off] = sl[l];
    }
}

// j[r][m] = y_n[r][m] + u[r][c+(m)] - u[r][c-(m)] in FP64, stored in FP32; finiteness check (the first
// bad step is kept); grid y: the steps to post-process; the last block to finish advances the step
// counter by adv (every block has read it before it arrives).
__global__ void k_project_out_tc(DevMesh m, Ctl* ctl, int adv, const double* y2,
                                 const double* u, int* __restrict__ done) {
    wait_prior();
    const int idx = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    const int64_t n = ctl->p0 + k;
    if (idx < m.ne * NR && k < post_count(ctl, adv)) {
        const int r = idx / m.ne, e = idx % m.ne;
        const double yv = y2[((int64_t)post_col(ctl, k) * 2 * NR + r) * m.ne + e];
        const double* uk = u + ((int64_t)k * NR + r) * m.nc;
        const double val = yv + uk[m.cplus_[e]] - uk[m.cminus_[e]];
        if (!isfinite(val)) {
            atomicCAS(&ctl->status, 0, (int)TDCFIE_E_NONFINITE);
            atomicMin(reinterpret_cast<unsigned long long*>(&ctl->bad_step), (unsigned long long)n);
        }
        const int64_t at = ((n - ctl->n0) * NR + r) * (int64_t)m.ne + e;
        if (ctl->out) reinterpret_cast<float*>(ctl->out)[at] = (float)val;
        if (ctl->yout) reinterpret_cast<float*>(ctl->yout)[at] = (float)yv;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(done, 1) == (int)(gridDim.x * gridDim.y) - 1) {
            *done = 0;
            ctl->n += adv;
            ctl->col = (ctl->col + adv) % TC_C;
            ctl->p0 = ctl->n;
            __threadfence();
        }
    }
}
__global__ void k_advance_tc(Ctl* ctl) {
    wait_prior();
    ctl->n += 1;
    ctl->col = (ctl->col + 1) % TC_C;
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiled encoder() {
    static EncodeTiled fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult q;
        void* p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiled)p;
    }
    return fn;
}

// 3-D 16-bit map {inner (K), rows, slices} with box {64, box_rows, 1}, 128-byte swizzle
static bool make_map(CUtensorMap* m, void* base, int64_t inner, int64_t rows, int64_t slices, int64_t ld,
                     int box_rows, bool fp16) {
    EncodeTiled enc = encoder();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)inner, (cuuint64_t)rows, (cuuint64_t)slices};
    cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)ld * 2 * rows};
    cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, fp16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides,
               box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct Gemm {
    CUtensorMap ah, al, x[3];
    GemmArgs a;
    int grid = 0;
    int* seg_ptr = nullptr;
    int* seg_slot = nullptr;
};

struct TcStep {
    bool fp16 = false;
    int xs = 2;
    int ld = 0, ldc = 0, R = 0, sms = 0;
    uint16_t *Ah = nullptr, *Al = nullptr;          // history blocks [nblk][ne][ld]
    uint16_t *Th = nullptr, *Tl = nullptr;          // T_0^-1
    uint16_t *Ph = nullptr, *Pl = nullptr;          // (Sigma^T Sigma)^+
    uint16_t* X[3] = {nullptr, nullptr, nullptr};   // history ring + e, h slots of a chunk [ring + 2 TC_C][R][ld]
    uint16_t* B[3] = {nullptr, nullptr, nullptr};   // b [R][ld]
    uint16_t* Z[3] = {nullptr, nullptr, nullptr};   // z [TC_C][R][ldc]
    float* env = nullptr;                           // envelope increments [npts][TC_C][R]
    float *sAh = nullptr, *sAs = nullptr, *sAp = nullptr;   // inverse row scales
    float *sXh = nullptr, *sXb = nullptr, *sXz = nullptr;   // inverse tile scales of the vectors
    double *y2 = nullptr, *u = nullptr;             // FP64 y_n, dy_n [TC_C][2][R][ne], u [TC_C][R][nc]
    int* done = nullptr;
    float* partial = nullptr;
    Gemm hist, solve, proj;
    std::vector<void*> owned;
    ~TcStep() {
        for (void* p : owned) cudaFree(p);
        for (Gemm* g : {&hist, &solve, &proj}) {
            if (g->seg_ptr) cudaFree(g->seg_ptr);
            if (g->seg_slot) cudaFree(g->seg_slot);
        }
    }
};

void destroy_tc(TcStep* g) { delete g; }

__global__ void k_fill(float* p, int64_t n, float v) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}

// history ring, e/h slots and the FP64 y pair start at zero (y_i = 0 for i <= 0)
cudaError_t reset_tc(TcStep* g, int ring, int ne, cudaStream_t s) {
    const size_t xs = sizeof(uint16_t) * (size_t)(ring + 2 * TC_C) * g->R * g->ld;
    cudaError_t e;
    for (int i = 0; i < g->xs; ++i)
        if ((e = cudaMemsetAsync(g->X[i], 0, xs, s)) != cudaSuccess) return e;
    const int64_t ns = (int64_t)(ring + 2 * TC_C) * (g->ld / 64) * g->R;
    k_fill<<<(unsigned)((ns + 255) / 256), 256, 0, s>>>(g->sXh, ns, 1.f);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return cudaMemsetAsync(g->y2, 0, sizeof(double) * 2 * TC_C * (size_t)g->R * ne, s);
}

template <class T>
static cudaError_t dalloc(TcStep* g, T** p, size_t count) {
    cudaError_t e = cudaMalloc((void**)p, sizeof(T) * (count ? count : 1));
    if (e == cudaSuccess) g->owned.push_back(*p);
    return e;
}

// stream-K partition and the per-row-tile list of partial slots (same traversal as the kernel)
static void plan_segments(GemmArgs& a, int& grid, int rows, int cols, int nblk, int reps, int sms, std::vector<int>& ptr,
                          std::vector<int>& slot) {
    a.rows = rows;
    a.cols = cols;
    a.nblk = nblk;
    a.reps = reps;
    a.ktiles = (cols + BK - 1) / BK;
    a.rtiles = (rows + BM - 1) / BM;
    const int tiles = a.rtiles;
    a.total = (int64_t)tiles * nblk * a.ktiles;
    a.grid = grid = (int)std::min<int64_t>(sms, a.total);
    const int64_t ipt = (int64_t)nblk * a.ktiles;
    std::vector<std::vector<std::pair<int, int>>> lists(tiles);
    int maxseg = 1;
    for (int c = 0; c < grid; ++c) {
        const int64_t b = (int64_t)c * a.total / grid, e = (int64_t)(c + 1) * a.total / grid;
        int seg = 0;
        for (int64_t it = b; it < e; ++seg) {
            const int64_t rt = it / ipt;
            lists[rt].push_back({c, seg});
            it = std::min<int64_t>(e, (rt + 1) * ipt);
        }
        maxseg = std::max(maxseg, seg);
    }
    a.maxseg = maxseg;
    ptr.assign(tiles + 1, 0);
    slot.clear();
    for (int t = 0; t < tiles; ++t) {
        for (auto& cs : lists[t]) slot.push_back(cs.first * maxseg + cs.second);
        ptr[t + 1] = (int)slot.size();
    }
}

static cudaError_t plan_gemm(Gemm& G, int rows, int cols, int nblk, int reps, int sms, cudaStream_t s) {
    std::vector<int> ptr, slot;
    plan_segments(G.a, G.grid, rows, cols, nblk, reps, sms, ptr, slot);
    cudaError_t e;
    if ((e = cudaMalloc(&G.seg_ptr, sizeof(int) * ptr.size())) != cudaSuccess) return e;
    if ((e = cudaMalloc(&G.seg_slot, sizeof(int) * slot.size())) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(G.seg_ptr, ptr.data(), sizeof(int) * ptr.size(), cudaMemcpyHostToDevice, s)) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(G.seg_slot, slot.data(), sizeof(int) * slot.size(), cudaMemcpyHostToDevice, s)) != cudaSuccess) return e;
    G.a.seg_ptr = G.seg_ptr;
    G.a.seg_slot = G.seg_slot;
    return cudaSuccess;
}

static size_t partial_floats(const Gemm& G) { return (size_t)G.a.reps * G.grid * G.a.maxseg * 2 * NR * BM; }

template <int XS, bool F16>
static void launch_gemm(const Gemm& G, cudaStream_t s) {
    launch_chained(k_tc_gemm<XS, F16>, G.grid * G.a.reps, NTHREADS, s, Cfg<XS>::SMEM, G.ah, G.al, G.x[0], G.x[1], G.x[2], G.a);
    launch_chained(k_tc_fix<XS, F16>, dim3(2 * G.a.rtiles * G.a.reps, NR / FIX_RB), 256, s, 0, G.a);
}

// the product and its sums: two kernels
static void run_gemm(const TcStep* g, const Gemm& G, cudaStream_t s) {
    if (g->fp16) {
        if (g->xs == 3) launch_gemm<3, true>(G, s);
        else launch_gemm<2, true>(G, s);
    } else {
        launch_gemm<2, false>(G, s);
    }
}

static cudaError_t set_smem_attrs() {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_tc_gemm<3, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<3>::SMEM)) !=
        cudaSuccess)
        return e;
    if ((e = cudaFuncSetAttribute(k_tc_gemm<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<2>::SMEM)) !=
        cudaSuccess)
        return e;
    if ((e = cudaFuncSetAttribute(k_rhs_tc<true, FP16_XS>, cudaFuncAttributeMaxDynamicSharedMemorySize, RHS_SMEM)) != cudaSuccess)
        return e;
    if ((e = cudaFuncSetAttribute(k_rhs_tc<false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, RHS_SMEM)) != cudaSuccess)
        return e;
    return cudaFuncSetAttribute(k_tc_gemm<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<2>::SMEM);
}

// Split a stack of blocks that share one scale per row: maxima over all blocks first
struct SplitBlock {
    const double* A;
    double scale;
    uint16_t *hi, *lo;
};
static cudaError_t split_blocks(bool f16, cudaStream_t s, const std::vector<SplitBlock>& blocks, int rows, int cols,
                                int ld, float* rowmax, float* inv_row) {
    cudaError_t e = cudaMemsetAsync(rowmax, 0, sizeof(float) * rows, s);
    if (e != cudaSuccess) return e;
    for (const SplitBlock& b : blocks) k_row_absmax<<<rows, 256, 0, s>>>(b.A, rows, cols, b.scale, rowmax);
    for (const SplitBlock& b : blocks) {
        if (f16) k_split_mat<true><<<rows, 256, 0, s>>>(b.A, rows, cols, ld, b.scale, rowmax, b.hi, b.lo, inv_row);
        else k_split_mat<false><<<rows, 256, 0, s>>>(b.A, rows, cols, ld, b.scale, rowmax, b.hi, b.lo, inv_row);
    }
    return cudaGetLastError();
}

#define CKB(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) return cuda_fail(h, e_, #x); } while (0)

static int round_up(int x, int m) { return (x + m - 1) / m * m; }

tdcfie_status build_tc(tdcfie_t h, StepPlan* p) {
    const int R = p->R, ne = p->ne, nc = p->nc, K = h->K;
    if (R != NR) return fail(h, TDCFIE_E_UNSUPPORTED, "tensor-core path is built for R = 64 right-hand sides");
    if (!encoder()) return fail(h, TDCFIE_E_CUDA, "cuTensorMapEncodeTiled entry point not available");
    auto* g = new TcStep();
    p->gemm = g;
    g->fp16 = (p->prec == TDCFIE_FP16X3);
    g->xs = g->fp16 ? FP16_XS : 2;
    const int XS = g->xs;
    cudaStream_t s = h->stream;
    int dev = 0;
    CKB(cudaGetDevice(&dev));
    CKB(cudaDeviceGetAttribute(&g->sms, cudaDevAttrMultiProcessorCount, dev));
    g->R = R;
    g->ld = round_up(ne, BK);
    g->ldc = round_up(nc, BK);
    const int ld = g->ld, ldc = g->ldc, nblk = p->nblk, ring = p->ring;
    const size_t blk = (size_t)ne * ld;
    CKB(dalloc(g, &g->Ah, blk * nblk));
    CKB(dalloc(g, &g->Al, blk * nblk));
    CKB(dalloc(g, &g->Th, blk));
    CKB(dalloc(g, &g->Tl, blk));
    CKB(dalloc(g, &g->Ph, (size_t)nc * ldc));
    CKB(dalloc(g, &g->Pl, (size_t)nc * ldc));
    for (int i = 0; i < XS; ++i) {
        CKB(dalloc(g, &g->X[i], (size_t)(ring + 2 * TC_C) * R * ld));
        CKB(dalloc(g, &g->B[i], (size_t)R * ld));
        CKB(dalloc(g, &g->Z[i], (size_t)TC_C * R * ldc));
        CKB(cudaMemsetAsync(g->B[i], 0, sizeof(uint16_t) * R * ld, s));
        CKB(cudaMemsetAsync(g->Z[i], 0, sizeof(uint16_t) * TC_C * R * ldc, s));
    }
    for (int i = XS; i < 3; ++i) { g->X[i] = g->X[0]; g->B[i] = g->B[0]; g->Z[i] = g->Z[0]; }   // unused maps
    CKB(dalloc(g, &g->sAh, (size_t)ne));
    CKB(dalloc(g, &g->sAs, (size_t)ne));
    CKB(dalloc(g, &g->sAp, (size_t)nc));
    float* rowmax = nullptr;
    CKB(dalloc(g, &rowmax, (size_t)std::max(ne, nc)));
    CKB(dalloc(g, &g->sXh, (size_t)(ring + 2 * TC_C) * (ld / 64) * R));
    CKB(dalloc(g, &g->sXb, (size_t)(ld / 64) * R));
    CKB(dalloc(g, &g->sXz, (size_t)TC_C * (ldc / 64) * R));
    CKB(cudaMemsetAsync(g->sXz, 0, sizeof(float) * TC_C * (ldc / 64) * R, s));
    CKB(dalloc(g, &g->y2, (size_t)2 * TC_C * R * ne));
    CKB(dalloc(g, &g->u, (size_t)TC_C * R * nc));
    CKB(dalloc(g, &g->env, (size_t)p->npts * TC_C * R));
    CKB(dalloc(g, &g->done, 1));
    CKB(cudaMemsetAsync(g->done, 0, sizeof(int), s));
    // matrices: -A, alpha L2, -T_1 .. -T_{K-1}, then T_0^-1 and the Laplacian pseudo-inverse
    const int64_t NN = (int64_t)ne * ne;
    const bool f16 = g->fp16;
    {
        std::vector<SplitBlock> hb;
        hb.push_back({h->A, -1.0, g->Ah, g->Al});
        hb.push_back({h->L2, h->alpha, g->Ah + blk, g->Al + blk});
        for (int k = 1; k < K; ++k) hb.push_back({h->T + k * NN, -1.0, g->Ah + (1 + k) * blk, g->Al + (1 + k) * blk});
        CKB(split_blocks(f16, s, hb, ne, ne, ld, rowmax, g->sAh));
        CKB(split_blocks(f16, s, {{h->T0inv, 1.0, g->Th, g->Tl}}, ne, ne, ld, rowmax, g->sAs));
        CKB(split_blocks(f16, s, {{h->PinvS, 1.0, g->Ph, g->Pl}}, nc, nc, ldc, rowmax, g->sAp));
    }
    CKB(cudaGetLastError());
    CKB(cudaStreamSynchronize(s));
    CKB(reset_tc(g, ring, ne, s));
    // GEMM plans and tensor maps
    CKB(plan_gemm(g->hist, ne, ne, nblk, 1, g->sms, s));
    CKB(plan_gemm(g->solve, ne, ne, 1, 1, g->sms, s));
    // The projector's blocks per step: those of a chunk's four steps fill the chip once (a quarter each),
    // so that a block's part is long against its partial sums (1920 edges, 200 k tiles: with all blocks each
    // a march of 100 steps takes 20.8 instead of 20.0 ms); on large meshes half each, so that a step taken
    // alone does not leave most of the chip idle (7680 edges, 3200 k tiles, 17 steps: 7.51 ms, a quarter
    // 7.58, all 7.66)
    const int64_t its = (int64_t)(ldc / BK) * ((nc + BM - 1) / BM);
    CKB(plan_gemm(g->proj, nc, nc, 1, TC_C, std::max(1, g->sms / (its < 1024 ? 4 : 2)), s));
    size_t pmax = 0;
    for (Gemm* G : {&g->hist, &g->solve, &g->proj}) pmax = std::max(pmax, partial_floats(*G));
    CKB(dalloc(g, &g->partial, pmax));
    bool ok = make_map(&g->hist.ah, g->Ah, ne, ne, nblk, ld, BM, f16) && make_map(&g->hist.al, g->Al, ne, ne, nblk, ld, BM, f16) &&
              make_map(&g->solve.ah, g->Th, ne, ne, 1, ld, BM, f16) && make_map(&g->solve.al, g->Tl, ne, ne, 1, ld, BM, f16) &&
              make_map(&g->proj.ah, g->Ph, nc, nc, 1, ldc, BM, f16) && make_map(&g->proj.al, g->Pl, nc, nc, 1, ldc, BM, f16);
    for (int i = 0; i < 3; ++i)
        ok = ok && make_map(&g->hist.x[i], g->X[i], ne, R, ring + 2 * TC_C, ld, R, f16) &&
             make_map(&g->solve.x[i], g->B[i], ne, R, 1, ld, R, f16) &&
             make_map(&g->proj.x[i], g->Z[i], nc, R, TC_C, ldc, R, f16);
    if (!ok) return fail(h, TDCFIE_E_CUDA, "cuTensorMapEncodeTiled failed");
    const uint32_t id = make_idesc(R, !f16);
    for (Gemm* G : {&g->hist, &g->solve, &g->proj}) {
        G->a.partial = g->partial;
        G->a.ctl = p->ctl;
        G->a.ring = ring;
        G->a.slot_mode = 1;
        G->a.off = 0;
        G->a.mark = 0;
        G->a.idesc = id;
        G->a.fx = FixOut{};
    }
    // history: d_n -> slices of the solve's vector operand
    g->hist.a.slot_mode = 0;
    g->hist.a.mark = 1;
    g->solve.a.mark = 2;
    g->hist.a.sA = g->sAh;
    g->hist.a.sX = g->sXh;
    g->hist.a.fx.mode = FIX_SPLIT;
    g->hist.a.fx.ld_x = ld;
    g->hist.a.fx.sx = g->sXb;
    for (int i = 0; i < 3; ++i) g->hist.a.fx.xs[i] = g->B[i];
    // solve: dy_n -> FP64 dy_n, y_n += dy_n (post-processing) and the history ring slot n mod (K - 1)
    g->solve.a.sA = g->sAs;
    g->solve.a.sX = g->sXb;
    g->solve.a.fx.mode = FIX_SOLVE;
    g->solve.a.fx.out = g->y2;
    g->solve.a.fx.ld_out = ne;
    g->solve.a.fx.ld_x = ld;
    g->solve.a.fx.sx = g->sXh;
    g->solve.a.fx.slot_ring = ring;
    for (int i = 0; i < 3; ++i) g->solve.a.fx.xs[i] = g->X[i];
    // projector: u = (Sigma^T Sigma)^+ z in FP64
    g->proj.a.sA = g->sAp;
    g->proj.a.sX = g->sXz;
    g->proj.a.fx.mode = FIX_PLAIN;
    g->proj.a.fx.out = g->u;
    g->proj.a.fx.ld_out = nc;
    CKB(set_smem_attrs());
    CKB(cudaStreamSynchronize(s));
    // algorithmic bytes of the history GEMM: every block (hi + lo) once, and its R vectors (XS slices)
    h->hist_bytes = (double)nblk * ne * ne * 4.0 + (double)nblk * R * ne * 2.0 * XS;
    // and of the whole step: the history, T_0^-1 and the pseudo-inverse (hi + lo each)
    h->step_bytes = h->hist_bytes + 4.0 * (double)ne * ne + 4.0 * (double)nc * nc;
    return TDCFIE_OK;
}

// tests of the steps that new_cols gives -> their e, h slots
int launch_tests_tc(tdcfie_t h, StepPlan* p, int most, cudaStream_t s) {
    TcStep* g = p->gemm;
    const int ne = p->ne, ring = p->ring, ld = g->ld;
    launch_chained(k_env_tc, (p->npts + ENV_PB - 1) / ENV_PB, NR * TC_C, s, 0, p->npts, h->dexc, h->dt, p->ctl, most,
                   (const float*)p->pts, g->env);
    const dim3 grhs(ld / 64, TC_C);
    const float4* ent = (const float4*)p->ecoef;
    if (g->fp16)
        launch_chained(k_rhs_tc<true, FP16_XS>, grhs, 32 * RHS_NW, s, RHS_SMEM, ne, h->dexc, p->ctl, most, p->eptr, g->env, ent, p->enE,
                       g->X[0], g->X[1], g->X[2], g->sXh, ring, ld);
    else
        launch_chained(k_rhs_tc<false, 2>, grhs, 32 * RHS_NW, s, RHS_SMEM, ne, h->dexc, p->ctl, most, p->eptr, g->env, ent, p->enE,
                       g->X[0], g->X[1], g->X[2], g->sXh, ring, ld);
    return 2;
}

// step ctl->n + off: d_n = -A de_n + alpha L2 dh_n - sum_k T_k dy_{n-k}, then dy_n = T_0^-1 d_n, y_n = y_{n-1} +
// dy_n (FP64) and dy_n's slices into history slot n % ring; advance: the step counter moves on
int launch_inner_tc(tdcfie_t h, StepPlan* p, int off, bool advance, cudaStream_t s) {
    (void)h;
    TcStep* g = p->gemm;
    Gemm hist = g->hist, solve = g->solve;
    hist.a.off = solve.a.off = off;
    run_gemm(g, hist, s);
    run_gemm(g, solve, s);
    if (advance) launch_chained(k_advance_tc, 1, 1, s, 0, p->ctl);
    return advance ? 5 : 4;
}

// projector of the `count` finished steps: z = Sigma^T w_n, u = (Sigma^T Sigma)^+ z, j_n = y_n + Sigma u = P^LH y_n +
// P^S dy_n / dtt; the step counter moves by adv
int launch_post_tc(tdcfie_t h, StepPlan* p, int adv, int count, cudaStream_t s) {
    TcStep* g = p->gemm;
    const int ne = p->ne, ldc = g->ldc;
    const dim3 gproj(ldc / 64, NR / PIN_RB, count);
    if (g->fp16)
        launch_chained(k_project_in_tc<true, FP16_XS>, gproj, 256, s, 0, h->dm, p->ctl, adv, g->y2, 1.0 / h->dtt, g->Z[0], g->Z[1],
                       g->Z[2], g->sXz, ldc);
    else
        launch_chained(k_project_in_tc<false, 2>, gproj, 256, s, 0, h->dm, p->ctl, adv, g->y2, 1.0 / h->dtt, g->Z[0], g->Z[1], g->Z[2],
                       g->sXz, ldc);
    Gemm proj = g->proj;
    proj.a.reps = count;
    run_gemm(g, proj, s);
    launch_chained(k_project_out_tc, dim3((ne * NR + 255) / 256, count), 256, s, 0, h->dm, p->ctl, adv, g->y2, g->u, g->done);
    return 4;
}
int tc_chunk() { return TC_C; }

// ---------------------------------------------------------------- stand-alone product
// out[r][i] = sum_q sum_j blocks[q][i][j] x[q][r][j] in the split format (see tdcfie.h)
tdcfie_status tc_gemm(int precision, const double* blocks, int64_t nblk, int64_t rows, int64_t cols, const double* x,
                      int64_t R, double* out, cudaStream_t s) {
    tdcfie_t h = nullptr;
    if (precision != TDCFIE_FP16X3 && precision != TDCFIE_BF16X3)
        return fail(h, TDCFIE_E_UNSUPPORTED, "tensor-core product supports TDCFIE_FP16X3 and TDCFIE_BF16X3");
    if (!blocks || !x || !out) return fail(h, TDCFIE_E_ARG, "NULL device pointer");
    if (R != NR) return fail(h, TDCFIE_E_UNSUPPORTED, "tensor-core product is built for R = 64");
    if (nblk < 1 || nblk > 4096 || rows < 1 || rows > (1 << 20) || cols < 1 || cols > (1 << 20))
        return fail(h, TDCFIE_E_ARG, "sizes out of range (1 <= nblk <= 4096, 1 <= rows, cols <= 2^20)");
    if (!encoder()) return fail(h, TDCFIE_E_CUDA, "cuTensorMapEncodeTiled entry point not available");
    const bool f16 = precision == TDCFIE_FP16X3;
    const int XS = f16 ? FP16_XS : 2;
    const int ld = round_up((int)cols, BK);
    int dev = 0, sms = 0;
    CKB(cudaGetDevice(&dev));
    CKB(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    TcStep g;   // owns the scratch below
    g.fp16 = f16;
    g.xs = XS;
    Gemm& G = g.hist;
    std::vector<int> ptr, slot;
    plan_segments(G.a, G.grid, (int)rows, (int)cols, (int)nblk, 1, sms, ptr, slot);
    CKB(dalloc(&g, &g.Ah, (size_t)nblk * rows * ld));
    CKB(dalloc(&g, &g.Al, (size_t)nblk * rows * ld));
    CKB(dalloc(&g, &g.sAh, (size_t)rows));
    float* rowmax = nullptr;
    CKB(dalloc(&g, &rowmax, (size_t)rows));
    for (int i = 0; i < XS; ++i) CKB(dalloc(&g, &g.X[i], (size_t)nblk * NR * ld));
    for (int i = XS; i < 3; ++i) g.X[i] = g.X[0];
    CKB(dalloc(&g, &g.sXh, (size_t)nblk * (ld / 64) * NR));
    CKB(dalloc(&g, &g.partial, partial_floats(G)));
    CKB(dalloc(&g, &G.seg_ptr, ptr.size()));
    CKB(dalloc(&g, &G.seg_slot, slot.size()));
    g.owned.erase(g.owned.end() - 2, g.owned.end());   // freed by ~TcStep's per-Gemm loop
    CKB(cudaMemcpyAsync(G.seg_ptr, ptr.data(), sizeof(int) * ptr.size(), cudaMemcpyHostToDevice, s));
    CKB(cudaMemcpyAsync(G.seg_slot, slot.data(), sizeof(int) * slot.size(), cudaMemcpyHostToDevice, s));
    {
        std::vector<SplitBlock> sb;
        for (int64_t q = 0; q < nblk; ++q) sb.push_back({blocks + q * rows * cols, 1.0, g.Ah + q * rows * ld, g.Al + q * rows * ld});
        CKB(split_blocks(f16, s, sb, (int)rows, (int)cols, ld, rowmax, g.sAh));
    }
    const dim3 gx(ld / 64, (unsigned)nblk);
    if (f16) k_split_x<true, FP16_XS><<<gx, 256, 0, s>>>(x, (int)cols, ld, g.X[0], g.X[1], g.X[2], g.sXh);
    else k_split_x<false, 2><<<gx, 256, 0, s>>>(x, (int)cols, ld, g.X[0], g.X[1], g.X[2], g.sXh);
    CKB(cudaGetLastError());
    bool ok = make_map(&G.ah, g.Ah, cols, rows, nblk, ld, BM, f16) && make_map(&G.al, g.Al, cols, rows, nblk, ld, BM, f16);
    for (int i = 0; i < 3; ++i) ok = ok && make_map(&G.x[i], g.X[i], cols, NR, nblk, ld, NR, f16);
    if (!ok) return fail(h, TDCFIE_E_CUDA, "cuTensorMapEncodeTiled failed");
    Ctl* ctl = nullptr;
    CKB(dalloc(&g, &ctl, 1));
    CKB(cudaMemsetAsync(ctl, 0, sizeof(Ctl), s));
    G.a.seg_ptr = G.seg_ptr;
    G.a.seg_slot = G.seg_slot;
    G.a.partial = g.partial;
    G.a.ctl = ctl;
    G.a.ring = 1;
    G.a.off = 0;
    G.a.mark = 0;
    G.a.slot_mode = 2;
    G.a.idesc = make_idesc(NR, !f16);
    G.a.sA = g.sAh;
    G.a.sX = g.sXh;
    G.a.fx = FixOut{};
    G.a.fx.mode = FIX_PLAIN;
    G.a.fx.out = out;
    G.a.fx.ld_out = (int)rows;
    CKB(set_smem_attrs());
    run_gemm(&g, G, s);
    CKB(cudaGetLastError());
    CKB(cudaStreamSynchronize(s));
    Ctl c;
    CKB(cudaMemcpy(&c, ctl, sizeof(Ctl), cudaMemcpyDeviceToHost));
    if (c.timeout) return fail(h, TDCFIE_E_TIMEOUT, "a bounded device-side wait ran out (tensor-core pipeline)");
    return TDCFIE_OK;
}

}  // namespace tdc
