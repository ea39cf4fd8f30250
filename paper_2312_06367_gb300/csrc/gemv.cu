// Stand-alone history sum of the MOT recurrence (Sec. IV-B) on caller-held blocks:
//   out[r][i] = sum_{q < nblk} sum_{j < n} blocks[q][i][j] x[q][r][j]
// A warp writes the per-block partial sums of a few rows of one block; a second kernel adds the
// blocks in a fixed order (deterministic result).
#include <cuda.h>
#include <cuda_runtime.h>

#include <mutex>

#include "simt.h"

namespace tdc {

// Streams the matrices once.  FP32 is bound by the memory: several loads per row are in flight, and with
// R > 1 a warp takes two rows, so that a value of x is fetched once for both (with one row per warp the
// fetches of x at R = 8 took eight times the matrix's).  41 blocks of 7680 rows, R = 1, FP32: 1300 us
// (7.4 TB/s); 1614 us with 4-byte loads.  FP64 is bound by its pipe from R = 3 on (0.62e12 multiply-adds/s),
// where vector loads only lengthen a row's last turn.  Every R has its own kernel: a bound on r that is not a
// constant costs a branch or an idle issue slot per product (R = 5, FP64, 7680 rows: 2.0 ms, 3.6 ms with room for 8).
template <typename T> struct Vec16;
template <> struct Vec16<float> { using V = float4; };
template <> struct Vec16<double> { using V = double2; };

// Rows per warp and turns unrolled, W entries per load: 1, or (rows and pointers on 16-byte boundaries)
// a 16-byte vector.  Measured over 1, 2, 4 rows x 1, 2, 4, 8 turns at 120 to 7680 rows per block:
//   FP32  vectors  R = 1: 1 row x 4 (41 blocks of 7680: 1296 us; 4 x 4 1390); R > 1: 2 x 1 (R = 8, 4 blocks: 219 us; 4 x 2 305)
//         scalars  R = 1: 1 x 8 (4 blocks of 7679: 167 us; 4 x 2 272); R > 1: 2 x 2 (R = 8: 391 us; 4 x 2 386, 1 x 2 725)
//   FP64  1 row (R = 8, 7679: 3.24 ms; 2 rows 3.27, 4 rows 3.7), 4 turns up to R = 4, above 1
template <typename T, int R, int W>
struct BgShape {
    static constexpr bool F32 = sizeof(T) == 4;
    static constexpr int ROWS = F32 && R > 1 ? 2 : 1;
    static constexpr int TURNS = !F32 ? (R <= 4 ? 4 : 1) : R > 1 ? (W > 1 ? 1 : 2) : W > 1 ? 4 : 8;
};

template <typename T, int R, int W>
__global__ void k_bg_partial(const T* __restrict__ blocks, int64_t n, const T* __restrict__ x,
                             T* __restrict__ partial) {
    constexpr int NR = BgShape<T, R, W>::ROWS;
    const int64_t row0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * NR;
    const int64_t q = blockIdx.y;
    const int lane = threadIdx.x & 31;
    if (row0 >= n) return;
    const T* a = blocks + (q * n + row0) * n;
    const T* xq = x + q * R * n;
    int64_t ro[NR];      // rows behind the last one read the last one
#pragma unroll
    for (int i = 0; i < NR; ++i) ro[i] = (row0 + i < n ? i : n - 1 - row0) * n;
    T s[NR][R] = {};
#pragma unroll(BgShape<T, R, W>::TURNS)
    for (int64_t j = W * lane; j < n; j += 32 * W) {
        T v[NR][W];
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            if constexpr (W == 1) v[i][0] = __ldcs(a + ro[i] + j);
            else *reinterpret_cast<typename Vec16<T>::V*>(v[i]) = __ldcs(reinterpret_cast<const typename Vec16<T>::V*>(a + ro[i] + j));
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            T u[W];
            if constexpr (W == 1) u[0] = xq[r * n + j];
            else *reinterpret_cast<typename Vec16<T>::V*>(u) = *reinterpret_cast<const typename Vec16<T>::V*>(xq + r * n + j);
#pragma unroll
            for (int i = 0; i < NR; ++i)
#pragma unroll
                for (int k = 0; k < W; ++k) s[i][r] += v[i][k] * u[k];
        }
    }
#pragma unroll
    for (int i = 0; i < NR; ++i)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            T v = s[i][r];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0 && row0 + i < n) partial[(q * R + r) * n + row0 + i] = v;
        }
}

template <typename T>
__global__ void k_bg_reduce(const T* partial, int64_t nblk, int64_t n, int R, T* out) {
    wait_prior();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * R) return;
    T s = 0;
#pragma unroll 8
    for (int64_t q = 0; q < nblk; ++q) s += __ldcg(partial + q * R * n + i);
    out[i] = s;
}

template <typename T, int R>
static void launch_bg_partial(const T* blocks, int64_t nblk, int64_t n, const T* x, T* partial, cudaStream_t s) {
    constexpr int V = 16 / (int)sizeof(T), W = sizeof(T) == 8 && R > 3 ? 1 : V;
    const auto grid = [&](int rows) { return dim3((unsigned)((n + 8 * rows - 1) / (8 * rows)), (unsigned)nblk); };
    if (W > 1 && n % W == 0 && (uintptr_t)blocks % 16 == 0 && (uintptr_t)x % 16 == 0)
        k_bg_partial<T, R, W><<<grid(BgShape<T, R, W>::ROWS), 256, 0, s>>>(blocks, n, x, partial);
    else
        k_bg_partial<T, R, 1><<<grid(BgShape<T, R, 1>::ROWS), 256, 0, s>>>(blocks, n, x, partial);
}

template <typename T>
static cudaError_t launch_block_gemv(const T* blocks, int64_t nblk, int64_t n, const T* x, int R, T* out, T* partial,
                                     cudaStream_t s) {
    using Launch = void (*)(const T*, int64_t, int64_t, const T*, T*, cudaStream_t);
    static const Launch by_r[] = {launch_bg_partial<T, 1>, launch_bg_partial<T, 2>, launch_bg_partial<T, 3>, launch_bg_partial<T, 4>,
                                  launch_bg_partial<T, 5>, launch_bg_partial<T, 6>, launch_bg_partial<T, 7>, launch_bg_partial<T, 8>};
    by_r[R - 1](blocks, nblk, n, x, partial, s);
    launch_chained(k_bg_reduce<T>, (unsigned)((n * R + 63) / 64), 64, s, 0, (const T*)partial, nblk, n, R, out);
    return cudaGetLastError();
}

// common argument checks; returns 0 when the call may proceed
static tdcfie_status check_gemv(int precision, const void* blocks, int64_t nblk, int64_t n, const void* x, int64_t R,
                                void* out) {
    if (precision != TDCFIE_FP64 && precision != TDCFIE_FP32)
        return fail(nullptr, TDCFIE_E_UNSUPPORTED, "block GEMV supports TDCFIE_FP64 and TDCFIE_FP32");
    if (!blocks || !x || !out) return fail(nullptr, TDCFIE_E_ARG, "NULL device pointer");
    if (nblk < 1 || nblk > 65535 || n < 1 || n > (1 << 24) || R < 1 || R > 8)
        return fail(nullptr, TDCFIE_E_ARG, "sizes out of range (1 <= nblk <= 65535, 1 <= n <= 2^24, 1 <= R <= 8)");
    return TDCFIE_OK;
}

}  // namespace tdc

using namespace tdc;

extern "C" tdcfie_status tdcfie_block_gemv(int precision, const void* blocks, int64_t nblk, int64_t n, const void* x,
                                           int64_t R, void* out, void* stream) {
    tdcfie_status st = check_gemv(precision, blocks, nblk, n, x, R, out);
    if (st != TDCFIE_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t es = precision == TDCFIE_FP64 ? 8 : 4;
    void* partial = nullptr;
    cudaError_t e = cudaMallocAsync(&partial, es * (size_t)nblk * R * n, s);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaMallocAsync (block GEMV scratch)");
    if (precision == TDCFIE_FP64)
        e = launch_block_gemv<double>((const double*)blocks, nblk, n, (const double*)x, (int)R, (double*)out,
                                      (double*)partial, s);
    else
        e = launch_block_gemv<float>((const float*)blocks, nblk, n, (const float*)x, (int)R, (float*)out,
                                     (float*)partial, s);
    cudaError_t e2 = cudaFreeAsync(partial, s);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "block GEMV launch");
    if (e2 != cudaSuccess) return cuda_fail(nullptr, e2, "cudaFreeAsync (block GEMV scratch)");
    return TDCFIE_OK;
}

// ---------------------------------------------------------------- variant without allocation
// Some callers cannot allocate device memory when they need this sum: a thread of a process in
// which another thread holds a global-mode stream capture (cudaMalloc is not permitted then),
// services whose caching allocator has reserved nearly all of the HBM up front, or loops that
// cannot take the implicit synchronisation of an allocation.  For them the per-block partial sums
// live in this file-scope device array.  Every GPU that loads the library holds it (32 MiB) until
// the process exits.  In host code the name below is only a host-side stand-in for the array;
// the kernels receive the device address obtained with cudaGetSymbolAddress.
namespace tdc {
constexpr size_t NOALLOC_SCRATCH_BYTES = size_t(32) << 20;
static __device__ __align__(256) unsigned char g_block_gemv_scratch[NOALLOC_SCRATCH_BYTES];

constexpr int NOALLOC_MAX_DEVICES = 64;
static void* g_scratch_addr[NOALLOC_MAX_DEVICES];
static CUcontext g_scratch_ctx[NOALLOC_MAX_DEVICES];
static std::mutex g_scratch_mu;

// cuCtxGetCurrent through the runtime's driver entry point, so that the library keeps no link-time
// dependency on the driver library (it loads on hosts without a GPU)
typedef CUresult (*CtxGetCurrent)(CUcontext*);
static CtxGetCurrent ctx_get_current() {
    static CtxGetCurrent fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult q;
        void* p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (CtxGetCurrent)p;
    }
    return fn;
}

// device address of the scratch array on the current device, looked up once per device and
// context (a cudaDeviceReset gives the device a new primary context and the array a new address)
static cudaError_t scratch_address(void** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return cudaErrorInvalidDevice;
    // no allocation and no synchronising call here: cudaGetDevice and cuCtxGetCurrent only, and
    // the symbol lookup (which also makes the primary context current) when the context is new
    const CtxGetCurrent get = ctx_get_current();
    if (!get) return cudaErrorDeviceUninitialized;
    CUcontext ctx = nullptr;
    if (get(&ctx) != CUDA_SUCCESS) return cudaErrorDeviceUninitialized;
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_addr[dev] || !ctx || g_scratch_ctx[dev] != ctx) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_block_gemv_scratch);
        if (e != cudaSuccess) return e;
        if (get(&ctx) != CUDA_SUCCESS) return cudaErrorDeviceUninitialized;
        g_scratch_addr[dev] = p;
        g_scratch_ctx[dev] = ctx;
    }
    *out = g_scratch_addr[dev];
    return cudaSuccess;
}
}  // namespace tdc

extern "C" tdcfie_status tdcfie_block_gemv_noalloc(int precision, const void* blocks, int64_t nblk, int64_t n,
                                                   const void* x, int64_t R, void* out, void* stream) {
    tdcfie_status st = check_gemv(precision, blocks, nblk, n, x, R, out);
    if (st != TDCFIE_OK) return st;
    const size_t es = precision == TDCFIE_FP64 ? 8 : 4;
    const double need = (double)es * (double)nblk * (double)R * (double)n;
    if (need > (double)NOALLOC_SCRATCH_BYTES)
        return fail(nullptr, TDCFIE_E_ARG,
                    "tdcfie_block_gemv_noalloc: nblk * R * n * element size exceeds the 32 MiB static scratch "
                    "(at most 4194304 FP64 or 8388608 FP32 partial sums); use tdcfie_block_gemv");
    void* partial = nullptr;
    cudaError_t e = scratch_address(&partial);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaGetSymbolAddress (static block GEMV scratch)");
    cudaStream_t s = (cudaStream_t)stream;
    if (precision == TDCFIE_FP64)
        e = launch_block_gemv<double>((const double*)blocks, nblk, n, (const double*)x, (int)R, (double*)out,
                                      (double*)partial, s);
    else
        e = launch_block_gemv<float>((const float*)blocks, nblk, n, (const float*)x, (int)R, (float*)out,
                                     (float*)partial, s);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "block GEMV launch");
    return TDCFIE_OK;
}
