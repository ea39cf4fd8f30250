// Restarted GMRES on T_0 for the per-step solve T_0 y_n = b_n (Sec. IV-B), mixed precision:
//   restart: true residual r = b - T_0 x with T_0 in FP64 (the assembled block), convergence when
//            ||r|| <= tol ||b||;
//   cycle:   Arnoldi with the path-precision T_0 (FP32 or FP64 matvec), classical Gram-Schmidt
//            applied twice (CGS2) in FP64, Givens rotations, up to m iterations or until the
//            residual estimate drops below max(inner_tol beta, tol ||b|| / 2); then x += V_m y.
// One cooperative kernel per step solves all right-hand sides, each by a group of co-resident blocks
// of its own (grid.y) that hold the rows in equal shares.  A group meets at three barriers per Arnoldi
// iteration (projections, their repetition, norm) and two per restart; between barriers a block only
// touches its rows, and what the group sums passes through one partial per block, added by every
// block in the same order: the Hessenberg column, the rotations and every decision are formed by all
// blocks alike, and the results do not depend on timing.  Latency bounds it; 100 steps at 768 unknowns,
// FP32, took 45.6 ms with an iteration as seven kernels in a graph loop, 22.8 ms so.
#include <cmath>

#include "gmres.h"
#include "plan.h"
#include "simt.h"

namespace tdc {

// stats: [0] Arnoldi iterations this march, [1] steps, [2] max per step, [3] this step,
//        [4] solves not converged, [5] groups done this step
enum { NSTATS = 8 };
constexpr int GM_T = 512, GM_W = GM_T / 32;       // threads and warps per block
// Rows per block, or more where the chip is full.  us per step at 4, 8, 16, 32: 120 unknowns FP64 204, 216,
// 229, 274; 480 FP32 196, 197, 203, 244; 768 FP32 226, 235, 253, 287; from 1920 on the chip is full.  Fewer rows
// are more partial sums to add per block, more rows a longer product; 4 and 8 are within 6 %.
constexpr int GM_ROWS = 8;
constexpr int GM_TILE = 8192;                     // entries of a vector staged at a time

struct GmDev {
    int R, ne, ld, m, maxit;
    int G, rpb, wpr;       // blocks per right-hand side, rows per block, warps per row of a product
    int tile;              // doubles of the staging buffer
    double tol, inner_tol;
    double *x, *r, *V, *w, *H, *part;      // part: per right-hand side (2 (m + 1) + 2) x G
    unsigned long long* sync;              // per right-hand side: arrivals so far; behind them: a wait ran out
    unsigned long long* stats;
};

__device__ __forceinline__ double warp_sum(double s) {
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// a . x over n entries by one warp; x in shared memory.  16-byte loads where the rows allow them
template <typename T>
__device__ __forceinline__ T dot(const T* __restrict__ a, const T* x, int n, bool vec) {
    const int lane = threadIdx.x & 31;
    T s = 0;
    if (vec) {
        if constexpr (sizeof(T) == 4) {
#pragma unroll 6
            for (int c = 4 * lane; c < n; c += 128) {
                const float4 u = *reinterpret_cast<const float4*>(a + c), v = *reinterpret_cast<const float4*>(x + c);
                s += u.x * v.x; s += u.y * v.y; s += u.z * v.z; s += u.w * v.w;
            }
        } else {
#pragma unroll 6
            for (int c = 2 * lane; c < n; c += 64) {
                const double2 u = *reinterpret_cast<const double2*>(a + c), v = *reinterpret_cast<const double2*>(x + c);
                s += u.x * v.x; s += u.y * v.y;
            }
        }
    } else {
#pragma unroll 8
        for (int c = lane; c < n; c += 32) s += a[c] * x[c];
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// out[i] = A (sc src) over the block's rows; the vector is staged in shared memory (xs) in tiles, a row
// is shared by d.wpr warps (psum: their parts).  Ends with a barrier of the block.
template <typename T>
__device__ __forceinline__ void block_product(const GmDev& d, const T* __restrict__ A, const double* src, double sc,
                                              int row0, int nloc, double* xs_, double* psum, double* out) {
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    constexpr int Q = 16 / (int)sizeof(T);      // entries of a 16-byte load
    T* xs = reinterpret_cast<T*>(xs_);
    const bool vec = d.ne % Q == 0;
    for (int c0 = 0; c0 < d.ne; c0 += GM_TILE) {
        const int nc = min(GM_TILE, d.ne - c0);
        if (c0) __syncthreads();
        for (int c = t; c < nc; c += GM_T) xs[c] = (T)(__ldcg(src + c0 + c) * sc);
        __syncthreads();
        const int per = (nc + d.wpr * Q - 1) / (d.wpr * Q) * Q;      // columns per warp
        for (int u = warp; u < nloc * d.wpr; u += GM_W) {
            const int row = u / d.wpr, c1 = u % d.wpr * per, n = min(per, nc - c1);
            const T v = n > 0 ? dot<T>(A + (int64_t)(row0 + row) * d.ne + c0 + c1, xs + c1, n, vec) : (T)0;
            if (lane == 0) psum[u] = c0 ? psum[u] + (double)v : (double)v;
        }
    }
    __syncthreads();
    for (int i = t; i < nloc; i += GM_T) {
        double s = psum[i * d.wpr];
        for (int k = 1; k < d.wpr; ++k) s += psum[i * d.wpr + k];
        out[i] = s;
    }
    __syncthreads();
}

// part[k][block] = V_k . w over the block's rows, k < cnt (w in shared memory)
__device__ __forceinline__ void block_dots(const GmDev& d, const double* V, int cnt, int nloc, const double* w, double* part) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = warp; k < cnt; k += GM_W) {
        const double* v = V + (int64_t)k * d.R * d.ne;
        double s = 0.0;
        for (int i = lane; i < nloc; i += 32) s += v[i] * w[i];
        s = warp_sum(s);
        if (lane == 0) __stcg(part + k * d.G + blockIdx.x, s);
    }
}
// part[block] = |v|^2 over the block's rows (first warp)
__device__ __forceinline__ void block_norm(const double* v, int nloc, double* part) {
    if (threadIdx.x >= 32) return;
    double s = 0.0;
    for (int i = threadIdx.x; i < nloc; i += 32) s += v[i] * v[i];
    s = warp_sum(s);
    if (threadIdx.x == 0) __stcg(part + blockIdx.x, s);
}
// out[k] = the sum of part[k][.], k < cnt.  Ends with a barrier of the block.
__device__ __forceinline__ void group_sums(const GmDev& d, const double* part, int cnt, double* out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = warp; k < cnt; k += GM_W) {
        double s = 0.0;
        for (int q = lane; q < d.G; q += 32) s += __ldcg(part + k * d.G + q);
        s = warp_sum(s);
        if (lane == 0) out[k] = s;
    }
    __syncthreads();
}
// w[i] += sign sum_k c[k] V_k over the block's rows: one warp per row, lanes along the vectors
__device__ __forceinline__ void add_vectors(const GmDev& d, const double* V, int cnt, int nloc, const double* c, double sign,
                                            double* w) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = warp; i < nloc; i += GM_W) {
        double s = 0.0;
        for (int k = lane; k < cnt; k += 32) s += c[k] * V[(int64_t)k * d.R * d.ne + i];
        s = warp_sum(s);
        if (lane == 0) w[i] += sign * s;
    }
    __syncthreads();
}

// One step's solves; the solution goes to ring slot (ctl->n + off) % ring.  mode: the initial guess, 0
// zero, 1 y_{n-1}, 2 and 4 the learned guess buffer, 3 cubic extrapolation of y_{n-1..n-4} (y_i = 0
// for i <= 0).  The first step with a solve left above the tolerance is recorded in the step state
// (returned as TDCFIE_E_NOCONV).
template <typename T>
__global__ void __launch_bounds__(GM_T, 1) k_gm_solve(const __grid_constant__ GmDev d, const double* __restrict__ T0,
                                                   const T* __restrict__ T0p, const T* __restrict__ b, int mode,
                                                   T* __restrict__ ringbuf, int ring, const T* __restrict__ learned, int off,
                                                   Ctl* ctl) {
    extern __shared__ __align__(16) double sm[];
    __shared__ double sc[4];      // ||r||^2 (or ||w||^2), ||b||^2, h_{j+1,j}
    __shared__ int failed, stop;
    const int t = threadIdx.x, lane = t & 31, r = blockIdx.y, m = d.m;
    const int row0 = blockIdx.x * d.rpb, nloc = min(d.rpb, d.ne - row0);
    double* xs = sm;
    double* cs = xs + d.tile;
    double* sn = cs + m;
    double* g = sn + m;
    double* hc = g + m + 1;      // the current column of H
    double* h1 = hc + m + 1;
    double* wl = h1 + m + 1;     // the block's part of a vector
    double* xl = wl + d.rpb;
    double* psum = xl + d.rpb;
    if (t == 0) failed = (int)__ldcg(d.sync + d.R);      // an earlier solve's wait ran out
    if (t == 0 && blockIdx.x == 0 && r == 0) ctl->hist_ns += device_ns() - ctl->t_mark;      // the history kernel is done
    __syncthreads();
    if (failed) {
        ctl->timeout = 1;
        return;
    }
    const int64_t n = ctl->n + off;
    const int64_t vec0 = (int64_t)r * d.ne;
    double* x = d.x + vec0;
    double* V = d.V + vec0 + row0;      // the block's rows of V_0
    double* H = d.H + (int64_t)r * (m + 1) * m;
    double* p0 = d.part + (int64_t)r * (2 * (m + 1) + 2) * d.G;
    double* p1 = p0 + (m + 1) * d.G;
    double* p2 = p1 + (m + 1) * d.G;
    const T* br = b + (int64_t)r * d.ld + row0;
#define MEET() if (!group_barrier(d.sync + r, d.G, d.sync + d.R, &failed)) { ctl->timeout = 1; return; }

    for (int i = t; i < nloc; i += GM_T) {
        const int64_t e = (int64_t)r * d.ld + row0 + i;
        double x0 = 0.0;
        if (mode == 1 && n > 1) x0 = (double)ringbuf[((n - 1) % ring) * (int64_t)d.R * d.ld + e];
        if ((mode == 2 || mode == 4) && n > 1) x0 = (double)learned[e];
        if (mode == 3) {
            const double c[4] = {4.0, -6.0, 4.0, -1.0};
            for (int k = 1; k <= 4 && k <= ring; ++k)
                if (n - k >= 1) x0 += c[k - 1] * (double)ringbuf[((n - k) % ring) * (int64_t)d.R * d.ld + e];
        }
        __stcg(x + row0 + i, x0);
        xl[i] = x0;
        wl[i] = (double)br[i];
    }
    __syncthreads();
    block_norm(wl, nloc, p2 + d.G);
    MEET();
    group_sums(d, p2 + d.G, 1, sc + 1);
    const double bn = sqrt(sc[1]);
    int iters = 0;
    bool conv = false;
    for (;;) {
        // restart: converged, out of iterations, or open a cycle with beta = ||r||
        block_product<double>(d, T0, x, 1.0, row0, nloc, xs, psum, wl);
        for (int i = t; i < nloc; i += GM_T) {
            wl[i] = (double)br[i] - wl[i];
            __stcg(d.r + vec0 + row0 + i, wl[i]);
        }
        __syncthreads();
        block_norm(wl, nloc, p2);
        MEET();
        group_sums(d, p2, 1, sc);
        const double beta = sqrt(sc[0]);
        conv = beta <= d.tol * bn || beta == 0.0;
        if (conv || iters >= d.maxit) break;
        if (t == 0) g[0] = beta;
        const double* src = d.r + vec0;
        double scale = 1.0 / beta;
        int j = 0;
        for (bool last = false; !last; ++j) {
            // w = T0p V_j, V_j = scale * src taken on the fly; the rows of V_j kept; first projections
            for (int i = t; i < nloc; i += GM_T) V[(int64_t)j * d.R * d.ne + i] = __ldcg(src + row0 + i) * scale;
            block_product<T>(d, T0p, src, scale, row0, nloc, xs, psum, wl);
            block_dots(d, V, j + 1, nloc, wl, p0);
            MEET();
            group_sums(d, p0, j + 1, hc);
            add_vectors(d, V, j + 1, nloc, hc, -1.0, wl);
            block_dots(d, V, j + 1, nloc, wl, p1);
            MEET();
            group_sums(d, p1, j + 1, h1);
            add_vectors(d, V, j + 1, nloc, h1, -1.0, wl);
            for (int i = t; i < nloc; i += GM_T) __stcg(d.w + vec0 + row0 + i, wl[i]);
            block_norm(wl, nloc, p2 + d.G);
            MEET();
            group_sums(d, p2 + d.G, 1, sc);
            ++iters;
            if (t == 0) {      // Givens rotations, residual estimate
                const double hn = sqrt(sc[0]);
                double a = hc[0] + h1[0];
                for (int k = 0; k < j; ++k) {
                    const double q = hc[k + 1] + h1[k + 1];
                    hc[k] = cs[k] * a + sn[k] * q;
                    a = -sn[k] * a + cs[k] * q;
                }
                const double rr = sqrt(a * a + hn * hn);
                const double c = rr > 0.0 ? a / rr : 1.0, s = rr > 0.0 ? hn / rr : 0.0;
                cs[j] = c;
                sn[j] = s;
                hc[j] = rr;
                g[j + 1] = -s * g[j];
                g[j] = c * g[j];
                // a cycle gains inner_tol, but never solves past half the outer target (the true FP64
                // residual decides at the restart whether another cycle runs)
                const double goal = fmax(d.inner_tol * beta, 0.5 * d.tol * bn);
                stop = fabs(g[j + 1]) <= goal || j + 1 == m || hn == 0.0 || iters >= d.maxit;
                sc[2] = 1.0 / hn;
            }
            __syncthreads();
            last = stop != 0;
            if (blockIdx.x == 0)
                for (int k = t; k <= j; k += GM_T) __stcg(H + (int64_t)k * m + j, hc[k]);
            src = d.w + vec0;
            scale = sc[2];
        }
        // H y = g: the columns before the last were written ahead of a barrier, the last is in hc
        for (int e = t; e < j * j; e += GM_T) {
            const int i = e / j, k = e % j;
            xs[e] = k < i ? 0.0 : k == j - 1 ? hc[i] : __ldcg(H + (int64_t)i * m + k);
        }
        __syncthreads();
        if (t < 32) {      // by columns, two right-hand sides per lane (j <= 60); y replaces g
            double u0 = lane < j ? g[lane] : 0.0, u1 = lane + 32 < j ? g[lane + 32] : 0.0;
            for (int i = j - 1; i >= 0; --i) {
                const double y = __shfl_sync(0xffffffffu, i < 32 ? u0 : u1, i & 31) / xs[i * j + i];
                if (lane < i) u0 -= xs[lane * j + i] * y;
                if (lane + 32 < i) u1 -= xs[(lane + 32) * j + i] * y;
                if (lane == 0) g[i] = y;
            }
        }
        __syncthreads();
        add_vectors(d, V, j, nloc, g, 1.0, xl);
        for (int i = t; i < nloc; i += GM_T) __stcg(x + row0 + i, xl[i]);
        MEET();
    }
#undef MEET
    for (int i = t; i < nloc; i += GM_T) ringbuf[(n % ring) * (int64_t)d.R * d.ld + (int64_t)r * d.ld + row0 + i] = (T)xl[i];
    if (t == 0 && blockIdx.x == 0) {
        atomicAdd(d.stats + 0, (unsigned long long)iters);
        atomicAdd(d.stats + 3, (unsigned long long)iters);
        if (!conv) {
            atomicAdd(d.stats + 4, 1ULL);
            if (atomicCAS(&ctl->noconv, 0, 1) == 0) ctl->noconv_step = n;
        }
        __threadfence();
        if (atomicAdd(d.stats + 5, 1ULL) == (unsigned long long)(d.R - 1)) {      // the step's last group
            __threadfence();
            atomicAdd(d.stats + 1, 1ULL);
            atomicMax(d.stats + 2, atomicExch(d.stats + 3, 0ULL));
            atomicExch(d.stats + 5, 0ULL);
        }
    }
}

// ---------------------------------------------------------------- host side
struct GmresPlan {
    GmDev d{};
    size_t smem = 0;
    std::vector<void*> owned;
    ~GmresPlan() {
        for (void* p : owned) cudaFree(p);
    }
};

void destroy_gmres(GmresPlan* g) { delete g; }

// The split of the rows.  GM_ROWS per block (two warps per row) until every SM has a block; then all
// SMs, more rows each.
template <typename T>
static cudaError_t split_rows(GmresPlan* g) {
    GmDev& d = g->d;
    int dev = 0, sms = 0, occ = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return e;
    auto shape = [&](int slots) {
        const int per = std::max(1, slots / d.R);
        d.rpb = std::max(GM_ROWS, (d.ne + per - 1) / per);
        d.G = (d.ne + d.rpb - 1) / d.rpb;
        d.wpr = d.rpb <= GM_W / 2 ? 2 : 1;
        // the staged vector, or a cycle's triangle
        d.tile = std::max(std::min(d.ne, GM_TILE), std::min(d.m, d.maxit) * std::min(d.m, d.maxit));
        d.tile += d.tile & 1;
        g->smem = sizeof(double) * (d.tile + 5 * d.m + 3 + (size_t)d.rpb * (2 + d.wpr));
    };
    shape(sms);
    if ((e = cudaFuncSetAttribute(k_gm_solve<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g->smem))) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_gm_solve<T>, GM_T, g->smem))) return e;
    return (int64_t)d.G * d.R <= (int64_t)occ * sms ? cudaSuccess : cudaErrorCooperativeLaunchTooLarge;
}

cudaError_t build_gmres(tdcfie_t h, StepPlan* p) {
    auto* g = new GmresPlan();
    p->gm = g;
    const int R = p->R, ne = p->ne;
    const int m = std::max(2, std::min(60, h->opts.gmres_restart));
    GmDev& d = g->d;
    d.R = R; d.ne = ne; d.ld = p->ld; d.m = m;
    d.tol = h->opts.gmres_tol;
    d.inner_tol = 1e-4;   // each cycle gains four digits; the restarts refine against the FP64 residual
    d.maxit = std::max(1, h->opts.gmres_maxit);
    cudaError_t e = p->prec == TDCFIE_FP64 ? split_rows<double>(g) : split_rows<float>(g);
    if (e != cudaSuccess) return e;
    auto al = [&](double** q, size_t n) -> cudaError_t {
        cudaError_t e = cudaMalloc((void**)q, sizeof(double) * (n ? n : 1));
        if (e == cudaSuccess) { g->owned.push_back(*q); e = cudaMemsetAsync(*q, 0, sizeof(double) * (n ? n : 1), h->stream); }
        return e;
    };
    if ((e = al(&d.x, (size_t)R * ne)) || (e = al(&d.r, (size_t)R * ne)) || (e = al(&d.V, (size_t)(m + 1) * R * ne)) ||
        (e = al(&d.w, (size_t)R * ne)) || (e = al(&d.H, (size_t)R * (m + 1) * m)) ||
        (e = al(&d.part, (size_t)R * (2 * (m + 1) + 2) * d.G)))
        return e;
    // the barriers' counters and the statistics in one piece
    if ((e = cudaMalloc(&d.sync, sizeof(unsigned long long) * (R + 1 + NSTATS))) != cudaSuccess) return e;
    g->owned.push_back(d.sync);
    d.stats = d.sync + R + 1;
    return reset_gmres_stats(g, h->stream);
}

void gmres_set_tol(GmresPlan* g, double tol) { g->d.tol = tol; }

// on the handle's stream, ahead of its next solve: the counters must stand while a solve runs
cudaError_t reset_gmres_stats(GmresPlan* g, cudaStream_t s) {
    return cudaMemsetAsync(g->d.sync, 0, sizeof(unsigned long long) * (g->d.R + 1 + NSTATS), s);
}

cudaError_t gmres_stats(GmresPlan* g, long long* out5) {
    unsigned long long st[NSTATS];
    const cudaError_t e = cudaMemcpy(st, g->d.stats, sizeof(st), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return e;
    for (int i = 0; i < 5; ++i) out5[i] = (long long)st[i];
    return cudaSuccess;
}

// Enqueue the solve of step ctl->n + off on s
template <typename T>
cudaError_t launch_gmres(tdcfie_t h, StepPlan* p, const T* b, const T* learned, const T* T0p, T* ringbuf, int off,
                         cudaStream_t s) {
    GmresPlan* g = p->gm;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g->d.G, g->d.R);
    cfg.blockDim = dim3(GM_T);
    cfg.dynamicSmemBytes = g->smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_gm_solve<T>, g->d, (const double*)h->T, T0p, b, h->opts.guess, ringbuf, p->ring, learned,
                              off, p->ctl);
}

template cudaError_t launch_gmres<double>(tdcfie_t, StepPlan*, const double*, const double*, const double*, double*, int,
                                          cudaStream_t);
template cudaError_t launch_gmres<float>(tdcfie_t, StepPlan*, const float*, const float*, const float*, float*, int,
                                         cudaStream_t);

}  // namespace tdc
