// Hot path of the marching-on-in-time solver (Sec. IV-B), CUDA graphs over chunks of steps.
//
// Per step n (t_n = n dt), with y_i = 0 for i <= 0:
//   rhs:      e_m(t_n) = int f_m . e_in(t_n),  h_m(t_n) = int g_m . h_in(t_n)         (Sec. II-C)
//   history:  b_n = -A e_n + alpha L2 h_n - sum_{k=1}^{K-1} T_k y_{n-k}                 (Sec. IV-B)
//             A = L1 (dtt P^LH + P^S) folds the rescaling of e (Sec. III-A) into L1
//   solve:    y_n = T_0^-1 b_n
//   project:  z = Sigma^T w_n, w_n = (1/dtt - 1) y_n - y_{n-1}/dtt;  u = (Sigma^T Sigma)^+ z
//   post:     j_n = y_n + Sigma u = P^LH y_n + P^S (y_n - y_{n-1})/dtt                (Eq. post_processing)
// How the steps of a chunk share the passes over the matrices: simt.h.
// Layouts (HBM): matrices row-major; vectors right-hand-side-major (R x ld per slot).  The ring holds
// the last K - 1 + C y, slot = i mod (K - 1 + C): the K - 1 that the history reads and those of the
// chunk, which the post-processing reads at its end.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>

#include "internal.h"
#include "gmres.h"
#include "simt.h"
#include "plan.h"
#include "umma.h"

namespace tdc {

// ---------------------------------------------------------------- kernels (arithmetic in simt.h)
// The tests and pre-sums of a chunk: no work where new_cols gives no columns
template <typename T>
__global__ void __launch_bounds__(128) k_env(const __grid_constant__ SimtDev<T> d, int most) {
    wait_prior();
    const int64_t n = d.ctl->n;
    const int col = d.ctl->col;
    const Cols cs = new_cols(d.ctl, d.C, n, col, most);
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int nc = cs.hi - cs.lo;
    if (idx >= (int64_t)d.npts * d.R * nc) return;
    const int i = cs.lo + (int)(idx % nc), r = (int)(idx / nc % d.R), pt = (int)(idx / nc / d.R);
    d.env[((int64_t)pt * d.R + r) * d.C + i] = env_point<T>(d.exc + 11 * r, n - col + i, d.dt, d.pts[3 * pt], d.pts[3 * pt + 1], d.pts[3 * pt + 2]);
}

template <typename T>
__global__ void __launch_bounds__(128) k_gather(const __grid_constant__ SimtDev<T> d, int most) {
    wait_prior();
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const Cols cs = new_cols(d.ctl, d.C, d.ctl->n, d.ctl->col, most);
    if (w >= d.ne * d.R || cs.lo == cs.hi) return;
    gather_edge<T>(d, cs, w / d.R, w % d.R, threadIdx.x & 31);
}

// grid: (column tiles x row blocks, groups), the column tiles fastest so that blocks that share rows
// run together
template <typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 4 : 3) k_pre(const __grid_constant__ SimtDev<T> d, int ctiles, int most) {
    wait_prior();
    const int col = d.ctl->col;
    const Cols cs = new_cols(d.ctl, d.C, d.ctl->n, col, most);
    if (cs.lo == cs.hi) return;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) d.ctl->t_mark = device_ns();
    const int tile = blockIdx.x % ctiles, rb = blockIdx.x / ctiles;
    const int row0 = (rb * 4 + (threadIdx.x >> 5)) * pre_rows<T>();
    if (row0 < d.ne) pre_item<T>(d, cs, ring_at(d.ctl->slot, -col, d.ring), row0, blockIdx.y, tile, threadIdx.x & 31);
}

// b_n; step n = ctl->n + off.  sums_ready: the pre-sums are older than the kernel in front
template <typename T, int RM>
__global__ void __launch_bounds__(128, 4) k_hist(const __grid_constant__ SimtDev<T> d, int off, bool sums_ready) {
    const StepPos pos = step_pos(d, off);
    auto wait = [&] {
        wait_prior();
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            const unsigned long long t = device_ns();
            if (pos.col == 0) d.ctl->hist_ns += t - d.ctl->t_mark;     // the chunk's pre-sums ran just before
            d.ctl->t_mark = t;
        }
    };
    hist_unit<T, RM>(d, pos, (blockIdx.x * blockDim.x + threadIdx.x) >> 5, threadIdx.x & 31, sums_ready, wait);
}

template <typename T, int RM>
__global__ void __launch_bounds__(128) k_solve(const __grid_constant__ SimtDev<T> d, int off) {
    const StepPos pos = step_pos(d, off);
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    auto wait = [&] {
        wait_prior();
        if (blockIdx.x == 0 && threadIdx.x == 0) d.ctl->hist_ns += device_ns() - d.ctl->t_mark;
    };
    if (row < d.ne) solve_unit<T, RM>(d, pos, row, threadIdx.x & 31, wait);
}

// Post-processing of the steps p0 .. ctl->n + adv - 1 (at most C); the last kernel advances the step
// counter by adv
template <typename T>
__device__ __forceinline__ bool post_step(const SimtDev<T>& d, int adv, int col, int64_t& n, int& slot) {
    const Ctl* c = d.ctl;
    n = c->p0 + col / d.R;
    slot = ring_at(c->slot, (int)(n - c->n), d.ring);
    return n < c->n + adv && col < d.C * d.R;
}
template <typename T>
__global__ void __launch_bounds__(256) k_pin(const __grid_constant__ SimtDev<T> d, int adv) {
    wait_prior();
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = idx % d.nc, col = idx / d.nc;
    int64_t n;
    int slot;
    if (post_step(d, adv, col, n, slot)) pin_value<T>(d, n, slot, col, col % d.R, c);
}

template <typename T>
__global__ void __launch_bounds__(128) k_pinv(const __grid_constant__ SimtDev<T> d, int adv, int ctiles) {
    wait_prior();
    const int ncol = min((int)(d.ctl->n + adv - d.ctl->p0), d.C) * d.R;
    const int col0 = blockIdx.x % ctiles * PRE_COLS, row0 = (blockIdx.x / ctiles * 4 + (threadIdx.x >> 5)) * pre_rows<T>();
    if (col0 < ncol && row0 < d.nc) pinv_item<T>(d, ncol, row0, col0, threadIdx.x & 31);
}

template <typename T>
__global__ void __launch_bounds__(256) k_pout(const __grid_constant__ SimtDev<T> d, int adv) {
    wait_prior();
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const int e = idx % d.ne, col = idx / d.ne;
    int64_t n;
    int slot;
    if (post_step(d, adv, col, n, slot)) pout_value<T>(d, n, slot, col, col % d.R, e);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(d.done, 1) == (int)gridDim.x - 1) {     // every block has read n and p0
            *d.done = 0;
            advance(d, adv);
            d.ctl->p0 = d.ctl->n;
            __threadfence();
        }
    }
}

template <typename T>
__global__ void k_advance(const __grid_constant__ SimtDev<T> d) {
    wait_prior();
    advance(d, 1);
}

// ---------------------------------------------------------------- launches
static size_t esize(int prec) { return prec == TDCFIE_FP64 ? 8 : 4; }

template <typename T>
SimtDev<T> simt_view(tdcfie_t h, const StepPlan& p) {
    SimtDev<T> d;
    d.ne = p.ne; d.nc = p.nc; d.R = p.R; d.C = p.C; d.K = p.K; d.ring = p.ring; d.ld = p.ld; d.ldc = p.ldc;
    d.ngroups = p.ngroups; d.npts = p.npts;
    d.blocks = (const T*)p.blocks; d.t0inv = (const T*)p.t0inv; d.pinv = (const T*)p.pinv;
    d.E = (T*)p.E; d.H = (T*)p.Hv; d.rbuf = (T*)p.ringbuf; d.b = (T*)p.b; d.z = (T*)p.z; d.u = (T*)p.u;
    using S = typename SumOf<T>::S;
    d.partial = (S*)p.partial; d.inner = (S*)p.inner; d.env = (T*)p.env; d.pts = (const T*)p.pts;
    d.eptr = p.eptr; d.enE = p.enE; d.eidx = p.eidx; d.ecoef = (const T*)p.ecoef;
    d.exc = h->dexc; d.m = h->dm; d.dt = h->dt; d.dtt = h->dtt; d.ctl = p.ctl; d.done = p.done;
    return d;
}
template SimtDev<float> simt_view<float>(tdcfie_t, const StepPlan&);

static unsigned div_up(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }

template <typename T>
int launch_tests(tdcfie_t h, StepPlan& p, int most, cudaStream_t s) {
    const SimtDev<T> d = simt_view<T>(h, p);
    k_env<T><<<div_up((int64_t)p.npts * p.R * p.C, 128), 128, 0, s>>>(d, most);
    launch_chained(k_gather<T>, div_up((int64_t)p.ne * p.R, 4), 128, s, 0, d, most);
    return 2;
}
template int launch_tests<double>(tdcfie_t, StepPlan&, int, cudaStream_t);
template int launch_tests<float>(tdcfie_t, StepPlan&, int, cudaStream_t);

template <typename T>
static int launch_pre(tdcfie_t h, StepPlan& p, int most, cudaStream_t s) {
    int n = launch_tests<T>(h, p, most, s);
    if (p.fact) return n;
    const int ctiles = (int)div_up(p.C * p.R, PRE_COLS);
    launch_chained(k_pre<T>, dim3(ctiles * div_up(p.ne, 4 * pre_rows<T>()), p.ngroups), 128, s, 0, simt_view<T>(h, p), ctiles, most);
    return n + 1;
}

// history and solve of step ctl->n + off (chunk: of a whole chunk that starts at ctl->n)
template <typename T>
static cudaError_t launch_inner(tdcfie_t h, StepPlan& p, bool chunk, int off, cudaStream_t s, int& kernels) {
    if (p.fact) {
        kernels += launch_step_fact<T>(h, p, s);
        return cudaGetLastError();
    }
    const SimtDev<T> d = simt_view<T>(h, p);
    const int units = (int)div_up(p.ne, p.R <= 2 ? 2 : 1);
    // units of the history: the step's rows, and the rows of every lag that can be pushed (chunk: the
    // step's column is known)
    const int lags = 1 + std::max(0, std::min(chunk ? p.C - off : p.C - 1, p.K - 1) - 1) * (chunk && off == 0 ? 0 : 1);
    unsigned g = div_up((int64_t)units * lags, 4);
#define BY_R(K, ...) launch_chained(p.R == 1 ? K<T, 1> : p.R == 2 ? K<T, 2> : p.R <= 4 ? K<T, 4> : K<T, 8>, g, 128, s, 0, __VA_ARGS__)
    BY_R(k_hist, d, off, chunk && off > 0);
    kernels += 1;
    g = div_up(p.ne, 4);
    if (p.mlp_on) kernels += launch_mlp_guess<T>(&p, off, s);
    if (p.gmres_on) {
        const cudaError_t e = launch_gmres<T>(h, &p, (const T*)p.b, (const T*)p.guessbuf, (const T*)p.t0mat,
                                              (T*)p.ringbuf, off, s);
        if (e != cudaSuccess) return e;
        kernels += 1;
    } else {
        BY_R(k_solve, d, off);
        kernels += 1;
    }
#undef BY_R
    return cudaGetLastError();
}

template <typename T>
static int launch_post(tdcfie_t h, StepPlan& p, int adv, cudaStream_t s) {
    if (p.fact) return 0;      // part of the step
    const SimtDev<T> d = simt_view<T>(h, p);
    const int CR = p.C * p.R, ctiles = (int)div_up(CR, PRE_COLS);
    launch_chained(k_pin<T>, div_up((int64_t)p.nc * CR, 256), 256, s, 0, d, adv);
    launch_chained(k_pinv<T>, ctiles * div_up(p.nc, 4 * pre_rows<T>()), 128, s, 0, d, adv, ctiles);
    launch_chained(k_pout<T>, div_up((int64_t)p.ne * CR, 256), 256, s, 0, d, adv);
    return 3;
}

// enqueue the kernels of one of the plan's graphs (s must be capturing)
template <typename T>
static cudaError_t launch_graph(tdcfie_t h, StepPlan& p, int which, cudaStream_t s, int& k) {
    cudaError_t e = cudaSuccess;
    const bool chunk = which == StepPlan::G_CHUNK;
    if (which == StepPlan::G_PRE || chunk) k += launch_pre<T>(h, p, chunk ? p.C : 0, s);
    if (which == StepPlan::G_STEP || which == StepPlan::G_LAST) e = launch_inner<T>(h, p, false, 0, s, k);
    if (which == StepPlan::G_STEP && !p.fact) {      // the factored step advances the counter itself
        launch_chained(k_advance<T>, 1, 1, s, 0, simt_view<T>(h, p));
        k += 1;
    }
    if (chunk)
        for (int i = 0; i < p.C && e == cudaSuccess; ++i) e = launch_inner<T>(h, p, true, p.fact ? 0 : i, s, k);
    if (which == StepPlan::G_LAST || chunk) k += launch_post<T>(h, p, chunk ? p.C : 1, s);
    return e == cudaSuccess ? cudaGetLastError() : e;
}
static cudaError_t launch_graph_tc(tdcfie_t h, StepPlan& p, int which, cudaStream_t s, int& k) {
    const bool chunk = which == StepPlan::G_CHUNK, last = which >= StepPlan::G_LAST;
    if (which == StepPlan::G_PRE || chunk) k += launch_tests_tc(h, &p, chunk ? p.C : 0, s);
    if (which == StepPlan::G_STEP || last) k += launch_inner_tc(h, &p, 0, which == StepPlan::G_STEP, s);
    if (chunk)
        for (int i = 0; i < p.C; ++i) k += launch_inner_tc(h, &p, i, false, s);
    if (chunk) k += launch_post_tc(h, &p, p.C, p.C, s);
    if (last) k += launch_post_tc(h, &p, 1, which - StepPlan::G_LAST + 1, s);
    return cudaGetLastError();
}

tdcfie_status plan_gmres_stats(tdcfie_t h, long long* out5) {
    StepPlan* p = h->plan;
    if (!p || !p->gm) return fail(h, TDCFIE_E_STATE, "GMRES solver not active on this handle");
    const cudaError_t e = gmres_stats(p->gm, out5);
    if (e != cudaSuccess) return cuda_fail(h, e, "gmres_stats");
    return TDCFIE_OK;
}

static void drop_graphs(StepPlan* p) {
    for (int g = 0; g < StepPlan::NGRAPH; ++g) {
        if (p->exec[g]) { cudaGraphExecDestroy(p->exec[g]); p->exec[g] = nullptr; }
        if (p->graph[g]) { cudaGraphDestroy(p->graph[g]); p->graph[g] = nullptr; }
    }
}

void free_plan(tdcfie_t h) {
    StepPlan* p = h->plan;
    if (!p) return;
    void* bufs[] = {p->blocks, p->t0inv, p->pinv, p->E, p->Hv, p->ringbuf, p->b, p->partial, p->inner, p->z, p->u, p->done,
                    p->ctl, p->env, p->pts, p->ecoef, p->eptr, p->enE, p->eidx};
    for (void* b : bufs) if (b) cudaFree(b);
    drop_graphs(p);
    if (p->ev0) cudaEventDestroy(p->ev0);
    if (p->ev1) cudaEventDestroy(p->ev1);
    if (p->gemm) destroy_tc(p->gemm);
    if (p->gm) destroy_gmres(p->gm);
    if (p->mlp) destroy_mlp(p->mlp);
    if (p->fact) destroy_fact(p->fact);
    if (p->t0mat) cudaFree(p->t0mat);
    if (p->guessbuf) cudaFree(p->guessbuf);
    delete p;
    h->plan = nullptr;
}

#define CK(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) return cuda_fail(h, e_, #x); } while (0)

// dst[i][j] = scale src[i][j] in the path precision, rows padded with zeros from cols to ld
template <typename T>
__global__ void k_to_path(const double* __restrict__ src, T* __restrict__ dst, int64_t rows, int cols, int ld, double scale) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= rows * ld) return;
    const int64_t i = t / ld;
    const int j = (int)(t - i * ld);
    dst[t] = j < cols ? (T)(scale * src[i * cols + j]) : (T)0;
}
void to_path(cudaStream_t s, int prec, const double* src, void* dst, int64_t rows, int cols, int ld, double scale) {
    const unsigned g = div_up(rows * ld, 256);
    if (prec == TDCFIE_FP64) k_to_path<double><<<g, 256, 0, s>>>(src, (double*)dst, rows, cols, ld, scale);
    else k_to_path<float><<<g, 256, 0, s>>>(src, (float*)dst, rows, cols, ld, scale);
}

tdcfie_status build_plan(tdcfie_t h) {
    free_plan(h);
    StepPlan* p = new StepPlan();
    h->plan = p;
    cudaStream_t s = h->stream;
    const tdc::Mesh& M = h->mesh;
    p->prec = h->opts.precision;
    p->R = (int)h->R;
    p->ne = M.ne; p->nc = M.nc; p->K = h->K;
    p->nblk = h->K + 1;              // -A, alpha L2, -T_1..-T_{K-1}
    p->esz = esize(p->prec);
    const int64_t ne = M.ne, nc = M.nc, R = p->R;
    const bool tensor = p->prec == TDCFIE_BF16X3 || p->prec == TDCFIE_FP16X3;
    if (h->formulation != TDCFIE_FORMULATION_QHP_CFIE && (tensor || h->history_form != TDCFIE_HISTORY_DENSE))
        return fail(h, TDCFIE_E_UNSUPPORTED, "the comparison formulation runs on the dense FP64 and FP32 paths");
    if (tensor) p->esz = 4;   // the tensor-core paths keep FP32 vectors, 16-bit hi/lo matrices
    const size_t es = p->esz;
    // Steps per chunk.  Matrix blocks read per step: (K + 1) / C + (C - 1) / 2 + 1 + 1 / C, least near
    // C = sqrt(2 (K + 2)) = 9 at K = 42; where the C matrices that a step re-reads sit in L2 the kernels
    // per chunk count, not the bytes, and 16 steps share them.  The tests' kernel needs a divisor of 32.
    // us per step with 8 and 16, R = 1, FP64 / FP32: 480 edges 22.6 and 19.2 / 8.9 and 7.8; 990 edges 66.2
    // and 64.5 / 19.7 and 17.6; 1920 edges, K = 42, 319 and 310 / 72.9 and 73.4; 3072 edges 469 and 455 /
    // 109 and 112.  R = 3: 990 edges 173 and 173 / 42.9 and 42.7; 1320 edges 284 and 289 / 68 and 71.  So 16 pays
    // clearly below the line, and beyond it little (FP64) or nothing.  Against every block in every step: 480 edges FP64 232 -> 20 us per step, 1920 edges
    // FP32 243 -> 74 us, with eight waves 990 -> 490 us.
    p->C = tensor ? tc_chunk() : (ne <= 1024 && R <= 2 ? 16 : 8);
    p->ring = tensor ? h->K - 1 : h->K - 1 + p->C;
    const int vw = (int)(16 / es);      // elements per 16-byte vector
    p->ld = (int)(ne + vw - 1) / vw * vw;
    p->ldc = (int)(nc + vw - 1) / vw * vw;
    p->ngroups = (h->K + 1 + 3) / 4;
    // rhs quadrature tables (host, FP64), uploaded in the path precision on the handle's stream (the legacy
    // stream has no order to it)
    {
        const double s15 = std::sqrt(15.0);
        const double a1 = (9.0 - 2.0 * s15) / 21.0, b1 = (6.0 + s15) / 21.0, w1 = (155.0 + s15) / 1200.0;
        const double a2 = (9.0 + 2.0 * s15) / 21.0, b2 = (6.0 - s15) / 21.0, w2 = (155.0 - s15) / 1200.0;
        const double r7[7][4] = {{1.0 / 3, 1.0 / 3, 1.0 / 3, 9.0 / 40.0}, {a1, b1, b1, w1}, {b1, a1, b1, w1},
                                 {b1, b1, a1, w1}, {a2, b2, b2, w2}, {b2, a2, b2, w2}, {b2, b2, a2, w2}};
        const double r3[3][4] = {{2.0 / 3, 1.0 / 6, 1.0 / 6, 1.0 / 3}, {1.0 / 6, 2.0 / 3, 1.0 / 6, 1.0 / 3},
                                 {1.0 / 6, 1.0 / 6, 2.0 / 3, 1.0 / 3}};
        // entries of every edge, e-points first (the coarse loop precedes the fine loop), over the
        // distinct points: 7 per triangle, 3 per fine triangle
        std::vector<std::vector<double>> cfs(ne);
        std::vector<std::vector<int>> ids(ne);
        std::vector<int> nE(ne, 0);
        std::vector<double> X(3 * (size_t)(7 * M.nc + 3 * M.nf));
        auto area = [](const double* a, const double* b, const double* c) {
            const double ex = b[0] - a[0], ey = b[1] - a[1], ez = b[2] - a[2];
            const double fx = c[0] - a[0], fy = c[1] - a[1], fz = c[2] - a[2];
            const double nx = ey * fz - ez * fy, ny = ez * fx - ex * fz, nz = ex * fy - ey * fx;
            return 0.5 * std::sqrt(nx * nx + ny * ny + nz * nz);
        };
        for (int c = 0; c < M.nc; ++c) {
            const double* v[3] = {&M.V[3 * M.F[3 * c]], &M.V[3 * M.F[3 * c + 1]], &M.V[3 * M.F[3 * c + 2]]};
            const double A = area(v[0], v[1], v[2]);
            for (int q = 0; q < 7; ++q) {
                const int id = 7 * c + q;
                for (int k = 0; k < 3; ++k) X[3 * (size_t)id + k] = r7[q][0] * v[0][k] + r7[q][1] * v[1][k] + r7[q][2] * v[2][k];
            }
            for (int j = 0; j < 3; ++j) {
                const int m = M.tedge[3 * c + j];
                const double sgn = M.tsign[3 * c + j] / (2.0 * A);
                for (int q = 0; q < 7; ++q) {
                    ids[m].push_back(7 * c + q);
                    for (int k = 0; k < 3; ++k) cfs[m].push_back(r7[q][3] * A * sgn * (X[3 * (size_t)(7 * c + q) + k] - v[j][k]));
                    nE[m]++;
                }
            }
        }
        for (int t = 0; t < M.nf; ++t) {
            const double* v[3] = {&M.fV[3 * M.fF[3 * t]], &M.fV[3 * M.fF[3 * t + 1]], &M.fV[3 * M.fF[3 * t + 2]]};
            const double A = area(v[0], v[1], v[2]);
            for (int q = 0; q < 3; ++q) {
                const size_t id = 7 * (size_t)M.nc + 3 * t + q;
                for (int k = 0; k < 3; ++k) X[3 * id + k] = r3[q][0] * v[0][k] + r3[q][1] * v[1][k] + r3[q][2] * v[2][k];
            }
            for (int e = M.bc_ptr[t]; e < M.bc_ptr[t + 1]; ++e) {
                const int m = M.bc_fn[e];
                const double* ph = &M.bc_phi[3 * e];
                for (int q = 0; q < 3; ++q) {
                    const int id = 7 * M.nc + 3 * t + q;
                    ids[m].push_back(id);
                    for (int k = 0; k < 3; ++k) {
                        double g = 0.0;
                        for (int j = 0; j < 3; ++j) g += ph[j] * (X[3 * (size_t)id + k] - v[j][k]);
                        cfs[m].push_back(r3[q][3] * A * g / (2.0 * A));
                    }
                }
            }
        }
        std::vector<int> ptr(ne + 1, 0);
        for (int64_t m = 0; m < ne; ++m) ptr[m + 1] = ptr[m] + (int)ids[m].size();
        std::vector<double> C(3 * (size_t)ptr[ne]);
        std::vector<int> I(ptr[ne]);
        for (int64_t m = 0; m < ne; ++m) {
            std::copy(ids[m].begin(), ids[m].end(), I.begin() + ptr[m]);
            std::copy(cfs[m].begin(), cfs[m].end(), C.begin() + 3 * (size_t)ptr[m]);
        }
        auto put = [&](void** dst, const std::vector<double>& v) -> cudaError_t {      // path precision
            const bool f64 = p->prec == TDCFIE_FP64;
            std::vector<float> vf;
            if (!f64) vf.assign(v.begin(), v.end());
            const size_t bytes = v.size() * (f64 ? 8 : 4);
            const cudaError_t e = cudaMalloc(dst, bytes);
            return e != cudaSuccess ? e : cudaMemcpyAsync(*dst, f64 ? (const void*)v.data() : vf.data(), bytes, cudaMemcpyHostToDevice, s);
        };
        auto puti = [&](int** dst, const std::vector<int>& v) -> cudaError_t {
            const cudaError_t e = cudaMalloc(dst, sizeof(int) * v.size());
            return e != cudaSuccess ? e : cudaMemcpyAsync(*dst, v.data(), sizeof(int) * v.size(), cudaMemcpyHostToDevice, s);
        };
        p->npts = (int)(X.size() / 3);
        CK(puti(&p->eptr, ptr));
        CK(puti(&p->enE, nE));
        CK(put(&p->pts, X));
        if (tensor) {       // {c, point index} together
            std::vector<float> ent(4 * I.size());
            for (size_t q = 0; q < I.size(); ++q) {
                for (int k = 0; k < 3; ++k) ent[4 * q + k] = (float)C[3 * q + k];
                std::memcpy(&ent[4 * q + 3], &I[q], sizeof(int));
            }
            CK(cudaMalloc(&p->ecoef, sizeof(float) * ent.size()));
            CK(cudaMemcpyAsync(p->ecoef, ent.data(), sizeof(float) * ent.size(), cudaMemcpyHostToDevice, s));
        } else {
            CK(puti(&p->eidx, I));
            CK(put(&p->ecoef, C));
        }
        if (!tensor) CK(cudaMalloc(&p->env, es * p->npts * R * p->C));
    }
    CK(cudaMalloc(&p->ctl, sizeof(Ctl)));
    if (!h->dexc) {     // with the plan, so that whoever keeps a view of the plan has its address
        CK(cudaMalloc(&h->dexc, sizeof(double) * 11 * R));
        CK(cudaMemsetAsync(h->dexc, 0, sizeof(double) * 11 * R, s));
    }
    if (!tensor) {
        const size_t CR = (size_t)p->C * R;
        struct { void** p; size_t n; } bufs[] = {{&p->E, es * CR * p->ld}, {&p->Hv, es * CR * p->ld},
                                                 {&p->ringbuf, es * (p->ring + 1) * R * p->ld}, {&p->b, es * R * p->ld},
                                                 {&p->partial, 8 * p->ngroups * CR * p->ld},
                                                 {&p->inner, 8 * p->C * CR * p->ld},
                                                 {&p->z, es * CR * p->ldc}, {&p->u, es * CR * p->ldc}, {(void**)&p->done, sizeof(int)}};
        for (auto& b : bufs) {      // the padding stays zero
            CK(cudaMalloc(b.p, b.n));
            CK(cudaMemsetAsync(*b.p, 0, b.n, s));
        }
    }
    if (tensor) {
        tdcfie_status st = build_tc(h, p);
        if (st != TDCFIE_OK) return st;
    } else if (h->formulation == TDCFIE_FORMULATION_MFIE) {
        // mixed TD-MFIE (a comparison formulation of Sec. V): sum_k MM'_k j_{n-k} = h_n with
        // MM'_0 = MM_0 + G/2; block 0 (e) zero, block 1 (h) the identity, block 1+k: -MM_k; the
        // unknown is j itself, so the projector product is zero and the post-processing returns y
        const int ld = p->ld, ldc = p->ldc;
        CK(cudaMalloc(&p->blocks, es * p->nblk * ne * ld));
        CK(cudaMalloc(&p->t0inv, es * ne * ld));
        CK(cudaMalloc(&p->pinv, es * nc * ldc));
        CK(cudaMemsetAsync(p->blocks, 0, es * ne * ld, s));
        CK(cudaMemsetAsync(p->pinv, 0, es * nc * ldc, s));
        double *tmp = nullptr, *work = nullptr;
        CK(cudaMalloc(&tmp, 8 * ne * ne));
        CK(cudaMalloc(&work, 8 * (2 * ne + 2)));
        fill_identity(s, tmp, (int)ne, 1.0);
        to_path(s, p->prec, tmp, (char*)p->blocks + es * ne * ld, ne, (int)ne, ld, 1.0);
        for (int k = 1; k < h->K; ++k)
            to_path(s, p->prec, h->MM + (int64_t)k * ne * ne, (char*)p->blocks + es * (1 + k) * ne * ld, ne, (int)ne, ld, -1.0);
        CK(cudaMemcpyAsync(tmp, h->MM, 8 * ne * ne, cudaMemcpyDeviceToDevice, s));
        axpby(s, ne * ne, 0.5, h->G, 1.0, tmp);
        const int singular = invert(s, tmp, (int)ne, work);
        to_path(s, p->prec, tmp, p->t0inv, ne, (int)ne, ld, 1.0);
        CK(cudaStreamSynchronize(s));
        cudaFree(tmp);
        cudaFree(work);
        if (singular) return fail(h, TDCFIE_E_STATE, "G/2 + MM_0 is singular");
    } else if (h->history_form == TDCFIE_HISTORY_FACTORED) {
        tdcfie_status st = build_fact(h, p);
        if (st != TDCFIE_OK) return st;
        h->step_bytes = fact_step_bytes(p);
    } else {
        // block 0: -A, block 1: alpha L2, block 1+k: -T_k
        const int ld = p->ld, ldc = p->ldc;
        CK(cudaMalloc(&p->blocks, es * p->nblk * ne * ld));
        CK(cudaMalloc(&p->t0inv, es * ne * ld));
        CK(cudaMalloc(&p->pinv, es * nc * ldc));
        to_path(s, p->prec, h->A, p->blocks, ne, (int)ne, ld, -1.0);
        to_path(s, p->prec, h->L2, (char*)p->blocks + es * ne * ld, ne, (int)ne, ld, h->alpha);
        to_path(s, p->prec, h->T + ne * ne, (char*)p->blocks + es * 2 * ne * ld, ne * (h->K - 1), (int)ne, ld, -1.0);
        to_path(s, p->prec, h->T0inv, p->t0inv, ne, (int)ne, ld, 1.0);
        to_path(s, p->prec, h->PinvS, p->pinv, nc, (int)nc, ldc, 1.0);
        CK(cudaStreamSynchronize(s));
    }
    CK(cudaEventCreate(&p->ev0));
    CK(cudaEventCreate(&p->ev1));
    if (!tensor && !p->fact) {
        h->hist_bytes = (double)p->nblk * ne * ne * es;
        h->step_bytes = h->hist_bytes + (double)ne * ne * es + (double)nc * nc * es;
    }
    if (h->opts.solver == TDCFIE_SOLVE_GMRES) {
        const tdcfie_status st = plan_set_solver(h, h->opts.solver, h->opts.guess, h->opts.gmres_tol);
        if (st != TDCFIE_OK) return st;
    }
    return plan_reset(h);
}

// Select the per-step solve of an existing plan; GMRES state, T_0 in the path precision and the
// learned-guess network are allocated on first use.  The step graph is captured again at the next
// step.
tdcfie_status plan_set_solver(tdcfie_t h, int solver, int guess, double tol) {
    StepPlan* p = h->plan;
    cudaStream_t s = h->stream;
    const int64_t ne = p->ne, R = p->R;
    const size_t es = p->esz;
    if (solver == TDCFIE_SOLVE_GMRES && (p->prec == TDCFIE_BF16X3 || p->prec == TDCFIE_FP16X3))
        return fail(h, TDCFIE_E_UNSUPPORTED, "GMRES runs on the FP64 and FP32 paths");
    if (solver == TDCFIE_SOLVE_GMRES && p->fact)
        return fail(h, TDCFIE_E_UNSUPPORTED, "the factored history form uses the direct solve");
    if (solver == TDCFIE_SOLVE_GMRES && h->formulation != TDCFIE_FORMULATION_QHP_CFIE)
        return fail(h, TDCFIE_E_UNSUPPORTED, "the comparison formulation uses the direct solve");
    const bool learned = guess == TDCFIE_GUESS_MLP || guess == TDCFIE_GUESS_MLP_EXTRAP;
    if (solver == TDCFIE_SOLVE_GMRES && guess == TDCFIE_GUESS_EXTRAP && p->K - 1 < 4)
        return fail(h, TDCFIE_E_UNSUPPORTED, "the extrapolated guess needs K - 1 >= 4 stored steps");
    if (solver == TDCFIE_SOLVE_GMRES && learned && p->K - 1 < 8)
        return fail(h, TDCFIE_E_UNSUPPORTED, "the learned guess needs K - 1 >= 8 stored steps");
    h->opts.solver = solver;
    h->opts.guess = guess;
    h->opts.gmres_tol = tol;
    if (solver == TDCFIE_SOLVE_GMRES) {
        if (!p->t0mat) {
            CK(cudaMalloc(&p->t0mat, es * ne * ne));
            to_path(s, p->prec, h->T, p->t0mat, ne, (int)ne, (int)ne, 1.0);
            CK(cudaMalloc(&p->guessbuf, es * R * p->ld));
            CK(cudaMemsetAsync(p->guessbuf, 0, es * R * p->ld, s));
        }
        if (!p->gm) CK(build_gmres(h, p));
        gmres_set_tol(p->gm, tol);
        if (learned && !p->mlp) CK(build_mlp(p, s));
        CK(cudaStreamSynchronize(s));
    }
    p->gmres_on = solver == TDCFIE_SOLVE_GMRES;
    p->mlp_on = p->gmres_on && learned;
    p->guess_extrap = guess == TDCFIE_GUESS_MLP_EXTRAP;
    drop_graphs(p);
    return TDCFIE_OK;
}

tdcfie_status plan_reset(tdcfie_t h) {
    StepPlan* p = h->plan;
    cudaStream_t s = h->stream;
    Ctl c{};
    c.n = c.n0 = c.p0 = 1;
    c.bad_step = INT64_MAX;
    c.slot = 1;      // n mod ring (ring > 1), column 0 of a chunk
    if (p->gm) CK(reset_gmres_stats(p->gm, s));
    CK(cudaMemcpyAsync(p->ctl, &c, sizeof(Ctl), cudaMemcpyHostToDevice, s));
    if (p->ringbuf) CK(cudaMemsetAsync(p->ringbuf, 0, p->esz * p->ring * p->R * p->ld, s));
    if (p->fact) {
        const tdcfie_status st = reset_fact(h, p);
        if (st != TDCFIE_OK) return st;
    }
    if (p->gemm) CK(reset_tc(p->gemm, p->ring, p->ne, s));
    CK(cudaStreamSynchronize(s));
    return TDCFIE_OK;
}

// Enqueue one whole step of h on s (s must be capturing a graph): the tests and pre-sums (which return
// at once unless a chunk starts or it is the march's first), the step, its post-processing.
cudaError_t capture_step(tdcfie_t h, cudaStream_t s) {
    StepPlan* p = h->plan;
    auto simt = [&](auto t) -> cudaError_t {
        using T = decltype(t);
        int k = launch_pre<T>(h, *p, 1, s);
        const cudaError_t e = launch_inner<T>(h, *p, false, 0, s, k);
        k += launch_post<T>(h, *p, 1, s);
        p->launches_per_step = k;
        return e == cudaSuccess ? cudaGetLastError() : e;
    };
    if (p->prec == TDCFIE_FP64) return simt(0.0);
    if (p->prec == TDCFIE_FP32) return simt(0.f);
    p->launches_per_step = launch_tests_tc(h, p, 1, s);
    p->launches_per_step += launch_inner_tc(h, p, 0, false, s);
    p->launches_per_step += launch_post_tc(h, p, 1, 1, s);
    return cudaGetLastError();
}

// the executable graph `which` of the plan, captured on first use
static tdcfie_status plan_graph(tdcfie_t h, int which) {
    StepPlan* p = h->plan;
    cudaStream_t s = h->stream;
    if (p->exec[which]) return TDCFIE_OK;
    CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    int kernels = 0;
    const cudaError_t ce = p->gemm ? launch_graph_tc(h, *p, which, s, kernels)
                           : p->prec == TDCFIE_FP64 ? launch_graph<double>(h, *p, which, s, kernels)
                                                    : launch_graph<float>(h, *p, which, s, kernels);
    const cudaError_t ee = cudaStreamEndCapture(s, &p->graph[which]);
    if (ce != cudaSuccess) {
        if (p->graph[which]) { cudaGraphDestroy(p->graph[which]); p->graph[which] = nullptr; }
        return cuda_fail(h, ce, "capturing the step graph");
    }
    CK(ee);
    CK(cudaGraphInstantiate(&p->exec[which], p->graph[which], 0));
    p->nodes[which] = kernels;
    return TDCFIE_OK;
}

// Output base of the next steps of h (synchronous on h's stream): step n writes row n - n0.
tdcfie_status plan_set_outputs(tdcfie_t h, void* out, void* yout) {
    StepPlan* p = h->plan;
    cudaStream_t s = h->stream;
    Ctl c;
    CK(cudaMemcpyAsync(&c, p->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    c.n0 = c.n;
    c.out = out;
    c.yout = yout;
    CK(cudaMemcpyAsync(p->ctl, &c, sizeof(Ctl), cudaMemcpyHostToDevice, s));
    CK(cudaStreamSynchronize(s));
    return TDCFIE_OK;
}

// Status of the step state words: device timeout, then a non-finite current, then a GMRES solve that
// stopped above its tolerance (each with the first step it happened at)
tdcfie_status plan_status(tdcfie_t h, const Ctl& c) {
    if (c.timeout)
        return fail(h, TDCFIE_E_TIMEOUT, "a bounded device-side wait ran out (tensor-core pipeline, or the GMRES solve)");
    if (c.status != 0)
        return fail(h, TDCFIE_E_NONFINITE, "non-finite current at step " + std::to_string(c.bad_step));
    if (c.noconv)
        return fail(h, TDCFIE_E_NOCONV, "GMRES stopped above gmres_tol (gmres_maxit reached) at step " +
                                            std::to_string(c.noconv_step));
    return TDCFIE_OK;
}

// Status words of the last steps of h (call after they completed)
tdcfie_status plan_check(tdcfie_t h) {
    StepPlan* p = h->plan;
    Ctl c;
    CK(cudaMemcpy(&c, p->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost));
    return plan_status(h, c);
}

int plan_launches_per_step(tdcfie_t h) { return h->plan ? h->plan->launches_per_step : 0; }

tdcfie_status plan_step(tdcfie_t h, int64_t nsteps, void* out, void* yout) {
    StepPlan* p = h->plan;
    cudaStream_t s = h->stream;
    if (h->own_stream) {
        // outputs may come from work queued on the caller's legacy default stream
        CK(cudaEventRecord(h->ev_in, 0));
        CK(cudaStreamWaitEvent(s, h->ev_in, 0));
    }
    // set the output base of this call: n0 = current n
    Ctl c;
    CK(cudaMemcpyAsync(&c, p->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    c.n0 = c.n;
    c.last = c.n + nsteps - 1;
    c.out = out;
    c.yout = yout;
    c.hist_ns = 0;
    CK(cudaMemcpyAsync(p->ctl, &c, sizeof(Ctl), cudaMemcpyHostToDevice, s));
    int64_t kernels = 0;
    auto run = [&](int which) -> tdcfie_status {
        const tdcfie_status st = plan_graph(h, which);
        if (st != TDCFIE_OK) return st;
        CK(cudaGraphLaunch(p->exec[which], s));
        kernels += p->nodes[which];
        return TDCFIE_OK;
    };
#define RUN(g) do { const tdcfie_status st_ = run(g); if (st_ != TDCFIE_OK) return st_; } while (0)
    // whole chunks by one graph, the rest step by step; the post-processing runs when a chunk ends and
    // when the call does (with its last step)
    const int64_t C = p->C;
    CK(cudaEventRecord(p->ev0, s));
    for (int64_t n = c.n, end = c.n + nsteps; n < end;) {
        const int64_t i = (n - 1) % C, m = std::min(C - i, end - n);
        if (m == C) {
            RUN(StepPlan::G_CHUNK);
        } else {
            if (i == 0 || n - i == 1) RUN(StepPlan::G_PRE);      // (new_cols)
            for (int64_t q = 1; q < m; ++q) RUN(StepPlan::G_STEP);
            RUN(p->fact ? StepPlan::G_STEP : StepPlan::G_LAST + (p->gemm ? (int)m - 1 : 0));
        }
        n += m;
    }
#undef RUN
    CK(cudaEventRecord(p->ev1, s));
    CK(cudaMemcpyAsync(&c, p->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, p->ev0, p->ev1);
    h->last_step_ms = ms / (nsteps > 0 ? nsteps : 1);
    h->last_hist_ms = 1e-6 * (double)c.hist_ns / (double)nsteps;
    h->last_launches = kernels;
    return plan_status(h, c);
}

}  // namespace tdc
