// Learned initial guess for the per-step GMRES solve (no counterpart in the paper).
//
// Per unknown m at step n: features x = (y_{n-1} .. y_{n-8})_m / s_n with s_n = RMS_m (y_{n-1})_m,
// network 8 -> 64 -> 64 -> 1 with tanh hidden layers, prediction y_{n,m} = y_{n-1,m} + s_n f(x) (the
// network learns the increment; a zero output is the previous-step guess).
// Parameters (FP32 master, 4801 floats): W1 (64 x 8), b1 (64), W2 (64 x 64), b2 (64), W3 (64), b3.
// Training: mini-batch squared error (1/2N) sum (f(x) - t)^2, gradient by these kernels (32-sample
// tiles, per-block gradients in registers added with atomics), Adam update in the next one's prologue.
// Inference (march and tdcfie_mlp_predict) uses FP16 copies of the weights with FP32 arithmetic.
#include <cuda_fp16.h>

#include <cmath>
#include <random>
#include <vector>

#include "gmres.h"
#include "plan.h"
#include "simt.h"

namespace tdc {

constexpr int NIN = 8, NH = 64, NP = 4801;
constexpr int OW1 = 0, OB1 = 512, OW2 = 576, OB2 = 4672, OW3 = 4736, OB3 = 4800;
// ---------------------------------------------------------------- gradient
// A block takes tiles of TS samples; its 256 threads hold the whole gradient in registers (19 parameters
// each) and add it to the global one once.  Latency bounds it (a batch of 4096 samples is 60 M
// multiply-adds), so every product is tiled in registers from shared memory with the operands in the
// order that gives 16-byte loads: H1 and D2 in both orders, W2 too.  An update of 4096 samples: 17 us; 69 us
// with one output per thread, a block per tile and Adam in a kernel of its own.
constexpr int TS = 32;        // samples per tile
constexpr int GT = 256;       // threads per block
struct GradSh {      // every array's size is a multiple of 16 bytes
    float W1[NH][NIN], b1[NH], b2[NH], w3[NH], b3[4];
    float W2[NH][NH], W2t[NH][NH + 4];      // [i][j], [j][i]; padded against bank conflicts of the stores
    float X[TS][NIN];
    float H1[TS][NH], H1t[NH][TS + 2];      // [s][j], [j][s]
    float H2[TS][NH];
    float D2[TS][NH], D2t[NH][TS + 2];      // [s][i], [i][s]
    float D1[TS][NH];
    float o[TS], dv[TS];
};

// parameters 4 q .. 4 q + 3 of the flat order into shared memory (a quad lies in one array)
constexpr int NQ = (NP + 3) / 4, NPS = 4 * NQ;      // quads, and the stride of a padded vector
__device__ __forceinline__ void put_quad(GradSh& sh, int q, float4 v) {
    q *= 4;
    if (q < OB1) *reinterpret_cast<float4*>(&sh.W1[q / NIN][q % NIN]) = v;
    else if (q < OW2) *reinterpret_cast<float4*>(&sh.b1[q - OB1]) = v;
    else if (q < OB2) {
        const int i = (q - OW2) / NH, j = (q - OW2) % NH;
        *reinterpret_cast<float4*>(&sh.W2[i][j]) = v;
        sh.W2t[j][i] = v.x;
        sh.W2t[j + 1][i] = v.y;
        sh.W2t[j + 2][i] = v.z;
        sh.W2t[j + 3][i] = v.w;
    } else if (q < OW3) *reinterpret_cast<float4*>(&sh.b2[q - OB2]) = v;
    else if (q < OB3) *reinterpret_cast<float4*>(&sh.w3[q - OW3]) = v;
    else sh.b3[0] = v.x;
}

// This thread's entry of a tile's inputs, and of its targets (first TS threads)
struct TileIn { float x, y; };
__device__ __forceinline__ TileIn tile_in(const float* __restrict__ X, const float* __restrict__ Y, int64_t n, int64_t off,
                                          int64_t count, int64_t base) {
    const int t = threadIdx.x;
    TileIn in{0.f, 0.f};
    auto at = [&](int64_t q) { return off + q < n ? off + q : off + q - n; };      // off < n, count <= n
    if (base + (t >> 3) < count) in.x = X[at(base + (t >> 3)) * NIN + (t & 7)];
    if (t < TS && base + t < count) in.y = Y[at(base + t)];
    return in;
}

// The gradient (added to grad) and the loss of samples off .. off + count - 1 (modulo n) with the
// parameters in sh; all blocks share the tiles; `in` is this block's first.  VEC: grad is 16-byte aligned
template <bool VEC>
__device__ __forceinline__ void grad_tiles(GradSh& sh, TileIn in, const float* __restrict__ X, const float* __restrict__ Y,
                                           int64_t n, int64_t off, int64_t count, float inv_total, float* grad, float* loss) {
    const int t = threadIdx.x;
    float g2[4][4] = {}, g1[2] = {}, gb = 0.f, g3 = 0.f;      // W2 tile, W1 pair, b1 | b2 | w3, b3
    const int gi = (t >> 4) * 4, gj = (t & 15) * 4;                      // W2 rows gi.., columns gj..
    for (int64_t base = (int64_t)blockIdx.x * TS; base < count; base += (int64_t)gridDim.x * TS) {
        __syncthreads();      // the parameters are there, the tile before is done with
        sh.X[t >> 3][t & 7] = in.x;
        const float y = in.y;
        if (base + (int64_t)gridDim.x * TS < count) in = tile_in(X, Y, n, off, count, base + (int64_t)gridDim.x * TS);
        __syncthreads();
        {      // H1: one unit per thread, eight samples
            const int i = t & (NH - 1);
            const float4 wa = *reinterpret_cast<const float4*>(&sh.W1[i][0]), wb = *reinterpret_cast<const float4*>(&sh.W1[i][4]);
            const float bi = sh.b1[i];
#pragma unroll
            for (int u = 0; u < TS * NH / GT; ++u) {
                const int s = (t >> 6) + u * (GT / NH);
                const float4 xa = *reinterpret_cast<const float4*>(&sh.X[s][0]), xb = *reinterpret_cast<const float4*>(&sh.X[s][4]);
                float z = fmaf(wa.x, xa.x, bi);
                z = fmaf(wa.y, xa.y, z); z = fmaf(wa.z, xa.z, z); z = fmaf(wa.w, xa.w, z);
                z = fmaf(wb.x, xb.x, z); z = fmaf(wb.y, xb.y, z); z = fmaf(wb.z, xb.z, z); z = fmaf(wb.w, xb.w, z);
                const float h = tanhf(z);
                sh.H1[s][i] = h;
                sh.H1t[i][s] = h;
            }
        }
        __syncthreads();
        const int s0 = (t >> 4) * 2, i0 = (t & 15) * 4;      // two samples, four units
        {
            float z[2][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) z[0][u] = z[1][u] = sh.b2[i0 + u];
#pragma unroll 8
            for (int j = 0; j < NH; ++j) {
                const float4 w = *reinterpret_cast<const float4*>(&sh.W2t[j][i0]);
                const float2 h = *reinterpret_cast<const float2*>(&sh.H1t[j][s0]);
                z[0][0] = fmaf(w.x, h.x, z[0][0]); z[0][1] = fmaf(w.y, h.x, z[0][1]);
                z[0][2] = fmaf(w.z, h.x, z[0][2]); z[0][3] = fmaf(w.w, h.x, z[0][3]);
                z[1][0] = fmaf(w.x, h.y, z[1][0]); z[1][1] = fmaf(w.y, h.y, z[1][1]);
                z[1][2] = fmaf(w.z, h.y, z[1][2]); z[1][3] = fmaf(w.w, h.y, z[1][3]);
            }
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                float o = 0.f;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    z[a][u] = tanhf(z[a][u]);
                    o = fmaf(sh.w3[i0 + u], z[a][u], o);
                }
                *reinterpret_cast<float4*>(&sh.H2[s0 + a][i0]) = make_float4(z[a][0], z[a][1], z[a][2], z[a][3]);
                for (int k = 8; k > 0; k >>= 1) o += __shfl_xor_sync(0xffffffffu, o, k);      // over the 16 lanes of a sample
                if ((t & 15) == 0) sh.o[s0 + a] = o;
            }
        }
        __syncthreads();
        if (t < TS) {
            const float r = base + t < count ? sh.o[t] + sh.b3[0] - y : 0.f;
            sh.dv[t] = r * inv_total;
            atomicAdd(loss, 0.5f * r * r * inv_total);
        }
        __syncthreads();
        for (int e = t; e < TS * NH; e += GT) {
            const int s = e / NH, i = e % NH;
            const float h = sh.H2[s][i], d = sh.dv[s] * sh.w3[i] * (1.f - h * h);
            sh.D2[s][i] = d;
            sh.D2t[i][s] = d;
        }
        __syncthreads();
        {
            float a0[4] = {}, a1[4] = {};
#pragma unroll 8
            for (int i = 0; i < NH; ++i) {
                const float4 w = *reinterpret_cast<const float4*>(&sh.W2[i][i0]);
                const float2 d = *reinterpret_cast<const float2*>(&sh.D2t[i][s0]);
                a0[0] = fmaf(w.x, d.x, a0[0]); a0[1] = fmaf(w.y, d.x, a0[1]); a0[2] = fmaf(w.z, d.x, a0[2]); a0[3] = fmaf(w.w, d.x, a0[3]);
                a1[0] = fmaf(w.x, d.y, a1[0]); a1[1] = fmaf(w.y, d.y, a1[1]); a1[2] = fmaf(w.z, d.y, a1[2]); a1[3] = fmaf(w.w, d.y, a1[3]);
            }
            const float4 h0 = *reinterpret_cast<const float4*>(&sh.H1[s0][i0]);
            const float4 h1 = *reinterpret_cast<const float4*>(&sh.H1[s0 + 1][i0]);
            *reinterpret_cast<float4*>(&sh.D1[s0][i0]) =
                make_float4(a0[0] * (1.f - h0.x * h0.x), a0[1] * (1.f - h0.y * h0.y), a0[2] * (1.f - h0.z * h0.z),
                            a0[3] * (1.f - h0.w * h0.w));
            *reinterpret_cast<float4*>(&sh.D1[s0 + 1][i0]) =
                make_float4(a1[0] * (1.f - h1.x * h1.x), a1[1] * (1.f - h1.y * h1.y), a1[2] * (1.f - h1.z * h1.z),
                            a1[3] * (1.f - h1.w * h1.w));
        }
        __syncthreads();
#pragma unroll 4
        for (int s = 0; s < TS; ++s) {
            const float4 d = *reinterpret_cast<const float4*>(&sh.D2[s][gi]);
            const float4 h = *reinterpret_cast<const float4*>(&sh.H1[s][gj]);
            const float dd[4] = {d.x, d.y, d.z, d.w}, hh[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) g2[a][b] = fmaf(dd[a], hh[b], g2[a][b]);
            // W1[i][k], i = t / 4, k = 2 (t % 4) + {0, 1}
            const float d1 = sh.D1[s][t >> 2];
            const float2 x = *reinterpret_cast<const float2*>(&sh.X[s][2 * (t & 3)]);
            g1[0] = fmaf(d1, x.x, g1[0]);
            g1[1] = fmaf(d1, x.y, g1[1]);
            gb += t < NH ? sh.D1[s][t] : t < 2 * NH ? sh.D2[s][t - NH] : t < 3 * NH ? sh.dv[s] * sh.H2[s][t - 2 * NH] : 0.f;
            if (t == GT - 1) g3 += sh.dv[s];
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        float* p = grad + OW2 + (gi + a) * NH + gj;
        if constexpr (VEC) atomicAdd(reinterpret_cast<float4*>(p), make_float4(g2[a][0], g2[a][1], g2[a][2], g2[a][3]));
        else
#pragma unroll
            for (int b = 0; b < 4; ++b) atomicAdd(p + b, g2[a][b]);
    }
    atomicAdd(grad + OW1 + (t >> 2) * NIN + 2 * (t & 3), g1[0]);
    atomicAdd(grad + OW1 + (t >> 2) * NIN + 2 * (t & 3) + 1, g1[1]);
    if (t < 3 * NH) atomicAdd(grad + (t < NH ? OB1 + t : t < 2 * NH ? OB2 + t - NH : OW3 + t - 2 * NH), gb);
    if (t == GT - 1) atomicAdd(grad + OB3, g3);
}

__global__ void __launch_bounds__(GT) k_mlp_grad(const float* __restrict__ prm, const float* __restrict__ X,
                                                 const float* __restrict__ Y, int64_t n, float inv_total,
                                                 float* __restrict__ grad, float* __restrict__ loss) {
    extern __shared__ __align__(16) unsigned char smem[];
    GradSh& sh = *reinterpret_cast<GradSh*>(smem);
    for (int q = threadIdx.x; q < NQ; q += GT)      // prm may have any alignment
        put_quad(sh, q, 4 * q < OB3 ? make_float4(prm[4 * q], prm[4 * q + 1], prm[4 * q + 2], prm[4 * q + 3])
                                    : make_float4(prm[OB3], 0.f, 0.f, 0.f));
    grad_tiles<false>(sh, tile_in(X, Y, n, 0, n, (int64_t)blockIdx.x * TS), X, Y, n, 0, n, inv_total, grad, loss);
}

struct AdamStep { float lr, b1, b2, eps, c1, c2; };
__device__ __forceinline__ float adam(const AdamStep& a, float p, float g, float& m1, float& m2) {
    m1 = a.b1 * m1 + (1.f - a.b1) * g;
    m2 = a.b2 * m2 + (1.f - a.b2) * g * g;
    return p - a.lr * (m1 / a.c1) / (sqrtf(m2 / a.c2) + a.eps);
}

// One training update in one kernel: every block forms the parameters after the update before (from
// that update's gradient; block 0 keeps them and the moments for the next kernel in the other of two
// slots), then adds its samples' gradient to this update's buffer, one of three in turn (block 0 clears
// the next one's).  Slot layout: params, m1, m2, each padded to NPS.
struct TrainStep {
    const float* cur;      // state before the update in front (this kernel's, if there is none)
    float* next;
    const float* gprev;    // its gradient (nullptr: none yet)
    float* grad;
    float* gclear;
    float* loss;
    AdamStep a;
    int64_t n, off, count;
};
__global__ void __launch_bounds__(GT) k_mlp_step(const __grid_constant__ TrainStep ts, const float* __restrict__ X,
                                                 const float* __restrict__ Y) {
    extern __shared__ __align__(16) unsigned char smem[];
    GradSh& sh = *reinterpret_cast<GradSh*>(smem);
    // the samples are the caller's: no kernel of the chain writes them
    const TileIn in = tile_in(X, Y, ts.n, ts.off, ts.count, (int64_t)blockIdx.x * TS);
    wait_prior();
    const float4* cur = reinterpret_cast<const float4*>(ts.cur);
    for (int q = threadIdx.x; q < NQ; q += GT) {
        float4 p = cur[q];
        if (ts.gprev) {
            float4 m1 = cur[NQ + q], m2 = cur[2 * NQ + q];
            const float4 g = reinterpret_cast<const float4*>(ts.gprev)[q];
            p.x = adam(ts.a, p.x, g.x, m1.x, m2.x);
            p.y = adam(ts.a, p.y, g.y, m1.y, m2.y);
            p.z = adam(ts.a, p.z, g.z, m1.z, m2.z);
            p.w = adam(ts.a, p.w, g.w, m1.w, m2.w);
            if (blockIdx.x == 0) {
                float4* next = reinterpret_cast<float4*>(ts.next);
                next[q] = p;
                next[NQ + q] = m1;
                next[2 * NQ + q] = m2;
            }
        }
        if (blockIdx.x == 0) reinterpret_cast<float4*>(ts.gclear)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        put_quad(sh, q, p);
    }
    grad_tiles<true>(sh, in, X, Y, ts.n, ts.off, ts.count, 1.f / (float)ts.count, ts.grad, ts.loss);
}
// the last update, into the caller's parameters
__global__ void k_mlp_last(const float* cur, const float* g, AdamStep a, float* prm) {
    wait_prior();
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= NP) return;
    float m1 = cur[NPS + q], m2 = cur[2 * NPS + q];
    prm[q] = adam(a, cur[q], g[q], m1, m2);
}

__global__ void k_to_half(const float* __restrict__ a, __half* __restrict__ b, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = __float2half_rn(a[i]);
}

// forward pass of one sample with FP16 weights staged in shared memory as FP32
__device__ __forceinline__ float mlp_forward(const float* P, const float* x) {
    float h1[NH];   // kept in registers: every loop that indexes it is fully unrolled
#pragma unroll
    for (int i = 0; i < NH; ++i) {
        float z = P[OB1 + i];
#pragma unroll
        for (int k = 0; k < NIN; ++k) z += P[OW1 + i * NIN + k] * x[k];
        h1[i] = tanhf(z);
    }
    float o = P[OB3];
    for (int i = 0; i < NH; ++i) {
        float z = P[OB2 + i];
#pragma unroll
        for (int j = 0; j < NH; ++j) z += P[OW2 + i * NH + j] * h1[j];
        o += P[OW3 + i] * tanhf(z);
    }
    return o;
}

__global__ void k_mlp_predict(const __half* __restrict__ wh, const float* __restrict__ X, int64_t n,
                              float* __restrict__ out) {
    __shared__ float P[NP];
    for (int i = threadIdx.x; i < NP; i += blockDim.x) P[i] = __half2float(wh[i]);
    __syncthreads();
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    float x[NIN];
    for (int k = 0; k < NIN; ++k) x[k] = X[s * NIN + k];
    out[s] = mlp_forward(P, x);
}

// RMS over ne entries of one vector, FP32 accumulation; block of 256 threads, result to all threads
// (1 for a zero vector).  Used both for the in-march guess and for training samples, so that the two
// scale their features identically.
template <typename T>
__device__ float block_rms(const T* __restrict__ y, int ne, float* red) {
    float a = 0.f;
    if (y)
        for (int i = threadIdx.x; i < ne; i += blockDim.x) a += (float)y[i] * (float)y[i];
    red[threadIdx.x] = a;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    const float s = sqrtf(red[0] / ne);
    __syncthreads();
    return s > 0.f ? s : 1.f;
}

// s_r = RMS over edges of y_{n-1} (one block of 256 threads per right-hand side)
template <typename T>
__global__ void k_mlp_rms(const T* __restrict__ ringbuf, int ring, int R, int ne, int ld, const Ctl* ctl, int off,
                          float* __restrict__ scale) {
    __shared__ float red[256];
    const int r = blockIdx.x;
    const int64_t n = ctl->n + off;
    const T* y = n > 1 ? ringbuf + (((n - 1) % ring) * R + r) * (int64_t)ld : nullptr;
    const float s = block_rms(y, ne, red);
    if (threadIdx.x == 0) scale[r] = s;
}

// Training samples from a stored trajectory y (nt x R x ne, step-major): for t = 8 .. nt-1 the
// sample ((t - 8) R + r) ne + m has X = (y[t-1] .. y[t-8])_{r,m} / s and the increment target
// Y = (y[t] - base)_{r,m} / s with s = RMS_m y[t-1]_r, base y[t-1] or the cubic extrapolation
// 4 y[t-1] - 6 y[t-2] + 4 y[t-3] - y[t-4]; the difference is formed in the
// trajectory's own precision before the division, so small increments keep their digits.  One
// block of 256 threads per (t, r).
template <typename T>
__global__ void k_mlp_samples(const T* __restrict__ y, int R, int ne, int base, float* __restrict__ X,
                              float* __restrict__ Y) {
    __shared__ float red[256];
    const int64_t q = blockIdx.x;          // (t - 8) * R + r
    const int r = (int)(q % R);
    const int64_t t = q / R + 8;
    auto at = [&](int64_t step) { return y + (step * R + r) * (int64_t)ne; };
    const float s = block_rms(at(t - 1), ne, red);
    for (int m = threadIdx.x; m < ne; m += blockDim.x) {
        const int64_t o = q * ne + m;
        for (int k = 1; k <= NIN; ++k) X[o * NIN + k - 1] = (float)at(t - k)[m] / s;
        const T b = base ? (T)4 * at(t - 1)[m] - (T)6 * at(t - 2)[m] + (T)4 * at(t - 3)[m] - at(t - 4)[m] : at(t - 1)[m];
        Y[o] = (float)((at(t)[m] - b) / (T)s);
    }
}

// guess[r][m] = base + s_r f((y_{n-1..n-8})_{r,m} / s_r), base = y_{n-1} or (extrap) the cubic
// extrapolation 4 y_{n-1} - 6 y_{n-2} + 4 y_{n-3} - y_{n-4}; y_i = 0 for i <= 0.  The base is formed in
// the path precision T, so a network that outputs zero reproduces it exactly.
template <typename T>
__global__ void k_mlp_guess(const __half* __restrict__ wh, const T* __restrict__ ringbuf, int ring, int R, int ne, int ld,
                            const Ctl* ctl, int off, const float* __restrict__ scale, int extrap, T* __restrict__ guess) {
    __shared__ float P[NP];
    for (int i = threadIdx.x; i < NP; i += blockDim.x) P[i] = __half2float(wh[i]);
    __syncthreads();
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= R * ne) return;
    const int r = idx / ne, m = idx % ne;
    const int64_t n = ctl->n + off;
    const float s = scale[r];
    float x[NIN];
    T yk[4] = {0, 0, 0, 0};
    for (int k = 1; k <= NIN; ++k) {
        T v = 0;
        if (n - k >= 1) {
            v = ringbuf[(((n - k) % ring) * R + r) * (int64_t)ld + m];
        }
        if (k <= 4) yk[k - 1] = v;
        x[k - 1] = (float)v / s;
    }
    const T base = extrap ? (T)4 * yk[0] - (T)6 * yk[1] + (T)4 * yk[2] - yk[3] : yk[0];
    guess[(int64_t)r * ld + m] = base + (T)(s * mlp_forward(P, x));   // base + predicted correction
}

// ---------------------------------------------------------------- march integration
struct MlpState {
    __half* wh = nullptr;
    float* scale = nullptr;
    bool loaded = false;
};

void destroy_mlp(MlpState* m) {
    if (!m) return;
    if (m->wh) cudaFree(m->wh);
    if (m->scale) cudaFree(m->scale);
    delete m;
}

template <typename T>
int launch_mlp_guess(StepPlan* p, int off, cudaStream_t s) {
    MlpState* m = p->mlp;
    k_mlp_rms<T><<<p->R, 256, 0, s>>>((const T*)p->ringbuf, p->ring, p->R, p->ne, p->ld, p->ctl, off, m->scale);
    k_mlp_guess<T><<<(p->R * p->ne + 127) / 128, 128, 0, s>>>(m->wh, (const T*)p->ringbuf, p->ring, p->R, p->ne,
                                                                p->ld, p->ctl, off, m->scale, p->guess_extrap ? 1 : 0,
                                                                (T*)p->guessbuf);
    return 2;
}
template int launch_mlp_guess<double>(StepPlan*, int, cudaStream_t);
template int launch_mlp_guess<float>(StepPlan*, int, cudaStream_t);

cudaError_t build_mlp(StepPlan* p, cudaStream_t s) {
    auto* m = new MlpState();
    p->mlp = m;
    cudaError_t e;
    if ((e = cudaMalloc(&m->wh, sizeof(__half) * NP)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(m->wh, 0, sizeof(__half) * NP, s)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&m->scale, sizeof(float) * p->R)) != cudaSuccess) return e;
    return cudaSuccess;
}

cudaError_t mlp_load(StepPlan* p, const float* host_params, cudaStream_t s) {
    float* d = nullptr;
    cudaError_t e = cudaMalloc(&d, sizeof(float) * NP);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(d, host_params, sizeof(float) * NP, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
        k_to_half<<<(NP + 255) / 256, 256, 0, s>>>(d, p->mlp->wh, NP);
        e = cudaStreamSynchronize(s);
    }
    cudaFree(d);
    p->mlp->loaded = (e == cudaSuccess);
    return e;
}

}  // namespace tdc

using namespace tdc;

// blocks of a gradient over `count` samples: two per SM at most (they share the tiles)
static int grad_blocks(int64_t count) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        sms = 148;
    return (int)std::min<int64_t>((count + TS - 1) / TS, 2 * sms);
}

extern "C" tdcfie_status tdcfie_mlp_grad(const float* params, const float* X, const float* Y, int64_t n, float* grad,
                                         float* loss, void* stream) {
    if (!params || !X || !Y || !grad || !loss) return fail(nullptr, TDCFIE_E_ARG, "NULL device pointer");
    if (n < 1) return fail(nullptr, TDCFIE_E_ARG, "n must be >= 1");
    cudaStream_t s = (cudaStream_t)stream;
    // the attribute is set on every call: it is per device
    cudaError_t e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSh));
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaFuncSetAttribute (MLP gradient)");
    e = cudaMemsetAsync(grad, 0, sizeof(float) * NP, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(loss, 0, sizeof(float), s);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaMemsetAsync");
    k_mlp_grad<<<grad_blocks(n), GT, sizeof(GradSh), s>>>(params, X, Y, n, 1.f / (float)n, grad, loss);
    e = cudaGetLastError();
    return e == cudaSuccess ? TDCFIE_OK : cuda_fail(nullptr, e, "MLP gradient launch");
}

extern "C" tdcfie_status tdcfie_mlp_train(float* params, const float* X, const float* Y, int64_t n, int epochs,
                                          int64_t batch, float lr, uint64_t seed, float* loss_history, void* stream) {
    if (!params || !X || !Y) return fail(nullptr, TDCFIE_E_ARG, "NULL device pointer");
    if (n < 1 || epochs < 1 || batch < 1 || !(lr > 0.f)) return fail(nullptr, TDCFIE_E_ARG, "bad training sizes");
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaFuncSetAttribute(k_mlp_step, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSh));
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaFuncSetAttribute (MLP training)");
    // two states (params, m1, m2), three gradients, the passes' losses
    float* buf = nullptr;
    const size_t bytes = sizeof(float) * (9 * (size_t)NPS + epochs);
    e = cudaMallocAsync((void**)&buf, bytes, s);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaMallocAsync (MLP training state)");
    float* state[2] = {buf, buf + 3 * NPS};
    float* grad = buf + 6 * NPS;
    float* loss = buf + 9 * NPS;
    e = cudaMemsetAsync(buf, 0, bytes, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(state[0], params, sizeof(float) * NP, cudaMemcpyDeviceToDevice, s);
    std::mt19937_64 rng(seed);
    const int64_t nb = (n + batch - 1) / batch;
    int64_t step = 0;
    TrainStep ts{};
    ts.a = AdamStep{lr, 0.9f, 0.999f, 1e-8f, 1.f, 1.f};
    ts.n = n;
    auto corrections = [&](int64_t k) {      // of update k
        ts.a.c1 = 1.f - std::pow(0.9f, (float)k);
        ts.a.c2 = 1.f - std::pow(0.999f, (float)k);
    };
    const int blocks = grad_blocks(std::min(n, batch));
    for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
        const int64_t rot = (int64_t)(rng() % (uint64_t)n);   // per-epoch rotation of the batch origin
        for (int64_t b = 0; b < nb && e == cudaSuccess; ++b, ++step) {
            // kernel `step` (from 0): state after step - 1 updates in slot (step + 1) & 1, from step 2 on
            ts.off = (rot + b * batch) % n;
            ts.count = std::min<int64_t>(batch, n - b * batch);
            ts.cur = state[step < 2 ? 0 : (step - 1) & 1];
            ts.next = state[step & 1];
            ts.gprev = step ? grad + (step - 1) % 3 * NPS : nullptr;
            ts.grad = grad + step % 3 * NPS;
            ts.gclear = grad + (step + 1) % 3 * NPS;
            ts.loss = loss + ep;
            corrections(step);
            launch_chained(k_mlp_step, blocks, GT, s, sizeof(GradSh), ts, X, Y);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess) {
        corrections(step);
        launch_chained(k_mlp_last, (NP + 255) / 256, 256, s, 0, (const float*)state[step < 2 ? 0 : (step - 1) & 1],
                       (const float*)(grad + (step - 1) % 3 * NPS), ts.a, params);
        e = cudaGetLastError();
    }
    tdcfie_status st = e == cudaSuccess ? TDCFIE_OK : cuda_fail(nullptr, e, "MLP training launch");
    if (loss_history && st == TDCFIE_OK) {
        e = cudaMemcpyAsync(loss_history, loss, sizeof(float) * epochs, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) st = cuda_fail(nullptr, e, "MLP loss readback");
        for (int ep = 0; ep < epochs; ++ep) loss_history[ep] /= (float)nb;
    }
    cudaFreeAsync(buf, s);
    return st;
}

extern "C" tdcfie_status tdcfie_mlp_predict(const float* params, const float* X, int64_t n, float* out, void* stream) {
    if (!params || !X || !out) return fail(nullptr, TDCFIE_E_ARG, "NULL device pointer");
    if (n < 1) return fail(nullptr, TDCFIE_E_ARG, "n must be >= 1");
    cudaStream_t s = (cudaStream_t)stream;
    __half* wh = nullptr;
    cudaError_t e = cudaMallocAsync((void**)&wh, sizeof(__half) * NP, s);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaMallocAsync (FP16 weights)");
    k_to_half<<<(NP + 255) / 256, 256, 0, s>>>(params, wh, NP);
    k_mlp_predict<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(wh, X, n, out);
    e = cudaGetLastError();
    cudaFreeAsync(wh, s);
    return e == cudaSuccess ? TDCFIE_OK : cuda_fail(nullptr, e, "MLP predict launch");
}

extern "C" tdcfie_status tdcfie_mlp_samples(int precision, int base, const void* y, int64_t nt, int64_t R,
                                            int64_t ne, float* X, float* Y, void* stream) {
    if (!y || !X || !Y) return fail(nullptr, TDCFIE_E_ARG, "NULL device pointer");
    if (precision != TDCFIE_FP64 && precision != TDCFIE_FP32) return fail(nullptr, TDCFIE_E_ARG, "y is float64 or float32");
    if (base != 0 && base != 1) return fail(nullptr, TDCFIE_E_ARG, "base is 0 (previous step) or 1 (extrapolation)");
    if (nt < 9 || R < 1 || ne < 1) return fail(nullptr, TDCFIE_E_ARG, "need nt >= 9, R >= 1, ne >= 1");
    if (ne > INT32_MAX || (nt - 8) * R > INT32_MAX) return fail(nullptr, TDCFIE_E_ARG, "sizes out of range");
    cudaStream_t s = (cudaStream_t)stream;
    const unsigned blocks = (unsigned)((nt - 8) * R);
    if (precision == TDCFIE_FP64)
        k_mlp_samples<double><<<blocks, 256, 0, s>>>((const double*)y, (int)R, (int)ne, base, X, Y);
    else
        k_mlp_samples<float><<<blocks, 256, 0, s>>>((const float*)y, (int)R, (int)ne, base, X, Y);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? TDCFIE_OK : cuda_fail(nullptr, e, "MLP sample launch");
}

extern "C" tdcfie_status tdcfie_mlp_load(tdcfie_t h, const float* params) {
    if (!h || !params) return fail(h, TDCFIE_E_ARG, "NULL argument");
    if (!h->plan) return fail(h, TDCFIE_E_STATE, "call tdcfie_assemble first");
    if (h->plan->K - 1 < 8) return fail(h, TDCFIE_E_UNSUPPORTED, "the learned guess needs K - 1 >= 8 stored steps");
    if (!h->plan->mlp) {
        const cudaError_t eb = build_mlp(h->plan, h->stream);
        if (eb != cudaSuccess) return cuda_fail(h, eb, "learned-guess state");
    }
    const cudaError_t e = mlp_load(h->plan, params, h->stream);
    return e == cudaSuccess ? TDCFIE_OK : cuda_fail(h, e, "tdcfie_mlp_load");
}
