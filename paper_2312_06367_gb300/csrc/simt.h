// Device arithmetic of the SIMT (FP64 / FP32) step, shared by the per-handle step kernels
// (march.cu) and the persistent uneven-batch kernel (batch.cu), so that both compute the same
// values bit for bit.
//
// The march is blocked in time.  Step n belongs to the chunk of C steps that starts at the absolute
// step n0 = n - i, i = (n - 1) mod C, so that the arithmetic of a step does not depend on how the
// caller cuts the march into calls.  Everything of a chunk that is known before its first solve is
// computed once for its C steps (columns) when n0 is reached:
//   tests    e_n, h_n of the C steps (the incident field does not depend on the march);
//   pre      the sums over the blocks -A e, alpha L2 h and over every lag k > i of column i, which
//            reaches back before n0: each block is read once per chunk instead of once per step;
// then step by step
//   hist     b_n = (pre-sums of column i) - sum_{k = i..1} T_k y_{n-k}, the lags inside the chunk: only
//            k = 1 waits for the solve before; the products T_k y_{n-1}, k >= 2, of the later columns
//            are formed beside it, one per row and lag, so that the step's chain stays short;
//   solve    y_n = T_0^-1 b_n (or GMRES);
// and the post-processing of the finished steps together (its projector is not part of the
// recurrence).  The first chunk of a march is the exception, see new_cols.  Matrix bytes per step at K = 42, C = 8: 43/8 + 3.5 + 1 + 1/8 blocks instead of 45.
//
// Rows of matrices and vectors are padded to 16 bytes (zeros), every load is a 16-byte vector.
#pragma once
#include <type_traits>

#include "internal.h"

namespace tdc {

constexpr int GQ = 4;         // blocks per group of the pre-sums

// Sums are carried in FP64 on the FP64 path and as unevaluated FP32 pairs (about 48 bits, as the lanes'
// error-free sums are) on the FP32 path: FP64 reductions there take the marches of 864 edges from 8.9 to
// 16.9 ms, of 1920 edges from 14.8 to 17.5 and, with eight waves, from 49.0 to 57.5 ms.  Rows of 30 to 7680
// entries, 1 to 44 blocks: the pairs' sums are within 9e-15 of sum |a x| (FP64 reductions 1e-15), and of
// 5160 sums rounded to FP32, in which form they leave, none differs: every one is the exact sum rounded.
struct Pair32 { float h, l; };
template <typename T> struct SumOf;
template <> struct SumOf<double> { using S = double; };
template <> struct SumOf<float> { using S = Pair32; };

template <typename T>
struct SimtDev {              // device view of one handle's step plan
    int ne, nc, R, C, K, ring, ld, ldc, ngroups, npts;
    const T *blocks, *t0inv, *pinv;     // (K + 1) x ne x ld (-A, alpha L2, -T_1 ..), ne x ld, nc x ldc
    T *E, *H;                           // tests of the chunk [C R][ld], column i R + r
    T *rbuf, *b;                        // ring [ring][R][ld], b_n [R][ld]
    T *z, *u;                           // projector vectors of the steps to post-process [C R][ldc]
    typename SumOf<T>::S* partial;      // pre-sums [ngroups][C R][ld]
    typename SumOf<T>::S* inner;        // T_k y of lag k >= 2 for column i of the chunk [i][k][R][ld]
    T* env;                             // envelopes [npts][R][C]
    const T* pts;                       // distinct quadrature points, npts x 3
    const int *eptr, *enE, *eidx;       // per edge: entries (e-points first), number of e-points, point index
    const T* ecoef;                     // weighted basis vector per entry
    const double* exc;
    DevMesh m;
    double dt, dtt;
    Ctl* ctl;
    int* done;
};

template <typename T> __device__ __forceinline__ T mul_rn(T a, T b);
template <> __device__ __forceinline__ float mul_rn<float>(float a, float b) { return __fmul_rn(a, b); }
template <> __device__ __forceinline__ double mul_rn<double>(double a, double b) { return __dmul_rn(a, b); }
template <typename T> __device__ __forceinline__ T add_rn(T a, T b);
template <> __device__ __forceinline__ float add_rn<float>(float a, float b) { return __fadd_rn(a, b); }
template <> __device__ __forceinline__ double add_rn<double>(double a, double b) { return __dadd_rn(a, b); }

// Position of a step in the march: its ring slot and its column of the chunk.  Both ride in the step
// state, so that no kernel of the chain starts with 64-bit divisions.
struct StepPos { int64_t n; int slot, col; };
__device__ __forceinline__ int ring_at(int slot, int delta, int ring) {      // |delta| <= ring
    const int t = slot + delta;
    return t < 0 ? t + ring : t >= ring ? t - ring : t;
}
// step ctl->n + off, which lies in the same chunk
template <typename T>
__device__ __forceinline__ StepPos step_pos(const SimtDev<T>& d, int off) {
    const Ctl* c = d.ctl;
    return StepPos{c->n + off, ring_at(c->slot, off, d.ring), c->col + off};
}
// the step counter moves by adv (at most C)
template <typename T>
__device__ __forceinline__ void advance(const SimtDev<T>& d, int adv) {
    Ctl* c = d.ctl;
    c->n += adv;
    c->slot = ring_at(c->slot, adv, d.ring);
    c->col = (c->col + adv) % d.C;
}

// Columns lo .. hi - 1 of the current chunk whose tests and pre-sums are formed at this step: all of them
// where a chunk starts.  In the march's first chunk (the steps 1 .. C), where the lags that reach back before
// it meet y_i = 0 and only the tests' blocks count, each call forms those of its own steps: a march may
// end there, and one of a few steps does not pay for C (one step, 1920 edges, K = 42, FP64: 2.33 ms with
// the chunk formed whole, 0.20 ms so; with eight waves 15.8 and 0.64 ms).  most: the call's steps from this
// one on, 0: up to ctl->last.
struct Cols { int lo, hi; bool first; };
__device__ __forceinline__ Cols new_cols(const Ctl* ctl, int C, int64_t n, int col, int most) {
    if (n - col != 1) return Cols{0, col ? 0 : C, false};
    const int64_t left = most ? most : ctl->last - n + 1;
    return Cols{col, (int)(left < C - col ? col + left : C), true};
}

// ---------------------------------------------------------------- plane-wave tests
// e_m(t_n) = sum_x c(x).p env(x, t_n) over the 7-point rule of the RWG triangles, h_m the same with
// c(x).(k x p) over the 3-point rule of the BC fine triangles; env(x, t) = amp exp(-((t - k.x - t0) /
// width)^2).  A point belongs to three RWG or about twelve BC functions, so the envelopes are taken
// once per point (one exponential each) and gathered per edge.  Every multiply-add is spelled out,
// so that all kernels that inline this round identically.
template <typename T>
__device__ __forceinline__ T env_point(const double* P, int64_t n, double dt, T x, T y, T z) {
    const T kx = (T)P[0], ky = (T)P[1], kz = (T)P[2];
    const T amp = (T)P[6], inv_w = (T)(1.0 / P[8]);
    const T tt = (T)((double)n * dt - P[7]);
    const T arg = mul_rn(add_rn(tt, -fma(kx, x, fma(ky, y, mul_rn(kz, z)))), inv_w);
    return mul_rn(amp, exp(-mul_rn(arg, arg)));
}

// e, h of edge m and wave r for the columns `cs` of the chunk's C (a divisor of 32): lane l takes column
// l % C and every (32 / C)-th entry; the parts are added by a fixed tree
template <typename T>
__device__ __forceinline__ void gather_edge(const SimtDev<T>& d, const Cols& cs, int m, int r, int lane) {
    const double* P = d.exc + 11 * r;
    const T kx = (T)P[0], ky = (T)P[1], kz = (T)P[2], qx = (T)P[3], qy = (T)P[4], qz = (T)P[5];
    const T hx = fma(ky, qz, -mul_rn(kz, qy)), hy = fma(kz, qx, -mul_rn(kx, qz)), hz = fma(kx, qy, -mul_rn(ky, qx));   // k x p
    const int i = lane % d.C, part = lane / d.C, parts = 32 / d.C;
    const bool mine = i >= cs.lo && i < cs.hi;
    const int b = d.eptr[m], me = b + d.enE[m], end = mine ? d.eptr[m + 1] : b;
    T e = 0, h = 0;
#pragma unroll 4
    for (int q = b + part; q < end; q += parts) {
        const T cx = d.ecoef[3 * q], cy = d.ecoef[3 * q + 1], cz = d.ecoef[3 * q + 2];
        const T env = d.env[((int64_t)d.eidx[q] * d.R + r) * d.C + i];
        if (q < me) e = fma(env, fma(cx, qx, fma(cy, qy, mul_rn(cz, qz))), e);
        else h = fma(env, fma(cx, hx, fma(cy, hy, mul_rn(cz, hz))), h);
    }
    for (int o = 16; o >= d.C; o >>= 1) {
        e = add_rn(e, __shfl_xor_sync(0xffffffffu, e, o));
        h = add_rn(h, __shfl_xor_sync(0xffffffffu, h, o));
    }
    if (part == 0 && mine) {
        d.E[(int64_t)(i * d.R + r) * d.ld + m] = e;
        d.H[(int64_t)(i * d.R + r) * d.ld + m] = h;
    }
}

// ---------------------------------------------------------------- row dot products (SIMT)
// One warp, lane l takes the 16-byte vectors l, l + 32, ... of a row.  FP64: plain FP64
// accumulation, one accumulator per vector component.  FP32: the products and their sums are carried
// error-free (each product's rounding error from an FMA, each addition's from Knuth's TwoSum), so the
// result equals the exact dot product of the FP32 inputs to about FP32 precision squared; the lanes
// are combined as pairs too.  The MOT recurrence turns y into the current through (y_n - y_{n-1}) / dtt
// (Eq. post_processing), which magnifies any per-step error of y by about |y| / |y_n - y_{n-1}|;
// plain FP32 accumulation over rows of thousands of entries is then far above the reduced-precision
// bar at small time steps.  The FP32 accumulators are packed pairs: ten two-lane instructions per two
// products, half the issue slots of scalar code (issue bounds FP32 with several columns).
template <typename T> struct VecOf;
template <> struct VecOf<double> { using V = double2; static constexpr int W = 2; };
template <> struct VecOf<float> { using V = float4; static constexpr int W = 4; };

template <typename T> struct Acc;
template <>
struct Acc<double> {
    double s0 = 0.0, s1 = 0.0;
    __device__ __forceinline__ void add(const double2& a, const double2&, const double2& x) {
        s0 = fma(a.x, x.x, s0);
        s1 = fma(a.y, x.y, s1);
    }
    __device__ __forceinline__ double sum() const { return s0 + s1; }
};

// sum of two sums; on pairs TwoSum of the leading parts (the same result for either order)
__device__ __forceinline__ double add_sum(double a, double b) { return a + b; }
__device__ __forceinline__ Pair32 add_sum(Pair32 a, Pair32 b) {
    const float t = __fadd_rn(a.h, b.h);
    const float bp = __fsub_rn(t, a.h);
    const float te = __fadd_rn(__fsub_rn(a.h, __fsub_rn(t, bp)), __fsub_rn(b.h, bp));
    return Pair32{t, __fadd_rn(__fadd_rn(a.l, b.l), te)};
}
__device__ __forceinline__ double shfl_sum(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ Pair32 shfl_sum(Pair32 a, int o) {
    return Pair32{__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
}
__device__ __forceinline__ double sum_value(double a) { return a; }
__device__ __forceinline__ double sum_value(Pair32 a) { return (double)a.h + (double)a.l; }

// hi + lo += a b on two lanes; na = -a.  Rounded intrinsics only: nothing may be contracted.
__device__ __forceinline__ void ff_add2(float2& hi, float2& lo, float2 a, float2 na, float2 b) {
    const float2 m1 = make_float2(-1.f, -1.f);
    const float2 p = __fmul2_rn(a, b);
    const float2 pe = __ffma2_rn(na, b, p);     // p - a b: minus the product's rounding error, exact
    const float2 t = __fadd2_rn(hi, p);         // TwoSum(hi, p) = t + te
    const float2 bp = __ffma2_rn(hi, m1, t);    // t - hi
    const float2 ap = __ffma2_rn(bp, m1, t);    // t - bp
    const float2 te = __fadd2_rn(__ffma2_rn(ap, m1, hi), __ffma2_rn(bp, m1, p));
    lo = __fadd2_rn(lo, __ffma2_rn(pe, m1, te));
    hi = t;
}
template <>
struct Acc<float> {
    float2 h0 = {0.f, 0.f}, h1 = {0.f, 0.f}, l0 = {0.f, 0.f}, l1 = {0.f, 0.f};
    __device__ __forceinline__ void add(const float4& a, const float4& na, const float4& x) {
        ff_add2(h0, l0, make_float2(a.x, a.y), make_float2(na.x, na.y), make_float2(x.x, x.y));
        ff_add2(h1, l1, make_float2(a.z, a.w), make_float2(na.z, na.w), make_float2(x.z, x.w));
    }
    __device__ __forceinline__ Pair32 sum() const {
        return add_sum(add_sum(Pair32{h0.x, l0.x}, Pair32{h0.y, l0.y}), add_sum(Pair32{h1.x, l1.x}, Pair32{h1.y, l1.y}));
    }
};
__device__ __forceinline__ double2 neg(double2 a) { return a; }    // unused by Acc<double>
__device__ __forceinline__ float4 neg(float4 a) { return make_float4(-a.x, -a.y, -a.z, -a.w); }

// acc[i][c] += row_i . x_c for ROWS rows and (at least) the first nv of COLS columns, nvec vectors per row.
// The loads do not branch on a column (one that is not wanted repeats another, whose sum nobody reads, or
// points at zeros), so that all loads of a turn are in flight together; the rows' next vectors are fetched a
// turn ahead.  A loop each for 1, 2, 4, 8 columns: a bound inside it is predicated and costs the pipe all of
// them (two blocks of 3072 rows, FP64: 302 us with one column as with eight, 69 us so).
// before_x() runs between the first loads of the rows and the first loads of x (a kernel whose x comes
// from the kernel before it waits there).
struct Nothing { __device__ __forceinline__ void operator()() const {} };
template <typename T, int ROWS, int COLS, class F = Nothing>
__device__ __forceinline__ void tile_rows(const T* const (&row)[ROWS], const T* x, const int (&off)[COLS], int nv,
                                          int nvec, int lane, Acc<T> (&acc)[ROWS][COLS], F before_x = F()) {
    using V = typename VecOf<T>::V;
    if constexpr (ROWS * COLS >= 8) {
        // pointers and byte offsets advance by additions: index arithmetic by multiply-add would take
        // the pipe that the packed FP32 instructions run on
        const V* ap[ROWS];
        V nx[ROWS];
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            ap[i] = reinterpret_cast<const V*>(row[i]) + lane;
            nx[i] = lane < nvec ? __ldg(ap[i]) : V{};
        }
        before_x();
        const char* xb = reinterpret_cast<const char*>(x);
        unsigned xo[COLS];
#pragma unroll
        for (int c = 0; c < COLS; ++c) xo[c] = (unsigned)off[c] * (unsigned)sizeof(T) + (unsigned)lane * 16u;
        auto turn = [&](bool more, auto cols) {
            constexpr int N = decltype(cols)::value;
            V a[ROWS], na[ROWS], xv[N];
#pragma unroll
            for (int c = 0; c < N; ++c) {
                xv[c] = *reinterpret_cast<const V*>(xb + xo[c]);
                xo[c] += 512u;
            }
#pragma unroll
            for (int i = 0; i < ROWS; ++i) {
                a[i] = nx[i];
                na[i] = neg(a[i]);
                ap[i] += 32;
                if (more) nx[i] = __ldg(ap[i]);
            }
#pragma unroll
            for (int c = 0; c < N; ++c)
#pragma unroll
                for (int i = 0; i < ROWS; ++i) acc[i][c].add(a[i], na[i], xv[c]);
        };
        auto loop = [&](auto cols) {
#pragma unroll 1
            for (int j = lane; j < nvec; j += 32) turn(j + 32 < nvec, cols);
        };
        if (2 * nv > COLS) loop(std::integral_constant<int, COLS>());
        else if (4 * nv > COLS) loop(std::integral_constant<int, COLS / 2>());
        else if (nv > 1) loop(std::integral_constant<int, COLS / 4>());
        else loop(std::integral_constant<int, 1>());
    } else {
        // turns whose loads are issued together: a whole row up to about 1000 entries
        constexpr int U = ROWS * COLS >= 4 ? 2 : ROWS * COLS == 2 ? 4 : 8;
        V a[U][ROWS], xv[U][COLS];
        auto load_rows = [&](int j0) {
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int i = 0; i < ROWS; ++i)
                    a[u][i] = j0 + 32 * u < nvec ? __ldg(reinterpret_cast<const V*>(row[i]) + j0 + 32 * u) : V{};
        };
        load_rows(lane);
        before_x();
        for (int j0 = lane; j0 < nvec; j0 += 32 * U) {
            if (j0 != lane) load_rows(j0);
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int c = 0; c < COLS; ++c)
                    xv[u][c] = j0 + 32 * u < nvec ? reinterpret_cast<const V*>(x + off[c])[j0 + 32 * u] : V{};
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j0 - lane + 32 * u < nvec)
#pragma unroll
                    for (int i = 0; i < ROWS; ++i) {
                        const V na = neg(a[u][i]);
#pragma unroll
                        for (int c = 0; c < COLS; ++c) acc[i][c].add(a[u][i], na, xv[u][c]);
                    }
        }
    }
}

// Sums over the warp of V values per lane (V a power of two up to 32): every sum is the same tree
// over lanes (strides 16, 8, 4, 2, 1) whatever V is, and the first log2 V strides halve the number of
// values a lane carries.  The lane returns the sum of value multi_index<V>(lane).
template <int V, typename S>
__device__ __forceinline__ S multi_reduce(S (&v)[V], int lane) {
    int n = V;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = lane & o;
#pragma unroll
            for (int j = 0; j < V / 2; ++j)
                if (j < n) {
                    const S keep = up ? v[j + n] : v[j], send = up ? v[j] : v[j + n];
                    v[j] = add_sum(keep, shfl_sum(send, o));
                }
        } else {
            v[0] = add_sum(v[0], shfl_sum(v[0], o));
        }
    }
    return v[0];
}
template <int V>
__device__ __forceinline__ int multi_index(int lane) {
    int id = 0, n = V;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (n > 1) {
            n >>= 1;
            if (lane & o) id += n;
        }
    return id;
}
// one lane per value: the one whose remaining bits are zero
template <int V>
__device__ __forceinline__ bool multi_owner(int lane) { return (lane & (32 / V - 1)) == 0; }

// ---------------------------------------------------------------- pre-sums of a chunk
constexpr int PRE_COLS = 8;
// rows per unit: two on the FP64 path (32 accumulator registers, the row's columns share the loads), one
// on the FP32 path, whose pair accumulators would leave 8 warps per SM at two rows (fused multiply-add
// pipe 62 % busy, 543 us for 8 columns at 1920 edges, K = 42; 433 us with one)
template <typename T> constexpr int pre_rows() { return sizeof(T) == 8 ? 2 : 1; }

// Rows row0 .. row0 + pre_rows - 1, the tile-th eight columns of `cs` and group g of the blocks in the
// order e, h, lag K-1, ..., lag 1: accumulated over the group's blocks, then over the warp, into partial[g].
// slot: ring slot of the chunk's first step
template <typename T>
__device__ __forceinline__ void pre_item(const SimtDev<T>& d, const Cols& cs, int slot, int row0, int g, int tile, int lane) {
    constexpr int PRE_ROWS = pre_rows<T>();
    const int CR = d.C * d.R, nvec = d.ld / VecOf<T>::W, end = cs.hi * d.R, col0 = cs.lo * d.R + tile * PRE_COLS;
    if (col0 >= end) return;
    int ci[PRE_COLS], co[PRE_COLS];      // step within the chunk, offset of the wave within a slot
#pragma unroll
    for (int c = 0; c < PRE_COLS; ++c) {
        ci[c] = d.R == 1 ? col0 + c : (col0 + c) / d.R;
        co[c] = (col0 + c - ci[c] * d.R) * d.ld;
    }
    Acc<T> acc[PRE_ROWS][PRE_COLS];
#pragma unroll 1
    for (int o = GQ * g; o < min(GQ * g + GQ, cs.first ? 2 : d.K + 1); ++o) {
        const int k = o < 2 ? 0 : d.K + 1 - o, q = o < 2 ? o : 1 + k;      // lag and block
        const int sk = ring_at(slot, -k, d.ring);
        int off[PRE_COLS], nv = 0;
#pragma unroll
        for (int c = 0; c < PRE_COLS; ++c) {
            // columns whose lag lies inside the chunk read the zero vectors behind the ring, those behind
            // the last one that is wanted repeat it
            const bool on = col0 + c < end && (o < 2 || ci[c] < k);
            nv += on;       // the first ones of the tile
            off[c] = o < 2 ? min(col0 + c, end - 1) * d.ld
                           : (on ? ring_at(sk, ci[c], d.ring) * d.R * d.ld + co[c] : d.ring * d.R * d.ld);
        }
        if (!nv) continue;
        const T* base = d.blocks + (int64_t)q * d.ne * d.ld;
        const T* row[PRE_ROWS];
#pragma unroll
        for (int i = 0; i < PRE_ROWS; ++i) row[i] = base + (int64_t)min(row0 + i, d.ne - 1) * d.ld;
        tile_rows<T, PRE_ROWS, PRE_COLS>(row, o == 0 ? d.E : o == 1 ? d.H : d.rbuf, off, nv, nvec, lane, acc);
    }
    typename SumOf<T>::S v[PRE_ROWS * PRE_COLS];
#pragma unroll
    for (int i = 0; i < PRE_ROWS; ++i)
#pragma unroll
        for (int c = 0; c < PRE_COLS; ++c) v[i * PRE_COLS + c] = acc[i][c].sum();
    const auto s = multi_reduce<PRE_ROWS * PRE_COLS>(v, lane);
    const int id = multi_index<PRE_ROWS * PRE_COLS>(lane), row = row0 + id / PRE_COLS, col = col0 + id % PRE_COLS;
    if (multi_owner<PRE_ROWS * PRE_COLS>(lane) && row < d.ne && col < end) d.partial[((int64_t)g * CR + col) * d.ld + row] = s;
}

// ---------------------------------------------------------------- one step
// rows per unit (one warp) of the history; the solve takes one (its chain is the step's)
template <int RM>
constexpr int step_rows() { return RM <= 2 ? 2 : 1; }

// lags k >= 2 whose product with y_{n-1} belongs to a later column of the chunk (n in column i)
__device__ __forceinline__ int push_lags(int i, int C, int K) { return i == 0 ? 0 : max(0, min(C - i, K - 1) - 1); }

// One unit of the history of step n (RM >= R columns): units 0 .. nu - 1 form b_n of their rows from the
// pre-sums, the inner products kept by earlier steps and lag 1; the units after them form T_k y_{n-1}
// for lag 2 + (u / nu - 1)
// wait() returns when y_{n-1} is there; sums_ready: the pre-sums and inner products are there before it
template <typename T, int RM, class F>
__device__ __forceinline__ void hist_unit(const SimtDev<T>& d, const StepPos& pos, int u, int lane, bool sums_ready, F wait) {
    using S = typename SumOf<T>::S;
    constexpr int ROWS = step_rows<RM>();
    const int CR = d.C * d.R, nvec = d.ld / VecOf<T>::W, nu = (d.ne + ROWS - 1) / ROWS;
    const int k = 1 + u / nu, row0 = (u - (k - 1) * nu) * ROWS, i = pos.col;
    if (k > 1 && k - 1 > push_lags(i, d.C, d.K)) return;
    S v[ROWS * RM];
#pragma unroll
    for (int q = 0; q < ROWS * RM; ++q) v[q] = S{};
    auto sums = [&] {
        const int kept = k > 1 ? 0 : d.ngroups + max(0, min(i, d.K - 1) - 1);
        for (int t = lane; t < kept; t += 32) {
            const S* src = t < d.ngroups ? d.partial + ((int64_t)t * CR + i * d.R) * d.ld
                                         : d.inner + (((int64_t)i * d.C + 2 + t - d.ngroups) * d.R) * d.ld;
#pragma unroll
            for (int q = 0; q < ROWS; ++q)
#pragma unroll
                for (int r = 0; r < RM; ++r)
                    if (r < d.R && row0 + q < d.ne) v[q * RM + r] = add_sum(v[q * RM + r], src[(int64_t)r * d.ld + row0 + q]);
        }
    };
    if (sums_ready) sums();
    Acc<T> acc[ROWS][RM];
    if (i > 0) {
        int off[RM];
        const int s0 = ring_at(pos.slot, -1, d.ring) * d.R;
#pragma unroll
        for (int r = 0; r < RM; ++r) off[r] = (s0 + min(r, d.R - 1)) * d.ld;
        const T* rp[ROWS];
#pragma unroll
        for (int q = 0; q < ROWS; ++q) rp[q] = d.blocks + ((int64_t)(1 + k) * d.ne + min(row0 + q, d.ne - 1)) * d.ld;
        tile_rows<T, ROWS, RM>(rp, d.rbuf, off, RM, nvec, lane, acc, wait);
    } else {
        wait();
    }
    if (!sums_ready) sums();
#pragma unroll
    for (int q = 0; q < ROWS; ++q)
#pragma unroll
        for (int r = 0; r < RM; ++r) v[q * RM + r] = add_sum(v[q * RM + r], acc[q][r].sum());
    const S s = multi_reduce<ROWS * RM>(v, lane);
    const int id = multi_index<ROWS * RM>(lane), row = row0 + id / RM, r = id % RM;
    if (!multi_owner<ROWS * RM>(lane) || r >= d.R || row >= d.ne) return;
    if (k == 1) d.b[(int64_t)r * d.ld + row] = (T)sum_value(s);
    else d.inner[(((int64_t)(i - 1 + k) * d.C + k) * d.R + r) * d.ld + row] = s;
}

// y_n of one row: T_0^-1 b_n into the ring; wait() returns when b_n is there
template <typename T, int RM, class F>
__device__ __forceinline__ void solve_unit(const SimtDev<T>& d, const StepPos& pos, int row, int lane, F wait) {
    Acc<T> acc[1][RM];
    int off[RM];
#pragma unroll
    for (int r = 0; r < RM; ++r) off[r] = min(r, d.R - 1) * d.ld;
    const T* rp[1] = {d.t0inv + (int64_t)row * d.ld};
    tile_rows<T, 1, RM>(rp, d.b, off, RM, d.ld / VecOf<T>::W, lane, acc, wait);
    typename SumOf<T>::S v[RM];
#pragma unroll
    for (int r = 0; r < RM; ++r) v[r] = acc[0][r].sum();
    const auto s = multi_reduce<RM>(v, lane);
    const int r = multi_index<RM>(lane);
    if (multi_owner<RM>(lane) && r < d.R) d.rbuf[((int64_t)pos.slot * d.R + r) * d.ld + row] = (T)sum_value(s);
}

// ---------------------------------------------------------------- post-processing of steps p0 .. p1 - 1
// z_c = sum_j tsign[c][j] w[tedge[c][j]], w = (1/dtt - 1) y_n - y_{n-1}/dtt (y_{n-1} = 0 at n = 1)
template <typename T>
__device__ __forceinline__ double project_in_value(const DevMesh& m, int c, const T* __restrict__ yn,
                                                   const T* __restrict__ yp, bool first, double dtt) {
    double s = 0.0;
    for (int j = 0; j < 3; ++j) {
        const int e = m.tedge[3 * c + j];
        const double w = fma(1.0 / dtt - 1.0, (double)yn[e], -((first ? 0.0 : (double)yp[e]) / dtt));
        s = fma(m.tsign[3 * c + j], w, s);
    }
    return s;
}
template <typename T>
__device__ __forceinline__ void pin_value(const SimtDev<T>& d, int64_t n, int slot, int col, int r, int c) {
    const T* yn = d.rbuf + ((int64_t)slot * d.R + r) * d.ld;
    const T* yp = d.rbuf + ((int64_t)ring_at(slot, -1, d.ring) * d.R + r) * d.ld;
    d.z[(int64_t)col * d.ldc + c] = (T)project_in_value<T>(d.m, c, yn, yp, n == 1, d.dtt);
}

// u = (Sigma^T Sigma)^+ z for pre_rows rows and eight columns (col0 ..) of ncol
template <typename T>
__device__ __forceinline__ void pinv_item(const SimtDev<T>& d, int ncol, int row0, int col0, int lane) {
    constexpr int PRE_ROWS = pre_rows<T>();
    Acc<T> acc[PRE_ROWS][PRE_COLS];
    int off[PRE_COLS];
#pragma unroll
    for (int c = 0; c < PRE_COLS; ++c) off[c] = min(col0 + c, ncol - 1) * d.ldc;
    const T* row[PRE_ROWS];
#pragma unroll
    for (int i = 0; i < PRE_ROWS; ++i) row[i] = d.pinv + (int64_t)min(row0 + i, d.nc - 1) * d.ldc;
    tile_rows<T, PRE_ROWS, PRE_COLS>(row, d.z, off, min(ncol - col0, PRE_COLS), d.ldc / VecOf<T>::W, lane, acc);
    typename SumOf<T>::S v[PRE_ROWS * PRE_COLS];
#pragma unroll
    for (int i = 0; i < PRE_ROWS; ++i)
#pragma unroll
        for (int c = 0; c < PRE_COLS; ++c) v[i * PRE_COLS + c] = acc[i][c].sum();
    const auto s = multi_reduce<PRE_ROWS * PRE_COLS>(v, lane);
    const int id = multi_index<PRE_ROWS * PRE_COLS>(lane), r = row0 + id / PRE_COLS, c = col0 + id % PRE_COLS;
    if (multi_owner<PRE_ROWS * PRE_COLS>(lane) && r < d.nc && c < ncol) d.u[(int64_t)c * d.ldc + r] = (T)sum_value(s);
}

// j_n = y_n + Sigma u -> outputs; finiteness check (the first bad step is kept)
template <typename T>
__device__ __forceinline__ void pout_value(const SimtDev<T>& d, int64_t n, int slot, int col, int r, int e) {
    const T y = d.rbuf[((int64_t)slot * d.R + r) * d.ld + e];
    const T* u = d.u + (int64_t)col * d.ldc;
    const T val = y + u[d.m.cplus_[e]] - u[d.m.cminus_[e]];
    Ctl* ctl = d.ctl;
    if (!isfinite((double)val)) {
        atomicCAS(&ctl->status, 0, (int)TDCFIE_E_NONFINITE);
        atomicMin(reinterpret_cast<unsigned long long*>(&ctl->bad_step), (unsigned long long)n);
    }
    const int64_t at = ((n - ctl->n0) * d.R + r) * (int64_t)d.ne + e;
    if (ctl->out) reinterpret_cast<T*>(ctl->out)[at] = val;
    if (ctl->yout) reinterpret_cast<T*>(ctl->yout)[at] = y;
}

// Programmatic dependent launch: a kernel of a step's chain is put on the SMs while the kernel before
// it finishes; wait_prior() returns when that kernel is complete and its results are visible (at once
// in a kernel launched without the attribute), and the next kernel may be put on the SMs after it.
// What a kernel reads ahead of it was complete before the kernel in front could pass its own wait:
// matrices, the step counter (it only moves in the last kernel of a graph) and sums two kernels old.
__device__ __forceinline__ void wait_prior() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// launch with programmatic stream serialization: the kernel may be put on the SMs before the one ahead
// of it has finished (it calls wait_prior before it touches anything that one writes)
template <class... P, class... A>
static void launch_chained(void (*kernel)(P...), dim3 grid, int threads, cudaStream_t s, size_t smem, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

__device__ __forceinline__ unsigned long long device_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

constexpr uint64_t WAIT_NS = 2000000000ull;      // limit of every device-side wait

// Barrier of the nb co-resident blocks (cooperative launch) that share the counter c, which only ever
// grows; false when a wait ran out.  One atomic and one load that waits; the timer is read once in a
// thousand turns.
__device__ __forceinline__ bool group_barrier(unsigned long long* c, unsigned long long nb, unsigned long long* err,
                                              int* failed) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned long long target = (atomicAdd(c, 1ULL) / nb + 1) * nb;
        unsigned long long v, t0 = 0;
        for (unsigned spin = 1;; ++spin) {
            asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(v) : "l"(c) : "memory");
            if (v >= target) break;
            if (spin % 1024 == 0) {
                const unsigned long long t = device_ns();
                if (t0 == 0) t0 = t;
                if (t - t0 > WAIT_NS) {
                    atomicExch(err, 1ULL);
                    *failed = 1;
                    break;
                }
            }
        }
        __threadfence();
    }
    __syncthreads();
    return !*failed;
}

}  // namespace tdc
