// FP64 device assembly of the space-time matrices (Sec. II-A..C, IV-A), natural units c = eta = 1.
//
//   S_k[m,n]    = -int int f_m(x).f_n(y) hdot_0(k dt - R) / (4 pi R)
//   Phi_k[c,c'] = -T0/(A_c A_c') int_c int_c' q_0(k dt - R) / (4 pi R)
//   MM_k[m,n]   =  int int g_m(x).[Rhat x f_n(y)] (h_0(k dt - R)/(4 pi R^2) + hdot_0(k dt - R)/(4 pi R))
//   Zs[m,n]     = -kappa int int g_m.g_n exp(-kappa R)/(4 pi R)
//   Psi[v,v']   = -(1/kappa) int int rho_v rho_v' exp(-kappa R)/(4 pi R),  rho_v = 1/(2 N_v A_t) on D_v
//   M[m,n]      =  int int g_m.[Rhat x f_n] (1 + kappa R) exp(-kappa R)/(4 pi R^2)
//   G[m,n]      =  int (n x g_m).f_n
//
// Quadrature rule (same rule as the reference implementation it is checked against):
//   outer: 7-point degree-5 rule on coarse triangles, 3-point degree-2 rule on fine triangles;
//   inner: polar decomposition about the projection of the outer point on the source plane,
//     one signed sub-triangle per edge, angular variable psi = asinh(lambda/h) split where the
//     breakpoint circles R = j dt cross the edge and into pieces of width <= 1, radial variable
//     u = asinh(rho/|d|) (rho when the pair is coplanar) split at the breakpoint radii and into
//     pieces of width <= 1; NANG and NRAD Gauss-Legendre points per piece;
//   retarded pairs other than a triangle with itself, when the projection p is well outside the
//     source triangle (every vertex at least two longest edges from p): polar coordinates about
//     p over the triangle's own angular range only (two halves split at the middle vertex, angle
//     variable psi = asinh(tan(theta - theta_f)) along the nearer boundary edge, split where
//     breakpoint circles cross a boundary edge and into pieces of width <= 1), radius from the
//     near to the far edge (split at breakpoint radii, u pieces of width <= 1); otherwise the
//     signed sub-triangle form above;
//   static pairs whose coarse parents share no vertex: 3 x 3 (fine-fine) and 3 x 7 (fine-coarse)
//     product rules; same-parent pairs are coplanar (d = 0) and the curl kernel vanishes there.
// Scatter: FP64 atomicAdd (order of summation is not fixed; results agree to rounding).
#include <cmath>
#include <cstdio>

#include "internal.h"

namespace tdc {

constexpr int MAXB = 64;   // breakpoint circles across one edge whose cuts are kept in a list (more: MANY)
__constant__ double c_ax[NANG], c_aw[NANG], c_rx[NRAD], c_rw[NRAD];
__constant__ double c_r7[7][4];   // barycentric a, b, c, weight
__constant__ double c_r3[3][4];

void triangle_rule7(double r7[7][4]) {
    const double s15 = std::sqrt(15.0);
    const double a1 = (9.0 - 2.0 * s15) / 21.0, b1 = (6.0 + s15) / 21.0, w1 = (155.0 + s15) / 1200.0;
    const double a2 = (9.0 + 2.0 * s15) / 21.0, b2 = (6.0 - s15) / 21.0, w2 = (155.0 - s15) / 1200.0;
    const double t[7][4] = {{1.0 / 3, 1.0 / 3, 1.0 / 3, 9.0 / 40.0},
                            {a1, b1, b1, w1}, {b1, a1, b1, w1}, {b1, b1, a1, w1},
                            {a2, b2, b2, w2}, {b2, a2, b2, w2}, {b2, b2, a2, w2}};
    for (int q = 0; q < 7; ++q)
        for (int c = 0; c < 4; ++c) r7[q][c] = t[q][c];
}

void set_rule_tables(const RuleTables& r, cudaStream_t s) {
    cudaMemcpyToSymbolAsync(c_ax, r.ax, sizeof(r.ax), 0, cudaMemcpyHostToDevice, s);
    cudaMemcpyToSymbolAsync(c_aw, r.aw, sizeof(r.aw), 0, cudaMemcpyHostToDevice, s);
    cudaMemcpyToSymbolAsync(c_rx, r.rx, sizeof(r.rx), 0, cudaMemcpyHostToDevice, s);
    cudaMemcpyToSymbolAsync(c_rw, r.rw, sizeof(r.rw), 0, cudaMemcpyHostToDevice, s);
    // symmetric rules: degree 5 (7 points) and degree 2 (3 points)
    double r7[7][4];
    triangle_rule7(r7);
    double r3[3][4] = {{2.0 / 3, 1.0 / 6, 1.0 / 6, 1.0 / 3}, {1.0 / 6, 2.0 / 3, 1.0 / 6, 1.0 / 3},
                       {1.0 / 6, 1.0 / 6, 2.0 / 3, 1.0 / 3}};
    cudaMemcpyToSymbolAsync(c_r7, r7, sizeof(r7), 0, cudaMemcpyHostToDevice, s);
    cudaMemcpyToSymbolAsync(c_r3, r3, sizeof(r3), 0, cudaMemcpyHostToDevice, s);
}

struct V3 { double x, y, z; };
__device__ __forceinline__ V3 mk(const double* p) { return {p[0], p[1], p[2]}; }
__device__ __forceinline__ V3 operator-(V3 a, V3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ V3 operator+(V3 a, V3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ V3 operator*(double s, V3 a) { return {s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ double dot(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ V3 cross(V3 a, V3 b) { return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x}; }
__device__ __forceinline__ double nrm(V3 a) { return sqrt(dot(a, a)); }

// Temporal basis (Sec. IV-A) on one interval R in [j dt, (j + 1) dt], v = j + 1 - R / dt in [0, 1]:
// block k = j + i sees t = k dt - R = (i - 1 + v) dt, so every basis function is a polynomial in v.
//   order 1 (the hat h_0 and the C1 quadratic q_0):
//     h_0 = v, 1 - v;  dt h_0' = 1, -1;  q_0 = v^2/2, 1/2 + v - v^2, (1 - v)^2/2      (i = 0, 1, 2)
//   order 2 (the remark closing Sec. IV-B: shifted quadratic Lagrange h_0 and the q_0 with
//   q_0' = (h_0(t) - h_0(t - dt)) / dt that vanishes before -dt):
//     h_0 = v(1 + v)/2, 1 - v^2, (v^2 - v)/2;  dt h_0' = 1/2 + v, -2v, v - 1/2;
//     q_0 = v^2/4 + v^3/6, 5/12 + v - v^2/4 - v^3/2, 2/3 - v - v^2/4 + v^3/2, -1/12 + v^2/4 - v^3/6
// The retarded kernels therefore sum moments in v per interval and form the blocks' values from
// them once per thread.

// ---------------------------------------------------------------- inner quadrature, shared parts
// The FP64 pipe (2 multiply-adds per clock and SM) bounds every kernel of this file, so the rules
// are evaluated with as few FP64 operations as they allow: the nodes of a piece are reached from its
// centre by the addition formulas, cosh and sinh of the node offsets are short series, and no
// inverse function is evaluated more than once per piece.

// C = cosh t, S = sinh t by their Taylor series, |t| <= 1/2 (truncation below 2^-53; short form
// below 1/8)
__device__ __forceinline__ void cosh_sinh(double t, double& C, double& S) {
    const double z = t * t;
    double c = 1.0 / 3628800.0, s = 1.0 / 362880.0;
    if (z > 1.0 / 64) {
        c = fma(z, fma(z, 1.0 / 87178291200.0, 1.0 / 479001600.0), c);
        s = fma(z, fma(z, 1.0 / 6227020800.0, 1.0 / 39916800.0), s);
    }
    c = fma(z, c, 1.0 / 40320.0);
    c = fma(z, c, 1.0 / 720.0);
    c = fma(z, c, 1.0 / 24.0);
    c = fma(z, c, 0.5);
    C = fma(z, c, 1.0);
    s = fma(z, s, 1.0 / 5040.0);
    s = fma(z, s, 1.0 / 120.0);
    s = fma(z, s, 1.0 / 6.0);
    S = fma(t * z, s, t);
}

// atanh w for 0 <= w <= tanh(1/2)
__device__ __forceinline__ double atanh_half(double w) {
    const double z = w * w;
    if (z > 1.0 / 64) return atanh(w);
    double s = fma(z, 1.0 / 17.0, 1.0 / 15.0);
    s = fma(z, s, 1.0 / 13.0);
    s = fma(z, s, 1.0 / 11.0);
    s = fma(z, s, 1.0 / 9.0);
    s = fma(z, s, 1.0 / 7.0);
    s = fma(z, s, 1.0 / 5.0);
    s = fma(z, s, 1.0 / 3.0);
    return fma(w * z, s, w);
}

// nodes of one radial piece with centre (rc, Rc) = |d| (sinh, cosh)(u_c) and half-width h in u:
// acc.node(R, W / R, rho) (node2: two at a time), W = cw h w_g rho R
template <class ACC>
__device__ __forceinline__ void radial_nodes(double rc, double Rc, double h, double cw, ACC& acc) {
    static_assert(NRAD == 5, "symmetric five-point rule");
    const double ch = cw * h;
    acc.node(Rc, ch * c_rw[2] * rc, rc);
#pragma unroll
    for (int g = 3; g < 5; ++g) {
        double C, S;
        cosh_sinh(h * c_rx[g], C, S);
        const double a = rc * C, b = Rc * S, e = Rc * C, f = rc * S, w = ch * c_rw[g];
        acc.node2(e + f, w * (a + b), a + b, e - f, w * (a - b), a - b);
    }
}

// the piece r0 <= rho <= r1 (R0, R1 the distances of its ends) of one ray with angular weight cw:
// u = asinh(rho / |d|) in pieces of width <= PIECE, or rho itself when the pair is coplanar
template <class ACC>
__device__ __forceinline__ void radial_piece(double r0, double R0, double r1, double R1, double ad, double cw, ACC& acc) {
    static_assert(PIECE == 1.0, "one piece up to tanh(1/2)");
    if (ad > 0.0) {
        const double N = (r1 - r0) + (R1 - R0);
        const double w = N / fma(2.0, r0 + R0, N);          // tanh((u1 - u0) / 2)
        if (w <= 0.46211715726000976) {
            const double sech = sqrt(fma(-w, w, 1.0));
            radial_nodes(0.5 * (r0 + r1) * sech, 0.5 * (R0 + R1) * sech, atanh_half(w), cw, acc);
        } else {
            const double u0 = asinh(r0 / ad), u1 = asinh(r1 / ad);
            const int ns = min(max((int)ceil((u1 - u0) / PIECE), 1), 1024);
            const double h = 0.5 * (u1 - u0) / ns;
            for (int k = 0; k < ns; ++k) {
                const double uc = u0 + (2 * k + 1) * h;
                radial_nodes(ad * sinh(uc), ad * cosh(uc), h, cw, acc);
            }
        }
    } else {
        const double hw = 0.5 * (r1 - r0);
#pragma unroll
        for (int g = 0; g < NRAD; ++g) {
            const double rho = r0 + hw * (c_rx[g] + 1.0);
            acc.node(rho, cw * hw * c_rw[g], rho);
        }
    }
}

// One (outer point, source triangle) pair in the plane of the source triangle
struct Pair {
    V3 v[3], n, p;      // vertices, unit normal, projection of the outer point
    double d, ad;       // signed height of the outer point, |d|
    __device__ void set(V3 x, V3 v0, V3 v1, V3 v2, bool coplanar) {
        v[0] = v0; v[1] = v1; v[2] = v2;
        n = cross(v1 - v0, v2 - v0);
        n = (1.0 / nrm(n)) * n;
        d = coplanar ? 0.0 : dot(x - v0, n);
        ad = fabs(d);
        p = x - d * n;
    }
    // the far form applies: p outside the triangle and at least two longest edges from every vertex
    __device__ bool far() const {
        bool inside = true;
        double l2 = 0.0, v2 = 1e300;
        for (int i = 0; i < 3; ++i) {
            const V3 a = v[i] - p, b = v[(i + 1) % 3] - p, e = b - a;
            if (dot(cross(a, b), n) < 0.0) inside = false;
            l2 = fmax(l2, dot(e, e));
            v2 = fmin(v2, dot(a, a));
        }
        return !inside && v2 >= 4.0 * l2;
    }
};

// ---------------------------------------------------------------- work items of a block
// Pairs differ in the number of their angular pieces and of the intervals that a ray crosses; with
// one thread per pair only 5 to 13 lanes of a warp were active.  A block therefore works in two
// phases per round: one thread per pair finds the pair's next fan (one per edge in the near form, one
// per half in the far form) and pushes its angular sub-pieces into a queue in shared memory; then every
// thread takes sub-pieces from the queue.  A sub-piece's six rays cross the same intervals (it was split
// where the circles R = j dt cross the fan's edges), so intervals that all rays cross whole are
// integrated once instead of six times, and the sums reach the pair's interval slots (shared memory)
// with one addition per sub-piece and interval.
constexpr int AB = 128;       // threads and pairs per block
constexpr int QCAP = 512;     // queue entries; what does not fit is worked on by the thread that found it

struct Fan {                  // rays om = (f + sinh(psi) g) / cosh(psi), psi = asinh(tan(angle from f))
    V3 f, g;
    double hn;                // rays start at hn cosh(psi); 0: at the projection (near form)
    double num, ex, ey;       // far: they end at num / ((ey - sinh(psi) ex) / cosh(psi)); near: at num cosh(psi), sign ex
};

struct BlockSh {
    double fan[10][AB];       // the pairs' fans of the current round
    double d[AB];             // signed heights
    int j0[AB];               // first interval of the pair's window
    double qc[QCAP], qh[QCAP];    // centre and half-width of a sub-piece
    unsigned short qe[QCAP];      // its pair
    int qn;
    int wsum[2 * AB / 32];
    unsigned short list[AB];
};

struct Steps { double dt, inv_dt; int ni; };   // time step, intervals per window

// one angular sub-piece of pair e's fan: add its sums to the slots [interval][component][pair]
template <class ACC>
__device__ __noinline__ void work_item(const BlockSh& sh, double* slots, int e, double pc, double hh, Steps st, double kappa) {
    static_assert(NANG == 6, "symmetric six-point rule");
    const double d = sh.d[e], ad = fabs(d), d2 = d * d;
    const V3 f = {sh.fan[0][e], sh.fan[1][e], sh.fan[2][e]}, g = {sh.fan[3][e], sh.fan[4][e], sh.fan[5][e]};
    const double hn = sh.fan[6][e], num = sh.fan[7][e], ex = sh.fan[8][e], ey = sh.fan[9][e];
    double cw[6], iv[6], sn[6], r0[6], r1[6], R0[6], R1[6];
    double A = 0.0, R0min = 1e300, R0max = 0.0, R1min = 1e300, R1max = 0.0;
    V3 B = {0, 0, 0};
    const double ep = exp(pc), em = 1.0 / ep, chc = 0.5 * (ep + em), shc = 0.5 * (ep - em);
#pragma unroll 1
    for (int gg = 3; gg < 6; ++gg) {
        double C, S;
        cosh_sinh(hh * c_ax[gg], C, S);
        const double w = hn > 0.0 ? hh * c_aw[gg] : ex * hh * c_aw[gg];
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
            const int k = 2 * gg - 6 + side;
            const double Sg = side ? -S : S;
            const double ch = fma(shc, Sg, chc * C), shp = fma(chc, Sg, shc * C), inv = 1.0 / ch, si = shp * inv;
            cw[k] = w * inv;
            iv[k] = inv;
            sn[k] = si;
            r0[k] = hn * ch;
            r1[k] = hn > 0.0 ? num / (inv * ey - si * ex) : num * ch;
            R1[k] = sqrt(fma(r1[k], r1[k], d2));
            if constexpr (ACC::RETARDED) {
                R0[k] = hn > 0.0 ? sqrt(fma(r0[k], r0[k], d2)) : ad;
                A += cw[k];
                B = B + cw[k] * (inv * f + si * g);
                R0min = fmin(R0min, R0[k]);
                R0max = fmax(R0max, R0[k]);
                R1min = fmin(R1min, R1[k]);
                R1max = fmax(R1max, R1[k]);
            }
        }
    }
    ACC acc;
    if constexpr (!ACC::RETARDED) {
        acc.kappa = kappa;
        acc.begin(0, st);
#pragma unroll 1
        for (int k = 0; k < 6; ++k) {
            if (!(r1[k] > 0.0)) continue;
            acc.ray();
            radial_piece(0.0, ad, r1[k], R1[k], ad, cw[k], acc);
            acc.turn(iv[k] * f + sn[k] * g);
        }
        acc.flush(slots + e);
    } else {
        const int j0 = sh.j0[e], j1 = j0 + st.ni;
        int j = max((int)(R0min * st.inv_dt), j0);
        double Ra = j * st.dt, ra = sqrt(fmax(fma(Ra, Ra, -d2), 0.0));
        // the intervals at the near edge, those that all rays cross whole, the rest: a warp's lanes meet
        // between the three, so that one ray's work is not done beside six rays'
#pragma unroll 1
        for (int ph = 0; ph < 3; ++ph)
#pragma unroll 1
        for (; j < j1 && Ra < R1max; ++j) {
            const double Rb = (j + 1) * st.dt;
            const bool whole = Rb <= R1min && (hn == 0.0 || R0max <= Ra);
            if (ph < 2 && whole != (ph == 1)) break;
            const double rb = sqrt(fmax(fma(Rb, Rb, -d2), 0.0)), Rs = fmax(Ra, ad);
            acc.begin(j, st);
#pragma unroll 1
            for (int k = 0; k < (whole ? 1 : 6); ++k) {
                const bool in = !whole && R0[k] > Rs, out = !whole && R1[k] < Rb;
                const double a = in ? r0[k] : ra, b = out ? r1[k] : rb;
                if (!(b > a)) continue;
                acc.ray();
                radial_piece(a, in ? R0[k] : Rs, b, out ? R1[k] : Rb, ad, whole ? 1.0 : cw[k], acc);
                if (!whole) acc.turn(iv[k] * f + sn[k] * g);
            }
            if (whole) {
                acc.scale(A);
                acc.turn(B);
            }
            acc.flush(slots + (int64_t)(j - j0) * ACC::NCOMP * AB + e);
            Ra = Rb;
            ra = rb;
        }
    }
}

// a piece [P0, P1] in psi of this thread's fan, in sub-pieces of width <= PIECE
template <class ACC>
__device__ __forceinline__ void push_piece(BlockSh& sh, double* slots, double P0, double P1, Steps st, double kappa) {
    const int nsub = min(max((int)ceil((P1 - P0) / PIECE), 1), 256);     // about 75 at most on valid pairs
    const double hh = 0.5 * (P1 - P0) / nsub;
    for (int sb = 0; sb < nsub; ++sb) {
        const double pc = P0 + (2 * sb + 1) * hh;
        const int at = atomicAdd(&sh.qn, 1);
        if (at < QCAP) {
            sh.qc[at] = pc;
            sh.qh[at] = hh;
            sh.qe[at] = (unsigned short)threadIdx.x;
        } else {
            work_item<ACC>(sh, slots, threadIdx.x, pc, hh, st, kappa);
        }
    }
}

__device__ __forceinline__ void store_fan(BlockSh& sh, const Fan& F) {
    const double v[10] = {F.f.x, F.f.y, F.f.z, F.g.x, F.g.y, F.g.z, F.hn, F.num, F.ex, F.ey};
#pragma unroll
    for (int i = 0; i < 10; ++i) sh.fan[i][threadIdx.x] = v[i];
}

// insert v into the ascending list a[0..n)
__device__ __forceinline__ void insert_sorted(double* a, int& n, double v) {
    int j = n++;
    while (j > 0 && a[j - 1] > v) { a[j] = a[j - 1]; --j; }
    a[j] = v;
}

// MANY (time steps below a 62nd of the longest edge): the circles R = j dt across an edge one after another
// in the edge's direction, inwards to its foot, then outwards, without a list.  It finds each circle twice and
// pushes pieces as it goes: on meshes that need no more than the list holds, 5 % slower than the list.
struct Circles {
    int j, jin, jend;       // next circle, innermost, behind the last one outwards
    bool out;
    // distances of the outer point from the edge's start, the point nearest to it and the end; whether
    // that point is the start or the end
    __device__ void set(double R0, double Rmin, double R1, bool start, bool end, double inv_dt) {
        out = start;
        jin = (int)(Rmin * inv_dt);
        j = start ? jin : (int)(R0 * inv_dt) + 1;
        jend = end ? jin : (int)(R1 * inv_dt) + 2;
    }
    // false: no more; inwards: the crossing lies before the foot
    __device__ bool next(int& circle, bool& inwards) {
        if (!out && j < jin) {
            out = true;
            j = jin;
        }
        if (out && j >= jend) return false;
        inwards = !out;
        circle = out ? j++ : j--;
        return true;
    }
};

// Polar rule about p: one signed sub-triangle (fan) per edge; round s is edge s
template <class ACC, bool MANY>
__device__ void push_near(BlockSh& sh, double* slots, int s, const Pair& P, Steps st, double kappa) {
    const V3 a = P.v[s], b = P.v[s == 2 ? 0 : s + 1];
    const V3 ab = b - a;
    const double L = nrm(ab);
    const V3 e = (1.0 / L) * ab;
    const double sig = dot(cross(a - P.p, b - P.p), P.n);
    if (sig == 0.0) return;
    const double t = dot(P.p - a, e);
    const V3 nu = a + t * e - P.p;
    const double h = nrm(nu);
    if (h <= 1e-14 * L) return;
    store_fan(sh, Fan{(1.0 / h) * nu, e, 0.0, h, sig > 0.0 ? 1.0 : -1.0, 1.0});
    const double psa = asinh(-t / h), psb = asinh((L - t) / h), d2 = P.d * P.d;
    double P0 = psa;
    if constexpr (ACC::RETARDED && MANY) {
        const double m2 = fma(h, h, d2), R0 = sqrt(fma(t, t, m2)), R1 = sqrt(fma(L - t, L - t, m2));
        Circles cir;
        cir.set(R0, t < 0.0 ? R0 : t > L ? R1 : sqrt(m2), R1, t < 0.0, t > L, st.inv_dt);
        int j;
        for (bool inwards; cir.next(j, inwards);) {
            const double R = j * st.dt, r2 = fma(R, R, -d2);
            if (!(r2 > h * h)) continue;
            const double c = acosh(sqrt(r2) / h), P1 = inwards ? -c : c;
            if (P1 > P0 && P1 < psb) {
                push_piece<ACC>(sh, slots, P0, P1, st, kappa);
                P0 = P1;
            }
        }
        if (psb > P0) push_piece<ACC>(sh, slots, P0, psb, st, kappa);
        return;
    }
    double sp[2 * MAXB + 2];
    int nsp = 0;
    if constexpr (ACC::RETARDED) {
        // breakpoint circles that cross the edge: between its foot and its farther end
        const double m = fmax(fabs(t), fabs(L - t));
        const double hi = sqrt(fma(m, m, fma(h, h, d2)));
        int j = (int)(sqrt(fma(h, h, d2)) * st.inv_dt);
        for (int nb = 0; nb < MAXB && j * st.dt < hi; ++j) {
            const double R = j * st.dt, r2 = fma(R, R, -d2);
            if (!(r2 > h * h)) continue;
            ++nb;
            const double c = acosh(sqrt(r2) / h);
            if (-c > psa && -c < psb) insert_sorted(sp, nsp, -c);
            if (c > psa && c < psb) insert_sorted(sp, nsp, c);
        }
    }
    for (int pc = 0; pc <= nsp; ++pc) {
        const double P1 = pc < nsp ? sp[pc] : psb;
        if (P1 > P0) push_piece<ACC>(sh, slots, P0, P1, st, kappa);
        P0 = P1;
    }
}

__device__ __forceinline__ double cr2(double ax, double ay, double bx, double by) { return ax * by - ay * bx; }

// Far form: polar coordinates about p over the triangle's own angular range (no signed
// cancellation), one fan per half.  Angles are measured from the foot of the half's near edge and
// carried as asinh(tan(angle)) = asinh(cross / dot), so that no angle itself is formed.  Round
// half is one half.
template <class ACC, bool MANY>
__device__ void push_far(BlockSh& sh, double* slots, int half, const Pair& P, Steps st) {
    V3 g = (1.0 / 3.0) * (P.v[0] + P.v[1] + P.v[2]) - P.p;
    const V3 u = (1.0 / nrm(g)) * g, w = cross(P.n, u);
    double X[3], Y[3];
    for (int i = 0; i < 3; ++i) {
        X[i] = dot(P.v[i] - P.p, u);
        Y[i] = dot(P.v[i] - P.p, w);
    }
    // by angle: the triangle subtends less than a half turn, so the sign of the cross product orders
    for (int i = 1; i < 3; ++i)
        for (int k = i; k > 0; --k)
            if (cr2(X[k - 1], Y[k - 1], X[k], Y[k]) < 0.0) {
                double t = X[k]; X[k] = X[k - 1]; X[k - 1] = t;
                t = Y[k]; Y[k] = Y[k - 1]; Y[k - 1] = t;
            }
    const double d2 = P.d * P.d;
    // the half between vertex half and vertex half + 1; its edges: that pair's and the long one (0, 2)
    const double x0 = X[half], y0 = Y[half], x1 = X[half + 1], y1 = Y[half + 1];
    if (!(cr2(x0, y0, x1, y1) > 0.0)) return;
    const double lx = X[2] - X[0], ly = Y[2] - Y[0], sx = x1 - x0, sy = y1 - y0;
    const double nl = cr2(X[0], Y[0], lx, ly), nsh = cr2(x0, y0, sx, sy);
    const double i0 = 1.0 / sqrt(x0 * x0 + y0 * y0), i1 = 1.0 / sqrt(x1 * x1 + y1 * y1);
    const double mx = i0 * x0 + i1 * x1, my = i0 * y0 + i1 * y1;     // along the bisector
    const bool lnear = nl / cr2(mx, my, lx, ly) < nsh / cr2(mx, my, sx, sy);
    const double ax = lnear ? X[0] : x0, ay = lnear ? Y[0] : y0;
    const double ndx = lnear ? lx : sx, ndy = lnear ? ly : sy;
    const double tf = -(ax * ndx + ay * ndy) / (ndx * ndx + ndy * ndy);
    const double fx = ax + tf * ndx, fy = ay + tf * ndy;
    const double hn = sqrt(fx * fx + fy * fy);
    if (!(hn > 0.0)) return;
    const double cf = fx / hn, sf = fy / hn;
    auto angle = [&](double vx, double vy) { return asinh((cf * vy - sf * vx) / (cf * vx + sf * vy)); };
    const double S0 = angle(x0, y0), S1 = angle(x1, y1);
    const double fdx = lnear ? sx : lx, fdy = lnear ? sy : ly;       // far edge
    store_fan(sh, Fan{cf * u + sf * w, cf * w - sf * u, hn, lnear ? nsh : nl, cf * fdx + sf * fdy, cf * fdy - sf * fdx});
    double P0 = S0;
    if constexpr (MANY) {
        // both edges run by ascending angle: a cut is the nearer of their next crossings
        Circles cir[2];
        for (int ei = 0; ei < 2; ++ei) {
            const double bx = ei ? x0 : X[0], by = ei ? y0 : Y[0], dx = ei ? sx : lx, dy = ei ? sy : ly;
            const double dd = dx * dx + dy * dy, bq = bx * dx + by * dy, aa = bx * bx + by * by, ee = aa + 2.0 * bq + dd;
            const double foot = bq < 0.0 && -bq < dd ? aa - bq * bq / dd : fmin(aa, ee);
            cir[ei].set(sqrt(aa + d2), sqrt(fmax(foot, 0.0) + d2), sqrt(fmax(ee, 0.0) + d2), bq >= 0.0, -bq >= dd, st.inv_dt);
        }
        auto crossing = [&](int ei) {       // the edge's next one inside the half, S1 if there is none
            const double bx = ei ? x0 : X[0], by = ei ? y0 : Y[0], dx = ei ? sx : lx, dy = ei ? sy : ly;
            const double dd = dx * dx + dy * dy, bq = bx * dx + by * dy, aa = bx * bx + by * by;
            int j;
            for (bool inwards; cir[ei].next(j, inwards);) {
                const double R = j * st.dt, r2 = fma(R, R, -d2);
                if (!(r2 > 0.0)) continue;
                const double disc = bq * bq - dd * (aa - r2);
                if (disc <= 0.0) continue;
                const double sq = sqrt(disc), ts = (inwards ? -bq - sq : sq - bq) / dd;
                if (ts <= 0.0 || ts >= 1.0) continue;
                const double S = angle(bx + ts * dx, by + ts * dy);
                if (S > S0 && S < S1) return S;
            }
            return S1;
        };
        for (double s0 = crossing(0), s1 = crossing(1); P0 < S1;) {
            const double P1 = fmin(s0, s1);
            if (P1 > P0) {
                push_piece<ACC>(sh, slots, P0, P1, st, 0.0);
                P0 = P1;
            }
            if (!(P1 < S1)) break;
            if (s0 <= s1) s0 = crossing(0);
            else s1 = crossing(1);
        }
        return;
    }
    double sp[4 * MAXB + 2];
    int nsp = 0;
#pragma unroll 1
    for (int ei = 0; ei < 2; ++ei) {
        const double bx = ei ? x0 : X[0], by = ei ? y0 : Y[0], dx = ei ? sx : lx, dy = ei ? sy : ly;
        const double dd = dx * dx + dy * dy, bq = bx * dx + by * dy, aa = bx * bx + by * by;
        // the edge's distances from the outer point lie between its foot (or ends) and its farther end
        const double ee = aa + 2.0 * bq + dd, foot = bq < 0.0 && -bq < dd ? aa - bq * bq / dd : fmin(aa, ee);
        const double hi = sqrt(fmax(aa, ee) + d2);
        int j = (int)(sqrt(fmax(foot, 0.0) + d2) * st.inv_dt);
        for (int nb = 0; nb < MAXB && j * st.dt < hi; ++j, ++nb) {
            const double R = j * st.dt, r2 = fma(R, R, -d2);
            if (!(r2 > 0.0)) continue;
            const double disc = bq * bq - dd * (aa - r2);
            if (disc <= 0.0) continue;
            const double sq = sqrt(disc);
            for (int k = 0; k < 2; ++k) {
                const double ts = (k ? sq - bq : -bq - sq) / dd;
                if (ts <= 0.0 || ts >= 1.0) continue;
                const double S = angle(bx + ts * dx, by + ts * dy);
                if (S > S0 && S < S1) insert_sorted(sp, nsp, S);
            }
        }
    }
    for (int pc = 0; pc <= nsp; ++pc) {
        const double P1 = pc < nsp ? sp[pc] : S1;
        if (P1 > P0) push_piece<ACC>(sh, slots, P0, P1, st, 0.0);
        P0 = P1;
    }
}

// the block's rounds for one window: kind 0 near, 1 far, other: no pair on this thread
template <class ACC, bool MANY>
__device__ __forceinline__ void run_rounds(BlockSh& sh, double* slots, int kind, const Pair& P, Steps st, double kappa) {
    const int rounds = __syncthreads_or(kind == 0) ? 3 : 2;
    for (int s = 0; s < rounds; ++s) {
        if (threadIdx.x == 0) sh.qn = 0;
        __syncthreads();
        if (kind == 0) push_near<ACC, MANY>(sh, slots, s, P, st, kappa);
        else if (ACC::RETARDED && kind == 1 && s < 2) push_far<ACC, MANY>(sh, slots, s, P, st);
        __syncthreads();
        const int n = min(sh.qn, QCAP);
        for (int i = threadIdx.x; i < n; i += AB) work_item<ACC>(sh, slots, sh.qe[i], sh.qc[i], sh.qh[i], st, kappa);
        __syncthreads();
    }
}

// Order of a block's pairs by form, so that warps hold one form: near pairs first, then far ones;
// kind 2 is left out.  Pair i of the block is list[i]; the numbers of near pairs and of all pairs
// come back.
__device__ __forceinline__ int sort_pairs(int kind, BlockSh& sh, int& nnear) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned mn = __ballot_sync(0xffffffffu, kind == 0), mf = __ballot_sync(0xffffffffu, kind == 1);
    if (lane == 0) { sh.wsum[warp] = __popc(mn); sh.wsum[AB / 32 + warp] = __popc(mf); }
    __syncthreads();
    int bn = 0, bf = 0, tn = 0, tf = 0;
    for (int w = 0; w < AB / 32; ++w) {
        if (w < warp) { bn += sh.wsum[w]; bf += sh.wsum[AB / 32 + w]; }
        tn += sh.wsum[w];
        tf += sh.wsum[AB / 32 + w];
    }
    const unsigned below = (1u << lane) - 1u;
    if (kind == 0) sh.list[bn + __popc(mn & below)] = (unsigned short)threadIdx.x;
    if (kind == 1) sh.list[tn + bf + __popc(mf & below)] = (unsigned short)threadIdx.x;
    __syncthreads();
    nnear = tn;
    return tn + tf;
}

__device__ __forceinline__ V3 tri_pt(const double (*r)[4], int q, V3 a, V3 b, V3 c) {
    return r[q][0] * a + r[q][1] * b + r[q][2] * c;
}
__device__ __forceinline__ double tri_area(V3 a, V3 b, V3 c) { return 0.5 * nrm(cross(b - a, c - a)); }

// distance bounds from x, at height ad over the source plane, to the triangle:
// lower = max(ad, min vertex distance - longest edge)
__device__ __forceinline__ void dist_bounds(V3 x, V3 a, V3 b, V3 c, double ad, double& lo, double& hi) {
    const double da = nrm(x - a), db = nrm(x - b), dc = nrm(x - c);
    const double L = fmax(nrm(b - a), fmax(nrm(c - b), nrm(a - c)));
    lo = fmax(ad, fmin(da, fmin(db, dc)) - L);
    lo = fmax(lo, 0.0);
    hi = fmax(da, fmax(db, dc));
}

// lags whose support meets the distances [lo, hi]
__device__ __forceinline__ void lag_range(double lo, double hi, double dt, int K, int order, int& klo, int& khi) {
    klo = max(0, (int)floor(lo / dt) - 1);
    khi = min(K - 1, (int)ceil(hi / dt) + order + 1);
}

// Shared memory of a pair kernel: BlockSh, then the interval slots [ni][NCOMP][AB]
extern __shared__ double dyn_sh[];
__device__ __forceinline__ BlockSh& block_sh() { return *reinterpret_cast<BlockSh*>(dyn_sh); }
constexpr size_t SLOT0 = (sizeof(BlockSh) + 7) / 8;
static size_t pair_smem(int ncomp, int ni) { return 8 * (SLOT0 + (size_t)ncomp * ni * AB); }

// ------------------------------------------------------------------ retarded EFIE
template <int ORDER>
struct EfieAcc {
    static constexpr bool RETARDED = true;
    static constexpr int NS = ORDER + 2, NV = ORDER, NCOMP = NS + 3 * NV;
    double inv_dt, jp;
    double c[NS], r[NV];     // sum W / R v^p; of the current ray sum W / R rho v^p
    V3 v[NV];                // sum of r over the rays, times om
    __device__ __forceinline__ void begin(int j, Steps st) {
        inv_dt = st.inv_dt;
        jp = j + 1;
#pragma unroll
        for (int p = 0; p < NS; ++p) c[p] = 0.0;
#pragma unroll
        for (int p = 0; p < NV; ++p) v[p] = {0, 0, 0};
    }
    __device__ __forceinline__ void ray() {
#pragma unroll
        for (int p = 0; p < NV; ++p) r[p] = 0.0;
    }
    __device__ __forceinline__ void node(double R, double Wr, double rho) {
        const double x = fma(-R, inv_dt, jp);
        double t = Wr;
        c[0] += t;
#pragma unroll
        for (int p = 1; p < NS; ++p) { t *= x; c[p] += t; }
        r[0] = fma(Wr, rho, r[0]);
        if constexpr (NV == 2) r[1] = fma(Wr * rho, x, r[1]);
    }
    __device__ __forceinline__ void node2(double Ra, double Wa, double rhoa, double Rb, double Wb, double rhob) {
        node(Ra, Wa, rhoa);
        node(Rb, Wb, rhob);
    }
    __device__ __forceinline__ void turn(V3 om) {
#pragma unroll
        for (int p = 0; p < NV; ++p) v[p] = v[p] + r[p] * om;
    }
    __device__ __forceinline__ void scale(double A) {
#pragma unroll
        for (int p = 0; p < NS; ++p) c[p] *= A;
    }
    __device__ __forceinline__ void flush(double* slot) const {
#pragma unroll
        for (int p = 0; p < NS; ++p) atomicAdd(slot + p * AB, c[p]);
#pragma unroll
        for (int p = 0; p < NV; ++p) {
            atomicAdd(slot + (NS + 3 * p) * AB, v[p].x);
            atomicAdd(slot + (NS + 3 * p + 1) * AB, v[p].y);
            atomicAdd(slot + (NS + 3 * p + 2) * AB, v[p].z);
        }
    }
    // from a pair's slots: sums of dt h_0'(t) W / R (scalar and times y - x) and of q_0(t) W / R for
    // the lag whose interval k - i is slot l - i
    __device__ static void lag(const double* slots, int l, const Pair& P, double& s0, V3& s1, double& q) {
        s0 = q = 0.0;
        V3 v = {0, 0, 0};
#pragma unroll
        for (int i = 0; i <= ORDER + 1; ++i) {
            const double* s = slots + (int64_t)(l - i) * NCOMP * AB;
            auto vec = [&](int p) { return V3{s[(NS + 3 * p) * AB], s[(NS + 3 * p + 1) * AB], s[(NS + 3 * p + 2) * AB]}; };
            if constexpr (ORDER == 1) {
                const double a = s[0], b = s[AB], c = s[2 * AB];
                q += i == 0 ? 0.5 * c : i == 1 ? 0.5 * a + b - c : 0.5 * a - b + 0.5 * c;
                if (i < 2) {
                    const double g = i == 0 ? 1.0 : -1.0;
                    s0 += g * a;
                    v = v + g * vec(0);
                }
            } else {
                const double a0 = i == 0 ? 0.0 : i == 1 ? 5.0 / 12 : i == 2 ? 2.0 / 3 : -1.0 / 12, a1 = i == 1 ? 1.0 : i == 2 ? -1.0 : 0.0;
                const double a2 = i == 0 || i == 3 ? 0.25 : -0.25, a3 = i == 0 ? 1.0 / 6 : i == 1 ? -0.5 : i == 2 ? 0.5 : -1.0 / 6;
                q += a0 * s[0] + a1 * s[AB] + a2 * s[2 * AB] + a3 * s[(NS - 1) * AB];
                if (i < 3) {
                    const double g0 = i == 0 ? 0.5 : i == 1 ? 0.0 : -0.5, g1 = i == 1 ? -2.0 : 1.0;
                    s0 += g0 * s[0] + g1 * s[AB];
                    v = v + g0 * vec(0) + g1 * vec(NV - 1);
                }
            }
        }
        s1 = v - (s0 * P.d) * P.n;
    }
};

// What bounds the retarded kernels is the FP64 pipe (a radial piece is some 120 operations, a near
// pair has about 30 of them), so the lanes have to be full and nothing may be computed twice; the
// queue of sub-pieces above is for that.  The sums of an interval of length dt are moments in v,
// turned into lags at the end, so that a node costs its own few multiply-adds whatever the number of
// lags.  Pairs that meet more than lagw lags take them in several windows.  480-edge sphere, 7 lags: the
// whole assembly 1524 -> 178 ms against one thread per pair, with the rays' intervals one by one and library
// functions at every node.
template <int ORDER, bool MANY>
__global__ void __launch_bounds__(AB) k_retarded_efie(DevMesh m, double dt, int K, int lagw, double T0, double* __restrict__ S,
                                                      double* __restrict__ Phi) {
    using ACC = EfieAcc<ORDER>;
    BlockSh& sh = block_sh();
    double* slots = dyn_sh + SLOT0;
    const int64_t total = (int64_t)m.nc * 7 * m.nc;
    Pair P;
    int c = 0, c2 = 0, q = 0;
    V3 x, wv[3];
    auto load = [&](int64_t it) {
        c2 = (int)(it % m.nc);
        const int64_t rest = it / m.nc;
        q = (int)(rest % 7);
        c = (int)(rest / 7);
        for (int i = 0; i < 3; ++i) wv[i] = mk(m.V + 3 * m.F[3 * c + i]);
        x = tri_pt(c_r7, q, wv[0], wv[1], wv[2]);
        P.set(x, mk(m.V + 3 * m.F[3 * c2]), mk(m.V + 3 * m.F[3 * c2 + 1]), mk(m.V + 3 * m.F[3 * c2 + 2]), c == c2);
    };
    const int64_t it = (int64_t)blockIdx.x * AB + threadIdx.x;
    int kind = 2, nnear;
    if (it < total) {
        load(it);
        kind = c != c2 && P.far() ? 1 : 0;
    }
    const int npairs = sort_pairs(kind, sh, nnear), tid = threadIdx.x;
    kind = tid < nnear ? 0 : tid < npairs ? 1 : 2;
    const Steps st{dt, 1.0 / dt, lagw + ORDER + 1};
    double A = 0.0, A2 = 0.0, wx = 0.0;
    int k0 = 0, khi = -1;
    if (kind < 2) {
        load((int64_t)blockIdx.x * AB + sh.list[tid]);
        A = tri_area(wv[0], wv[1], wv[2]);
        A2 = tri_area(P.v[0], P.v[1], P.v[2]);
        wx = c_r7[q][3] * A;
        double lo, hi;
        dist_bounds(x, P.v[0], P.v[1], P.v[2], P.ad, lo, hi);
        lag_range(lo, hi, dt, K, ORDER, k0, khi);
        sh.d[tid] = P.d;
    }
    const double fs = -1.0 / (4.0 * M_PI * dt), fq = -T0 / (4.0 * M_PI);
    for (; __syncthreads_or(k0 <= khi); k0 += lagw) {
        const int kd = k0 <= khi ? kind : 2;
        sh.j0[tid] = k0 - ORDER - 1;
        for (int i = 0; i < st.ni * ACC::NCOMP; ++i) slots[i * AB + tid] = 0.0;
        run_rounds<ACC, MANY>(sh, slots, kd, P, st, 0.0);
        if (kd == 2) continue;
        const int nk = min(lagw, khi - k0 + 1);
        for (int l = 0; l < nk; ++l) {
            const int k = k0 + l;
            double s0, qv;
            V3 s1;
            ACC::lag(slots + tid, l + ORDER + 1, P, s0, s1, qv);
            if (qv != 0.0) atomicAdd(Phi + ((int64_t)k * m.nc + c) * m.nc + c2, wx * fq * qv / (A * A2));
            if (s0 == 0.0 && s1.x == 0.0 && s1.y == 0.0 && s1.z == 0.0) continue;
            for (int jj = 0; jj < 3; ++jj) {
                const V3 Iy = (fs * m.tsign[3 * c2 + jj] / (2.0 * A2)) * (s1 + s0 * (x - P.v[jj]));
                const int n = m.tedge[3 * c2 + jj];
                for (int ii = 0; ii < 3; ++ii) {
                    const V3 Lx = (m.tsign[3 * c + ii] / (2.0 * A)) * (x - wv[ii]);
                    atomicAdd(S + ((int64_t)k * m.ne + m.tedge[3 * c + ii]) * m.ne + n, wx * dot(Lx, Iy));
                }
            }
        }
    }
}

// ------------------------------------------------------------------ retarded MFIE
// (h_0 / R + h_0') / (4 pi R^2) W (y - x): with R = (j + 1 - v) dt both terms share W / R^3, times
//   order 1: j + 1, -j;   order 2: (j + 1)(1/2 + v) - v^2/2, 1 - 2 (j + 1) v + v^2, (j + 1)(v - 1/2) - v^2/2
template <int ORDER>
struct MfieAcc {
    static constexpr bool RETARDED = true;
    static constexpr int NB = ORDER == 1 ? 1 : 3, NCOMP = 4 * NB;
    double inv_dt, jp;
    double c[NB], r[NB];     // sum W / R^3 v^p; of the current ray sum W / R^3 rho v^p
    V3 v[NB];
    __device__ __forceinline__ void begin(int j, Steps st) {
        inv_dt = st.inv_dt;
        jp = j + 1;
#pragma unroll
        for (int p = 0; p < NB; ++p) { c[p] = 0.0; v[p] = {0, 0, 0}; }
    }
    __device__ __forceinline__ void ray() {
#pragma unroll
        for (int p = 0; p < NB; ++p) r[p] = 0.0;
    }
    __device__ __forceinline__ void add(double R, double t, double rho) {
#pragma unroll
        for (int p = 0; p < NB; ++p) {
            if (p) t *= fma(-R, inv_dt, jp);
            c[p] += t;
            r[p] = fma(t, rho, r[p]);
        }
    }
    __device__ __forceinline__ void node(double R, double Wr, double rho) { add(R, Wr / (R * R), rho); }
    // one division for two nodes
    __device__ __forceinline__ void node2(double Ra, double Wa, double rhoa, double Rb, double Wb, double rhob) {
        const double qa = Ra * Ra, qb = Rb * Rb, inv = 1.0 / (qa * qb);
        add(Ra, Wa * (qb * inv), rhoa);
        add(Rb, Wb * (qa * inv), rhob);
    }
    __device__ __forceinline__ void turn(V3 om) {
#pragma unroll
        for (int p = 0; p < NB; ++p) v[p] = v[p] + r[p] * om;
    }
    __device__ __forceinline__ void scale(double A) {
#pragma unroll
        for (int p = 0; p < NB; ++p) c[p] *= A;
    }
    __device__ __forceinline__ void flush(double* slot) const {
#pragma unroll
        for (int p = 0; p < NB; ++p) {
            atomicAdd(slot + 4 * p * AB, c[p]);
            atomicAdd(slot + (4 * p + 1) * AB, v[p].x);
            atomicAdd(slot + (4 * p + 2) * AB, v[p].y);
            atomicAdd(slot + (4 * p + 3) * AB, v[p].z);
        }
    }
    // sum over the pair of (h_0 + R h_0') W / R^3 (y - x) for lag k, interval k - i in slot l - i
    __device__ static V3 lag(const double* slots, int l, int k, const Pair& P) {
        double s = 0.0;
        V3 v = {0, 0, 0};
#pragma unroll
        for (int i = 0; i <= ORDER; ++i) {
            const double* b = slots + (int64_t)(l - i) * NCOMP * AB;
            const double J = k - i + 1;
            const double g[3] = {ORDER == 1 ? (i == 0 ? J : 1.0 - J) : (i == 0 ? 0.5 * J : i == 1 ? 1.0 : -0.5 * J),
                                 i == 1 ? -2.0 * J : J, i == 1 ? 1.0 : -0.5};
#pragma unroll
            for (int p = 0; p < NB; ++p) {
                s += g[p] * b[4 * p * AB];
                v = v + g[p] * V3{b[(4 * p + 1) * AB], b[(4 * p + 2) * AB], b[(4 * p + 3) * AB]};
            }
        }
        return v - (s * P.d) * P.n;
    }
};

template <int ORDER, bool MANY>
__global__ void __launch_bounds__(AB) k_retarded_mfie(DevMesh m, double dt, int K, int lagw, double* __restrict__ MM) {
    using ACC = MfieAcc<ORDER>;
    BlockSh& sh = block_sh();
    double* slots = dyn_sh + SLOT0;
    const int64_t total = (int64_t)m.nf * 3 * m.nc;
    Pair P;
    int t = 0, c2 = 0, q = 0;
    V3 x, wv[3];
    auto load = [&](int64_t it) {
        c2 = (int)(it % m.nc);
        const int64_t rest = it / m.nc;
        q = (int)(rest % 3);
        t = (int)(rest / 3);
        for (int i = 0; i < 3; ++i) wv[i] = mk(m.fV + 3 * m.fF[3 * t + i]);
        x = tri_pt(c_r3, q, wv[0], wv[1], wv[2]);
        P.set(x, mk(m.V + 3 * m.F[3 * c2]), mk(m.V + 3 * m.F[3 * c2 + 1]), mk(m.V + 3 * m.F[3 * c2 + 2]), false);
    };
    const int64_t it = (int64_t)blockIdx.x * AB + threadIdx.x;
    int kind = 2, nnear;
    if (it < total) {
        load(it);
        if (m.fparent[t] != c2) kind = P.far() ? 1 : 0;   // coplanar: the curl kernel vanishes
    }
    const int npairs = sort_pairs(kind, sh, nnear), tid = threadIdx.x;
    kind = tid < nnear ? 0 : tid < npairs ? 1 : 2;
    const Steps st{dt, 1.0 / dt, lagw + ORDER};
    double A = 0.0, A2 = 0.0, wx = 0.0;
    int k0 = 0, khi = -1;
    if (kind < 2) {
        load((int64_t)blockIdx.x * AB + sh.list[tid]);
        A = tri_area(wv[0], wv[1], wv[2]);
        A2 = tri_area(P.v[0], P.v[1], P.v[2]);
        wx = c_r3[q][3] * A / (4.0 * M_PI);
        double lo, hi;
        dist_bounds(x, P.v[0], P.v[1], P.v[2], P.ad, lo, hi);
        lag_range(lo, hi, dt, K, ORDER, k0, khi);
        sh.d[tid] = P.d;
    }
    for (; __syncthreads_or(k0 <= khi); k0 += lagw) {
        const int kd = k0 <= khi ? kind : 2;
        sh.j0[tid] = k0 - ORDER;
        for (int i = 0; i < st.ni * ACC::NCOMP; ++i) slots[i * AB + tid] = 0.0;
        run_rounds<ACC, MANY>(sh, slots, kd, P, st, 0.0);
        if (kd == 2) continue;
        const int nk = min(lagw, khi - k0 + 1);
        for (int l = 0; l < nk; ++l) {
            const int k = k0 + l;
            const V3 m1 = ACC::lag(slots + tid, l + ORDER, k, P);
            if (m1.x == 0.0 && m1.y == 0.0 && m1.z == 0.0) continue;
            double val[3][3];   // [local outer field i][inner edge jj]
            for (int jj = 0; jj < 3; ++jj) {
                const V3 cr = (m.tsign[3 * c2 + jj] / (2.0 * A2)) * cross(x - P.v[jj], m1);
                for (int ii = 0; ii < 3; ++ii) val[ii][jj] = wx * dot((1.0 / (2.0 * A)) * (x - wv[ii]), cr);
            }
            for (int e = m.bc_ptr[t]; e < m.bc_ptr[t + 1]; ++e) {
                const int fn = m.bc_fn[e];
                const double* ph = m.bc_phi + 3 * e;
                for (int jj = 0; jj < 3; ++jj) {
                    const double v = ph[0] * val[0][jj] + ph[1] * val[1][jj] + ph[2] * val[2][jj];
                    if (v != 0.0) atomicAdd(MM + ((int64_t)k * m.ne + fn) * m.ne + m.tedge[3 * c2 + jj], v);
                }
            }
        }
    }
}

// ------------------------------------------------------------------ static matrices
// sums of W exp(-kappa R) / R, or (M) W (1 + kappa R) exp(-kappa R) / R^3, scalar and times rho om
template <bool M>
struct YukAcc {
    static constexpr bool RETARDED = false;
    static constexpr int NCOMP = 4;
    double kappa, c, r;
    V3 v;
    __device__ __forceinline__ void begin(int, Steps) { c = 0.0; v = {0, 0, 0}; }
    __device__ __forceinline__ void ray() { r = 0.0; }
    __device__ __forceinline__ void node(double R, double Wr, double rho) {
        double g = Wr * exp(-kappa * R);
        if constexpr (M) g *= fma(kappa, R, 1.0) / (R * R);
        c += g;
        r = fma(g, rho, r);
    }
    __device__ __forceinline__ void node2(double Ra, double Wa, double rhoa, double Rb, double Wb, double rhob) {
        node(Ra, Wa, rhoa);
        node(Rb, Wb, rhob);
    }
    __device__ __forceinline__ void turn(V3 om) { v = v + r * om; }
    __device__ __forceinline__ void flush(double* slot) const {
        atomicAdd(slot, c);
        atomicAdd(slot + AB, v.x);
        atomicAdd(slot + 2 * AB, v.y);
        atomicAdd(slot + 3 * AB, v.z);
    }
    // near form of the pair of this thread (valid: it has one): sums / (4 pi)
    __device__ static void run(bool valid, const Pair& P, double kappa, double& z0, V3& z1) {
        BlockSh& sh = block_sh();
        double* slots = dyn_sh + SLOT0;
        const int t = threadIdx.x;
        if (valid) sh.d[t] = P.d;
#pragma unroll
        for (int i = 0; i < NCOMP; ++i) slots[i * AB + t] = 0.0;
        run_rounds<YukAcc, false>(sh, slots, valid ? 0 : 2, P, Steps{0.0, 0.0, 1}, kappa);
        const double f = 1.0 / (4.0 * M_PI);
        z0 = f * slots[t];
        z1 = f * (V3{slots[AB + t], slots[2 * AB + t], slots[3 * AB + t]} - (slots[t] * P.d) * P.n);
    }
};

__device__ __forceinline__ bool parents_touch(const int* F, int a, int b) {
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            if (F[3 * a + i] == F[3 * b + j]) return true;
    return false;
}

// I[i][j] += wx (x - w_i) . (z1 + z0 (x - v_j)) / (4 A A2)
__device__ __forceinline__ void add_moments(double I[3][3], V3 x, const V3* w, const V3* v, double f, double z0, V3 z1) {
    for (int j = 0; j < 3; ++j) {
        const V3 Iy = f * (z1 + z0 * (x - v[j]));
        for (int i = 0; i < 3; ++i) I[i][j] += dot(x - w[i], Iy);
    }
}

// the pair's moments into Psi and Zs
__device__ __forceinline__ void scatter_zs(const DevMesh& m, double kappa, int t, int t2, double A, double A2,
                                           const double I[3][3], double Is, double* Zs, double* Psi) {
    const double rv = 1.0 / (2.0 * m.valence[m.fvert[t]] * A), rv2 = 1.0 / (2.0 * m.valence[m.fvert[t2]] * A2);
    atomicAdd(Psi + (int64_t)m.fvert[t] * m.nv + m.fvert[t2], -(1.0 / kappa) * rv * rv2 * Is);
    for (int e1 = m.bc_ptr[t]; e1 < m.bc_ptr[t + 1]; ++e1) {
        const double* p1 = m.bc_phi + 3 * e1;
        double u[3];
        for (int j = 0; j < 3; ++j) u[j] = -kappa * (p1[0] * I[0][j] + p1[1] * I[1][j] + p1[2] * I[2][j]);
        for (int e2 = m.bc_ptr[t2]; e2 < m.bc_ptr[t2 + 1]; ++e2) {
            const double* p2 = m.bc_phi + 3 * e2;
            atomicAdd(Zs + (int64_t)m.bc_fn[e1] * m.ne + m.bc_fn[e2], p2[0] * u[0] + p2[1] * u[1] + p2[2] * u[2]);
        }
    }
}

// Zs and Psi, pairs whose parents touch (polar rule): one thread per (outer fine triangle, point,
// inner fine triangle), from the list of touching parents; 36 x 3 per pair of parents
__global__ void __launch_bounds__(AB) k_static_efie_near(DevMesh m, double kappa, double* __restrict__ Zs, double* __restrict__ Psi) {
    const int64_t u = (int64_t)blockIdx.x * AB + threadIdx.x;
    const bool valid = u < (int64_t)m.ntouch * 108;
    const int64_t r = valid ? u / 3 : 0;
    const int q = valid ? (int)(u % 3) : 0;
    const int pa = m.touch[2 * (r / 36)], pb = m.touch[2 * (r / 36) + 1];
    const int t = 6 * pa + (int)(r % 36) / 6, t2 = 6 * pb + (int)(r % 6);
    const V3 w[3] = {mk(m.fV + 3 * m.fF[3 * t]), mk(m.fV + 3 * m.fF[3 * t + 1]), mk(m.fV + 3 * m.fF[3 * t + 2])};
    const V3 v[3] = {mk(m.fV + 3 * m.fF[3 * t2]), mk(m.fV + 3 * m.fF[3 * t2 + 1]), mk(m.fV + 3 * m.fF[3 * t2 + 2])};
    const double A = tri_area(w[0], w[1], w[2]), A2 = tri_area(v[0], v[1], v[2]);
    const V3 x = tri_pt(c_r3, q, w[0], w[1], w[2]);
    Pair P;
    P.set(x, v[0], v[1], v[2], pa == pb);
    double z0;
    V3 z1;
    YukAcc<false>::run(valid, P, kappa, z0, z1);
    if (!valid) return;
    const double wx = c_r3[q][3] * A;
    double I[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    add_moments(I, x, w, v, wx / (4.0 * A * A2), z0, z1);
    scatter_zs(m, kappa, t, t2, A, A2, I, wx * z0, Zs, Psi);
}

// Zs and Psi, all other pairs (product rule): one thread per (outer, inner) fine triangle
__global__ void __launch_bounds__(AB) k_static_efie(DevMesh m, double kappa, double* __restrict__ Zs, double* __restrict__ Psi) {
    const int64_t tid = (int64_t)blockIdx.x * AB + threadIdx.x;
    if (tid >= (int64_t)m.nf * m.nf) return;
    const int t2 = (int)(tid % m.nf), t = (int)(tid / m.nf);
    if (parents_touch(m.F, t / 6, t2 / 6)) return;
    const V3 w[3] = {mk(m.fV + 3 * m.fF[3 * t]), mk(m.fV + 3 * m.fF[3 * t + 1]), mk(m.fV + 3 * m.fF[3 * t + 2])};
    const V3 v[3] = {mk(m.fV + 3 * m.fF[3 * t2]), mk(m.fV + 3 * m.fF[3 * t2 + 1]), mk(m.fV + 3 * m.fF[3 * t2 + 2])};
    const double A = tri_area(w[0], w[1], w[2]), A2 = tri_area(v[0], v[1], v[2]);
    double I[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    double Is = 0.0;
    for (int q = 0; q < 3; ++q) {
        const V3 x = tri_pt(c_r3, q, w[0], w[1], w[2]);
        double z0 = 0.0;
        V3 z1 = {0, 0, 0};
        for (int q2 = 0; q2 < 3; ++q2) {
            const V3 ymx = tri_pt(c_r3, q2, v[0], v[1], v[2]) - x;
            const double R = nrm(ymx);
            const double g = c_r3[q2][3] * A2 * exp(-kappa * R) / (4.0 * M_PI * R);
            z0 += g;
            z1 = z1 + g * ymx;
        }
        const double wx = c_r3[q][3] * A;
        Is += wx * z0;
        add_moments(I, x, w, v, wx / (4.0 * A * A2), z0, z1);
    }
    scatter_zs(m, kappa, t, t2, A, A2, I, Is, Zs, Psi);
}

// val[i][j] += f (x - w_i) . (s_j (x - v_j) x m1)
__device__ __forceinline__ void add_curl(double val[3][3], const DevMesh& m, V3 x, const V3* w, const V3* v, int c2, double f, V3 m1) {
    for (int jj = 0; jj < 3; ++jj) {
        const V3 cr = (f * m.tsign[3 * c2 + jj]) * cross(x - v[jj], m1);
        for (int ii = 0; ii < 3; ++ii) val[ii][jj] += dot(x - w[ii], cr);
    }
}
__device__ __forceinline__ void scatter_m(const DevMesh& m, int t, int c2, const double val[3][3], double* M) {
    for (int e = m.bc_ptr[t]; e < m.bc_ptr[t + 1]; ++e) {
        const double* ph = m.bc_phi + 3 * e;
        for (int jj = 0; jj < 3; ++jj) {
            const double vv = ph[0] * val[0][jj] + ph[1] * val[1][jj] + ph[2] * val[2][jj];
            if (vv != 0.0) atomicAdd(M + (int64_t)m.bc_fn[e] * m.ne + m.tedge[3 * c2 + jj], vv);
        }
    }
}

// M, touching parents: one thread per (outer fine triangle, point, inner coarse triangle), 6 x 3 per
// pair of parents (a triangle with itself is coplanar: the curl kernel vanishes)
__global__ void __launch_bounds__(AB) k_static_mfie_near(DevMesh m, double kappa, double* __restrict__ M) {
    const int64_t u = (int64_t)blockIdx.x * AB + threadIdx.x;
    const bool in = u < (int64_t)m.ntouch * 18;
    const int64_t r = in ? u / 3 : 0;
    const int q = in ? (int)(u % 3) : 0;
    const int pa = m.touch[2 * (r / 6)], c2 = m.touch[2 * (r / 6) + 1], t = 6 * pa + (int)(r % 6);
    const bool valid = in && pa != c2;
    const V3 w[3] = {mk(m.fV + 3 * m.fF[3 * t]), mk(m.fV + 3 * m.fF[3 * t + 1]), mk(m.fV + 3 * m.fF[3 * t + 2])};
    const V3 v[3] = {mk(m.V + 3 * m.F[3 * c2]), mk(m.V + 3 * m.F[3 * c2 + 1]), mk(m.V + 3 * m.F[3 * c2 + 2])};
    const double A = tri_area(w[0], w[1], w[2]), A2 = tri_area(v[0], v[1], v[2]);
    const V3 x = tri_pt(c_r3, q, w[0], w[1], w[2]);
    Pair P;
    P.set(x, v[0], v[1], v[2], false);
    double z0;
    V3 m1;
    YukAcc<true>::run(valid, P, kappa, z0, m1);
    if (!valid) return;
    double val[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    add_curl(val, m, x, w, v, c2, c_r3[q][3] * A / (4.0 * A * A2), m1);
    scatter_m(m, t, c2, val, M);
}

// M, all other pairs (product rule): one thread per (outer fine triangle, inner coarse triangle)
__global__ void __launch_bounds__(AB) k_static_mfie(DevMesh m, double kappa, double* __restrict__ M) {
    const int64_t tid = (int64_t)blockIdx.x * AB + threadIdx.x;
    if (tid >= (int64_t)m.nf * m.nc) return;
    const int c2 = (int)(tid % m.nc), t = (int)(tid / m.nc);
    if (parents_touch(m.F, t / 6, c2)) return;
    const V3 w[3] = {mk(m.fV + 3 * m.fF[3 * t]), mk(m.fV + 3 * m.fF[3 * t + 1]), mk(m.fV + 3 * m.fF[3 * t + 2])};
    const V3 v[3] = {mk(m.V + 3 * m.F[3 * c2]), mk(m.V + 3 * m.F[3 * c2 + 1]), mk(m.V + 3 * m.F[3 * c2 + 2])};
    const double A = tri_area(w[0], w[1], w[2]), A2 = tri_area(v[0], v[1], v[2]);
    double val[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    for (int q = 0; q < 3; ++q) {
        const V3 x = tri_pt(c_r3, q, w[0], w[1], w[2]);
        V3 m1 = {0, 0, 0};
        for (int q2 = 0; q2 < 7; ++q2) {
            const V3 ymx = tri_pt(c_r7, q2, v[0], v[1], v[2]) - x;
            const double R = nrm(ymx);
            const double g = c_r7[q2][3] * A2 * (1.0 + kappa * R) * exp(-kappa * R) / (4.0 * M_PI * R * R * R);
            m1 = m1 + g * ymx;
        }
        add_curl(val, m, x, w, v, c2, c_r3[q][3] * A / (4.0 * A * A2), m1);
    }
    scatter_m(m, t, c2, val, M);
}

// G: one thread per fine triangle (degree-2 rule, exact for the quadratic integrand)
__global__ void k_gram(DevMesh m, double* __restrict__ G) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m.nf) return;
    const int c = m.fparent[t];
    const V3 w[3] = {mk(m.fV + 3 * m.fF[3 * t]), mk(m.fV + 3 * m.fF[3 * t + 1]), mk(m.fV + 3 * m.fF[3 * t + 2])};
    const V3 cv[3] = {mk(m.V + 3 * m.F[3 * c]), mk(m.V + 3 * m.F[3 * c + 1]), mk(m.V + 3 * m.F[3 * c + 2])};
    V3 nc = cross(cv[1] - cv[0], cv[2] - cv[0]);
    const double Ac = 0.5 * nrm(nc);
    nc = (1.0 / (2.0 * Ac)) * nc;
    const double A = tri_area(w[0], w[1], w[2]);
    for (int e = m.bc_ptr[t]; e < m.bc_ptr[t + 1]; ++e) {
        const double* ph = m.bc_phi + 3 * e;
        double acc[3] = {0, 0, 0};
        for (int q = 0; q < 3; ++q) {
            const V3 x = tri_pt(c_r3, q, w[0], w[1], w[2]);
            const V3 g = (1.0 / (2.0 * A)) * (ph[0] * (x - w[0]) + ph[1] * (x - w[1]) + ph[2] * (x - w[2]));
            const V3 ng = cross(nc, g);
            for (int j = 0; j < 3; ++j) {
                const V3 f = (m.tsign[3 * c + j] / (2.0 * Ac)) * (x - cv[j]);
                acc[j] += c_r3[q][3] * A * dot(ng, f);
            }
        }
        for (int j = 0; j < 3; ++j) atomicAdd(G + (int64_t)m.bc_fn[e] * m.ne + m.tedge[3 * c + j], acc[j]);
    }
}

static unsigned blocks(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// launch a pair kernel with its shared memory (over 48 KB: the attribute is set on every call, it is
// per device)
template <class K, class... A>
static void launch_pairs(K kernel, int64_t n, size_t smem, cudaStream_t s, A... args) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kernel<<<blocks(n, AB), AB, smem, s>>>(args...);
}

// lags per window: what a pair of the mesh can meet (its distances span at most twice the longest
// edge), at most LAGW, so that blocks of 128 pairs fit the shared memory of an SM: two (EFIE, 83 KB) and
// three (MFIE, 58 KB) at order 1, one at order 2 (134 and 144 KB)
static int lag_window(double lmax, double dt, int order) {
    const double span = std::ceil(2.0 * lmax / dt) + order + 4.0;
    return span < LAGW ? (int)span : LAGW;
}

// a circle and a half of room for the ends' rounding
static bool many_circles(double lmax, double dt) { return lmax / dt + 2.5 > MAXB; }

template <int ORDER>
static void launch_efie(const DevMesh& m, double dt, int K, double T0, double lmax, double* S, double* Phi, cudaStream_t s) {
    const int w = lag_window(lmax, dt, ORDER);
    launch_pairs(many_circles(lmax, dt) ? k_retarded_efie<ORDER, true> : k_retarded_efie<ORDER, false>, (int64_t)m.nc * 7 * m.nc,
                 pair_smem(EfieAcc<ORDER>::NCOMP, w + ORDER + 1), s, m, dt, K, w, T0, S, Phi);
}
void launch_retarded_efie(const DevMesh& m, double dt, int K, double T0, double lmax, double* S, double* Phi, int order,
                          cudaStream_t s) {
    if (order == 1) launch_efie<1>(m, dt, K, T0, lmax, S, Phi, s);
    else launch_efie<2>(m, dt, K, T0, lmax, S, Phi, s);
}

template <int ORDER>
static void launch_mfie(const DevMesh& m, double dt, int K, double lmax, double* MM, cudaStream_t s) {
    const int w = lag_window(lmax, dt, ORDER);
    launch_pairs(many_circles(lmax, dt) ? k_retarded_mfie<ORDER, true> : k_retarded_mfie<ORDER, false>, (int64_t)m.nf * 3 * m.nc,
                 pair_smem(MfieAcc<ORDER>::NCOMP, w + ORDER), s, m, dt, K, w, MM);
}
void launch_retarded_mfie(const DevMesh& m, double dt, int K, double lmax, double* MM, int order, cudaStream_t s) {
    if (order == 1) launch_mfie<1>(m, dt, K, lmax, MM, s);
    else launch_mfie<2>(m, dt, K, lmax, MM, s);
}

void launch_static(const DevMesh& m, double kappa, double* Zs, double* Psi, double* M, double* G, cudaStream_t s) {
    launch_pairs(k_static_efie_near, (int64_t)m.ntouch * 108, pair_smem(4, 1), s, m, kappa, Zs, Psi);
    k_static_efie<<<blocks((int64_t)m.nf * m.nf, AB), AB, 0, s>>>(m, kappa, Zs, Psi);
    launch_pairs(k_static_mfie_near, (int64_t)m.ntouch * 18, pair_smem(4, 1), s, m, kappa, M);
    k_static_mfie<<<blocks((int64_t)m.nf * m.nc, AB), AB, 0, s>>>(m, kappa, M);
    k_gram<<<blocks(m.nf, 128), 128, 0, s>>>(m, G);
}

}  // namespace tdc
