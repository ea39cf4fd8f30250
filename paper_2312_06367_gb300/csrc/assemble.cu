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

constexpr int MAXB = 64;   // breakpoint circles that may cross one edge of a source triangle
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
// acc.node(R, W / R, rho), W = cw h w_g rho R
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
        acc.node(e + f, w * (a + b), a + b);
        acc.node(e - f, w * (a - b), a - b);
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

// Angular nodes of the piece [P0, P1] in psi, in sub-pieces of width <= PIECE: ray(cosh psi,
// sinh psi, 1 / cosh psi, weight / cosh psi)
template <class RAY>
__device__ __forceinline__ void angular_piece(double P0, double P1, RAY& ray) {
    static_assert(NANG == 6, "symmetric six-point rule");
    const int nsub = min(max((int)ceil((P1 - P0) / PIECE), 1), 256);     // about 75 at most on valid pairs
    const double hh = 0.5 * (P1 - P0) / nsub;
    for (int sb = 0; sb < nsub; ++sb) {
        const double ep = exp(P0 + (2 * sb + 1) * hh), em = 1.0 / ep;
        const double chc = 0.5 * (ep + em), shc = 0.5 * (ep - em);
#pragma unroll 1
        for (int g = 3; g < 6; ++g) {
            double C, S;
            cosh_sinh(hh * c_ax[g], C, S);
            const double w = hh * c_aw[g];
#pragma unroll 1
            for (int side = 0; side < 2; ++side) {
                const double Sg = side ? -S : S;
                const double ch = fma(shc, Sg, chc * C), sh = fma(chc, Sg, shc * C), inv = 1.0 / ch;
                ray(ch, sh, inv, w * inv);
            }
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

// radial integrals of the retarded kernels: pieces split at R = j dt, each piece in one interval
// of the accumulator (pieces outside its window of intervals are left out)
template <class ACC>
__device__ __forceinline__ void radial_split(double r0, double r1, const Pair& P, double cw, V3 om, ACC& acc) {
    const double d2 = P.d * P.d;
    double ra = r0, Ra = P.ad > 0.0 ? sqrt(fma(r0, r0, d2)) : r0;
    const double R1 = P.ad > 0.0 ? sqrt(fma(r1, r1, d2)) : r1;
    int j = (int)(Ra * acc.inv_dt);
    if (j < acc.j0) {
        j = acc.j0;
        Ra = j * acc.dt;
        if (Ra >= R1) return;
        ra = sqrt(fmax(fma(Ra, Ra, -d2), 0.0));
    }
    for (; j < acc.j1; ++j) {
        const double Rb = (j + 1) * acc.dt;
        const bool end = Rb >= R1;
        const double rb = end ? r1 : sqrt(fmax(fma(Rb, Rb, -d2), 0.0));
        if (rb > ra) {
            acc.begin(j);
            radial_piece(ra, Ra, rb, end ? R1 : Rb, P.ad, cw, acc);
            acc.flush(j, om);
            ra = rb;
            Ra = Rb;
        }
        if (end) break;
    }
}

// static kernels: one radial piece, no breakpoints
template <class ACC>
__device__ __forceinline__ void radial_whole(double r1, const Pair& P, double cw, V3 om, ACC& acc) {
    if (!(r1 > 0.0)) return;
    acc.begin(0);
    radial_piece(0.0, P.ad, r1, P.ad > 0.0 ? sqrt(fma(r1, r1, P.d * P.d)) : r1, P.ad, cw, acc);
    acc.flush(0, om);
}

// insert v into the ascending list a[0..n)
__device__ __forceinline__ void insert_sorted(double* a, int& n, double v) {
    int j = n++;
    while (j > 0 && a[j - 1] > v) { a[j] = a[j - 1]; --j; }
    a[j] = v;
}

template <class ACC>
struct NearRay {
    const Pair& P;
    ACC& acc;
    V3 nu, e;
    double h, sig;
    __device__ __forceinline__ void operator()(double ch, double sh, double inv, double w) {
        const V3 om = inv * (nu + sh * e);
        if constexpr (ACC::RETARDED) radial_split(0.0, h * ch, P, sig * w, om, acc);
        else radial_whole(h * ch, P, sig * w, om, acc);
    }
};

// Polar rule about p: one signed sub-triangle per edge
template <class ACC>
__device__ void polar_near(const Pair& P, ACC& acc) {
    double sp[2 * MAXB + 2];
#pragma unroll 1
    for (int s = 0; s < 3; ++s) {
        const V3 a = P.v[s], b = P.v[s == 2 ? 0 : s + 1];
        const V3 ab = b - a;
        const double L = nrm(ab);
        const V3 e = (1.0 / L) * ab;
        double sig = dot(cross(a - P.p, b - P.p), P.n);
        if (sig == 0.0) continue;
        sig = sig > 0.0 ? 1.0 : -1.0;
        const double t = dot(P.p - a, e);
        V3 nu = a + t * e - P.p;
        const double h = nrm(nu);
        if (h <= 1e-14 * L) continue;
        nu = (1.0 / h) * nu;
        const double psa = asinh(-t / h), psb = asinh((L - t) / h);
        int nsp = 0;
        if constexpr (ACC::RETARDED) {
            // breakpoint circles that cross the edge: between its foot and its farther end
            const double d2 = P.d * P.d, m = fmax(fabs(t), fabs(L - t));
            const double hi = sqrt(fma(m, m, fma(h, h, d2)));
            int j = (int)(sqrt(fma(h, h, d2)) * acc.inv_dt);
            for (int nb = 0; nb < MAXB && j * acc.dt < hi; ++j) {
                const double R = j * acc.dt, r2 = fma(R, R, -d2);
                if (!(r2 > h * h)) continue;
                ++nb;
                const double c = acosh(sqrt(r2) / h);
                if (-c > psa && -c < psb) insert_sorted(sp, nsp, -c);
                if (c > psa && c < psb) insert_sorted(sp, nsp, c);
            }
        }
        NearRay<ACC> ray{P, acc, nu, e, h, sig};
        double P0 = psa;
        for (int pc = 0; pc <= nsp; ++pc) {
            const double P1 = pc < nsp ? sp[pc] : psb;
            if (P1 > P0) angular_piece(P0, P1, ray);
            P0 = P1;
        }
    }
}

__device__ __forceinline__ double cr2(double ax, double ay, double bx, double by) { return ax * by - ay * bx; }

template <class ACC>
struct FarRay {
    const Pair& P;
    ACC& acc;
    V3 f, g;                 // foot direction of the near edge and the direction a quarter turn on
    double hn, num, ex, ey;  // near edge's distance; far edge: cross(a, d) and its direction in (f, g)
    __device__ __forceinline__ void operator()(double ch, double sh, double inv, double w) {
        const double sn = sh * inv;
        const double r1 = num / (inv * ey - sn * ex);
        radial_split(hn * ch, r1, P, w, inv * f + sn * g, acc);
    }
};

// Far form: polar coordinates about p over the triangle's own angular range (no signed
// cancellation).  Angles are measured from the foot of the half's near edge and carried as
// asinh(tan(angle)) = asinh(cross / dot), so that no angle itself is formed.
template <class ACC>
__device__ void polar_far(const Pair& P, ACC& acc) {
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
    double sp[4 * MAXB + 2];
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
        // the half between vertex half and vertex half + 1; its edges: that pair's and the long one (0, 2)
        const double x0 = X[half], y0 = Y[half], x1 = X[half + 1], y1 = Y[half + 1];
        if (!(cr2(x0, y0, x1, y1) > 0.0)) continue;
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
        if (!(hn > 0.0)) continue;
        const double cf = fx / hn, sf = fy / hn;
        auto angle = [&](double vx, double vy) { return asinh((cf * vy - sf * vx) / (cf * vx + sf * vy)); };
        const double S0 = angle(x0, y0), S1 = angle(x1, y1);
        int nsp = 0;
#pragma unroll 1
        for (int ei = 0; ei < 2; ++ei) {
            const double bx = ei ? x0 : X[0], by = ei ? y0 : Y[0], dx = ei ? sx : lx, dy = ei ? sy : ly;
            const double dd = dx * dx + dy * dy, bq = bx * dx + by * dy, aa = bx * bx + by * by;
            // the edge's distances from the outer point lie between its foot (or ends) and its farther end
            const double ee = aa + 2.0 * bq + dd, foot = bq < 0.0 && -bq < dd ? aa - bq * bq / dd : fmin(aa, ee);
            const double hi = sqrt(fmax(aa, ee) + d2);
            int j = (int)(sqrt(fmax(foot, 0.0) + d2) * acc.inv_dt);
            for (int nb = 0; nb < MAXB && j * acc.dt < hi; ++j, ++nb) {
                const double R = j * acc.dt, r2 = fma(R, R, -d2);
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
        const double fdx = lnear ? sx : lx, fdy = lnear ? sy : ly;       // far edge
        FarRay<ACC> ray{P, acc, cf * u + sf * w, cf * w - sf * u, hn, lnear ? nsh : nl, cf * fdx + sf * fdy, cf * fdy - sf * fdx};
        double P0 = S0;
        for (int pc = 0; pc <= nsp; ++pc) {
            const double P1 = pc < nsp ? sp[pc] : S1;
            if (P1 > P0) angular_piece(P0, P1, ray);
            P0 = P1;
        }
    }
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

// Order of a block's items by kind, so that warps hold one kind: near pairs first, then far ones;
// kind 2 is left out.  Returns the number of items; item i of the block is list[i].
constexpr int AB = 128;     // threads per block of the pair kernels
__device__ __forceinline__ int sort_items(int kind, unsigned short* list, int* wsum, int* nnear) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned mn = __ballot_sync(0xffffffffu, kind == 0), mf = __ballot_sync(0xffffffffu, kind == 1);
    if (lane == 0) { wsum[warp] = __popc(mn); wsum[AB / 32 + warp] = __popc(mf); }
    __syncthreads();
    int bn = 0, bf = 0, tn = 0, tf = 0;
    for (int w = 0; w < AB / 32; ++w) {
        if (w < warp) { bn += wsum[w]; bf += wsum[AB / 32 + w]; }
        tn += wsum[w];
        tf += wsum[AB / 32 + w];
    }
    const unsigned below = (1u << lane) - 1u;
    if (kind == 0) list[bn + __popc(mn & below)] = (unsigned short)threadIdx.x;
    if (kind == 1) list[tn + bf + __popc(mf & below)] = (unsigned short)threadIdx.x;
    __syncthreads();
    *nnear = tn;
    return tn + tf;
}

// lags whose support meets the distances [lo, hi]
__device__ __forceinline__ void lag_range(double lo, double hi, double dt, int K, int order, int& klo, int& khi) {
    klo = max(0, (int)floor(lo / dt) - 1);
    khi = min(K - 1, (int)ceil(hi / dt) + order + 1);
}

// What bounds the retarded kernels is the FP64 pipe: about 20 (far) to 40 (near) radial pieces per
// pair, 120 FP64 operations each.  One thread per (outer point, source triangle); the pieces of an
// interval of length dt are summed as moments in v (local memory, one slot per interval) and turned
// into lags at the end, so that a node costs its own few multiply-adds whatever the number of lags.
// Measured on the 480-edge sphere, dt 0.4 (K = 7): see the launchers below.
//
// ------------------------------------------------------------------ retarded EFIE
template <int ORDER>
struct EfieAcc {
    static constexpr bool RETARDED = true;
    static constexpr int NS = ORDER + 2, NV = ORDER, NI = LAGW + ORDER + 1;
    double dt, inv_dt;
    int j0, j1;                  // window of intervals [j0, j1)
    double sc[NI][NS];           // sum W / R v^p
    double vc[NI][NV][3];        // sum W / R rho v^p om
    double c[NS], r[NV], jp;     // the current piece
    __device__ __forceinline__ void begin(int j) {
        jp = j + 1;
#pragma unroll
        for (int p = 0; p < NS; ++p) c[p] = 0.0;
#pragma unroll
        for (int p = 0; p < NV; ++p) r[p] = 0.0;
    }
    __device__ __forceinline__ void node(double R, double Wr, double rho) {
        const double v = fma(-R, inv_dt, jp);
        double t = Wr;
        c[0] += t;
#pragma unroll
        for (int p = 1; p < NS; ++p) { t *= v; c[p] += t; }
        r[0] = fma(Wr, rho, r[0]);
        if constexpr (NV == 2) r[1] = fma(Wr * rho, v, r[1]);
    }
    __device__ __forceinline__ void flush(int j, V3 om) {
        double* s = sc[j - j0];
#pragma unroll
        for (int p = 0; p < NS; ++p) s[p] += c[p];
#pragma unroll
        for (int p = 0; p < NV; ++p) {
            double* v = vc[j - j0][p];
            v[0] = fma(r[p], om.x, v[0]);
            v[1] = fma(r[p], om.y, v[1]);
            v[2] = fma(r[p], om.z, v[2]);
        }
    }
    __device__ __forceinline__ void clear(int n) {
        for (int i = 0; i < n; ++i) {
#pragma unroll
            for (int p = 0; p < NS; ++p) sc[i][p] = 0.0;
#pragma unroll
            for (int p = 0; p < NV; ++p) vc[i][p][0] = vc[i][p][1] = vc[i][p][2] = 0.0;
        }
    }
    // sums over the pair of dt h_0'(t) W / R (scalar and times y - x) and q_0(t) W / R for lag k
    __device__ __forceinline__ void lag(int k, const Pair& P, double& s0, V3& s1, double& q) const {
        s0 = q = 0.0;
        V3 v = {0, 0, 0};
#pragma unroll
        for (int i = 0; i <= ORDER + 1; ++i) {
            const int sl = k - i - j0;
            const double* s = sc[sl];
            if constexpr (ORDER == 1) {
                q += i == 0 ? 0.5 * s[2] : i == 1 ? 0.5 * s[0] + s[1] - s[2] : 0.5 * s[0] - s[1] + 0.5 * s[2];
                if (i < 2) {
                    const double g = i == 0 ? 1.0 : -1.0;
                    s0 += g * s[0];
                    v = v + g * V3{vc[sl][0][0], vc[sl][0][1], vc[sl][0][2]};
                }
            } else {
                const double a0 = i == 0 ? 0.0 : i == 1 ? 5.0 / 12 : i == 2 ? 2.0 / 3 : -1.0 / 12, a1 = i == 1 ? 1.0 : i == 2 ? -1.0 : 0.0;
                const double a2 = i == 0 || i == 3 ? 0.25 : -0.25, a3 = i == 0 ? 1.0 / 6 : i == 1 ? -0.5 : i == 2 ? 0.5 : -1.0 / 6;
                q += a0 * s[0] + a1 * s[1] + a2 * s[2] + a3 * s[3];
                if (i < 3) {
                    const double g0 = i == 0 ? 0.5 : i == 1 ? 0.0 : -0.5, g1 = i == 1 ? -2.0 : 1.0;
                    s0 += g0 * s[0] + g1 * s[1];
                    v = v + g0 * V3{vc[sl][0][0], vc[sl][0][1], vc[sl][0][2]} + g1 * V3{vc[sl][NV - 1][0], vc[sl][NV - 1][1], vc[sl][NV - 1][2]};
                }
            }
        }
        s1 = v - (s0 * P.d) * P.n;
    }
};

template <int ORDER>
__global__ void __launch_bounds__(AB) k_retarded_efie(DevMesh m, double dt, int K, double T0, double* __restrict__ S,
                                                      double* __restrict__ Phi) {
    __shared__ unsigned short list[AB];
    __shared__ int wsum[2 * AB / 32];
    const int64_t total = (int64_t)m.nc * 7 * m.nc;
    Pair P;
    int c, c2, q;
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
    int64_t it = (int64_t)blockIdx.x * AB + threadIdx.x;
    int kind = 2, nnear;
    if (it < total) {
        load(it);
        kind = c != c2 && P.far() ? 1 : 0;
    }
    if ((int)threadIdx.x >= sort_items(kind, list, wsum, &nnear)) return;
    load((int64_t)blockIdx.x * AB + list[threadIdx.x]);
    const double A = tri_area(wv[0], wv[1], wv[2]), A2 = tri_area(P.v[0], P.v[1], P.v[2]);
    const double wx = c_r7[q][3] * A;
    double lo, hi;
    dist_bounds(x, P.v[0], P.v[1], P.v[2], P.ad, lo, hi);
    int klo, khi;
    lag_range(lo, hi, dt, K, ORDER, klo, khi);
    EfieAcc<ORDER> acc;
    acc.dt = dt;
    acc.inv_dt = 1.0 / dt;
    const double fs = -1.0 / (4.0 * M_PI * dt), fq = -T0 / (4.0 * M_PI);
    for (int k0 = klo; k0 <= khi; k0 += LAGW) {
        const int nk = min(LAGW, khi - k0 + 1);
        acc.j0 = k0 - ORDER - 1;
        acc.j1 = k0 + nk;
        acc.clear(nk + ORDER + 1);
        if ((int)threadIdx.x < nnear) polar_near(P, acc);
        else polar_far(P, acc);
        for (int k = k0; k < k0 + nk; ++k) {
            double s0, qv;
            V3 s1;
            acc.lag(k, P, s0, s1, qv);
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
    static constexpr int NB = ORDER == 1 ? 1 : 3, NI = LAGW + ORDER;
    double dt, inv_dt;
    int j0, j1;
    double bc[NI][NB];           // sum W / R^3 v^p
    double bv[NI][NB][3];        // sum W / R^3 rho v^p om
    double c[NB], r[NB], jp;
    __device__ __forceinline__ void begin(int j) {
        jp = j + 1;
#pragma unroll
        for (int p = 0; p < NB; ++p) c[p] = r[p] = 0.0;
    }
    __device__ __forceinline__ void node(double R, double Wr, double rho) {
        double t = Wr / (R * R);
#pragma unroll
        for (int p = 0; p < NB; ++p) {
            if (p) t *= fma(-R, inv_dt, jp);
            c[p] += t;
            r[p] = fma(t, rho, r[p]);
        }
    }
    __device__ __forceinline__ void flush(int j, V3 om) {
#pragma unroll
        for (int p = 0; p < NB; ++p) {
            bc[j - j0][p] += c[p];
            double* v = bv[j - j0][p];
            v[0] = fma(r[p], om.x, v[0]);
            v[1] = fma(r[p], om.y, v[1]);
            v[2] = fma(r[p], om.z, v[2]);
        }
    }
    __device__ __forceinline__ void clear(int n) {
        for (int i = 0; i < n; ++i)
#pragma unroll
            for (int p = 0; p < NB; ++p) bc[i][p] = bv[i][p][0] = bv[i][p][1] = bv[i][p][2] = 0.0;
    }
    // sum over the pair of (h_0 + R h_0') W / R^3 (y - x) for lag k
    __device__ __forceinline__ V3 lag(int k, const Pair& P) const {
        double s = 0.0;
        V3 v = {0, 0, 0};
#pragma unroll
        for (int i = 0; i <= ORDER; ++i) {
            const int j = k - i, sl = j - j0;
            if constexpr (ORDER == 1) {
                const double g = i == 0 ? j + 1 : -j;
                s += g * bc[sl][0];
                v = v + g * V3{bv[sl][0][0], bv[sl][0][1], bv[sl][0][2]};
            } else {
                const double J = j + 1;
                const double g[3] = {i == 0 ? 0.5 * J : i == 1 ? 1.0 : -0.5 * J, i == 1 ? -2.0 * J : J, i == 1 ? 1.0 : -0.5};
#pragma unroll
                for (int p = 0; p < NB; ++p) {
                    s += g[p] * bc[sl][p];
                    v = v + g[p] * V3{bv[sl][p][0], bv[sl][p][1], bv[sl][p][2]};
                }
            }
        }
        return v - (s * P.d) * P.n;
    }
};

template <int ORDER>
__global__ void __launch_bounds__(AB) k_retarded_mfie(DevMesh m, double dt, int K, double* __restrict__ MM) {
    __shared__ unsigned short list[AB];
    __shared__ int wsum[2 * AB / 32];
    const int64_t total = (int64_t)m.nf * 3 * m.nc;
    Pair P;
    int t, c2, q;
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
    int64_t it = (int64_t)blockIdx.x * AB + threadIdx.x;
    int kind = 2, nnear;
    if (it < total) {
        load(it);
        if (m.fparent[t] != c2) kind = P.far() ? 1 : 0;   // coplanar: the curl kernel vanishes
    }
    if ((int)threadIdx.x >= sort_items(kind, list, wsum, &nnear)) return;
    load((int64_t)blockIdx.x * AB + list[threadIdx.x]);
    const double A = tri_area(wv[0], wv[1], wv[2]), A2 = tri_area(P.v[0], P.v[1], P.v[2]);
    const double wx = c_r3[q][3] * A / (4.0 * M_PI);
    double lo, hi;
    dist_bounds(x, P.v[0], P.v[1], P.v[2], P.ad, lo, hi);
    int klo, khi;
    lag_range(lo, hi, dt, K, ORDER, klo, khi);
    MfieAcc<ORDER> acc;
    acc.dt = dt;
    acc.inv_dt = 1.0 / dt;
    for (int k0 = klo; k0 <= khi; k0 += LAGW) {
        const int nk = min(LAGW, khi - k0 + 1);
        acc.j0 = k0 - ORDER;
        acc.j1 = k0 + nk;
        acc.clear(nk + ORDER);
        if ((int)threadIdx.x < nnear) polar_near(P, acc);
        else polar_far(P, acc);
        for (int k = k0; k < k0 + nk; ++k) {
            const V3 m1 = acc.lag(k, P);
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
struct YukAcc {
    static constexpr bool RETARDED = false;
    double kappa;
    bool want_m;           // (1 + kappa R) exp(-kappa R) / R^3 (times y - x), else exp(-kappa R) / R
    double s0;
    V3 s1;
    double c, r;
    __device__ __forceinline__ void begin(int) { c = r = 0.0; }
    __device__ __forceinline__ void node(double R, double Wr, double rho) {
        double g = Wr * exp(-kappa * R);
        if (want_m) g *= fma(kappa, R, 1.0) / (R * R);
        c += g;
        r = fma(g, rho, r);
    }
    __device__ __forceinline__ void flush(int, V3 om) {
        s0 += c;
        s1 = s1 + r * om;
    }
    // sums over the triangle of the kernel / (4 pi), scalar and times y - x
    __device__ __forceinline__ void run(const Pair& P, double& z0, V3& z1) {
        s0 = 0.0;
        s1 = {0, 0, 0};
        polar_near(P, *this);
        z0 = s0 / (4.0 * M_PI);
        z1 = (1.0 / (4.0 * M_PI)) * (s1 - (s0 * P.d) * P.n);
    }
};

__device__ __forceinline__ bool parents_touch(const int* F, int a, int b) {
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            if (F[3 * a + i] == F[3 * b + j]) return true;
    return false;
}

// Zs and Psi: one thread per (outer fine triangle, inner fine triangle); the few near pairs cost
// some fifty times a far one, so a block's near pairs share warps
__global__ void __launch_bounds__(AB) k_static_efie(DevMesh m, double kappa, double* __restrict__ Zs, double* __restrict__ Psi) {
    __shared__ unsigned short list[AB];
    __shared__ int wsum[2 * AB / 32];
    const int64_t total = (int64_t)m.nf * m.nf;
    int64_t tid = (int64_t)blockIdx.x * AB + threadIdx.x;
    int kind = 2, nnear;
    if (tid < total) kind = parents_touch(m.F, m.fparent[tid / m.nf], m.fparent[tid % m.nf]) ? 0 : 1;
    if ((int)threadIdx.x >= sort_items(kind, list, wsum, &nnear)) return;
    tid = (int64_t)blockIdx.x * AB + list[threadIdx.x];
    const int t2 = (int)(tid % m.nf), t = (int)(tid / m.nf);
    const V3 w[3] = {mk(m.fV + 3 * m.fF[3 * t]), mk(m.fV + 3 * m.fF[3 * t + 1]), mk(m.fV + 3 * m.fF[3 * t + 2])};
    const V3 v[3] = {mk(m.fV + 3 * m.fF[3 * t2]), mk(m.fV + 3 * m.fF[3 * t2 + 1]), mk(m.fV + 3 * m.fF[3 * t2 + 2])};
    const double A = tri_area(w[0], w[1], w[2]), A2 = tri_area(v[0], v[1], v[2]);
    const bool near = (int)threadIdx.x < nnear;
    const bool copl = m.fparent[t] == m.fparent[t2];
    double I[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    double Is = 0.0;
    for (int q = 0; q < 3; ++q) {
        const V3 x = tri_pt(c_r3, q, w[0], w[1], w[2]);
        const double wx = c_r3[q][3] * A;
        double z0 = 0.0;
        V3 z1 = {0, 0, 0};
        if (near) {
            Pair P;
            P.set(x, v[0], v[1], v[2], copl);
            YukAcc acc{kappa, false};
            acc.run(P, z0, z1);
        } else {
            for (int q2 = 0; q2 < 3; ++q2) {
                const V3 ymx = tri_pt(c_r3, q2, v[0], v[1], v[2]) - x;
                const double R = nrm(ymx);
                const double g = c_r3[q2][3] * A2 * exp(-kappa * R) / (4.0 * M_PI * R);
                z0 += g;
                z1 = z1 + g * ymx;
            }
        }
        Is += wx * z0;
        for (int j = 0; j < 3; ++j) {
            const V3 Iy = (1.0 / (2.0 * A2)) * (z1 + z0 * (x - v[j]));
            for (int i = 0; i < 3; ++i) I[i][j] += wx * dot((1.0 / (2.0 * A)) * (x - w[i]), Iy);
        }
    }
    const double rv = 1.0 / (2.0 * m.valence[m.fvert[t]] * A), rv2 = 1.0 / (2.0 * m.valence[m.fvert[t2]] * A2);
    atomicAdd(Psi + (int64_t)m.fvert[t] * m.nv + m.fvert[t2], -(1.0 / kappa) * rv * rv2 * Is);
    for (int e1 = m.bc_ptr[t]; e1 < m.bc_ptr[t + 1]; ++e1) {
        const double* p1 = m.bc_phi + 3 * e1;
        double u[3];
        for (int j = 0; j < 3; ++j) u[j] = p1[0] * I[0][j] + p1[1] * I[1][j] + p1[2] * I[2][j];
        for (int e2 = m.bc_ptr[t2]; e2 < m.bc_ptr[t2 + 1]; ++e2) {
            const double* p2 = m.bc_phi + 3 * e2;
            const double acc = p2[0] * u[0] + p2[1] * u[1] + p2[2] * u[2];
            atomicAdd(Zs + (int64_t)m.bc_fn[e1] * m.ne + m.bc_fn[e2], -kappa * acc);
        }
    }
}

// M: one thread per (outer fine triangle, inner coarse triangle)
__global__ void __launch_bounds__(AB) k_static_mfie(DevMesh m, double kappa, double* __restrict__ M) {
    __shared__ unsigned short list[AB];
    __shared__ int wsum[2 * AB / 32];
    const int64_t total = (int64_t)m.nf * m.nc;
    int64_t tid = (int64_t)blockIdx.x * AB + threadIdx.x;
    int kind = 2, nnear;
    if (tid < total) {
        const int a = m.fparent[tid / m.nc], b = (int)(tid % m.nc);
        if (a != b) kind = parents_touch(m.F, a, b) ? 0 : 1;
    }
    if ((int)threadIdx.x >= sort_items(kind, list, wsum, &nnear)) return;
    tid = (int64_t)blockIdx.x * AB + list[threadIdx.x];
    const int c2 = (int)(tid % m.nc), t = (int)(tid / m.nc);
    const V3 w[3] = {mk(m.fV + 3 * m.fF[3 * t]), mk(m.fV + 3 * m.fF[3 * t + 1]), mk(m.fV + 3 * m.fF[3 * t + 2])};
    const V3 v[3] = {mk(m.V + 3 * m.F[3 * c2]), mk(m.V + 3 * m.F[3 * c2 + 1]), mk(m.V + 3 * m.F[3 * c2 + 2])};
    const double A = tri_area(w[0], w[1], w[2]), A2 = tri_area(v[0], v[1], v[2]);
    const bool near = (int)threadIdx.x < nnear;
    double val[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    for (int q = 0; q < 3; ++q) {
        const V3 x = tri_pt(c_r3, q, w[0], w[1], w[2]);
        const double wx = c_r3[q][3] * A;
        V3 m1 = {0, 0, 0};
        if (near) {
            Pair P;
            P.set(x, v[0], v[1], v[2], false);
            YukAcc acc{kappa, true};
            double m0;
            acc.run(P, m0, m1);
        } else {
            for (int q2 = 0; q2 < 7; ++q2) {
                const V3 ymx = tri_pt(c_r7, q2, v[0], v[1], v[2]) - x;
                const double R = nrm(ymx);
                const double g = c_r7[q2][3] * A2 * (1.0 + kappa * R) * exp(-kappa * R) / (4.0 * M_PI * R * R * R);
                m1 = m1 + g * ymx;
            }
        }
        for (int jj = 0; jj < 3; ++jj) {
            const V3 cr = (m.tsign[3 * c2 + jj] / (2.0 * A2)) * cross(x - v[jj], m1);
            for (int ii = 0; ii < 3; ++ii) val[ii][jj] += wx * dot((1.0 / (2.0 * A)) * (x - w[ii]), cr);
        }
    }
    for (int e = m.bc_ptr[t]; e < m.bc_ptr[t + 1]; ++e) {
        const double* ph = m.bc_phi + 3 * e;
        for (int jj = 0; jj < 3; ++jj) {
            const double vv = ph[0] * val[0][jj] + ph[1] * val[1][jj] + ph[2] * val[2][jj];
            if (vv != 0.0) atomicAdd(M + (int64_t)m.bc_fn[e] * m.ne + m.tedge[3 * c2 + jj], vv);
        }
    }
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

void launch_retarded_efie(const DevMesh& m, double dt, int K, double T0, double* S, double* Phi, int order,
                          cudaStream_t s) {
    const unsigned g = blocks((int64_t)m.nc * 7 * m.nc, AB);
    if (order == 1) k_retarded_efie<1><<<g, AB, 0, s>>>(m, dt, K, T0, S, Phi);
    else k_retarded_efie<2><<<g, AB, 0, s>>>(m, dt, K, T0, S, Phi);
}

void launch_retarded_mfie(const DevMesh& m, double dt, int K, double* MM, int order, cudaStream_t s) {
    const unsigned g = blocks((int64_t)m.nf * 3 * m.nc, AB);
    if (order == 1) k_retarded_mfie<1><<<g, AB, 0, s>>>(m, dt, K, MM);
    else k_retarded_mfie<2><<<g, AB, 0, s>>>(m, dt, K, MM);
}

void launch_static(const DevMesh& m, double kappa, double* Zs, double* Psi, double* M, double* G, cudaStream_t s) {
    k_static_efie<<<blocks((int64_t)m.nf * m.nf, AB), AB, 0, s>>>(m, kappa, Zs, Psi);
    k_static_mfie<<<blocks((int64_t)m.nf * m.nc, AB), AB, 0, s>>>(m, kappa, M);
    k_gram<<<blocks(m.nf, 128), 128, 0, s>>>(m, G);
}

}  // namespace tdc
