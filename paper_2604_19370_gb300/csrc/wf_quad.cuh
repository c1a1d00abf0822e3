// Explicit residual of a (sub)step by Gauss quadrature:
//
//   R_ij   = Rscale sum_points w [ s B_i B_j - v_x T_x B_i' B_j - v_y T_y B_i B_j' ]
//   Phi_ij = -tau k_f sum_points w E phi B_i B_j
//
// with (Sec. 3, normalised form and Eq. termsPR; Sec. 7 listing "compute_rhs")
//   s   = K_ign E + c_rad (T_amb^4 - T^4) + c_chi (T_amb - T) - c_W (b + b').grad T
//   v   = C_nld T^3 + C_d
//   E   = [T > T_ig and phi > phi_min] T exp(-T_a / T),
// b the slot's mean wind and b' its variation.  This is Rscale (F - A_x (x) M^y T - M^x (x) A_y T): the
// linear terms of the 1-D operators are integrated exactly by the q = p+1 point rule, so they are
// summed with the nonlinear ones at the points instead of by band products afterwards (no band
// windows, and the gradient of a constant field is exactly zero in every precision).  XO: only the x
// operator (v_y = C_nld T^3, no mean wind along y), the first and last substeps of Strang splitting.
//
// On an element a spline is a polynomial of degree p in t = xi - 1/2 per direction.  Everything works on
// its p+1 (scaled) monomial components instead of on basis values: with uniform knots they are a few
// sums and differences of the coefficients, the Gauss nodes come in pairs +-t, so values at a pair share
// their even part, and so do derivatives; the test side is the transposed computation.  Operations per
// element, p = 2: 4 for a coefficient row along x, 12 + 15 + 24 to T, T_x, T_y at the nine points, 81
// at the points, 33 + 24 + 21 to the test rows, 8 to finish a row: 222, against 345 multiply-adds
// with basis tables.
//
// Two schedules.  Serial: one warp per work item, a strip of 32 element columns (lane L <-> element column
// X0 - p + L, outputs from lane p on) walking down a segment of rows.  Registers hold sliding windows
// of p rows: x components of the coefficient rows and x components of the unfinished test rows,
// 2 p (p+1) values in all.  Neighbour coefficients are loaded directly (the second and third load of a
// row hit L1); a finished row takes p shuffles.
//
// Boundary: with C^(p-1) continuity the splines on open uniform knots are, on the domain, the splines on
// unclamped uniform knots, so the elements next to the boundary take the same sums and differences once
// their outermost coefficients are exchanged for the unclamped ones (blossom values: p = 2:
// u0 = 2 c0 - c1; p = 3: u0 = 6 c0 - 6 c1 + c2, u1 = (3 c1 - c2) / 2), and the test side takes the
// transpose.  Both are written with differences of neighbours, which leave a constant field exact.
//
// The reaction needs T above T_ig.  B-splines are nonnegative and sum to one, so no point of an element
// row exceeds the largest coefficient of its rows: one warp vote per coefficient row decides whether
// the reaction (fuel loads, exponential, fuel row sums in shared memory) runs for an element row.  It
// adds its load to the sums of the rest, so a row gives the same bits whichever warp evaluates it.
#pragma once
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "wf_internal.h"

namespace wf {

namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }

__device__ __forceinline__ float larger(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double larger(double a, double b) { return a > b ? a : b; }

// A constant kept in a register: a multiply-add takes one operand from the constant bank, so where two
// are constants the second one would be moved to a register at every use.
__device__ __forceinline__ float held(float a) {
    asm volatile("" : "+f"(a));
    return a;
}
__device__ __forceinline__ double held(double a) { return a; }

// exp(-T_a / T).  FP32: 2^(-T_a log2(e) / T) with the fast divide and the hardware base-2
// exponential (PTX ex2.approx, relative error about 2^-22); FP64: exp of the exact quotient.
__device__ __forceinline__ float arrhenius(float Ta_l2, float, float T) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(-__fdividef(Ta_l2, T)));
    return y;
}
__device__ __forceinline__ double arrhenius(double, double T_a, double T) { return exp(-T_a / T); }

// Constants of the element algebra (see El); kx and ky hold flux / value ratios of a direction:
// kap = -(derivative scale)^2.
template <typename P>
struct ElK {
    P a[13];         // of the nodes and weights
    P kx[3], ky[3];  // flux coefficients of the test sums along x and along y
};

// Element algebra of degree p: components c_j of the p+1 coefficients x_k, values v and (scaled)
// derivatives d at the Gauss points in ascending order, and the transposed sums.  Point weights are
// normalised by the outermost point's; component j of a test sum m carries the factor 1 / scl[j].
template <int PD, typename P>
struct El;

// p = 1: T = c0 + c1 t, points -+t0
//   a = {t0}; dT/dx = c1 / h; k[0] = kap / t0
template <typename P>
struct El<1, P> {
    static __device__ __forceinline__ void comps(const P (&x)[2], P (&c)[2]) {
        c[1] = x[1] - x[0];
        c[0] = mad(P(0.5), c[1], x[0]);
    }
    static __device__ __forceinline__ void value(const P (&c)[2], P (&v)[2], const ElK<P>& K) {
        v[0] = mad(-K.a[0], c[1], c[0]);
        v[1] = mad(K.a[0], c[1], c[0]);
    }
    static __device__ __forceinline__ void deriv(const P (&c)[2], P (&d)[2], const ElK<P>&) { d[0] = d[1] = c[1]; }
    static __device__ __forceinline__ void sums(const P (&s)[2], P (&m)[2], const ElK<P>&) {
        m[0] = s[1] + s[0];
        m[1] = s[1] - s[0];
    }
    static __device__ __forceinline__ void sums_flux(const P (&s)[2], const P (&g)[2], P (&m)[2], const ElK<P>&,
                                                     const P (&k)[3]) {
        m[0] = s[1] + s[0];
        m[1] = mad(k[0], g[1] + g[0], s[1] - s[0]);
    }
    static __device__ __forceinline__ void scatter(const P (&m)[2], P (&x)[2], const ElK<P>& K) {
        const P e = P(0.5) * m[0];
        x[0] = mad(-K.a[0], m[1], e);
        x[1] = mad(K.a[0], m[1], e);
    }
};

// p = 2: T = c0 + c1 t / 2 + c2 t^2 / 2 (c1 = x2 - x0, c2 = x0 - 2 x1 + x2), points -t0, 0, t0
//   a = {t0 / 2, t0^2 / 2, 2 t0, rho}; dT/dx = (c1 + 2 t c2) / (2h); k[0] = 2 kap / t0, k[1] = 4 kap / t0
template <typename P>
struct El<2, P> {
    static __device__ __forceinline__ void comps(const P (&x)[3], P (&c)[3]) {
        c[2] = mad(P(-2), x[1], x[0] + x[2]);
        c[1] = x[2] - x[0];
        c[0] = mad(P(0.125), c[2], x[1]);
    }
    static __device__ __forceinline__ void value(const P (&c)[3], P (&v)[3], const ElK<P>& K) {
        const P e = mad(K.a[1], c[2], c[0]);
        v[0] = mad(-K.a[0], c[1], e);
        v[1] = c[0];
        v[2] = mad(K.a[0], c[1], e);
    }
    static __device__ __forceinline__ void deriv(const P (&c)[3], P (&d)[3], const ElK<P>& K) {
        d[0] = mad(-K.a[2], c[2], c[1]);
        d[1] = c[1];
        d[2] = mad(K.a[2], c[2], c[1]);
    }
    static __device__ __forceinline__ void sums(const P (&s)[3], P (&m)[3], const ElK<P>& K) {
        m[2] = s[0] + s[2];
        m[1] = s[2] - s[0];
        m[0] = mad(K.a[3], s[1], m[2]);
    }
    static __device__ __forceinline__ void sums_flux(const P (&s)[3], const P (&g)[3], P (&m)[3], const ElK<P>& K,
                                                     const P (&k)[3]) {
        const P S = s[0] + s[2];
        m[0] = mad(K.a[3], s[1], S);
        m[1] = mad(k[0], mad(K.a[3], g[1], g[0] + g[2]), s[2] - s[0]);
        m[2] = mad(k[1], g[2] - g[0], S);
    }
    static __device__ __forceinline__ void scatter(const P (&m)[3], P (&x)[3], const ElK<P>& K) {
        // c0 = x1 + c2 / 8
        const P r = mad(K.a[1], m[2], P(0.125) * m[0]);
        x[0] = mad(-K.a[0], m[1], r);
        x[1] = mad(P(-2), r, m[0]);
        x[2] = mad(K.a[0], m[1], r);
    }
};

// p = 3: T = c0 + c1 t + c2 t^2 / 4 + c3 t^3 / 6, points -t2, -t1, t1, t2 (t2 outer)
//   (c2 = x0 - x1 - x2 + x3, c3 = x3 - 3 x2 + 3 x1 - x0, c0 = (x1 + x2) / 2 + c2 / 48,
//    c1 = x2 - x1 + c3 / 8); dT/dx = (c1 + c2 t / 2 + c3 t^2 / 2) / h
//   a = {t1, t2, t1^2/4, t2^2/4, t1^2/6, t2^2/6, t1^2/2, t2^2/2, rho, rho t1/t2, (t1/t2)^2, t2^3/6, t2/8};
//   k[0] = kap / t2, k[1] = 2 kap / t2, k[2] = 3 kap / t2
template <typename P>
struct El<3, P> {
    static __device__ __forceinline__ void comps(const P (&x)[4], P (&c)[4]) {
        const P s1 = x[1] + x[2], d1 = x[2] - x[1];
        c[2] = (x[0] + x[3]) - s1;
        c[3] = mad(P(-3), d1, x[3] - x[0]);
        c[0] = mad(P(0.5), s1, P(1.0 / 48.0) * c[2]);
        c[1] = mad(P(0.125), c[3], d1);
    }
    static __device__ __forceinline__ void value(const P (&c)[4], P (&v)[4], const ElK<P>& K) {
        const P e1 = mad(K.a[2], c[2], c[0]), e2 = mad(K.a[3], c[2], c[0]);
        const P o1 = mad(K.a[4], c[3], c[1]), o2 = mad(K.a[5], c[3], c[1]);
        v[0] = mad(-K.a[1], o2, e2);
        v[1] = mad(-K.a[0], o1, e1);
        v[2] = mad(K.a[0], o1, e1);
        v[3] = mad(K.a[1], o2, e2);
    }
    static __device__ __forceinline__ void deriv(const P (&c)[4], P (&d)[4], const ElK<P>& K) {
        const P f1 = mad(K.a[6], c[3], c[1]), f2 = mad(K.a[7], c[3], c[1]), h = P(0.5) * c[2];
        d[0] = mad(-K.a[1], h, f2);
        d[1] = mad(-K.a[0], h, f1);
        d[2] = mad(K.a[0], h, f1);
        d[3] = mad(K.a[1], h, f2);
    }
    static __device__ __forceinline__ void sums(const P (&s)[4], P (&m)[4], const ElK<P>& K) {
        const P S2 = s[0] + s[3], A2 = s[3] - s[0], S1 = s[1] + s[2], A1 = s[2] - s[1];
        const P R1 = K.a[8] * S1, B1 = K.a[9] * A1;
        m[0] = S2 + R1;
        m[1] = A2 + B1;
        m[2] = mad(K.a[10], R1, S2);
        m[3] = mad(K.a[10], B1, A2);
    }
    static __device__ __forceinline__ void sums_flux(const P (&s)[4], const P (&g)[4], P (&m)[4], const ElK<P>& K,
                                                     const P (&k)[3]) {
        sums(s, m, K);
        const P G2 = g[0] + g[3], G1 = K.a[8] * (g[1] + g[2]);
        m[1] = mad(k[0], G2 + G1, m[1]);
        m[2] = mad(k[1], mad(K.a[9], g[2] - g[1], g[3] - g[0]), m[2]);
        m[3] = mad(k[2], mad(K.a[10], G1, G2), m[3]);
    }
    static __device__ __forceinline__ void scatter(const P (&m)[4], P (&x)[4], const ElK<P>& K) {
        const P s0 = mad(K.a[3], m[2], P(1.0 / 48.0) * m[0]);    // weight of x0 + x3
        const P s1 = mad(P(0.5), m[0], -s0);                     // of x1 + x2
        const P d0 = mad(K.a[11], m[3], K.a[12] * m[1]);         // of x3 - x0
        const P d1 = mad(P(-3), d0, K.a[1] * m[1]);              // of x2 - x1
        x[0] = s0 - d0;
        x[1] = s1 - d1;
        x[2] = s1 + d1;
        x[3] = s0 + d0;
    }
};

// Exchange of the outermost coefficients of an element for the unclamped ones, with the factors of one
// element (all zero away from the boundary; l: its left end, r: its right end):
//   p = 2: x0 += l0 (x0 - x1), x2 += r0 (x2 - x1)
//   p = 3: x0 += l0 (x0 - x1) + l1 (x1 - x2), x1 += l2 (x1 - x2), and mirrored
// end() gives the factors d elements from an end of a line of n elements.
template <int PD, typename P>
struct Ends {
    P l[3], r[3];
    static __device__ __forceinline__ void end(int d, int n, P (&f)[3]) {
        f[0] = f[1] = f[2] = P(0);
        if (PD == 2) f[0] = d == 0 ? P(1) : P(0);
        if (PD == 3) {
            // a single cubic element is clamped at both ends: c2 = f[0,1,1] instead of f[0,1,2]
            f[0] = d == 0 ? P(5) : (d == 1 ? P(0.5) : P(0));
            f[1] = d == 0 ? (n == 1 ? P(-2) : P(-1)) : P(0);
            f[2] = d == 0 ? (n == 1 ? P(1) : P(0.5)) : P(0);
        }
    }
    __device__ __forceinline__ Ends(int e, int n) {
        end(e, n, l);
        end(n - 1 - e, n, r);
    }
    __device__ __forceinline__ void apply(P (&x)[PD + 1]) const {
        if constexpr (PD == 2) {
            const P a = x[0] - x[1], b = x[2] - x[1];
            x[0] = mad(l[0], a, x[0]);
            x[2] = mad(r[0], b, x[2]);
        }
        if constexpr (PD == 3) {
            const P a = x[0] - x[1], b = x[1] - x[2], c = x[3] - x[2];
            x[0] = mad(l[0], a, mad(l[1], b, x[0]));
            x[1] = mad(l[2], b, x[1]);
            x[2] = mad(-r[2], b, x[2]);
            x[3] = mad(r[0], c, mad(-r[1], b, x[3]));
        }
    }
    __device__ __forceinline__ void transpose(P (&y)[PD + 1]) const {
        if constexpr (PD == 2) {
            y[1] = mad(-l[0], y[0], mad(-r[0], y[2], y[1]));
            y[0] = mad(l[0], y[0], y[0]);
            y[2] = mad(r[0], y[2], y[2]);
        }
        if constexpr (PD == 3) {
            // weights of the differences x0 - x1, x1 - x2, x3 - x2
            const P a = l[0] * y[0], c = r[0] * y[3];
            const P b = mad(l[1], y[0], mad(l[2], y[1], mad(-r[2], y[2], -r[1] * y[3])));
            y[0] += a;
            y[1] += b - a;
            y[2] -= b + c;
            y[3] += c;
        }
    }
};

template <typename P>
struct QuadArgs {
    int nx, ny, Nx, Ny, pitch;
    int h, nstrips;  // rows per segment; strips of the domain
    int s0, ns;      // strips of this launch: s0 .. s0 + ns - 1
    const P* T;
    const P* phi;
    P* Phi;
    P* R;
    const P *fxq, *gxq, *fyq, *gyq;
    const P* mw;       // mean wind of the slot: (b_x, b_y)
    P cwx, cwy;        // -c_W x derivative scale
    P T_ig, T_ig_lo, phi_min, Ta_l2, T_a;
    P fscale;          // -tau k_f x weights
    int heat_by_fuel;
    P Rw;              // Rscale x weights
    P K0, c_rad, c_chi, C_nld, C_d, K_ign;
    ElK<P> K;
    Batch b;
};

template <typename T>
__device__ __forceinline__ T* at_slot(T* p, long long off) {
    return p ? reinterpret_cast<T*>((char*)p + off) : p;
}

// One item: the strip at X0, rows [Y0, Y0 + h).  Rows and columns outside the domain are read at the
// nearest one inside: the elements that use them lie outside themselves and contribute zero.
template <typename P, int PD, int WR, bool XO>
__device__ __forceinline__ void quad_strip(const QuadArgs<P>& a, long long off, int lane, int X0, int Y0, P* accg, P* wsm) {
    using E = El<PD, P>;
    constexpr int NB = PD + 1, Q = PD + 1, WRm = WR > 0 ? WR : 1;
    const ElK<P>& K = a.K;
    const P* T0 = at_slot(a.T, off);
    P* Phi0 = at_slot(a.Phi, off);
    P* R0 = at_slot(a.R, off);
    const P* mw = at_slot(a.mw, off);
    const int ex = X0 - PD + lane;  // element column of this lane; also its DOF column
    const bool ex_ok = ex >= 0 && ex < a.nx;
    const bool out_col = lane >= PD && ex < a.Nx;
    const bool xb = X0 < 2 * PD || X0 + 31 >= a.nx;  // the strip reaches the x boundary
    const Ends<PD, P> xe(ex, a.nx);
    const int rows = min(a.h, a.Ny - Y0);  // output rows of this item

    // wind: factors of the lane's x points in registers, of the segment's y points in shared memory,
    // scaled by -c_W and the derivative scale; the mean wind is their constant term
    P fx[WRm][Q], fy[WRm][Q];
    const P mwx = a.cwx * mw[0], mwy = XO ? P(0) : a.cwy * mw[1];
    if constexpr (WR > 0) {
        const P* fxq = at_slot(a.fxq, off);
        const P* fyq = at_slot(a.fyq, off);
        const P* gxq = at_slot(a.gxq, off);
        const P* gyq = at_slot(a.gyq, off);
#pragma unroll
        for (int r = 0; r < WR; ++r)
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const size_t o = (size_t)r * a.nx * Q + (size_t)(ex_ok ? ex : 0) * Q + q;
                fx[r][q] = ex_ok ? a.cwx * fxq[o] : P(0);
                fy[r][q] = ex_ok ? a.cwy * fyq[o] : P(0);
            }
        // [row][x, y][r][point]
        for (int i = lane; i < (rows + PD) * WR * Q; i += 32) {
            const int row = i / (WR * Q), rq = i - row * WR * Q, r = rq / Q, q = rq - r * Q;
            const int ey = Y0 - PD + row;
            const bool ok = ey >= 0 && ey < a.ny;
            const size_t o = (size_t)r * a.ny * Q + (size_t)(ok ? ey : 0) * Q + q;
            wsm[(row * 2 + 0) * WR * Q + rq] = ok ? gxq[o] : P(0);
            wsm[(row * 2 + 1) * WR * Q + rq] = ok ? gyq[o] : P(0);
        }
        __syncwarp();
    }

    // the element's coefficients start at column ex, at the nearest one whose taps exist outside the domain
    const int shift = min(max(ex, 0), a.nx - 1) - ex;
    auto row_of = [&](const P* f, int r) {
        return f + ((long long)min(max(r, 0), a.Ny - 1) * a.pitch + ex);
    };
    auto fetch = [&](const P* row, P (&x)[NB]) {
        const P* c = row + shift;
#pragma unroll
        for (int k = 0; k < NB; ++k) x[k] = field_load(c + k);
    };
    auto xcomps = [&](P (&x)[NB], P (&c)[NB]) {
        if (PD > 1 && xb) xe.apply(x);
        E::comps(x, c);
    };
    // column ex of a finished row: basis k of element ex - k, from the lane k to its left
    auto gather = [&](const P (&m)[NB]) {
        P kx[NB];
        E::scatter(m, kx, K);
        if (xb) {
            xe.transpose(kx);
#pragma unroll
            for (int k = 0; k < NB; ++k) kx[k] = ex_ok ? kx[k] : P(0);
        }
        P r = kx[0];
#pragma unroll
        for (int k = 1; k < NB; ++k) r += __shfl_up_sync(kFull, kx[k], k);
        return r;
    };
    // Element rows next to the y boundary exchange their outermost coefficients, those outside the
    // domain contribute nothing.
    auto edge_comps = [&](int e, P (&x)[NB], P (&c)[NB]) {
        Ends<PD, P>(e, a.ny).apply(x);
        E::comps(x, c);
    };
    auto edge_rows = [&](int e, const P (&eta)[NB], P (&add)[NB]) {
        E::scatter(eta, add, K);
        Ends<PD, P>(e, a.ny).transpose(add);
#pragma unroll
        for (int l = 0; l < NB; ++l) add[l] = (e >= 0 && e < a.ny) ? add[l] : P(0);
    };

    // windows, [row][x component]: coefficient rows ey .. ey+p-1 and test rows ey .. ey+p-1
    P win[PD][NB], acc[PD][NB];
#pragma unroll
    for (int l = 0; l < PD; ++l)
#pragma unroll
        for (int j = 0; j < NB; ++j) acc[l][j] = P(0);

    // hot: coefficient rows left in the window's reach of the last one above T_ig (the first and the
    // last tap of 32 lanes cover every coefficient of a row); fuel_to: last iteration whose finished
    // row has fuel sums
    int hot = 0, fuel_to = -1;
    auto see = [&](const P (&x)[NB]) {
        const bool h = __any_sync(kFull, larger(x[0], x[PD]) > a.T_ig_lo);
        hot = h ? NB : hot - 1;
    };
    const P c_chi = held(a.c_chi), C_d = held(a.C_d);
    P nxt[NB];
#pragma unroll
    for (int l = 0; l < PD; ++l) {
        fetch(row_of(T0, Y0 - PD + l), nxt);
        xcomps(nxt, win[l]);
        see(nxt);
    }
    // The running coefficient row ey + p (+ 1 once fetched); row ey of R and Phi lies dR and dPhi elements
    // from it.  Past the last row nothing is fetched (the element rows that would use it are outside).
    const P* tp = row_of(T0, Y0);
    const long long back = (long long)(PD + 1) * a.pitch;
    const long long dR = (R0 - T0) - back, dPhi = Phi0 ? (Phi0 - T0) - back : 0;
    fetch(tp, nxt);
    // iterations lo <= i < hi have interior element rows
    const int lo = 2 * PD - Y0, hi = a.ny - Y0;
    int left = a.Ny - 1 - Y0;  // coefficient rows below the running one
    for (int i = 0; i < rows + PD; ++i) {
        const int ey = Y0 - PD + i;
        const bool edge = i < lo || i >= hi;
        P nw[NB];
        xcomps(nxt, nw);
        see(nxt);
        // the next coefficient row, one iteration ahead
        tp += a.pitch;
        if (--left >= 0) fetch(tp, nxt);

        // tensor components of the element: [y component][x component]
        P tc[NB][NB];
        auto tensor = [&](auto comps) {
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                P x[NB], c[NB];
#pragma unroll
                for (int l = 0; l < PD; ++l) x[l] = win[l][j];
                x[PD] = nw[j];
                comps(x, c);
#pragma unroll
                for (int m = 0; m < NB; ++m) tc[m][j] = c[m];
            }
        };
        if (__builtin_expect(edge, 0))
            tensor([&](P(&x)[NB], P(&c)[NB]) { edge_comps(ey, x, c); });
        else
            tensor([&](P(&x)[NB], P(&c)[NB]) { E::comps(x, c); });
#pragma unroll
        for (int j = 0; j < NB; ++j) {
#pragma unroll
            for (int l = 0; l + 1 < PD; ++l) win[l][j] = win[l + 1][j];
            win[PD - 1][j] = nw[j];
        }
        P yv[Q][NB], yd[Q][NB];  // [y point][x component]: T and its y derivative
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            P c[NB], v[Q], d[Q];
#pragma unroll
            for (int m = 0; m < NB; ++m) c[m] = tc[m][j];
            E::value(c, v, K);
            E::deriv(c, d, K);
#pragma unroll
            for (int b = 0; b < Q; ++b) {
                yv[b][j] = v[b];
                yd[b][j] = d[b];
            }
        }
        P mu[Q][NB], nu[Q][NB];  // x sums of the value and x-flux terms, of the y flux
#pragma unroll
        for (int b = 0; b < Q; ++b) {
            P T[Q], Tx[Q], Ty[Q], s[Q], gx[Q], gy[Q];
            E::value(yv[b], T, K);
            E::deriv(yv[b], Tx, K);
            E::value(yd[b], Ty, K);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const P T3 = (T[q] * T[q]) * T[q];
                P src = mad(T[q], mad(-a.c_rad, T3, -c_chi), a.K0);
                P bx = mwx, by = mwy;
#pragma unroll
                for (int r = 0; r < WR; ++r) {
                    bx = mad(fx[r][q], wsm[(i * 2 + 0) * WR * Q + r * Q + b], bx);
                    by = mad(fy[r][q], wsm[(i * 2 + 1) * WR * Q + r * Q + b], by);
                }
                src = mad(bx, Tx[q], src);
                if (!XO || WR > 0) src = mad(by, Ty[q], src);
                s[q] = src;
                const P vx = mad(a.C_nld, T3, C_d), vy = XO ? a.C_nld * T3 : vx;
                gx[q] = vx * Tx[q];
                gy[q] = vy * Ty[q];
            }
            E::sums_flux(s, gx, mu[b], K, K.kx);
            E::sums(gy, nu[b], K);
        }
        P done[NB];  // x components of the row this element row finishes
        auto to_rows = [&](auto scatter) {
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                P s[Q], f[Q], eta[NB], add[NB];
#pragma unroll
                for (int b = 0; b < Q; ++b) {
                    s[b] = mu[b][j];
                    f[b] = nu[b][j];
                }
                E::sums_flux(s, f, eta, K, K.ky);
                scatter(eta, add);
                done[j] = acc[0][j] + add[0];
#pragma unroll
                for (int l = 0; l + 1 < PD; ++l) acc[l][j] = acc[l + 1][j] + add[l + 1];
                acc[PD - 1][j] = add[PD];
            }
        };
        if (__builtin_expect(edge, 0))
            to_rows([&](const P(&eta)[NB], P(&add)[NB]) { edge_rows(ey, eta, add); });
        else
            to_rows([&](const P(&eta)[NB], P(&add)[NB]) { E::scatter(eta, add, K); });
        if (__builtin_expect(hot > 0, 0)) {
            // reaction: E and E phi at the points, their loads into R and into the fuel sums
            const P* phi0 = at_slot(a.phi, off);
            P pv[Q][NB];
            {
                P pw[NB][NB];
#pragma unroll
                for (int l = 0; l < NB; ++l) {
                    P x[NB];
                    fetch(row_of(phi0, ey + l), x);
                    xcomps(x, pw[l]);
                }
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    P x[NB], c[NB], v[Q];
#pragma unroll
                    for (int l = 0; l < NB; ++l) x[l] = pw[l][j];
                    if (edge) edge_comps(ey, x, c);
                    else E::comps(x, c);
                    E::value(c, v, K);
#pragma unroll
                    for (int b = 0; b < Q; ++b) pv[b][j] = v[b];
#pragma unroll
                    for (int m = 0; m < NB; ++m) c[m] = tc[m][j];
                    E::value(c, v, K);
#pragma unroll
                    for (int b = 0; b < Q; ++b) yv[b][j] = v[b];
                }
            }
            P me[Q][NB], mp[Q][NB];
#pragma unroll
            for (int b = 0; b < Q; ++b) {
                P T[Q], ph[Q], Ev[Q], Ep[Q];
                E::value(yv[b], T, K);
                E::value(pv[b], ph, K);
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const bool burn = T[q] > a.T_ig && ph[q] > a.phi_min;
                    const P e = burn ? T[q] * arrhenius(a.Ta_l2, a.T_a, T[q]) : P(0);
                    Ep[q] = e * ph[q];
                    Ev[q] = a.heat_by_fuel ? Ep[q] : e;
                }
                E::sums(Ev, me[b], K);
                E::sums(Ep, mp[b], K);
            }
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                P s[Q], eta[NB], add[NB];
#pragma unroll
                for (int b = 0; b < Q; ++b) s[b] = me[b][j];
                E::sums(s, eta, K);
                if (edge) edge_rows(ey, eta, add);
                else E::scatter(eta, add, K);
                done[j] = mad(a.K_ign, add[0], done[j]);
#pragma unroll
                for (int l = 0; l < PD; ++l) acc[l][j] = mad(a.K_ign, add[l + 1], acc[l][j]);
                if (Phi0) {
#pragma unroll
                    for (int b = 0; b < Q; ++b) s[b] = mp[b][j];
                    E::sums(s, eta, K);
                    if (edge) edge_rows(ey, eta, add);
                    else E::scatter(eta, add, K);
                    // sums of test row ey + l at ring slot (i + l) mod (p + 1)
                    int sl = i % NB;
#pragma unroll
                    for (int l = 0; l < NB; ++l) {
                        P* g = accg + (sl * NB + j) * 32 + lane;
                        *g = i + l <= fuel_to ? *g + add[l] : add[l];
                        sl = sl + 1 < NB ? sl + 1 : 0;
                    }
                }
            }
            fuel_to = i + PD;
        }
        const P r = a.Rw * gather(done);
        P f = P(0);
        if (__builtin_expect(i <= fuel_to, 0)) {
            if (Phi0) {
                P m[NB];
#pragma unroll
                for (int j = 0; j < NB; ++j) m[j] = accg[((i % NB) * NB + j) * 32 + lane];
                f = a.fscale * gather(m);
            }
        }
        if (out_col && i >= PD) {
            const_cast<P*>(tp)[dR] = r;
            if (Phi0) const_cast<P*>(tp)[dPhi] = f;
        }
    }
}

// Resident warps (one-warp CTAs) per SM the registers are budgeted for.
template <int PD>
struct QuadOcc {
    static constexpr int value = PD <= 2 ? 24 : 16;
};

template <typename P, int PD, int WR, bool XO>
__global__ void __launch_bounds__(32, QuadOcc<PD>::value) k_quad(const __grid_constant__ QuadArgs<P> a) {
    constexpr int NB = PD + 1;
    __shared__ P accg[NB * NB * 32];  // fuel sums of the unfinished rows: [row mod NB][x component][lane]
    extern __shared__ __align__(16) unsigned char wind_rows[];
    long long off = (long long)blockIdx.z * a.b.sbytes;
    grid_wait(off);
    if (!scene_active(a.b)) return;
    const int lane = threadIdx.x;
    const int sg = blockIdx.x / a.ns, strip = a.s0 + (blockIdx.x - sg * a.ns);
    const int X0 = strip * (32 - PD), Y0 = sg * a.h;
    P* wsm = reinterpret_cast<P*>(wind_rows);
    quad_strip<P, PD, WR, XO>(a, off, lane, X0, Y0, accg, wsm);
}

// Row-parallel form: a CTA of NW warps walks down a strip NW element rows a round, a row per warp; x components
// of the coefficient rows and the loads of the element rows go through rings in shared memory, and each warp
// finishes the output row of its element row (the same sums in the same order as the serial form: the same
// bits).  A segment recomputes p element rows once per CTA instead of once per warp, a small domain has the
// latency of one row instead of 1 + p of them, and the rows of a fire, two to three times as long, are spread over
// the warps of a CTA.  FP64 always takes it: the pipe issues a warp's instruction in 16 cycles, a quarter
// of that per scheduler, so the warp with the fire's rows was alone at the end (8 x 259^2 cubic: FP64
// pipe 71% of the kernel's time, quadrature 1135 us; now 867 us; 66^2: 57 -> 30; 1026^2: 640 -> 626).
// In FP32 the shared-memory traffic costs about a tenth more instructions: see the rule in run_quad.
template <typename P, int PD, int NW>
struct RowsSmem {
    static constexpr int NB = PD + 1, RS = NW + PD;  // ring of rows
    static constexpr bool kApart = sizeof(P) == 4;
    P comps[RS][NB][32];      // x components of coefficient rows
    P add[RS][NB * NB][32];   // loads of an element row: [test row][x component]
    P fuel[RS][NB * NB][32];  // its fuel sums
    // FP32: its reaction loads, added last as the serial form does; FP64, which has this form alone, adds them
    // to the others at once (1026^2: step 688 us, 708 with the third array)
    P react[kApart ? RS : 1][NB * NB][32];
    int hot_c[RS], hot_e[RS]; // coefficient rows above T_ig, element rows with fuel sums
};

// A barrier of the CTA whose warps arrive from different branches.  PTX counts the threads at barrier 0, by whichever
// instruction they arrive; __syncthreads asks in addition that the whole CTA takes the same branch.  (One barrier ahead of the
// reaction, in no branch, makes FP64 steps up to 5 % longer; one after it, with the loads kept across, spills.)
__device__ __forceinline__ void cta_barrier() { asm volatile("barrier.sync 0;" ::: "memory"); }

template <typename P, int PD, int WR, bool XO, int NW, typename SM>
__device__ __forceinline__ void quad_rows(const QuadArgs<P>& a, long long off, int lane, int w, int X0, int Y0, SM& sm, P* wsm) {
    using E = El<PD, P>;
    constexpr int NB = PD + 1, Q = PD + 1, WRm = WR > 0 ? WR : 1, RS = NW + PD;
    const ElK<P>& K = a.K;
    const P* T0 = at_slot(a.T, off);
    P* Phi0 = at_slot(a.Phi, off);
    P* R0 = at_slot(a.R, off);
    const P* mw = at_slot(a.mw, off);
    const int ex = X0 - PD + lane;  // element column of this lane; also its DOF column
    const bool ex_ok = ex >= 0 && ex < a.nx;
    const bool out_col = lane >= PD && ex < a.Nx;
    const bool xb = X0 < 2 * PD || X0 + 31 >= a.nx;  // the strip reaches the x boundary
    const Ends<PD, P> xe(ex, a.nx);
    const int rows = min(a.h, a.Ny - Y0);  // output rows of this item
    const int e0 = Y0 - PD, ne = rows + PD;  // element rows e0 .. e0 + ne - 1

    P fx[WRm][Q], fy[WRm][Q];
    const P mwx = a.cwx * mw[0], mwy = XO ? P(0) : a.cwy * mw[1];
    if constexpr (WR > 0) {
        const P* fxq = at_slot(a.fxq, off);
        const P* fyq = at_slot(a.fyq, off);
        const P* gxq = at_slot(a.gxq, off);
        const P* gyq = at_slot(a.gyq, off);
#pragma unroll
        for (int r = 0; r < WR; ++r)
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const size_t o = (size_t)r * a.nx * Q + (size_t)(ex_ok ? ex : 0) * Q + q;
                fx[r][q] = ex_ok ? a.cwx * fxq[o] : P(0);
                fy[r][q] = ex_ok ? a.cwy * fyq[o] : P(0);
            }
        // [row][x, y][r][point]
        for (int i = threadIdx.x; i < ne * WR * Q; i += 32 * NW) {
            const int row = i / (WR * Q), rq = i - row * WR * Q, r = rq / Q, q = rq - r * Q;
            const int ey = e0 + row;
            const bool ok = ey >= 0 && ey < a.ny;
            const size_t o = (size_t)r * a.ny * Q + (size_t)(ok ? ey : 0) * Q + q;
            wsm[(row * 2 + 0) * WR * Q + rq] = ok ? gxq[o] : P(0);
            wsm[(row * 2 + 1) * WR * Q + rq] = ok ? gyq[o] : P(0);
        }
    }
    const int shift = min(max(ex, 0), a.nx - 1) - ex;
    auto row_of = [&](const P* f, int r) {
        return f + ((long long)min(max(r, 0), a.Ny - 1) * a.pitch + ex);
    };
    auto fetch = [&](const P* row, P (&x)[NB]) {
        const P* c = row + shift;
#pragma unroll
        for (int k = 0; k < NB; ++k) x[k] = field_load(c + k);
    };
    auto xcomps = [&](P (&x)[NB], P (&c)[NB]) {
        if (PD > 1 && xb) xe.apply(x);
        E::comps(x, c);
    };
    auto gather = [&](const P (&m)[NB]) {
        P kx[NB];
        E::scatter(m, kx, K);
        if (xb) {
            xe.transpose(kx);
#pragma unroll
            for (int k = 0; k < NB; ++k) kx[k] = ex_ok ? kx[k] : P(0);
        }
        P r = kx[0];
#pragma unroll
        for (int k = 1; k < NB; ++k) r += __shfl_up_sync(kFull, kx[k], k);
        return r;
    };
    auto ycomps = [&](bool edge, int e, P (&x)[NB], P (&c)[NB]) {
        if (__builtin_expect(edge, 0)) Ends<PD, P>(e, a.ny).apply(x);
        E::comps(x, c);
    };
    auto yrows = [&](bool edge, int e, const P (&eta)[NB], P (&add)[NB]) {
        E::scatter(eta, add, K);
        if (__builtin_expect(edge, 0)) Ends<PD, P>(e, a.ny).transpose(add);
    };
    // x components of coefficient row e0 + c into its slot
    auto put = [&](int slot, P (&x)[NB]) {
        const bool h = __any_sync(kFull, larger(x[0], x[PD]) > a.T_ig_lo);
        P c[NB];
        xcomps(x, c);
#pragma unroll
        for (int j = 0; j < NB; ++j) sm.comps[slot][j][lane] = c[j];
        if (lane == 0) sm.hot_c[slot] = h;
    };
    const P c_chi = held(a.c_chi), C_d = held(a.C_d);
    P nxt[NB];
    for (int c = w; c < RS; c += NW) {
        fetch(row_of(T0, e0 + c), nxt);
        put(c, nxt);
    }
    fetch(row_of(T0, e0 + RS + w), nxt);
    if (w < PD && lane == 0) sm.hot_e[RS - 1 - w] = 0;
    __syncthreads();
    int si = w;  // slot of row i: i mod RS
    for (int i0 = 0; i0 < ne; i0 += NW) {
        const int i = i0 + w, ey = e0 + i;
        const bool edge = ey < PD || ey >= a.ny - PD;
        const bool in = i < ne && ey >= 0 && ey < a.ny;
        P add[NB][NB];  // [test row][x component]
        P tc[NB][NB];   // tensor components of the element: [y component][x component]
        bool hot = false;
        if (in) {
            int sl[NB];
#pragma unroll
            for (int l = 0; l < NB; ++l) sl[l] = si + l < RS ? si + l : si + l - RS;
#pragma unroll
            for (int l = 0; l < NB; ++l) hot = hot || sm.hot_c[sl[l]];
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                P x[NB], c[NB];
#pragma unroll
                for (int l = 0; l < NB; ++l) x[l] = sm.comps[sl[l]][j][lane];
                ycomps(edge, ey, x, c);
#pragma unroll
                for (int m = 0; m < NB; ++m) tc[m][j] = c[m];
            }
            P yv[Q][NB], yd[Q][NB];  // [y point][x component]: T and its y derivative
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                P c[NB], v[Q], d[Q];
#pragma unroll
                for (int m = 0; m < NB; ++m) c[m] = tc[m][j];
                E::value(c, v, K);
                E::deriv(c, d, K);
#pragma unroll
                for (int b = 0; b < Q; ++b) {
                    yv[b][j] = v[b];
                    yd[b][j] = d[b];
                }
            }
            P mu[Q][NB], nu[Q][NB];  // x sums of the value and x-flux terms, of the y flux
#pragma unroll
            for (int b = 0; b < Q; ++b) {
                P T[Q], Tx[Q], Ty[Q], s[Q], gx[Q], gy[Q];
                E::value(yv[b], T, K);
                E::deriv(yv[b], Tx, K);
                E::value(yd[b], Ty, K);
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const P T3 = (T[q] * T[q]) * T[q];
                    P src = mad(T[q], mad(-a.c_rad, T3, -c_chi), a.K0);
                    P bx = mwx, by = mwy;
#pragma unroll
                    for (int r = 0; r < WR; ++r) {
                        bx = mad(fx[r][q], wsm[(i * 2 + 0) * WR * Q + r * Q + b], bx);
                        by = mad(fy[r][q], wsm[(i * 2 + 1) * WR * Q + r * Q + b], by);
                    }
                    src = mad(bx, Tx[q], src);
                    if (!XO || WR > 0) src = mad(by, Ty[q], src);
                    s[q] = src;
                    const P vx = mad(a.C_nld, T3, C_d), vy = XO ? a.C_nld * T3 : vx;
                    gx[q] = vx * Tx[q];
                    gy[q] = vy * Ty[q];
                }
                E::sums_flux(s, gx, mu[b], K, K.kx);
                E::sums(gy, nu[b], K);
            }
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                P s[Q], f[Q], eta[NB], t[NB];
#pragma unroll
                for (int b = 0; b < Q; ++b) {
                    s[b] = mu[b][j];
                    f[b] = nu[b][j];
                }
                E::sums_flux(s, f, eta, K, K.ky);
                yrows(edge, ey, eta, t);
#pragma unroll
                for (int l = 0; l < NB; ++l) add[l][j] = t[l];
            }
        } else {
#pragma unroll
            for (int l = 0; l < NB; ++l)
#pragma unroll
                for (int j = 0; j < NB; ++j) add[l][j] = P(0);
        }
        if (__builtin_expect(hot, 0)) {
            // reaction: E and E phi at the points, their loads
            const P* phi0 = at_slot(a.phi, off);
            P pv[Q][NB], yv[Q][NB];
            {
                P pw[NB][NB];
#pragma unroll
                for (int l = 0; l < NB; ++l) {
                    P x[NB];
                    fetch(row_of(phi0, ey + l), x);
                    xcomps(x, pw[l]);
                }
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    P x[NB], c[NB], v[Q];
#pragma unroll
                    for (int l = 0; l < NB; ++l) x[l] = pw[l][j];
                    ycomps(edge, ey, x, c);
                    E::value(c, v, K);
#pragma unroll
                    for (int b = 0; b < Q; ++b) pv[b][j] = v[b];
#pragma unroll
                    for (int m = 0; m < NB; ++m) c[m] = tc[m][j];
                    E::value(c, v, K);
#pragma unroll
                    for (int b = 0; b < Q; ++b) yv[b][j] = v[b];
                }
            }
            P me[Q][NB], mp[Q][NB];
#pragma unroll
            for (int b = 0; b < Q; ++b) {
                P T[Q], ph[Q], Ev[Q], Ep[Q];
                E::value(yv[b], T, K);
                E::value(pv[b], ph, K);
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const bool burn = T[q] > a.T_ig && ph[q] > a.phi_min;
                    const P e = burn ? T[q] * arrhenius(a.Ta_l2, a.T_a, T[q]) : P(0);
                    Ep[q] = e * ph[q];
                    Ev[q] = a.heat_by_fuel ? Ep[q] : e;
                }
                E::sums(Ev, me[b], K);
                E::sums(Ep, mp[b], K);
            }
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                P s[Q], eta[NB], t[NB];
#pragma unroll
                for (int b = 0; b < Q; ++b) s[b] = me[b][j];
                E::sums(s, eta, K);
                yrows(edge, ey, eta, t);
#pragma unroll
                for (int l = 0; l < NB; ++l) {
                    if (SM::kApart) me[l][j] = t[l];  // (Q = NB)
                    else add[l][j] = mad(a.K_ign, t[l], add[l][j]);
                }
                if (Phi0) {
#pragma unroll
                    for (int b = 0; b < Q; ++b) s[b] = mp[b][j];
                    E::sums(s, eta, K);
                    yrows(edge, ey, eta, t);
#pragma unroll
                    for (int l = 0; l < NB; ++l) mp[l][j] = t[l];
                }
            }
            cta_barrier();
#pragma unroll
            for (int l = 0; l < NB; ++l)
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    if (SM::kApart) sm.react[si][l * NB + j][lane] = me[l][j];
                    if (Phi0) sm.fuel[si][l * NB + j][lane] = mp[l][j];
                }
        } else {
            cta_barrier();
        }
#pragma unroll
        for (int l = 0; l < NB; ++l)
#pragma unroll
            for (int j = 0; j < NB; ++j) sm.add[si][l * NB + j][lane] = add[l][j];
        if (lane == 0) sm.hot_e[si] = hot;
        put(si, nxt);  // coefficient row i + RS
        __syncthreads();
        if (i0 + NW < ne) fetch(row_of(T0, ey + RS + NW), nxt);
        if (i >= PD && i < ne) {
            P m[NB];
            int sl = si - PD < 0 ? si - PD + RS : si - PD;
            int any = 0;
#pragma unroll
            for (int l = PD; l >= 0; --l) {
#pragma unroll
                for (int j = 0; j < NB; ++j) m[j] = l == PD ? sm.add[sl][l * NB + j][lane] : m[j] + sm.add[sl][l * NB + j][lane];
                if (__builtin_expect(sm.hot_e[sl], 0)) {
                    any = 1;
                    if constexpr (SM::kApart)
#pragma unroll
                        for (int j = 0; j < NB; ++j) m[j] = mad(a.K_ign, sm.react[sl][l * NB + j][lane], m[j]);
                }
                sl = sl + 1 < RS ? sl + 1 : 0;
            }
            const P r = a.Rw * gather(m);
            P f = P(0);
            if (Phi0 && __builtin_expect(any, 0)) {
#pragma unroll
                for (int j = 0; j < NB; ++j) m[j] = P(0);
                sl = si - PD < 0 ? si - PD + RS : si - PD;
#pragma unroll
                for (int l = PD; l >= 0; --l) {
                    if (sm.hot_e[sl])
#pragma unroll
                        for (int j = 0; j < NB; ++j) m[j] += sm.fuel[sl][l * NB + j][lane];
                    sl = sl + 1 < RS ? sl + 1 : 0;
                }
                f = a.fscale * gather(m);
            }
            if (out_col) {
                const size_t o = (size_t)ey * a.pitch + ex;
                R0[o] = r;
                if (Phi0) Phi0[o] = f;
            }
        }
        si = si + NW < RS ? si + NW : si + NW - RS;
    }
}

constexpr int kRowWarps = 4;

template <typename P, int PD>
struct RowOcc {  // CTAs per SM
    static constexpr int value = sizeof(P) == 4 ? (PD <= 2 ? 6 : 4) : 2;
};

template <typename P, int PD, int WR, bool XO, int NW>
__global__ void __launch_bounds__(32 * NW, RowOcc<P, PD>::value) k_quad_rows(const __grid_constant__ QuadArgs<P> a) {
    extern __shared__ __align__(16) unsigned char wind_rows[];
    long long off = (long long)blockIdx.z * a.b.sbytes;
    grid_wait<sizeof(P) == 4>(off);  // (FP64: see even_smem)
    if (!scene_active(a.b)) return;
    using SM = RowsSmem<P, PD, NW>;
    SM& sm = *reinterpret_cast<SM*>(wind_rows);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int sg = blockIdx.x / a.ns, strip = a.s0 + (blockIdx.x - sg * a.ns);
    quad_rows<P, PD, WR, XO, NW>(a, off, lane, w, strip * (32 - PD), sg * a.h, sm,
                                 reinterpret_cast<P*>(wind_rows + sizeof(SM)));
}

// Shared memory a CTA asks for so that `ctas` CTAs spread evenly: no SM holds more than ctas / sms of them, rounded up.
// The FP64 quadrature is few long CTAs (rounds of element rows on the busiest SM set its time, run_quad).  Started beside the
// last CTAs of a y pass, they all went to the SMs that were free then, two or three to an SM beside idle
// ones: 8 x 258^2, PR step 866 us, 377 with this; 64 x 42^2 Strang 885 and 315; 402^2 cubic 514 and 355.
// Its own CTAs do not let the next kernel start early: x tiles waiting beside them made it slower (8 x 67 x 303 cubic
// 410 us, 393 without).
inline size_t even_smem(size_t need, long ctas, int sms) {
    constexpr size_t per_sm = 228 * 1024, per_cta = 227 * 1024, reserved = 1024;  // of an SM; at most, and by the system, of a CTA
    const size_t fit = (size_t)((ctas + sms - 1) / sms);
    const size_t most = per_sm / (fit + 1) / 128 * 128 + 128 - reserved;  // fit + 1 of them are more than an SM holds
    return most > need && most <= per_cta ? most : need;
}

template <typename P>
void fill_elk(int p, double gx, double gy, ElK<P>& K) {
    double a[13] = {0}, k[3] = {0};
    if (p == 1) {
        a[0] = 0.5 / sqrt(3.0);
        k[0] = 1.0 / a[0];
    } else if (p == 2) {
        const double t = 0.5 * sqrt(0.6);
        a[0] = 0.5 * t, a[1] = 0.5 * t * t, a[2] = 2.0 * t, a[3] = 1.6;
        k[0] = 2.0 / t, k[1] = 4.0 / t;
    } else {
        const double r = 2.0 / 7.0 * sqrt(1.2);
        const double t1 = 0.5 * sqrt(3.0 / 7.0 - r), t2 = 0.5 * sqrt(3.0 / 7.0 + r);
        const double rho = (18.0 + sqrt(30.0)) / (18.0 - sqrt(30.0)), u = t1 / t2;
        a[0] = t1, a[1] = t2, a[2] = 0.25 * t1 * t1, a[3] = 0.25 * t2 * t2, a[4] = t1 * t1 / 6.0, a[5] = t2 * t2 / 6.0;
        a[6] = 0.5 * t1 * t1, a[7] = 0.5 * t2 * t2, a[8] = rho, a[9] = rho * u, a[10] = u * u;
        a[11] = t2 * t2 * t2 / 6.0, a[12] = 0.125 * t2;
        k[0] = 1.0 / t2, k[1] = 2.0 / t2, k[2] = 3.0 / t2;
    }
    for (int i = 0; i < 13; ++i) K.a[i] = (P)a[i];
    for (int i = 0; i < 3; ++i) {
        K.kx[i] = (P)(-gx * gx * k[i]);
        K.ky[i] = (P)(-gy * gy * k[i]);
    }
}

// weight of the outermost Gauss point on [0, 1]
inline double outer_weight(int p) {
    return p == 1 ? 0.5 : (p == 2 ? 5.0 / 18.0 : (18.0 - sqrt(30.0)) / 72.0);
}

template <typename P, int PD, int WR, bool XO>
cudaError_t run_quad(const RhsArgs& r, cudaStream_t s) {
    QuadArgs<P> a;
    a.nx = r.nx;
    a.ny = r.ny;
    a.Nx = r.Nx;
    a.Ny = r.Ny;
    a.pitch = r.pitch;
    a.T = (const P*)r.T;
    a.phi = (const P*)r.phi;
    a.Phi = (P*)r.Phi;
    a.R = (P*)r.R;
    a.fxq = (const P*)r.fxq;
    a.gxq = (const P*)r.gxq;
    a.fyq = (const P*)r.fyq;
    a.gyq = (const P*)r.gyq;
    a.mw = (const P*)r.mw;
    // dT/dx = derivative of El / (h or 2h)
    const double gx = 1.0 / ((PD == 2 ? 2.0 : 1.0) * r.hx), gy = 1.0 / ((PD == 2 ? 2.0 : 1.0) * r.hy);
    const double w = r.hx * r.hy * outer_weight(PD) * outer_weight(PD);
    const Phys& c = r.phys;
    a.cwx = (P)(-c.c_W * gx);
    a.cwy = (P)(-c.c_W * gy);
    a.T_ig = (P)c.T_ig;
    a.T_ig_lo = (P)(c.T_ig * (1.0 - 1e-5));
    a.phi_min = (P)c.phi_min;
    a.Ta_l2 = (P)(c.T_a * 1.4426950408889634074);  // log2(e)
    a.T_a = (P)c.T_a;
    a.fscale = (P)(-r.tau * c.k_f * w);
    a.heat_by_fuel = c.heat_by_fuel;
    a.Rw = (P)(r.Rscale * w);
    a.K0 = (P)(c.c_chi * c.T_amb + c.c_rad * c.T_amb * c.T_amb * c.T_amb * c.T_amb);
    a.c_rad = (P)c.c_rad;
    a.c_chi = (P)c.c_chi;
    a.C_nld = (P)c.C_nld;
    a.C_d = (P)c.C_d;
    a.K_ign = (P)c.K_ign;
    fill_elk<P>(PD, gx, gy, a.K);
    a.b = r.b;
    a.nstrips = (r.Nx + (32 - PD) - 1) / (32 - PD);
    int sms = 152, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // interior strips: X0 >= 2p and X0 + 31 < nx
    int lo = (2 * PD + (32 - PD) - 1) / (32 - PD), hi = r.nx > 31 ? (r.nx - 32) / (32 - PD) + 1 : 0;
    if (lo > a.nstrips) lo = a.nstrips;
    if (hi < lo) hi = lo;
    // one launch over every strip; r.parts: the strips left of the interior ones, the interior ones and
    // the strips right of them in launches of their own (FP32 with interior strips)
    const bool parts = r.parts && sizeof(P) == 4 && hi > lo;
    const int cut[4] = {0, parts ? lo : a.nstrips, parts ? hi : a.nstrips, a.nstrips};
    // the segment's wind factors stay within 48 KB of shared memory, beside the sums
    auto wind_bytes = [](int h) { return (size_t)2 * WR * (PD + 1) * (h + PD) * sizeof(P); };
    const long strips = (long)a.nstrips * r.b.S;
    auto launch = [&](auto kern, int hgt, int threads, size_t ring) {
        if (r.seg > 0) hgt = r.seg;
        if (hgt > r.Ny) hgt = r.Ny;
        while (hgt > 1 && wind_bytes(hgt) > 48 * 1024) hgt /= 2;
        const int nseg = (r.Ny + hgt - 1) / hgt;
        a.h = threads == 32 ? (r.Ny + nseg - 1) / nseg : hgt;
        size_t smem = ring + wind_bytes(a.h);
        if (sizeof(P) == 8) smem = even_smem(smem, strips * nseg, sms);
        if (smem > 24 * 1024) {
            cudaError_t e = allow_dynamic_smem(kern, smem);
            if (e != cudaSuccess) return e;
        }
        for (int k = 0; k < 3; ++k) {
            a.s0 = cut[k];
            a.ns = cut[k + 1] - cut[k];
            if (a.ns <= 0) continue;
            const cudaError_t e =
                launch_overlapped(kern, dim3((unsigned)(a.ns * nseg), 1, r.b.S), threads, smem, s, a);
            if (e != cudaSuccess) return e;
            count_launches(1);
        }
        return cudaSuccess;
    };
    constexpr int NW = kRowWarps;
    const size_t ring = sizeof(RowsSmem<P, PD, NW>);
    if constexpr (sizeof(P) == 8) {
        // Height by the FP64 pipe: rounds of NW element rows on the busiest SM, fewest first, then the lower
        // segment (8 x 259^2 cubic, step at height 65 (its rule): 932 us, 1096 at 52, 963 at 33).
        int h = r.Ny;
        long best = 0;
        for (int n = 1; n <= r.Ny && strips * (n - 1) < 8L * sms; ++n) {
            const int hn = (r.Ny + n - 1) / n;
            const long ctas = strips * ((r.Ny + hn - 1) / hn);
            const long cost = (ctas + sms - 1) / sms * ((hn + PD + NW - 1) / NW);
            if (best == 0 || cost <= best) best = cost, h = hn;
        }
        return launch(k_quad_rows<P, PD, WR, XO, NW>, h, 32 * NW, ring);
    } else {
        const double rows_sm = (double)strips * r.Ny / sms;  // element rows per SM
        // Row-parallel while the rows are few enough for latency to decide; its height weighs the rounds of a
        // segment against the element rows recomputed (a round is one row's latency; eight rows per SM take
        // about as long to issue).  Step, serial / row-parallel: 130^2 16.4 / 13.9 us, 402^2 25.4 / 24.1
        // (37 rows per SM), 642^2 26.7 / 28.5 (93); cubic 100 x 64 Strang 53 / 37, 515^2 46.9 / 37.2 (61), 643^2
        // 47.7 / 42.0 (97), 803^2 50.5 / 52.3 (148); linear within 0.8 us up to 60.
        if (rows_sm <= (PD <= 2 ? 48 : 128)) {
            int h = NW - PD;
            double best = 1e30;
            for (int g = 1; g <= 16; ++g) {
                const int hn = NW * g - PD;
                const double cost = g + 0.125 * rows_sm * (hn + PD) / hn;
                if (hn >= 1 && cost < best) best = cost, h = hn;
            }
            return launch(k_quad_rows<P, PD, WR, XO, NW>, h, 32 * NW, ring);
        }
        // Segment height of the serial form: a segment recomputes p element rows, so high ones do less work;
        // but below about the resident number of warps per SM the SMs idle on latency.  The largest power of two
        // from 64 down that gives nine tenths of the resident warps an item, then equal segments.
        // Step, 1026^2: 34.7 us at height 8 (its rule), 34.5 at 13, 36.6 at 20, 38.9 at 30; 8 x 515^2
        // cubic: 102.9 at 31 (its rule), 109 at 24, 118 at 52; 4099^2 cubic: 537 at 64 (its rule), 554 at 32, 550 at 128.
        int h = 64;
        const long want = (long)QuadOcc<PD>::value * sms * 9 / 10;
        while (h > 1 && strips * ((r.Ny + h - 1) / h) < want) h /= 2;
        return launch(k_quad<P, PD, WR, XO>, h, 32, 0);
    }
}

// instantiations by wind rank (ranks 3 and 4 run as 4, rank 1 as 2: the unused factors are zero) and
// by operator
template <typename P, int PD>
cudaError_t quad_by_rank(const RhsArgs& r, cudaStream_t s) {
    if (r.wind_rank < 0 || r.wind_rank > kMaxRank) return cudaErrorInvalidValue;
    if (r.xonly) {
        if (r.wind_rank == 0) return run_quad<P, PD, 0, true>(r, s);
        if (r.wind_rank <= 2) return run_quad<P, PD, 2, true>(r, s);
        return run_quad<P, PD, 4, true>(r, s);
    }
    if (r.wind_rank == 0) return run_quad<P, PD, 0, false>(r, s);
    if (r.wind_rank <= 2) return run_quad<P, PD, 2, false>(r, s);
    return run_quad<P, PD, 4, false>(r, s);
}

}  // namespace
}  // namespace wf
