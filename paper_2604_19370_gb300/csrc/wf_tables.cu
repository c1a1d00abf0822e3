// Tables and 1-D factorisations, computed on the GPU in FP64 once per handle.
//
// Paper: the 1-D mass, stiffness and advection matrices of Sec. 3.1 ("Matrix
// formulation") and the banded direct solvers of Sec. 4 ("Cost of directional
// implicit solves").  Every directional operator is a combination
// aM M + aK K + aG G of these matrices; its LU factors are computed here
// together with the transfers of a recursion's state through chunks of rows, so
// that the line solves of every step run with many chunks per line at once.
#include <math.h>

#include "wf_internal.h"

namespace wf {

namespace {

// Gauss-Legendre nodes and weights on [0, 1] by Newton's method on the
// Legendre polynomial P_q (three-term recurrence), one thread per node.
__global__ void k_gauss(double* xi, double* w, int q) {
    int i = threadIdx.x;
    if (i >= q) return;
    const double pi = 3.14159265358979323846;
    double x = cos(pi * (i + 0.75) / (q + 0.5));
    double dp = 1.0;
    for (int it = 0; it < 100; ++it) {
        double p0 = 1.0, p1 = x;
        for (int k = 2; k <= q; ++k) {
            double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        dp = q * (x * p1 - p0) / (x * x - 1.0);
        double dx = p1 / dp;
        x -= dx;
        if (fabs(dx) < 1e-16) break;
    }
    {
        double p0 = 1.0, p1 = x;
        for (int k = 2; k <= q; ++k) {
            double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        dp = q * (x * p1 - p0) / (x * x - 1.0);
    }
    xi[i] = 0.5 * (1.0 - x);
    w[i] = 1.0 / ((1.0 - x * x) * dp * dp);  // (2 / ((1-x^2) P_q'^2)) / 2
}

// Knot t_j of the open uniform knot vector relative to the start of element e, as
// (integer) * h: the same bits for every interior element, so the tables, the
// assembled bands and the chunk factors of interior rows are exactly translation
// invariant.
__device__ inline double knot_rel(int j, int e, int n, int p, double h) {
    int m = j - p;
    m = m < 0 ? 0 : (m > n ? n : m);
    return (double)(m - e) * h;
}

// Basis values and derivatives at the Gauss points of every element, by the
// triangular (left/right difference) evaluation of the nonzero B-splines of
// a knot span, in coordinates relative to the element start.  One thread per
// (element, point).
__global__ void k_basis(const double* __restrict__ xi, int q, int n, int p, double L, double* B, double* D) {
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * q) return;
    const int e = idx / q, a = idx % q;
    const double h = L / n;
    const int span = e + p;
    const double x = xi[a] * h;  // offset of the point inside element e
    double left[kMaxP + 1], right[kMaxP + 1], Nv[kMaxP + 1], Nm[kMaxP + 1];
    Nv[0] = 1.0;
    Nm[0] = 1.0;
    for (int j = 1; j <= p; ++j) {
        left[j] = x - knot_rel(span + 1 - j, e, n, p, h);
        right[j] = knot_rel(span + j, e, n, p, h) - x;
        double saved = 0.0;
        for (int r = 0; r < j; ++r) {
            double tmp = Nv[r] / (right[r + 1] + left[j - r]);
            Nv[r] = saved + right[r + 1] * tmp;
            saved = left[j - r] * tmp;
        }
        Nv[j] = saved;
        if (j == p - 1)
            for (int r = 0; r <= j; ++r) Nm[r] = Nv[r];
    }
    for (int l = 0; l <= p; ++l) {
        const int i = span - p + l;
        double d = 0.0;
        if (p > 0) {
            if (l >= 1) {
                double den = knot_rel(i + p, e, n, p, h) - knot_rel(i, e, n, p, h);
                if (den > 0.0) d += p * Nm[l - 1] / den;
            }
            if (l <= p - 1) {
                double den = knot_rel(i + p + 1, e, n, p, h) - knot_rel(i + 1, e, n, p, h);
                if (den > 0.0) d -= p * Nm[l] / den;
            }
        }
        B[(size_t)(e * q + a) * (p + 1) + l] = Nv[l];
        D[(size_t)(e * q + a) * (p + 1) + l] = d;
    }
}

// 1-D matrices by Gauss quadrature, one thread per band entry (row i, diagonal d).
// Row = test function, column = trial function (G carries the trial derivative).
__global__ void k_assemble(const double* __restrict__ B, const double* __restrict__ D, const double* __restrict__ w,
                           int q, int n, int p, double h, double* Mb, double* Kb, double* Gb) {
    const int N = n + p, W = 2 * p + 1;
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= N * W) return;
    const int i = idx / W, d = idx % W, k = i + d - p;
    double m = 0.0, kk = 0.0, g = 0.0;
    if (k >= 0 && k < N) {
        int lo = (i > k ? i : k) - p;
        int hi = i < k ? i : k;
        lo = lo < 0 ? 0 : lo;
        hi = hi > n - 1 ? n - 1 : hi;
        for (int e = lo; e <= hi; ++e) {
            const int li = i - e, lk = k - e;
            for (int a = 0; a < q; ++a) {
                const double wa = w[a] * h;
                const size_t o = (size_t)(e * q + a) * (p + 1);
                const double bi = B[o + li], bk = B[o + lk], di = D[o + li], dk = D[o + lk];
                m += wa * bi * bk;
                kk += wa * di * dk;
                g += wa * bi * dk;
            }
        }
    }
    Mb[idx] = m;
    Kb[idx] = kk;
    Gb[idx] = g;
}

__device__ __forceinline__ bool same_bits(double a, double b) {
    return __double_as_longlong(a) == __double_as_longlong(b);
}

// Factor tables of one operator per block (layout: wf_internal.h).  A thread owns a chunk of rows and runs the
// banded LU recursion (FP64, no pivoting) from the first row of the line down to its chunk, so every row has
// the factors of one sequential elimination; one division a row.  The FP64 pipe bounds it (a warp instruction takes
// 64 cycles of a scheduler, and a row has 25 to 90), so rows are what counts: those away from the ends of the line are the same,
// the recursion maps its state (the last p rows of U) to itself there, and once the state comes back bit for
// bit, after a few dozen rows, the ones left before the chunk are so many turns of the same cycle and are passed
// over (Brent's cycle search: the state is compared with a kept one, which is replaced after 1, 3, 7, ... rows).
// wf_set_mean_wind with every row / now, ms: 1024 x 4 quadratic FP32 2.0 / 0.33, 16000 x 4 63.5 / 0.76, 32768 x 4 cubic FP64
// 319 / 2.2; where no state comes back within the line, 300 x 200, kappa = 3e6: linear FP64 0.34 / 0.38, cubic 0.86 / 0.69.
template <typename P, int PD>
__global__ void __launch_bounds__(128) k_line_tables(const __grid_constant__ TabJobs jobs) {
    constexpr int W = 2 * PD + 1, NF = PD == 3 ? 4 : PD, NU = PD == 1 ? 2 : 4, S = PD * PD;
    const TabJob& jb = jobs.job[blockIdx.x];
    const long long off = (long long)blockIdx.y * jobs.sbytes;
    const int N = jb.N, M = jb.chunk, C = (N + M - 1) / M, tid = threadIdx.x;
    char* out = static_cast<char*>(jb.out) + off;
    auto entry = [&](int r, int d) {
        const int col = r + d - PD;
        const size_t o = (size_t)r * W + d;
        return (col >= 0 && col < N) ? jb.aM * jb.M[o] + jb.aK * jb.K[o] + jb.aG * jb.G[o] : 0.0;
    };
    if (blockIdx.x == 0 && tid == 0) {
        P* mw = reinterpret_cast<P*>(static_cast<char*>(jobs.mw) + off);
        mw[0] = (P)jobs.wind_x;
        mw[1] = (P)jobs.wind_y;
    }
    if (jb.band) {
        P* b = reinterpret_cast<P*>(out);
        for (int i = tid; i < N * 2 * PD; i += blockDim.x) {
            const int r = i / (2 * PD), e = i % (2 * PD), col = r + e - PD;  // factor of T[col + 1] - T[col]
            double v = 0.0;
            if (col >= 0 && col + 1 < N)
                for (int d = e + 1; d < W; ++d) v += entry(r, d);
            b[i] = (P)v;
        }
        return;
    }
    constexpr int NV = PD == 1 ? 2 : (PD == 2 ? 4 : 8), D = 2 * PD, EW = 2 * kEndRows;
    __shared__ int s_uni, s_J, s_bad, s_Ju;
    __shared__ double s_l[PD], s_u[PD], s_inv, s_T[2][PD][PD];  // uniform factors and transfers
    __shared__ double s_W[2 * D][EW];   // columns of B^{-1} at the first and last 2p unknowns, near each end
    __shared__ double s_H[2 * D][4 * D];
    if (tid == 0) s_uni = 0, s_J = 0, s_bad = 0, s_Ju = 0;
    __syncthreads();
    int* hdr = reinterpret_cast<int*>(out);
    P* gl = reinterpret_cast<P*>(out + kTabHeader);
    P* gu = gl + 4;
    P* gT = gu + 4;
    P* VT = gT + 2 * tab_round(S);
    P* VB = VT + (kEndRows + M) * NV;
    P* F = VB + (kEndRows + 2 * M) * NV;
    P* U = F + tab_round(C * M * NF);
    P* Pf = U + tab_round(C * M * NU);
    P* Pb = Pf + tab_round(C * S);
    for (int k = tid; k < C; k += blockDim.x) {
        double u[PD][PD], inv[PD];  // rows r-1 .. r-p: u_{r-i,r-i+j} and 1 / u_{r-i,r-i}
        double st[PD][PD];          // unit states carried through the chunk: [basis][value, nearest first]
        for (int a = 0; a < PD; ++a) {
            inv[a] = 0.0;
            for (int b = 0; b < PD; ++b) {
                u[a][b] = 0.0;
                st[a][b] = a == b ? 1.0 : 0.0;
            }
        }
        double anorm = 0.0;
        // row r of the elimination: its multipliers l, its row of U in w[p+1 ..], returns 1 / u_rr
        auto eliminate = [&](int r, double (&w)[W], double (&l)[PD]) {
            bool pad = r >= N;
            double rs = 0.0;
            for (int d = 0; d < W; ++d) {
                w[d] = pad ? (d == PD ? 1.0 : 0.0) : entry(r, d);
                rs += fabs(w[d]);
            }
            if (!pad && rs > anorm) anorm = rs;
#pragma unroll
            for (int i = PD; i >= 1; --i) {
                l[i - 1] = w[PD - i] * inv[i - 1];
#pragma unroll
                for (int j = 1; j <= PD; ++j) w[PD - i + j] -= l[i - 1] * u[i - 1][j - 1];
            }
            double piv = w[PD];
            if (!(fabs(piv) > 1e-300 * anorm)) {
                s_bad = 1;
                piv = 1.0;
            }
            const double iv = 1.0 / piv;
            for (int a = PD - 1; a > 0; --a) {
                inv[a] = inv[a - 1];
                for (int b = 0; b < PD; ++b) u[a][b] = u[a - 1][b];
            }
            inv[0] = iv;
            for (int b = 0; b < PD; ++b) u[0][b] = w[PD + 1 + b];
            return iv;
        };
        // the rows before the chunk; those from 2p to `stop` are the same
        const int stop = min(k * M, N - 2 * PD);
        double seen[PD][PD + 1];
        int mark = 2 * PD, span = 0;  // row of the state kept in `seen`, rows after which it is replaced
        for (int r = 0; r < k * M; ++r) {
            if (r >= mark && r < stop) {
                bool same = r > mark && same_bits(seen[0][PD], inv[0]);
                if (same)
                    for (int a = 0; a < PD; ++a) {
                        same = same && same_bits(seen[a][PD], inv[a]);
                        for (int b = 0; b < PD; ++b) same = same && same_bits(seen[a][b], u[a][b]);
                    }
                if (same) {
                    r += (stop - r) / (r - mark) * (r - mark);
                    mark = N;  // one time is enough
                    if (r == k * M) break;
                } else if (r - mark == span) {
                    for (int a = 0; a < PD; ++a) {
                        seen[a][PD] = inv[a];
                        for (int b = 0; b < PD; ++b) seen[a][b] = u[a][b];
                    }
                    mark = r;
                    span = 2 * span + 1;
                }
            }
            double w[W], l[PD];
            eliminate(r, w, l);
        }
        for (int r = k * M; r < (k + 1) * M; ++r) {
            double w[W], l[PD];
            const double iv = eliminate(r, w, l);
            for (int c = 0; c < NF; ++c) F[(size_t)r * NF + c] = c < PD ? (P)l[c < PD ? c : 0] : P(0);
            U[(size_t)r * NU] = (P)iv;
            for (int c = 1; c < NU; ++c) U[(size_t)r * NU + c] = c <= PD ? (P)(w[c <= PD ? PD + c : 0] * iv) : P(0);
            for (int b = 0; b < PD; ++b) {
                double y = 0.0;
                for (int a = 0; a < PD; ++a) y -= l[a] * st[b][a];
                for (int a = PD - 1; a > 0; --a) st[b][a] = st[b][a - 1];
                st[b][0] = y;
            }
        }
        for (int a = 0; a < PD; ++a)
            for (int b = 0; b < PD; ++b) Pf[(size_t)k * S + a * PD + b] = (P)st[b][a];
        // backward: the chunk's own U rows from its last one up
        for (int a = 0; a < PD; ++a)
            for (int b = 0; b < PD; ++b) st[a][b] = a == b ? 1.0 : 0.0;
        for (int r = (k + 1) * M - 1; r >= k * M; --r)
            for (int b = 0; b < PD; ++b) {
                double z = 0.0;
                for (int a = 0; a < PD; ++a) z -= (double)U[(size_t)r * NU + 1 + a] * st[b][a];
                for (int a = PD - 1; a > 0; --a) st[b][a] = st[b][a - 1];
                st[b][0] = z;
            }
        for (int a = 0; a < PD; ++a)
            for (int b = 0; b < PD; ++b) Pb[(size_t)k * S + a * PD + b] = (P)st[b][a];
    }
    __syncthreads();
    // Uniform factors: the fixed point of the elimination of an interior row (row 2p), if it converges.
    // (FP32: kUniformFactors, wf_internal.h)
    const double ulp = 1e-12;
    if (kUniformFactors<P> && tid == 0 && N > 4 * PD) {
        double u[PD][PD], inv[PD], l[PD], w[W];
        for (int a = 0; a < PD; ++a) {
            inv[a] = 0.0;
            for (int b = 0; b < PD; ++b) u[a][b] = 0.0;
        }
        int still = 0;
        for (int it = 0; it < 4096 && still < PD + 2; ++it) {
            for (int d = 0; d < W; ++d) w[d] = entry(2 * PD, d);
            for (int i = PD; i >= 1; --i) {
                l[i - 1] = w[PD - i] * inv[i - 1];
                for (int j = 1; j <= PD; ++j) w[PD - i + j] -= l[i - 1] * u[i - 1][j - 1];
            }
            const double iv = 1.0 / w[PD];
            bool same = fabs(iv - inv[0]) <= ulp * fabs(iv);
            for (int b = 0; b < PD; ++b)
                same = same && fabs(w[PD + 1 + b] - u[0][b]) <= ulp * fabs(w[PD]);
            still = same ? still + 1 : 0;
            for (int a = PD - 1; a > 0; --a) {
                inv[a] = inv[a - 1];
                for (int b = 0; b < PD; ++b) u[a][b] = u[a - 1][b];
            }
            inv[0] = iv;
            for (int b = 0; b < PD; ++b) u[0][b] = w[PD + 1 + b];
        }
        bool ok = still >= PD + 2 && isfinite(inv[0]);
        // multipliers and rows as they will be stored, then the transfers through M rows and J
        for (int a = 0; a < PD; ++a) {
            s_l[a] = (double)(P)l[a];
            s_u[a] = (double)(P)(u[0][a] * inv[0]);
        }
        s_inv = (double)(P)inv[0];
        for (int dir = 0; dir < 2; ++dir) {
            const double* c = dir ? s_u : s_l;
            for (int b = 0; b < PD; ++b) {
                double st[PD];
                for (int a = 0; a < PD; ++a) st[a] = a == b ? 1.0 : 0.0;
                for (int i = 0; i < M; ++i) {
                    double y = 0.0;
                    for (int a = 0; a < PD; ++a) y -= c[a] * st[a];
                    for (int a = PD - 1; a > 0; --a) st[a] = st[a - 1];
                    st[0] = y;
                }
                for (int a = 0; a < PD; ++a) s_T[dir][a][b] = st[a];
            }
            double prod[PD][PD], big = 1.0;
            for (int a = 0; a < PD; ++a)
                for (int b = 0; b < PD; ++b) prod[a][b] = a == b ? 1.0 : 0.0;
            int J = 0;
            while (ok && big > jobs.tol && (J + 1) * M <= kEndRows) {
                double nx[PD][PD];
                big = 0.0;
                for (int a = 0; a < PD; ++a)
                    for (int b = 0; b < PD; ++b) {
                        nx[a][b] = 0.0;
                        for (int q = 0; q < PD; ++q) nx[a][b] += prod[a][q] * s_T[dir][q][b];
                        big = fmax(big, fabs(nx[a][b]));
                    }
                for (int a = 0; a < PD; ++a)
                    for (int b = 0; b < PD; ++b) prod[a][b] = nx[a][b];
                ++J;
            }
            ok = ok && big <= jobs.tol;
            s_Ju = J > s_Ju ? J : s_Ju;
        }
        s_uni = ok ? 1 : 0;
    }
    __syncthreads();
    const bool uni = s_uni != 0;
    if (uni) {
        // The ends: the system B has constant factors, E = A - B is nonzero in the first and last 2p x 2p
        // blocks.  Rows 0 .. n1-1 and n - n2 .. of the line are kept (all of a short line, where both ends see
        // each other); s_W[c]: column of B^{-1} at unknown c (c < 2p: the first ones, then the last ones).
        const bool all = N <= EW;
        const int len = all ? N : EW;  // rows of s_W: 0 .. len-1, for the last ones N - len .. N-1
        if (tid < 2 * D) {
            const bool bot = tid >= D;
            double* w = s_W[tid];
            const int at = bot ? len - 2 * D + tid : tid;
            for (int i = 0; i < len; ++i) {
                double y = i == at ? 1.0 : 0.0;
                for (int a = 0; a < PD; ++a)
                    if (i - 1 - a >= 0) y -= s_l[a] * w[i - 1 - a];
                w[i] = y;
            }
            for (int i = len - 1; i >= 0; --i) {
                double z = w[i] * s_inv;
                for (int a = 0; a < PD; ++a)
                    if (i + 1 + a < len) z -= s_u[a] * w[i + 1 + a];
                w[i] = z;
            }
        }
        __syncthreads();
        if (tid == 0) {
            // g = H z: H = (I + E W)^{-1} E over the end unknowns (first 2p, last 2p)
            double E[2 * D][2 * D];
            for (int a = 0; a < 2 * D; ++a)
                for (int b = 0; b < 2 * D; ++b) {
                    E[a][b] = 0.0;
                    if ((a < D) != (b < D)) continue;
                    const int i = a < D ? a : N - 2 * D + a, j = b < D ? b : N - 2 * D + b;
                    const int d = j - i + PD;
                    if (d < 0 || d >= W) continue;
                    double lu = 0.0;  // (L U)_ij
                    for (int m = (i > j ? i : j) - PD; m <= (i < j ? i : j); ++m) {
                        if (m < 0) continue;
                        const double lm = i == m ? 1.0 : s_l[i - m - 1];
                        const double um = (j == m ? 1.0 : s_u[j - m - 1]) / s_inv;
                        lu += lm * um;
                    }
                    E[a][b] = entry(i, d) - lu;
                }
            auto Wat = [&](int a, int c) {  // row of end unknown a, column of end unknown c
                const bool ba = a >= D, bc = c >= D;
                if (!all && ba != bc) return 0.0;
                return s_W[c][ba ? len - 2 * D + a : a];
            };
            const int n = 2 * D;
            for (int a = 0; a < n; ++a)
                for (int b = 0; b < n; ++b) {
                    double v = a == b ? 1.0 : 0.0;
                    for (int q = 0; q < n; ++q) v += E[a][q] * Wat(q, b);
                    s_H[a][b] = v;
                    s_H[a][n + b] = E[a][b];
                }
            bool ok = true;
            for (int col = 0; col < n; ++col) {
                int pv = col;
                for (int r = col + 1; r < n; ++r)
                    if (fabs(s_H[r][col]) > fabs(s_H[pv][col])) pv = r;
                ok = ok && fabs(s_H[pv][col]) > 1e-300;
                for (int c = 0; c < 2 * n; ++c) {
                    const double t = s_H[col][c];
                    s_H[col][c] = s_H[pv][c];
                    s_H[pv][c] = t;
                }
                const double iv = 1.0 / s_H[col][col];
                for (int c = 0; c < 2 * n; ++c) s_H[col][c] *= iv;
                for (int r = 0; r < n; ++r) {
                    if (r == col) continue;
                    const double f = s_H[r][col];
                    for (int c = 0; c < 2 * n; ++c) s_H[r][c] -= f * s_H[col][c];
                }
            }
            if (!ok) s_uni = 0;
        }
        __syncthreads();
        const int J = s_Ju, kB = C - J - 1 > 0 ? C - J - 1 : 0, n = 2 * D;
        for (int i = tid; i < (J < C ? J : C) * M; i += blockDim.x)
            for (int c = 0; c < NV; ++c) {
                double v = 0.0;
                if (c < D && i < N)
                    for (int a = 0; a < n; ++a)
                        if (a < D || all) v += s_W[a][i] * s_H[a][n + c];
                VT[(size_t)i * NV + c] = (P)v;
            }
        for (int i = tid; i < (C - kB) * M; i += blockDim.x) {
            const int row = kB * M + i, o = row - (N - len);
            for (int c = 0; c < NV; ++c) {
                double v = 0.0;
                if (c < D && row < N && o >= 0)
                    for (int a = 0; a < n; ++a)
                        if (a >= D || all) v += s_W[a][o] * s_H[a][n + D + c];
                VB[(size_t)i * NV + c] = (P)v;
            }
        }
        if (tid < 4) {
            gl[tid] = tid < PD ? (P)s_l[tid < PD ? tid : 0] : P(0);
            gu[tid] = tid == 0 ? (P)s_inv : (tid <= PD ? (P)s_u[tid - 1 < PD ? tid - 1 : 0] : P(0));
        }
        for (int i = tid; i < 2 * S; i += blockDim.x)
            gT[(i / S) * tab_round(S) + i % S] = (P)s_T[i / S][(i % S) / PD][i % PD];
    }
    __syncthreads();
    // J: the smallest count of transfers whose product is below tol, for every chunk and direction (as
    // many as there are chunks on that side where none is)
    for (int q = tid; q < 2 * C; q += blockDim.x) {
        const int k = q >> 1, step = (q & 1) ? 1 : -1;
        const P* T = (q & 1) ? Pb : Pf;
        double prod[PD][PD];
        for (int a = 0; a < PD; ++a)
            for (int b = 0; b < PD; ++b) prod[a][b] = a == b ? 1.0 : 0.0;
        int J = 0;
        for (int i = k + step; i >= 0 && i < C; i += step) {
            // the state of chunk i counts as long as the transfers between it and chunk k do
            double big = 0.0;
            for (int a = 0; a < PD; ++a)
                for (int b = 0; b < PD; ++b) big = fmax(big, fabs(prod[a][b]));
            if (J > 0 && big <= jobs.tol) break;
            ++J;
            double nx[PD][PD];
            for (int a = 0; a < PD; ++a)
                for (int b = 0; b < PD; ++b) {
                    nx[a][b] = 0.0;
                    for (int c = 0; c < PD; ++c) nx[a][b] += prod[a][c] * (double)T[(size_t)i * S + c * PD + b];
                }
            for (int a = 0; a < PD; ++a)
                for (int b = 0; b < PD; ++b) prod[a][b] = nx[a][b];
        }
        atomicMax(&s_J, J);
    }
    __syncthreads();
    if (tid == 0) {
        hdr[0] = s_uni;
        hdr[1] = s_Ju;
        hdr[2] = s_J;
        hdr[3] = s_bad;
    }
}

template <typename P>
__global__ void k_factor_points(const double* __restrict__ coef, int rank, int n, int p, const double* __restrict__ B,
                                P* out) {
    const int q = p + 1, N = n + p;
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rank * n * q) return;
    const int r = idx / (n * q), eq = idx % (n * q), e = eq / q;
    double v = 0.0;
    for (int l = 0; l <= p; ++l) v += B[(size_t)eq * (p + 1) + l] * coef[(size_t)r * N + e + l];
    out[idx] = (P)v;
}

template <typename P, typename H>
__global__ void k_convert_in(const H* __restrict__ src, P* dst, int Nx, int Ny, int pitch) {
    size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)Ny * pitch) return;
    const int j = (int)(idx / pitch), i = (int)(idx % pitch);
    dst[idx] = (i < Nx) ? (P)src[(size_t)j * Nx + i] : (P)0;
}

// every slot of a batch at once: blockIdx.z = slot, host arrays [S][Ny][Nx], slot fields sbytes apart
template <typename P, typename H>
__global__ void k_convert_in_batch(const H* __restrict__ src, P* dst0, long long sbytes, int Nx, int Ny, int pitch) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)Ny * pitch) return;
    const int z = blockIdx.z;
    P* dst = reinterpret_cast<P*>(reinterpret_cast<char*>(dst0) + (long long)z * sbytes);
    const int j = (int)(idx / pitch), i = (int)(idx % pitch);
    dst[idx] = (i < Nx) ? (P)src[(size_t)z * Nx * Ny + (size_t)j * Nx + i] : (P)0;
}

template <typename P, typename H>
__global__ void k_convert_out_batch(const P* src0, H* dst, long long sbytes, int Nx, int Ny, int pitch) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)Ny * Nx) return;
    const int z = blockIdx.z;
    const P* src = reinterpret_cast<const P*>(reinterpret_cast<const char*>(src0) + (long long)z * sbytes);
    const int j = (int)(idx / Nx), i = (int)(idx % Nx);
    dst[(size_t)z * Nx * Ny + idx] = (H)src[(size_t)j * pitch + i];
}

template <typename P, typename H>
__global__ void k_convert_out(const P* __restrict__ src, H* dst, int Nx, int Ny, int pitch) {
    size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)Ny * Nx) return;
    const int j = (int)(idx / Nx), i = (int)(idx % Nx);
    dst[idx] = (H)src[(size_t)j * pitch + i];
}

// Guard flags of S scenarios (each in its own block, sbytes apart) gathered into out[S],
// and cleared when clear != 0.
__global__ void k_gather_status(int* status0, long long sbytes, int S, int* out, int clear) {
    const int z = blockIdx.x * blockDim.x + threadIdx.x;
    if (z >= S) return;
    int* st = reinterpret_cast<int*>(reinterpret_cast<char*>(status0) + (long long)z * sbytes);
    out[z] = st[0];
    if (clear) st[0] = 0;
}

// Per-slot step budgets (end of a step): an active slot with a positive budget spends one step of
// it; at zero the slot is skipped until its budget is set again; a negative budget is unlimited.
__global__ void k_step_budget(const int* active, int* budget, int S) {
    const int z = blockIdx.x * blockDim.x + threadIdx.x;
    if (z >= S || !active[z]) return;
    const int b = budget[z];
    if (b > 0) budget[z] = b - 1;
}

template <typename P>
__global__ void k_fill(P* dst, size_t n, P v) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = v;
}

inline unsigned blocks(size_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t launch_gauss(double* xi, double* w, int q, cudaStream_t s) {
    k_gauss<<<1, 32, 0, s>>>(xi, w, q);
    return cudaGetLastError();
}

cudaError_t launch_basis(const double* xi, int q, int n, int p, double L, double* B, double* D, cudaStream_t s) {
    k_basis<<<blocks((size_t)n * q, 128), 128, 0, s>>>(xi, q, n, p, L, B, D);
    return cudaGetLastError();
}

cudaError_t launch_assemble(const double* B, const double* D, const double* w, int q, int n, int p, double h,
                            double* Mb, double* Kb, double* Gb, cudaStream_t s) {
    const size_t cnt = (size_t)(n + p) * (2 * p + 1);
    k_assemble<<<blocks(cnt, 128), 128, 0, s>>>(B, D, w, q, n, p, h, Mb, Kb, Gb);
    return cudaGetLastError();
}

cudaError_t launch_line_tables(int prec, int p, const TabJobs& jobs, cudaStream_t s) {
    const dim3 grid(jobs.n, jobs.slots);
    const bool f32 = prec == 0;
    switch (p) {
        case 1: f32 ? k_line_tables<float, 1><<<grid, 128, 0, s>>>(jobs) : k_line_tables<double, 1><<<grid, 128, 0, s>>>(jobs); break;
        case 2: f32 ? k_line_tables<float, 2><<<grid, 128, 0, s>>>(jobs) : k_line_tables<double, 2><<<grid, 128, 0, s>>>(jobs); break;
        case 3: f32 ? k_line_tables<float, 3><<<grid, 128, 0, s>>>(jobs) : k_line_tables<double, 3><<<grid, 128, 0, s>>>(jobs); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_factor_points(int prec, const double* coef, int rank, int n, int p, const double* B, void* out,
                                 cudaStream_t s) {
    const size_t cnt = (size_t)rank * n * (p + 1);
    if (cnt == 0) return cudaSuccess;
    if (prec == 0)
        k_factor_points<float><<<blocks(cnt, 128), 128, 0, s>>>(coef, rank, n, p, B, (float*)out);
    else
        k_factor_points<double><<<blocks(cnt, 128), 128, 0, s>>>(coef, rank, n, p, B, (double*)out);
    return cudaGetLastError();
}

cudaError_t launch_convert_in(int prec, const void* src, int host32, void* dst, int Nx, int Ny, int pitch,
                              cudaStream_t s) {
    const size_t cnt = (size_t)Ny * pitch;
    if (prec == 0) {
        if (host32) k_convert_in<float, float><<<blocks(cnt, 256), 256, 0, s>>>((const float*)src, (float*)dst, Nx, Ny, pitch);
        else k_convert_in<float, double><<<blocks(cnt, 256), 256, 0, s>>>((const double*)src, (float*)dst, Nx, Ny, pitch);
    } else {
        if (host32) k_convert_in<double, float><<<blocks(cnt, 256), 256, 0, s>>>((const float*)src, (double*)dst, Nx, Ny, pitch);
        else k_convert_in<double, double><<<blocks(cnt, 256), 256, 0, s>>>((const double*)src, (double*)dst, Nx, Ny, pitch);
    }
    return cudaGetLastError();
}

cudaError_t launch_convert_batch(int dir_in, int prec, const void* host_stage, int host32, void* field0,
                                 long long sbytes, int S, int Nx, int Ny, int pitch, cudaStream_t s) {
    const size_t cnt = dir_in ? (size_t)Ny * pitch : (size_t)Ny * Nx;
    dim3 g(blocks(cnt, 256), 1, S);
#define WF_CB(P, H)                                                                                        \
    if (dir_in)                                                                                            \
        k_convert_in_batch<P, H><<<g, 256, 0, s>>>((const H*)host_stage, (P*)field0, sbytes, Nx, Ny, pitch); \
    else                                                                                                   \
        k_convert_out_batch<P, H><<<g, 256, 0, s>>>((const P*)field0, (H*)host_stage, sbytes, Nx, Ny, pitch)
    if (prec == 0) {
        if (host32) { WF_CB(float, float); } else { WF_CB(float, double); }
    } else {
        if (host32) { WF_CB(double, float); } else { WF_CB(double, double); }
    }
#undef WF_CB
    return cudaGetLastError();
}

cudaError_t launch_convert_out(int prec, const void* src, void* dst, int host32, int Nx, int Ny, int pitch,
                               cudaStream_t s) {
    const size_t cnt = (size_t)Ny * Nx;
    if (prec == 0) {
        if (host32) k_convert_out<float, float><<<blocks(cnt, 256), 256, 0, s>>>((const float*)src, (float*)dst, Nx, Ny, pitch);
        else k_convert_out<float, double><<<blocks(cnt, 256), 256, 0, s>>>((const float*)src, (double*)dst, Nx, Ny, pitch);
    } else {
        if (host32) k_convert_out<double, float><<<blocks(cnt, 256), 256, 0, s>>>((const double*)src, (float*)dst, Nx, Ny, pitch);
        else k_convert_out<double, double><<<blocks(cnt, 256), 256, 0, s>>>((const double*)src, (double*)dst, Nx, Ny, pitch);
    }
    return cudaGetLastError();
}

cudaError_t launch_gather_status(int* status0, long long sbytes, int S, int* out, int clear, cudaStream_t s) {
    k_gather_status<<<blocks(S, 128), 128, 0, s>>>(status0, sbytes, S, out, clear);
    return cudaGetLastError();
}

cudaError_t launch_step_budget(const int* active, int* budget, int S, cudaStream_t s) {
    k_step_budget<<<blocks(S, 128), 128, 0, s>>>(active, budget, S);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_fill(int prec, void* dst, size_t n, double v, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (prec == 0)
        k_fill<float><<<blocks(n, 256), 256, 0, s>>>((float*)dst, n, (float)v);
    else
        k_fill<double><<<blocks(n, 256), 256, 0, s>>>((double*)dst, n, v);
    return cudaGetLastError();
}

}  // namespace wf
