// Internal declarations shared by the CUDA translation units of libwf.
//
// Data layout on the device (all fields of one handle):
//   - coefficient fields T, phi, Phi, R: [Ny][pitch] in the handle's
//     precision P (float or double), pitch = Nx rounded up to 32 elements
//     so every row starts on a 128-byte boundary;
//   - 1-D Gauss tables per direction: B[e][a][l] = B_{e+l}(x_{e,a}) and the
//     derivative D[e][a][l], e < n, a < q = p+1, l <= p;
//   - 1-D banded matrices: band[r][d] = A[r][r+d-p], d in [0, 2p], zero
//     outside the matrix;
//   - LU factors of a 1-D operator (see the factor tables below).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <mutex>
#include <type_traits>

namespace wf {

constexpr int kMaxP = 3;
constexpr int kMaxRank = 4;

// Scenario batching.  Every per-scenario pointer handed to a kernel addresses scenario 0;
// scenario z's copy lies z * sbytes bytes further (each scenario owns one block of device
// memory with the same internal layout).  Launches cover all S scenarios with grid.z = S;
// a scenario whose active flag is 0, or whose step budget is spent (0), is skipped.
// Slots of one launch (its grid.z); every per-slot pointer of the launch refers to the launch's
// first slot, the next ones follow sbytes apart (a launch over a group of slots gets pointers to
// the group's first slot).
struct Batch {
    int S;
    long long sbytes;
    const int* active;  // [S] or nullptr (all active)
    const int* budget;  // [S] step budgets (negative: unlimited) or nullptr (none)
};
#ifdef __CUDACC__
__device__ __forceinline__ bool scene_active(const Batch& b) {
    return (!b.active || b.active[blockIdx.z] != 0) && (!b.budget || b.budget[blockIdx.z] != 0);
}
#endif

// Normalised model coefficients (equation divided by rho*c_p).
struct Phys {
    double C_d, C_nld, c_rad, c_chi, c_W, K_ign, k_f, T_a, T_amb, T_ig, phi_min;
    int heat_by_fuel;
};

// ---- factor tables of the line solves ------------------------------------------------
// A line of N unknowns is cut into C = ceil(N / M) chunks of M (the last one padded).  The table of one
// operator A = aM M + aK K + aG G (half-bandwidth p), written once per operator in the working precision from
// FP64 LU factors without pivoting (wf_lines.cuh has the method):
//   header (kTabHeader bytes of ints): [0] 1: uniform factors and end corrections, 0: exact factors of every
//     row; [1] J, the chunks whose states a chunk's entering state takes in, with uniform factors, [2] with
//     exact ones; [3] 1 if a pivot was below 1e-300 ||A||
//   l[4], u[4]                uniform rows of F and U
//   Tf[p][p], Tb[p][p]        transfer of a state (the last p values of a forward, the first p of a backward
//                             recursion, nearest first) through a chunk of uniform rows
//   VT[kEndRows + M][V], VB[kEndRows + 2M][V]  (V = 2, 4, 8) end corrections of the first J and last J + 1 chunks
//   F[C*M][p (4 for p = 3)]   multipliers: row r subtracts F[r][i-1] * y[r-i], i = 1..p
//   U[C*M][2 (p = 1) or 4]    1 / u_rr, then u_r,r+j / u_rr, j = 1..p
//   Pf[C][p][p], Pb[C][p][p]  transfers through every chunk
// every part rounded up to a multiple of four elements.
constexpr int kTabHeader = 64;
// FP32 takes uniform factors where an operator has them.  FP64 reads every row's factors: its pipe bounds the
// passes, loads are free beside it, and the end corrections are a tenth to a half more multiply-adds (step, uniform /
// table: 66^2 quadratic 53.6 / 48.6 us, 8 x 259^2 cubic 949 / 932, 1026^2 695 / 688).
template <typename P>
constexpr bool kUniformFactors = sizeof(P) == 4;
constexpr int kEndRows = 128;  // J * M at most for the uniform form
__host__ __device__ constexpr int tab_round(int n) { return (n + 3) & ~3; }
inline int line_chunks(int N, int M) { return (N + M - 1) / M; }
inline size_t line_tab_bytes(size_t es, int p, int N, int M) {
    const int C = line_chunks(N, M), NF = p == 3 ? 4 : p, NU = p == 1 ? 2 : 4, NV = p == 1 ? 2 : (p == 2 ? 4 : 8);
    return kTabHeader + es * (size_t)(8 + 2 * tab_round(p * p) + (2 * kEndRows + 3 * M) * NV + tab_round(C * M * NF) +
                                      tab_round(C * M * NU) + 2 * tab_round(C * p * p) + 8);
}
// One operator of a direction; band: instead of factors, the rows of an operator without a mass term (the explicit
// operator of the middle y pass) as factors of differences, [N][2p]: its rows sum to zero, so row r applied to T is the
// sum over e of (the row's entries right of column r - p + e) * (T[r-p+e+1] - T[r-p+e]).  Rounding then scales
// with the differences: with the entries times T, FP32 steps of a large diffusivity lost the ambient temperature's last
// digits (kappa = 3e6, 300 x 200 linear, one step against FP64: 4.6e-5 relative, with this 5.8e-8).
struct TabJob {
    const double *M, *K, *G;
    double aM, aK, aG;
    int N, chunk;
    void* out;
    int band;
};
struct TabJobs {
    TabJob job[5];
    int n;
    void* mw;  // the slot's mean wind in the working precision (2 values)
    double wind_x, wind_y;
    double tol;  // products of transfers below it are dropped
    int slots;   // slots written, sbytes apart (the same operators in each)
    long long sbytes;
};

// ---- tables and factorisation (FP64, wf_tables.cu) ---------------------------------
cudaError_t launch_gauss(double* xi, double* w, int q, cudaStream_t s);
cudaError_t launch_basis(const double* xi, int q, int n, int p, double L, double* B, double* D, cudaStream_t s);
cudaError_t launch_assemble(const double* B, const double* D, const double* w, int q, int n, int p, double h,
                            double* Mb, double* Kb, double* Gb, cudaStream_t s);
// every table of jobs.job[0 .. n-1], for jobs.slots slots
cudaError_t launch_line_tables(int prec, int p, const TabJobs& jobs, cudaStream_t s);
// out[r][e*q+a] = sum_l B[e][a][l] coef[r][e+l]  (1-D spline factor at Gauss points)
cudaError_t launch_factor_points(int prec, const double* coef, int rank, int n, int p, const double* B,
                                 void* out, cudaStream_t s);
// host layout [Ny][Nx] in FP64 (host32 = 0) or FP32 (host32 = 1) <-> device [Ny][pitch] in the
// handle's precision (padding columns written as zeros)
cudaError_t launch_convert_in(int prec, const void* src, int host32, void* dst, int Nx, int Ny, int pitch,
                              cudaStream_t s);
cudaError_t launch_convert_out(int prec, const void* src, void* dst, int host32, int Nx, int Ny, int pitch,
                               cudaStream_t s);
// every slot at once (dir_in 1: staged host arrays [S][Ny][Nx] -> slot fields field0 + z * sbytes;
// 0: the reverse)
cudaError_t launch_convert_batch(int dir_in, int prec, const void* host_stage, int host32, void* field0,
                                 long long sbytes, int S, int Nx, int Ny, int pitch, cudaStream_t s);
cudaError_t launch_fill(int prec, void* dst, size_t n, double v, cudaStream_t s);
cudaError_t launch_gather_status(int* status0, long long sbytes, int S, int* out, int clear, cudaStream_t s);
// end of a step: every active slot with a positive budget spends one step (at zero the slot is
// skipped by every kernel until its budget is set again)
cudaError_t launch_step_budget(const int* active, int* budget, int S, cudaStream_t s);

// ---- quadrature (wf_quad.cuh) -------------------------------------------------------
struct RhsArgs {
    int nx, ny, Nx, Ny, pitch;
    double hx, hy;  // element sizes
    const void* T;
    const void* phi;
    void* Phi;  // fuel increment load vector -tau k_f int(E phi B_i B_j) (optional)
    void* R;    // Rscale (F - A_x (x) M^y T - M^x (x) A_y T), or with xonly Rscale (F - A_x (x) M^y T)
    int xonly;
    double Rscale;
    double tau;  // full time step (fuel update)
    int wind_rank;
    const void *fxq, *gxq, *fyq, *gyq;  // [rank][n*q] factor values at Gauss points
    const void* mw;                     // mean wind (b_x, b_y)
    int seg;    // rows per segment (0: the launcher's rule)
    int parts;  // FP32: the strips at either x boundary in launches of their own
    Phys phys;
    Batch b;  // per scenario: T, phi, Phi, R, mw, fxq, gxq, fyq, gyq
};
cudaError_t launch_rhs(int prec, int p, const RhsArgs& a, cudaStream_t s);
cudaError_t launch_quad_p1_f32(const RhsArgs& a, cudaStream_t s);
cudaError_t launch_quad_p2_f32(const RhsArgs& a, cudaStream_t s);
cudaError_t launch_quad_p3_f32(const RhsArgs& a, cudaStream_t s);
cudaError_t launch_quad_p1_f64(const RhsArgs& a, cudaStream_t s);
cudaError_t launch_quad_p2_f64(const RhsArgs& a, cudaStream_t s);
cudaError_t launch_quad_p3_f64(const RhsArgs& a, cudaStream_t s);
// process-wide count of the time-step kernels launched (wf_launch_count)
void count_launches(int n);

// ---- manufactured-solution forcing (wf_mms.cu) --------------------------------------
struct MmsArgs {
    int nmodes;
    double amp[4], kx[4], ky[4], lambda[4], base;  // u* = base + sum amp (1-cos)(1-cos) exp(-lambda t)
    double Lx, Ly, hx, hy;
    int nx, ny, Nx, Ny, pitch, p, q;
    const double *Bx, *By;  // FP64 basis tables [n][q][p+1]
    double xi[8], w[8];     // Gauss nodes and weights on [0, 1]
    double C_d, c_W, c_chi, T_amb, T_amb4, c_rad, C_nld, wind_x, wind_y;
    const double* t;        // device: start time of the step being enqueued
};
// out += s1 * int f B_i B_j
cudaError_t launch_forcing(int prec, const MmsArgs& a, void* out, double s1, cudaStream_t s);
cudaError_t launch_advance_time(double* t, double dt, cudaStream_t s);

// ---- line passes (wf_lines.cuh) -------------------------------------------------------
struct LineArgs {
    int N, M, C, J;  // line length, chunk length and count; J: see the factor tables (largest of the slots)
    int uni;     // every operator of the handle has uniform factors
    int G;       // x pass: rows per CTA at most (0: the launcher's rule)
    int nlines;  // number of independent lines
    int pitch;   // row pitch of the fields (elements)
    int narr;    // 1 or 2 arrays (blockIdx.y)
    const void* in[2];
    void* out[2];
    const void* tab[2];     // factor tables
    const void* base[2];    // y pass: out = base + solution (or NULL: out = solution)
    const void* band;       // middle y pass: rows of the explicit operator
    int* status;            // y pass: guard flag for out[0] (or NULL)
    int* tstatus;           // x pass: flag word whose bit 4 records a bounded wait that gave up
    long long wait_ns;      // limit of a bounded device wait (ns of %globaltimer; 0: give up at once)
    double tmax;
    Batch b;  // per scenario: in, out, tab, base, band, status, tstatus
};
// kind 0: x pass; 1: y pass; 2: middle y pass of a Strang step (in: the x-solved right-hand side, base: T,
// tab: M^y and Y_+, out: T**, a field of its own)
cudaError_t launch_lines_p1_f32(int kind, const LineArgs& l, cudaStream_t s);
cudaError_t launch_lines_p2_f32(int kind, const LineArgs& l, cudaStream_t s);
cudaError_t launch_lines_p3_f32(int kind, const LineArgs& l, cudaStream_t s);
cudaError_t launch_lines_p1_f64(int kind, const LineArgs& l, cudaStream_t s);
cudaError_t launch_lines_p2_f64(int kind, const LineArgs& l, cudaStream_t s);
cudaError_t launch_lines_p3_f64(int kind, const LineArgs& l, cudaStream_t s);
// Raise (never lower) the dynamic shared memory a kernel may be launched with.  The limit is a
// property of the kernel, read when a launch is made; the launches captured in a graph keep the
// size each needed, so a later, smaller request for the same kernel (another pass, other launch
// shapes) must not take the limit below them, nor may one of another thread (another handle) that read the limit
// before this one raised it.
template <typename K>
inline cudaError_t allow_dynamic_smem(K kern, size_t bytes) {
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, reinterpret_cast<const void*>(kern));
    if (e != cudaSuccess) return e;
    if ((size_t)fa.maxDynamicSharedSizeBytes >= bytes) return cudaSuccess;
    return cudaFuncSetAttribute(reinterpret_cast<const void*>(kern), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)bytes);
}

// A launch that may begin while the last CTAs of the kernel before it in the stream drain (programmatic dependent
// launch; the kernel begins with grid_wait): the launch latency and the start of the CTAs overlap that tail.
template <typename... KA, typename... A>
inline cudaError_t launch_overlapped(void (*kern)(KA...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                                     A... args) {
    cudaLaunchConfig_t c = {};
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kern, KA(args)...);
}
#ifdef __CUDACC__
// First statement of such a kernel: waits until the kernel before it is complete and its writes are visible.
// `off` is added to every address the kernel reads, and passes through the wait, so that no load (a read-only one
// neither) can be moved above it.  EARLY: a grid of at most kEarlyCtas CTAs then lets the next kernel's CTAs start
// beside it; larger ones leave that to their end, where the next kernel's CTAs no longer take room from theirs.  us per
// step, no overlap / at the end / always early: 130^2 13.9 / 13.0 / 12.9, 100 x 64 cubic Strang 37.7 / 36.7 /
// 35.2, 1026^2 34.8 / 33.9 / 35.6, 8 x 515^2 cubic 105.3 / 104.3 / 107.5.
constexpr unsigned kEarlyCtas = 2 * 152;
template <bool EARLY = true>
__device__ __forceinline__ void grid_wait(long long& off) {
    asm volatile("griddepcontrol.wait;" : "+l"(off)::"memory");
    if (EARLY && gridDim.x * gridDim.y * gridDim.z <= kEarlyCtas)
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// A value of a field.  The kernels of a step live while the one before them still writes fields, and the read-only
// path (__ldg) is for data that nothing writes while a kernel lives: tables and factors.  Steps take as long with
// either kind of load (88 grids of both precisions: 0.05 % apart in the mean).
template <typename T>
__device__ __forceinline__ T field_load(const T* p) {
    return __ldca(p);
}
#endif

// ---- persistent line passes (wf_persist.cu) -----------------------------------------
// After the quadrature launch of a Peaceman-Rachford step (one F per step), one launch runs the
// step's x and y passes for every active slot, over the (pass, slot, tile) items listed
// by persist_items; the arguments are those of the per-pass launches of the same step.
struct PersistHost {
    int prec, p;
    LineArgs x, y;            // two arrays each (R, Phi)
    int nslots_cap;           // slot capacity of the handle (counter blocks)
    long long wait_ns;
    int* status;              // slot-0 flag word
    const int4* items;        // device: work items in their order
    int* ctl;                 // device: [0] ticket, [1] abort flag, [2] items, [3] items per slot
    int* cnt;                 // device: nslots_cap x cstride arrival counters
    size_t cnt_cap;           // ints allocated at cnt (the launch refuses a larger plan)
    const int* active;        // device: per-slot activity flags (an inactive slot's items are skipped)
    int* budget;              // device: per-slot step budgets, or NULL (a spent budget, 0, skips too)
};
struct PersistPlan {
    int nxg, nyg, narr, cstride, ctas;
};
cudaError_t persist_p1(const PersistHost& h, PersistPlan* plan, bool launch, cudaStream_t s);
cudaError_t persist_p2(const PersistHost& h, PersistPlan* plan, bool launch, cudaStream_t s);
cudaError_t persist_p3(const PersistHost& h, PersistPlan* plan, bool launch, cudaStream_t s);
// plan (and, with launch, enqueue: counter reset + one kernel) of one step; cudaErrorNotSupported
// when the persistent form cannot take these arguments
cudaError_t persist_step(const PersistHost& h, PersistPlan* plan, bool launch, cudaStream_t s);
// work items of one step for the given active slots, groups of gs slots in wavefront order;
// returns the count (entries past cap are not written) and the items of one slot
int persist_items(const PersistPlan& plan, const int* slots, int nslots, int gs, int4* out, int cap,
                  int* items_per_slot);

}  // namespace wf
