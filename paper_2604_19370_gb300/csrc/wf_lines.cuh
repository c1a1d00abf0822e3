// Line solves of the directional operators (Sec. 4, "Cost of directional implicit solves": independent
// banded 1-D systems along x or y), device code shared by the per-pass kernels (wf_lines_body.cuh) and the
// persistent one (wf_persist.cuh).
//
// A line of N values is cut into C chunks of M; one thread owns one chunk of one line and keeps its M values in
// registers from load to store.  The operator's LU factors are those of the whole line (wf_tables.cu).
// Forward elimination y_i = x_i - sum_j l_ij y_{i-j} is a recursion whose state are the last p values:
//   1. run it over the chunk from a zero state: the state f_k it ends with;
//   2. the state entering chunk k is f_{k-1} + P_{k-1} (f_{k-2} + P_{k-2} (f_{k-3} + ...)), P_k the (p x p)
//      transfer of a state through chunk k, from the neighbours' f in shared memory;
//   3. run it again from that state.
// Backward substitution does the same from the other end.  The inverse of these operators decays by a
// factor of 0.2 to 0.6 a row, so products of J transfers below the truncation tolerance (1e-8 FP32,
// 1e-15 FP64) are dropped; J is found when the operator is factored (2 chunks of 17 rows in FP32,
// p = 2) and may be as large as C - 1, where nothing is dropped.
//
// Uniform factors and end corrections.  Away from the ends of the line the rows of an operator A are the
// same (uniform knots), and its LU factors converge to constant ones l, u within a few dozen rows.  With B
// the product of constant bidiagonal-like factors, A - B is nonzero only in the first and last 2p x 2p
// blocks, so A^{-1} r = z - VT z_top - VB z_bottom with z = B^{-1} r and z_top, z_bottom its first and last
// 2p values (Woodbury's identity, tables in wf_tables.cu); the rows of VT and VB decay like the states and
// are kept for J chunks from either end.  Every chunk then runs its recursions with factors in registers;
// reading each row's factors from a table in the chunks near the ends made those the slowest of their CTA
// (256 scenarios of 258^2, FP32: x pass 66, y pass 93 us).  Operators whose factors do not converge, whose
// states reach further than kEndRows rows, lines of less than 4p + 1 values, and FP64 (kUniformFactors) take the table
// of exact factors.
//
// Against a chunk-local LU with spike corrections (three sweeps over shared memory, about 50 warp
// instructions a value) this is about 9 multiply-adds a value from registers, and the chunk's loads are all
// in flight at once.
#pragma once
#include "wf_internal.h"

namespace wf {

namespace {

// Row widths of the factor tables, padded for vector loads: the p multipliers; 1/u_rr and u_r,r+j / u_rr.
template <int PD>
struct TabW {
    static constexpr int F = PD == 3 ? 4 : PD;
    static constexpr int U = PD == 1 ? 2 : 4;
    static constexpr int V = PD == 1 ? 2 : (PD == 2 ? 4 : 8);  // 2p end values
};

// Parts of an operator's table (layout: wf_internal.h), in elements from the end of the header.
template <int PD, int M>
struct TabAt {
    static constexpr int l = 0, u = 4, Tf = 8, Tb = Tf + tab_round(PD * PD), VT = Tb + tab_round(PD * PD),
                         VB = VT + (kEndRows + M) * TabW<PD>::V, F = VB + (kEndRows + 2 * M) * TabW<PD>::V;
    static __device__ __forceinline__ int U(int C) { return F + tab_round(C * M * TabW<PD>::F); }
    static __device__ __forceinline__ int Pf(int C) { return U(C) + tab_round(C * M * TabW<PD>::U); }
    static __device__ __forceinline__ int Pb(int C) { return Pf(C) + tab_round(C * PD * PD); }
};

// W consecutive table values (aligned to W values, at most 16 bytes a load)
template <int W>
__device__ __forceinline__ void tab_load(const float* p, float (&o)[W]) {
    if constexpr (W % 4 == 0) {
#pragma unroll
        for (int i = 0; i < W; i += 4) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(p + i));
            o[i] = v.x, o[i + 1] = v.y, o[i + 2] = v.z, o[i + 3] = v.w;
        }
    } else if constexpr (W == 2) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(p));
        o[0] = v.x, o[1] = v.y;
    } else {
        o[0] = __ldg(p);
    }
}
template <int W>
__device__ __forceinline__ void tab_load(const double* p, double (&o)[W]) {
    if constexpr (W == 1) {
        o[0] = __ldg(p);
    } else {
#pragma unroll
        for (int i = 0; i < W; i += 2) {
            const double2 v = __ldg(reinterpret_cast<const double2*>(p + i));
            o[i] = v.x, o[i + 1] = v.y;
        }
    }
}

// Factors of the rows of a chunk: the same in every row, or read from the table.
template <typename P, int PD>
struct RowsUniform {
    P l[TabW<PD>::F], u[TabW<PD>::U];
    __device__ __forceinline__ RowsUniform(const P* l_, const P* u_) {
        tab_load(l_, l);
        tab_load(u_, u);
    }
    __device__ __forceinline__ P pivot(int) const { return u[0]; }
    __device__ __forceinline__ void low(int, P (&o)[TabW<PD>::F]) const {
#pragma unroll
        for (int j = 0; j < TabW<PD>::F; ++j) o[j] = l[j];
    }
    __device__ __forceinline__ void up(int, P (&o)[TabW<PD>::U]) const {
#pragma unroll
        for (int j = 0; j < TabW<PD>::U; ++j) o[j] = u[j];
    }
};
template <typename P, int PD>
struct RowsTable {
    const P *F, *U;
    __device__ __forceinline__ RowsTable(const P* F_, const P* U_, int row)
        : F(F_ + (size_t)row * TabW<PD>::F), U(U_ + (size_t)row * TabW<PD>::U) {}
    __device__ __forceinline__ P pivot(int i) const { return __ldg(U + i * TabW<PD>::U); }
    __device__ __forceinline__ void low(int i, P (&o)[TabW<PD>::F]) const { tab_load(F + i * TabW<PD>::F, o); }
    __device__ __forceinline__ void up(int i, P (&o)[TabW<PD>::U]) const { tab_load(U + i * TabW<PD>::U, o); }
};

// s[j]: the value j+1 rows back (forward) or ahead (backward)
template <bool KEEP, typename P, int PD, int M, typename R>
__device__ __forceinline__ void forward(P (&x)[M], const R& rows, P (&s)[PD]) {
#pragma unroll
    for (int i = 0; i < M; ++i) {
        P l[TabW<PD>::F];
        rows.low(i, l);
        P y = x[i];
#pragma unroll
        for (int j = PD - 1; j >= 0; --j) y -= l[j] * s[j];
#pragma unroll
        for (int j = PD - 1; j > 0; --j) s[j] = s[j - 1];
        s[0] = y;
        if (KEEP) x[i] = y;
    }
}
template <typename P, int PD, int M, typename R>
__device__ __forceinline__ void scale(P (&x)[M], const R& rows) {
#pragma unroll
    for (int i = 0; i < M; ++i) x[i] *= rows.pivot(i);
}
template <bool KEEP, typename P, int PD, int M, typename R>
__device__ __forceinline__ void backward(P (&x)[M], const R& rows, P (&s)[PD]) {
#pragma unroll
    for (int i = M - 1; i >= 0; --i) {
        P u[TabW<PD>::U];
        rows.up(i, u);
        P z = x[i];  // scaled by 1 / u_ii
#pragma unroll
        for (int j = PD - 1; j >= 0; --j) z -= u[1 + j] * s[j];
#pragma unroll
        for (int j = PD - 1; j > 0; --j) s[j] = s[j - 1];
        s[0] = z;
        if (KEEP) x[i] = z;
    }
}

template <typename P, int PD>
__device__ __forceinline__ void clear(P (&s)[PD]) {
#pragma unroll
    for (int j = 0; j < PD; ++j) s[j] = P(0);
}

// s = f + T s
template <bool FIRST, typename P, int PD>
__device__ __forceinline__ void add_state(const P* f, int jstride, const P* T, P (&s)[PD]) {
    P o[PD];
#pragma unroll
    for (int a = 0; a < PD; ++a) {
        o[a] = f[a * jstride];
        if (!FIRST)
#pragma unroll
            for (int b = 0; b < PD; ++b) o[a] += __ldg(T + a * PD + b) * s[b];
    }
#pragma unroll
    for (int j = 0; j < PD; ++j) s[j] = o[j];
}

// The sweeps of chunk k: forward1 leaves the state after the chunk from a zero state in s, forward2 runs from
// the entering state in s; backward1 and backward2 likewise (have: values of the chunk that exist).  enter:
// the state entering the chunk from the chunks before it (step -1) or after it (step +1), of which those
// from kb to ke - 1 have their zero-state results st[(chunk - kb) * stride + j * jstride].
// UNI: constant factors, end corrections.  Otherwise every row's own factors (no end corrections).
template <typename P, int PD, int M, bool UNI>
struct Sweeps;

template <typename P, int PD, int M>
struct Sweeps<P, PD, M, true> {
    using At = TabAt<PD, M>;
    const P* t;
    RowsUniform<P, PD> ru;
    int k, J;
    __device__ __forceinline__ Sweeps(const void* tab, int k_, int)
        : t(reinterpret_cast<const P*>(static_cast<const char*>(tab) + kTabHeader)), ru(t + At::l, t + At::u), k(k_),
          J(__ldg(static_cast<const int*>(tab) + 1)) {}
    __device__ __forceinline__ void forward1(P (&x)[M], P (&s)[PD]) const {
        clear(s);
        forward<false, P, PD, M>(x, ru, s);
    }
    __device__ __forceinline__ void forward2(P (&x)[M], P (&s)[PD]) const { forward<true, P, PD, M>(x, ru, s); }
    __device__ __forceinline__ void backward1(P (&x)[M], P (&s)[PD], int have) const {
        clear(s);
        // nothing follows the last row of the line
        if (have < M)
#pragma unroll
            for (int i = 0; i < M; ++i) x[i] = i < have ? x[i] : P(0);
        scale<P, PD, M>(x, ru);
        backward<false, P, PD, M>(x, ru, s);
    }
    __device__ __forceinline__ void backward2(P (&x)[M], P (&s)[PD]) const { backward<true, P, PD, M>(x, ru, s); }
    __device__ __forceinline__ void enter(const P* st, int stride, int jstride, int kb, int ke, int step,
                                          P (&s)[PD]) const {
        clear(s);
        const P* T = t + (step < 0 ? At::Tf : At::Tb);
        int i = k + step * J;
        if (i >= kb && i < ke) add_state<true, P, PD>(st + (i - kb) * stride, jstride, T, s);
        for (int d = J - 1; d >= 1; --d) {
            i = k + step * d;
            if (i >= kb && i < ke) add_state<false, P, PD>(st + (i - kb) * stride, jstride, T, s);
        }
    }
    // End corrections: the chunks that hold the first and last 2p values put them into e ([2][2p], estride
    // apart); after a barrier the chunks in reach of an end take them off.
    __device__ __forceinline__ void ends_put(const P (&x)[M], P* e, int estride, int N, int have) const {
        if (k == 0 && have > 0)
#pragma unroll
            for (int c = 0; c < 2 * PD; ++c) e[c * estride] = x[c];
        const int b0 = N - 2 * PD - k * M;  // chunk row of the first of the last 2p values
        if (have > 0 && b0 < M)
#pragma unroll
            for (int i = 0; i < M; ++i)
                if (i >= b0 && i < b0 + 2 * PD) e[(2 * PD + i - b0) * estride] = x[i];
    }
    __device__ __forceinline__ void take(P (&x)[M], const P* V, const P* z, int estride) const {
        P zc[2 * PD];
#pragma unroll
        for (int c = 0; c < 2 * PD; ++c) zc[c] = z[c * estride];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            P v[TabW<PD>::V];
            tab_load(V + i * TabW<PD>::V, v);
#pragma unroll
            for (int c = 0; c < 2 * PD; ++c) x[i] -= v[c] * zc[c];
        }
    }
    __device__ __forceinline__ void ends_take(P (&x)[M], const P* e, int estride, int C) const {
        const int kB = max(0, C - J - 1);
        if (k < J) take(x, t + At::VT + k * M * TabW<PD>::V, e, estride);
        if (k >= kB) take(x, t + At::VB + (k - kB) * M * TabW<PD>::V, e + 2 * PD * estride, estride);
    }
};

template <typename P, int PD, int M>
struct Sweeps<P, PD, M, false> {
    using At = TabAt<PD, M>;
    const P* t;
    int k, C, J;
    __device__ __forceinline__ Sweeps(const void* tab, int k_, int C_)
        : t(reinterpret_cast<const P*>(static_cast<const char*>(tab) + kTabHeader)), k(k_), C(C_),
          J(__ldg(static_cast<const int*>(tab) + 2)) {}
    __device__ __forceinline__ RowsTable<P, PD> rt() const { return RowsTable<P, PD>(t + At::F, t + At::U(C), k * M); }
    __device__ __forceinline__ void forward1(P (&x)[M], P (&s)[PD]) const {
        clear(s);
        forward<false, P, PD, M>(x, rt(), s);
    }
    __device__ __forceinline__ void forward2(P (&x)[M], P (&s)[PD]) const { forward<true, P, PD, M>(x, rt(), s); }
    __device__ __forceinline__ void backward1(P (&x)[M], P (&s)[PD], int) const {
        clear(s);
        scale<P, PD, M>(x, rt());
        backward<false, P, PD, M>(x, rt(), s);
    }
    __device__ __forceinline__ void backward2(P (&x)[M], P (&s)[PD]) const { backward<true, P, PD, M>(x, rt(), s); }
    __device__ __forceinline__ void enter(const P* st, int stride, int jstride, int kb, int ke, int step,
                                          P (&s)[PD]) const {
        clear(s);
        const P* T = t + (step < 0 ? At::Pf(C) : At::Pb(C));
        for (int d = J; d >= 1; --d) {
            const int i = k + step * d;
            if (i < kb || i >= ke) continue;
            add_state<false, P, PD>(st + (size_t)(i - kb) * stride, jstride, T + (size_t)i * PD * PD, s);
        }
    }
    __device__ __forceinline__ void ends_put(const P (&)[M], P*, int, int, int) const {}
    __device__ __forceinline__ void ends_take(P (&)[M], const P*, int, int) const {}
};

// The M values of a chunk, `step` elements apart, of which the first n exist (n <= 0: none; the others are zero);
// whole chunks take no per-value check.  Returns false if every bit of every value is zero.
template <bool CG, typename P, int M>
__device__ __forceinline__ bool chunk_load(const P* p, size_t step, int n, P (&x)[M]) {
    auto get = [](const P* q) { return CG ? __ldcg(q) : *q; };
    if (n >= M) {
#pragma unroll
        for (int i = 0; i < M; ++i, p += step) x[i] = get(p);
    } else {
#pragma unroll
        for (int i = 0; i < M; ++i, p += step) x[i] = i < n ? get(p) : P(0);
    }
    if constexpr (sizeof(P) == 4) {
        unsigned bits = 0;
#pragma unroll
        for (int i = 0; i < M; ++i) bits |= __float_as_uint(x[i]);
        return bits != 0;
    } else {
        long long bits = 0;
#pragma unroll
        for (int i = 0; i < M; ++i) bits |= __double_as_longlong(x[i]);
        return bits != 0;
    }
}

// out = base + x (base: NULL or as many values), true if some |value| is above tmax or not a number.  Rows
// are taken in batches whose base values are all in flight at once.
template <typename P, int M>
__device__ __forceinline__ bool chunk_store(P* out, const P* base, size_t step, int n, const P (&x)[M], P tmax) {
    constexpr int B = 12;
    bool bad = false;
#pragma unroll
    for (int i0 = 0; i0 < M; i0 += B) {
        P y[B];
#pragma unroll
        for (int i = i0; i < i0 + B && i < M; ++i) {
            y[i - i0] = x[i];
            if (base) y[i - i0] += (i < n) ? base[i * step] : P(0);
        }
#pragma unroll
        for (int i = i0; i < i0 + B && i < M; ++i)
            if (i < n) {
                out[i * step] = y[i - i0];
                bad |= !(fabs(y[i - i0]) <= tmax);
            }
    }
    return bad;
}

// ---- TMA bulk copies and mbarrier (PTX) ------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// global -> shared, completion signalled on the mbarrier (16-byte aligned, size multiple of 16)
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// shared -> global, tracked by the bulk async-group of the issuing thread
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit_and_wait_read() {
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Bounded mbarrier wait: gives up after the handle's wait limit (ns of the SM's global timer); the kernel then
// sets bit 4 of the slot's flag word and drains the copies still in flight with kDrainPolls polls (each
// try_wait may suspend the thread for a while), so that no copy lands in shared memory after the CTA exits.
constexpr uint32_t kDrainPolls = 1u << 20;
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// true once the barrier's phase `parity` completed; false if limit_ns passed first (limit 0: no poll)
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, long long limit_ns) {
    if (limit_ns <= 0) return false;
    const unsigned long long t0 = global_ns();
    for (uint32_t it = 0;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 15u) == 15u && (long long)(global_ns() - t0) > limit_ns) return false;
    }
}
__device__ __forceinline__ void mbar_drain(uint64_t* bar, uint32_t parity) {
    for (uint32_t it = 0; it < kDrainPolls; ++it)
        if (mbar_try_wait(bar, parity)) return;
}

// ---- arguments -------------------------------------------------------------------------
template <typename P>
struct PassArgs {
    int N, C, nlines, pitch;
    // x: G rows per CTA (a power of two up to 8), lanes of a warp = G rows x 32/G chunks, row stride in
    // shared memory; y: G columns and CK chunks per CTA, of which those of its tile of KO are written
    int G, sp, CK, KO, halo;
    int cells;  // x: states of a CTA in values / p
    int staged, bulk;  // x: rows go through shared memory; by bulk copies of row_values values
    const P* in[2];
    P* out[2];
    const P* base[2];
    const void* tab[2];
    int* status;
    int* tstatus;
    long long wait_ns;
    P tmax;
    Batch b;
};

template <typename T>
__device__ __forceinline__ T* shift(T* p, long long off) {
    return p ? reinterpret_cast<T*>(reinterpret_cast<char*>(const_cast<typename std::remove_const<T>::type*>(p)) + off)
             : p;
}

// Values of a row in shared memory: its N values up to a multiple of 16 bytes, whatever the row pitch of the field (a
// caller of the allocation-free step chooses that).  Bulk copies move as many: rows of a multiple of 16 bytes have them.
template <typename P>
__host__ __device__ __forceinline__ int row_values(int N) {
    constexpr int per = 16 / (int)sizeof(P);
    return (N + per - 1) / per * per;
}

// ---- x tile: G rows of one array, the whole CTA (G * chunks threads, the chunks rounded up to whole
// warps) -----------------------------------------------------------------------------------
// shared memory: [16] mbarrier, [G][sp] rows (staged), [chunks][G][p] states, [4p][G] end values
template <typename P, int PD, int M, bool UNI, bool STAGED>
__device__ __forceinline__ void x_tile(const PassArgs<P>& a, long long off, int arr, int tile, unsigned char* smem,
                                       int tid, int nt) {
    const bool one = arr != 0;
    const P* in = shift(one ? a.in[1] : a.in[0], off);
    P* out = shift(one ? a.out[1] : a.out[0], off);
    const void* tab = shift(one ? a.tab[1] : a.tab[0], off);
    const int N = a.N, C = a.C, G = a.G, L = 32 / G;
    const int j0 = tile * G, rows = min(G, a.nlines - j0);
    const size_t row_bytes = (size_t)row_values<P>(N) * sizeof(P);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
    P* rowbuf = reinterpret_cast<P*>(smem + 16);
    P* st = rowbuf + (STAGED ? (size_t)G * a.sp : 0);
    const int warp = tid >> 5, lane = tid & 31;
    const int r = lane / L, k = warp * L + (lane - r * L);
    const bool active = tid < nt && r < rows && k < C;

    if constexpr (STAGED) {
        if (a.bulk) {
            if (tid == 0) {
                mbar_init(bar, 1);
                mbar_fence_init();
                mbar_expect_tx(bar, (uint32_t)(rows * row_bytes));
                for (int q = 0; q < rows; ++q)
                    bulk_load(rowbuf + (size_t)q * a.sp, in + (size_t)(j0 + q) * a.pitch, (uint32_t)row_bytes, bar);
            }
            __syncthreads();
            const bool ok = __syncthreads_and(mbar_wait_bounded(bar, 0, a.wait_ns));
            if (!ok) {
                // drain the copies in flight before the shared memory is released; the step's output is
                // not valid (bit 4 invalidates it for the whole handle)
                mbar_drain(bar, 0);
                int* ts = shift(a.tstatus, off);
                if (tid == 0 && ts) atomicOr(ts, 4);
                return;
            }
        } else {
            for (int q = 0; q < rows; ++q)
                for (int x = tid; x < N; x += blockDim.x)
                    rowbuf[(size_t)q * a.sp + x] = __ldcg(in + (size_t)(j0 + q) * a.pitch + x);
            __syncthreads();
        }
    }
    P x[M];
    const int o0 = k * M, have = active ? N - o0 : 0;
    P* g = rowbuf + (active ? (size_t)r * a.sp + o0 : 0);
    const size_t go = active ? (size_t)(j0 + r) * a.pitch + o0 : 0;
    const bool any = STAGED ? chunk_load<false>(g, 1, have, x) : chunk_load<false>(in + go, 1, have, x);
    // rows of zeros (the fuel increment away from a fire) are their own solution
    if (!__syncthreads_or(any)) {
        if (in == out) return;
    }
    const int kc = active ? k : 0;
    const Sweeps<P, PD, M, UNI> sw(tab, kc, C);
    P* fs = st + ((size_t)kc * G + r) * PD;
    P* ends = st + (size_t)a.cells * PD;
    P s[PD];
    sw.forward1(x, s);
    if (active)
#pragma unroll
        for (int j = 0; j < PD; ++j) fs[j] = s[j];
    __syncthreads();
    sw.enter(st + r * PD, G * PD, 1, 0, C, -1, s);
    sw.forward2(x, s);
    sw.backward1(x, s, have);
    __syncthreads();
    if (active)
#pragma unroll
        for (int j = 0; j < PD; ++j) fs[j] = s[j];
    __syncthreads();
    sw.enter(st + r * PD, G * PD, 1, 0, C, 1, s);
    sw.backward2(x, s);
    sw.ends_put(x, ends + r, G, N, have);
    __syncthreads();
    if (active) sw.ends_take(x, ends + r, G, C);
    auto put = [&](P* o) {
        if (have >= M) {
#pragma unroll
            for (int i = 0; i < M; ++i) o[i] = x[i];
        } else {
#pragma unroll
            for (int i = 0; i < M; ++i)
                if (i < have) o[i] = x[i];
        }
    };
    if constexpr (STAGED) {
        put(g);
        if (a.bulk) {
            fence_proxy_async_smem();
            __syncthreads();
            if (tid == 0) {
                for (int q = 0; q < rows; ++q)
                    bulk_store(out + (size_t)(j0 + q) * a.pitch, rowbuf + (size_t)q * a.sp, (uint32_t)row_bytes);
                bulk_commit_and_wait_read();
            }
        } else {
            __syncthreads();
            for (int q = 0; q < rows; ++q)
                for (int c = tid; c < N; c += blockDim.x)
                    out[(size_t)(j0 + q) * a.pitch + c] = rowbuf[(size_t)q * a.sp + c];
        }
    } else {
        put(out + go);
    }
}

// ---- y tile: G columns x CK chunks of threads ----------------------------------------------------
// The chunks [ko, ke) of the tile are written; up to `halo` chunks on either side are solved as far as
// the states that enter the tile need (lines of more chunks than a CTA holds).  shared memory:
// [p][CK][G] states, [4p][G] end values.
template <typename P, int PD, int M, bool UNI, bool CG>
__device__ __forceinline__ void y_tile(const PassArgs<P>& a, long long off, int arr, int cg, int tile,
                                       unsigned char* smem, int tid) {
    const bool one = arr != 0;
    const P* in = shift(one ? a.in[1] : a.in[0], off);
    P* out = shift(one ? a.out[1] : a.out[0], off);
    const P* base = shift(one ? a.base[1] : a.base[0], off);
    const void* tab = shift(one ? a.tab[1] : a.tab[0], off);
    const int N = a.N, C = a.C, G = a.G;
    const int ko = tile * a.KO, ke = min(C, ko + a.KO);
    const int kb = max(0, ko - a.halo), kn = min(C, ke + a.halo);
    const int kk = tid / G, c = tid - kk * G, k = kb + kk;
    const int line = cg * G + c;
    const bool active = k < kn && kk < a.CK && line < a.nlines;
    const int kc = active ? k : kb, row0 = kc * M;
    const size_t pitch = (size_t)a.pitch;
    P* st = reinterpret_cast<P*>(smem);
    const int cells = a.CK * G;
    P x[M];
    const int have = active ? N - row0 : 0;
    const size_t o0 = (size_t)row0 * pitch + (active ? line : 0);
    const bool any = chunk_load<CG>(in + o0, pitch, have, x);
    // columns of zeros (the fuel increment away from a fire) add nothing to their base
    if (!__syncthreads_or(any)) {
        if (base == out && (arr != 0 || a.status == nullptr)) return;
    }
    const Sweeps<P, PD, M, UNI> sw(tab, kc, C);
    P s[PD];
    P* fs = st + kk * G + c;
    P* ends = st + (size_t)cells * PD;
    const bool mine = kk < a.CK, mine_out = active && k >= ko && k < ke;
    sw.forward1(x, s);
    if (mine)
#pragma unroll
        for (int j = 0; j < PD; ++j) fs[j * cells] = s[j];
    __syncthreads();
    sw.enter(st + c, G, cells, kb, kn, -1, s);
    sw.forward2(x, s);
    sw.backward1(x, s, have);
    __syncthreads();
    if (mine)
#pragma unroll
        for (int j = 0; j < PD; ++j) fs[j * cells] = s[j];
    __syncthreads();
    if (mine_out) {
        sw.enter(st + c, G, cells, kb, kn, 1, s);
        sw.backward2(x, s);
        sw.ends_put(x, ends + c, G, N, have);
    }
    __syncthreads();
    if (!mine_out) return;  // no barrier follows in this tile
    sw.ends_take(x, ends + c, G, C);
    const P* bs = base ? base + o0 : nullptr;
    const bool bad = have >= M ? chunk_store(out + o0, bs, pitch, M, x, a.tmax)
                               : chunk_store(out + o0, bs, pitch, have, x, a.tmax);
    if (bad && a.status != nullptr && arr == 0) atomicOr(shift(a.status, off), 1);
}

// ---- y tile of the middle of a Strang / Crank-Nicolson step ----------------------------------------
// With u the x-solved right-hand side of the first substep, T* = T + (M^y)^{-1} u, and the y substep
// Y_+ T** = (2 M^y - Y_+) T* becomes
//   T** = T - (M^y)^{-1} u + Y_+^{-1} (2 u + 2 B T),   B = -theta_y A_y:
// two solves of one column in one pass instead of a pass for T* and a second one for T**.  T** goes to a
// field of its own (tiles read the rows of T around theirs).  in: u, base: T, tab: M^y and Y_+, band:
// factors of B's rows on differences of T (TabJob), out: T**.
template <typename P, int PD, int M, bool UNI>
__device__ __forceinline__ void y_mid_tile(const PassArgs<P>& a, const P* band0, long long off, int cg, int tile,
                                           unsigned char* smem, int tid) {
    constexpr int W = 2 * PD;
    const P* in = shift(a.in[0], off);
    P* out = shift(a.out[0], off);
    const P* base = shift(a.base[0], off);
    const P* band = shift(band0, off);
    const int N = a.N, C = a.C, G = a.G;
    const int ko = tile * a.KO, ke = min(C, ko + a.KO);
    const int kb = max(0, ko - a.halo), kn = min(C, ke + a.halo);
    const int kk = tid / G, c = tid - kk * G, k = kb + kk;
    const int line = cg * G + c;
    const bool active = k < kn && kk < a.CK && line < a.nlines, mine = kk < a.CK;
    const int kc = active ? k : kb, row0 = kc * M;
    const size_t pitch = (size_t)a.pitch;
    P* st = reinterpret_cast<P*>(smem);
    const int cells = a.CK * G;
    P* st2 = st + (size_t)PD * cells + 4 * PD * G;
    P u[M], v[M];
    {
        const P* src = in + (active ? line : 0);
        const P* T = base + (active ? line : 0);
        auto row_of = [&](int r) { return (active && r >= 0 && r < N) ? field_load(T + r * pitch) : P(0); };
        P dif[W];  // T[i - p + e + 1] - T[i - p + e]
        P last = row_of(row0 - PD);
#pragma unroll
        for (int e = 0; e + 1 < W; ++e) {
            const P next = row_of(row0 - PD + e + 1);
            dif[e] = next - last;
            last = next;
        }
        P bi[W];  // the rows of B away from the ends of the line
        const bool inner = N > 4 * PD;
#pragma unroll
        for (int e = 0; e < W; ++e) bi[e] = inner ? __ldg(band + (size_t)(2 * PD) * W + e) : P(0);
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const int row = row0 + i;
            const P next = row_of(row + PD);
            dif[W - 1] = next - last;
            last = next;
            u[i] = (active && row < N) ? field_load(src + row * pitch) : P(0);
            P t = P(0);
            if (inner && row >= 2 * PD && row < N - 2 * PD) {
#pragma unroll
                for (int e = 0; e < W; ++e) t += bi[e] * dif[e];
            } else if (row < N) {
#pragma unroll
                for (int e = 0; e < W; ++e) t += __ldg(band + (size_t)row * W + e) * dif[e];
            }
            v[i] = P(2) * (u[i] + t);
#pragma unroll
            for (int e = 0; e + 1 < W; ++e) dif[e] = dif[e + 1];
        }
    }
    const Sweeps<P, PD, M, UNI> sm(shift(a.tab[0], off), kc, C), sy(shift(a.tab[1], off), kc, C);
    const int have = active ? N - row0 : 0;
    P s[PD], s2[PD];
    P* fs = st + kk * G + c;
    P* fs2 = st2 + kk * G + c;
    auto put = [&] {
        if (mine)
#pragma unroll
            for (int j = 0; j < PD; ++j) {
                fs[j * cells] = s[j];
                fs2[j * cells] = s2[j];
            }
    };
    P* ends = st + (size_t)PD * cells;
    P* ends2 = st2 + (size_t)PD * cells;
    const bool mine_out = active && k >= ko && k < ke;
    sm.forward1(u, s);
    sy.forward1(v, s2);
    put();
    __syncthreads();
    sm.enter(st + c, G, cells, kb, kn, -1, s);
    sy.enter(st2 + c, G, cells, kb, kn, -1, s2);
    sm.forward2(u, s);
    sy.forward2(v, s2);
    sm.backward1(u, s, have);
    sy.backward1(v, s2, have);
    __syncthreads();
    put();
    __syncthreads();
    if (mine_out) {
        sm.enter(st + c, G, cells, kb, kn, 1, s);
        sy.enter(st2 + c, G, cells, kb, kn, 1, s2);
        sm.backward2(u, s);
        sy.backward2(v, s2);
        sm.ends_put(u, ends + c, G, N, have);
        sy.ends_put(v, ends2 + c, G, N, have);
    }
    __syncthreads();
    if (!mine_out) return;
    sm.ends_take(u, ends + c, G, C);
    sy.ends_take(v, ends2 + c, G, C);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        const size_t o = (size_t)(row0 + i) * pitch + line;
        if (row0 + i < N) out[o] = base[o] + (v[i] - u[i]);
    }
}

// Tiles of handles in which some operator has no uniform factors (UNI false): each table says what it has, so
// that a slot's bits do not depend on the other slots.
__device__ __forceinline__ bool uniform_table(const void* tab, long long off) {
    return __ldg(static_cast<const int*>(shift(tab, off))) == 1;
}
template <typename P, int PD, int M, bool UNI, bool STAGED>
__device__ __forceinline__ void x_any(const PassArgs<P>& a, long long off, int arr, int tile, unsigned char* smem, int tid,
                                      int nt) {
    if constexpr (!kUniformFactors<P>)
        x_tile<P, PD, M, false, STAGED>(a, off, arr, tile, smem, tid, nt);
    else if (UNI || uniform_table(arr ? a.tab[1] : a.tab[0], off))
        x_tile<P, PD, M, true, STAGED>(a, off, arr, tile, smem, tid, nt);
    else
        x_tile<P, PD, M, false, STAGED>(a, off, arr, tile, smem, tid, nt);
}
template <typename P, int PD, int M, bool UNI, bool CG>
__device__ __forceinline__ void y_any(const PassArgs<P>& a, long long off, int arr, int cg, int tile, unsigned char* smem,
                                      int tid) {
    if constexpr (!kUniformFactors<P>)
        y_tile<P, PD, M, false, CG>(a, off, arr, cg, tile, smem, tid);
    else if (UNI || uniform_table(arr ? a.tab[1] : a.tab[0], off))
        y_tile<P, PD, M, true, CG>(a, off, arr, cg, tile, smem, tid);
    else
        y_tile<P, PD, M, false, CG>(a, off, arr, cg, tile, smem, tid);
}
template <typename P, int PD, int M, bool UNI>
__device__ __forceinline__ void y_mid_any(const PassArgs<P>& a, const P* band, long long off, int cg, int tile,
                                          unsigned char* smem, int tid) {
    if constexpr (!kUniformFactors<P>)
        y_mid_tile<P, PD, M, false>(a, band, off, cg, tile, smem, tid);
    else if (UNI || (uniform_table(a.tab[0], off) && uniform_table(a.tab[1], off)))
        y_mid_tile<P, PD, M, true>(a, band, off, cg, tile, smem, tid);
    else
        y_mid_tile<P, PD, M, false>(a, band, off, cg, tile, smem, tid);
}

// Geometry of a pass (host): fills the fields of `a` that do not come from LineArgs; false when the line
// does not fit one CTA.
template <typename P, int PD, int M>
bool x_geometry(const LineArgs& l, int max_threads, size_t smem_budget, PassArgs<P>& a, int* threads, size_t* smem) {
    // Rows per CTA: eight (full use of a warp's banks and one barrier for many rows: 256 scenarios of 258^2,
    // step 318 us; 343 at 2, 402 at 1), fewer while that leaves less than four CTAs per SM (1026^2: 34.8 us
    // at 2, 35.5 at 8).
    int G = 8;
    if (l.G > 0)
        while (G > 1 && G > l.G) G /= 2;
    else
        while (G > 1 && (long)((l.nlines + G - 1) / G) * l.narr * l.b.S < 4L * 152) G /= 2;
    for (;; G /= 2) {
        const int L = 32 / G, slots = sizeof(P) == 4 ? 32 : 16;
        // shared-memory row stride: the rows of a warp start L banks apart (chunk lengths are odd), so its
        // lanes hit distinct banks; 16-byte multiple for bulk copies
        int sp = row_values<P>(l.N);
        if (L < slots)
            while (sp % (2 * L) != L || (sp * sizeof(P)) % 16 != 0) ++sp;
        else
            while ((sp * sizeof(P)) % 16 != 0) ++sp;
        const int nt = ((a.C + L - 1) / L) * 32;
        a.cells = (nt / 32) * L * G;
        const size_t states = ((size_t)a.cells * PD + 4 * PD * G) * sizeof(P);
        size_t need = 16 + (size_t)G * sp * sizeof(P) + states;
        a.staged = 1;
        if (G == 1 && need > 227 * 1024) {
            a.staged = 0;  // a row that does not fit the shared memory is read in place
            need = 16 + states;
        }
        if (nt <= max_threads && need <= (G > 1 ? smem_budget : (size_t)227 * 1024)) {
            a.G = G;
            a.sp = sp;
            *threads = nt;
            *smem = need;
            return true;
        }
        if (G == 1) return false;
    }
}

// most: threads a CTA may have.  Whole columns where a CTA holds them with at least 64 bytes of columns side
// by side, else tiles of chunks with a halo (1026^2 FP32, 61 chunks: step 35.5 us in tiles of 32 columns, 37.7
// with whole columns eight at a time).
template <typename P, int PD, int M>
bool y_geometry(const LineArgs& l, int most, PassArgs<P>& a, int* threads, size_t* smem) {
    int G = 32;
    while (G > 64 / (int)sizeof(P) && G * a.C > most) G /= 2;
    a.halo = 0;
    a.CK = a.KO = a.C;
    if (G * a.C > most) {
        // tiles of equal height; the first holds the J chunks from the top, the last the J + 1 from the
        // bottom that the end corrections reach
        const int CK = most / 32, J = l.J < a.C ? l.J : a.C;
        int KO = CK - 2 * J;
        if (KO > J) {
            const int n = (a.C + KO - 1) / KO;
            KO = (a.C + n - 1) / n;
            while (KO > J && a.C - (a.C - 1) / KO * KO < J + 1) --KO;
        }
        if (KO > J) {
            G = 32;
            a.CK = KO + 2 * J;
            a.halo = J;
            a.KO = KO;
        } else {
            // the states reach further than a tile of chunks: whole columns, fewer of them
            while (G > 1 && G * a.C > most) G /= 2;
            if (G * a.C > most) return false;
        }
    }
    a.G = G;
    *threads = (G * a.CK + 31) / 32 * 32;
    *smem = ((size_t)PD * a.CK * G + 4 * PD * G) * sizeof(P);
    return true;
}

template <typename P>
void pass_args(const LineArgs& l, int N, PassArgs<P>& a) {
    a.N = N;
    a.C = l.C;
    a.nlines = l.nlines;
    a.pitch = l.pitch;
    a.G = a.sp = a.CK = a.KO = a.halo = a.cells = 0;
    a.staged = a.bulk = 0;
    for (int q = 0; q < 2; ++q) {
        a.in[q] = (const P*)l.in[q];
        a.out[q] = (P*)l.out[q];
        a.base[q] = (const P*)l.base[q];
        a.tab[q] = l.tab[q];
    }
    a.status = l.status;
    a.tstatus = l.tstatus;
    a.wait_ns = l.wait_ns;
    a.tmax = (P)l.tmax;
    a.b = l.b;
}

}  // namespace
}  // namespace wf
