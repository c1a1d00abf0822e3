// Chunked line solves (TMA-staged x pass, column-parallel y pass).
//
// Paper: Sec. 4 ("Cost of directional implicit solves"): each directional system
// is a set of independent banded 1-D solves (half-bandwidth p) along x or y.
//
// Every line is cut into at most 32 chunks; one thread owns one chunk (`base`
// values, or the last chunk of at most base + 2p values), runs the chunk-local LU
// substitution with the recurrence in registers, solves the p x p interface
// systems of truncated SPIKE with its neighbours' boundary values and applies the
// spike corrections.  LU factors and spikes come from shared memory in their
// compact form: with uniform open knots every interior chunk has the same factors,
// so a CTA stages three chunk types (first, interior, last) whatever the length.
//
// x pass: one warp per row, one lane per chunk.  The rows of a CTA are contiguous
// in memory and move with one TMA bulk copy each way (cp.async.bulk with an
// mbarrier); neighbouring chunks exchange boundary values by warp shuffles.
// y pass: a CTA owns G columns; lanes of neighbouring columns read and write
// contiguous runs of G elements per row, 16 or 32 loads in flight per thread.
#include "wf_internal.h"

#include "wf_line_blocks.cuh"

namespace wf {

namespace {

// x pass.  CTA = G lines; a warp solves 32 / lanes lines, lane k of a line's group owns chunk k
// (C <= lanes per line).
// The G rows are contiguous in memory: one bulk copy stages them, one bulk store writes them back.
// Chunk lengths are odd, so the 32 lanes of a warp read 32 distinct shared-memory banks.
template <typename P, int PD>
__global__ void __launch_bounds__(256) k_xsolve_warp(const FastArgs<P> a) {
    if (!scene_active(a.b)) return;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Chunks ch = a.ch;
    const int N = ch.N, C = ch.C, base = ch.base, G = a.G;
    const int mmax = base + 2 * PD;
    const int arr = blockIdx.y;
    const LineView<P> v = scene_line(a, arr);
    const int j0 = blockIdx.x * G;
    const int rows = min(G, a.nlines - j0);
    const size_t row_bytes = (size_t)a.pitch * sizeof(P);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);
    const int sp = a.sp;                                           // shared-memory row stride
    P* rowbuf = reinterpret_cast<P*>(smem_raw + 128);             // [G][sp]
    const FacSmem<P, PD> fm(rowbuf + (size_t)G * sp, mmax);
    const P* __restrict__ in = v.in;
    P* out = v.out;
    // factors: one bulk copy of the operator's padded block beside the rows, else staged element
    // by element
    const bool fbulk = a.tma && v.fpad != nullptr;
    const uint32_t fbytes = (uint32_t)(fac_elems<PD>(mmax) * sizeof(P));
    bool staged = true;
    if (a.tma) {
        // one bulk copy per row (the shared-memory stride differs from the global pitch);
        // thread 0 arms the barrier with the total, the lanes of warp 0 issue the copies
        if (tid == 0) {
            mbar_init(bar, 1);
            mbar_fence_init();
            const uint32_t bytes = (uint32_t)(rows * row_bytes);
            mbar_expect_tx(bar, bytes + (fbulk ? fbytes : 0u));
        }
        __syncwarp();
        if (warp == 0) {
            if (fbulk && lane == 31) bulk_load(fm.F, v.fpad, fbytes, bar);
            for (int r = lane; r < rows; r += 32)
                bulk_load(rowbuf + (size_t)r * sp, in + (size_t)(j0 + r) * a.pitch, (uint32_t)row_bytes, bar);
        }
    } else {
        for (int r = 0; r < rows; ++r)
            for (int x = tid; x < N; x += blockDim.x) rowbuf[(size_t)r * sp + x] = in[(size_t)(j0 + r) * a.pitch + x];
    }
    if (!fbulk) stage_factors<P, PD>(v, mmax, fm);
    __syncthreads();  // mbarrier initialised, factors staged
    if (a.tma) staged = mbar_wait_bounded(bar, 0, a.wait_ns);
    staged = __syncthreads_and(staged);  // one decision for the whole CTA (barriers follow)
    if (!staged) {
        // drain the copies in flight before the shared memory is released; the step's output is
        // not valid (bit 4 invalidates it for the whole handle)
        mbar_drain(bar, 0);
        if (tid == 0 && v.tstatus) atomicOr(v.tstatus, 4);
        return;
    }
    // lanes per line: 32 >> (5 - lsh); line r of the CTA = warp * lines-per-warp + lane / lanes
    const int k = lane & ((1 << a.lsh) - 1);
    const int r = (warp << (5 - a.lsh)) + (lane >> a.lsh);
    const bool active = r < rows && k < C;
    const int m = (k < C - 1) ? base : ch.last;
    P* g = rowbuf + (size_t)(r < rows ? r : 0) * sp + (size_t)k * base;
    const int t = chunk_type(ch, k < C ? k : 0);
    if (active) {
        lu_forward<P, PD>(g, m, fm.F + t * mmax * FacW<PD>::F);
        lu_backward<P, PD>(g, m, fm.U + t * mmax * FacW<PD>::U);
    }
    __syncwarp();
    P top[PD], bot[PD], nxt_top[PD], prv_bot[PD];
#pragma unroll
    for (int q = 0; q < PD; ++q) {
        top[q] = active ? g[q] : P(0);
        bot[q] = (active && k + 1 < C) ? g[base - PD + q] : P(0);
    }
#pragma unroll
    for (int q = 0; q < PD; ++q) {
        nxt_top[q] = __shfl_down_sync(0xffffffffu, top[q], 1);
        prv_bot[q] = __shfl_up_sync(0xffffffffu, bot[q], 1);
    }
    P tn[PD], bp[PD];
    interface_solve<P, PD>(ch, k < C ? k : 0, mmax, fm.S, fm.E, top, bot, nxt_top, prv_bot, tn, bp);
    if (active) spike_fix<P, PD>(g, m, fm.S + t * mmax * FacW<PD>::S, tn, bp);
    if (a.tma) {
        fence_proxy_async_smem();
        __syncthreads();
        if (warp == 0) {
            bool issued = false;
            for (int r = lane; r < rows; r += 32) {
                bulk_store(out + (size_t)(j0 + r) * a.pitch, rowbuf + (size_t)r * sp, (uint32_t)row_bytes);
                issued = true;
            }
            if (issued) bulk_commit_and_wait_read();
        }
    } else {
        __syncthreads();
        for (int r = 0; r < rows; ++r)
            for (int x = tid; x < N; x += blockDim.x) out[(size_t)(j0 + r) * a.pitch + x] = rowbuf[(size_t)r * sp + x];
    }
}

// y pass.  CTA = G columns x C chunks (blockDim = G*C <= 256); thread tid = k*G + c owns chunk k
// of column c in its private shared-memory strip (odd stride: distinct banks).  The column values
// are loaded 16 or 32 rows at a time and eliminated forward as they arrive, so the strip is written
// once before the backward sweep; the increment base is added on the final store.  Threads of
// columns past the last line solve a copy of the last line and store nothing.
template <typename P, int PD, int B>
__global__ void __launch_bounds__(256) k_ysolve_cols(const FastArgs<P> a) {
    constexpr int W = 2 * PD + 1, B2 = 8;
    constexpr int NF = FacW<PD>::F, NU = FacW<PD>::U, NS = FacW<PD>::S;
    if (!scene_active(a.b)) return;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x;
    const Chunks ch = a.ch;
    const int N = ch.N, C = ch.C, base = ch.base, G = a.G, mpad = a.mpad;
    const int mmax = base + 2 * PD;
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);  // 16 bytes: the factors' mbarrier
    const FacSmem<P, PD> fm(reinterpret_cast<P*>(smem_raw + 16), mmax);
    P* buf = fm.end();  // [nt][mpad]
    const int arr = blockIdx.y;
    const int k = tid / G, c = tid - k * G;
    const int s = k * base;
    const int m = (k < C - 1) ? base : ch.last;
    const int t = chunk_type(ch, k);
    const int line_raw = blockIdx.x * G + c;
    const bool valid = line_raw < a.nlines;
    const int line = valid ? line_raw : a.nlines - 1;
    const LineView<P> v = scene_line(a, arr);
    const size_t pitch = (size_t)a.pitch;
    P* g = buf + (size_t)tid * mpad;

    // factors: one bulk copy of the operator's padded block (bounded wait; a CTA that gives up
    // stores nothing and sets bit 4 of the slot's flag word), else staged element by element
    const bool fbulk = v.fpad != nullptr;
    if (fbulk) {
        if (tid == 0) {
            const uint32_t fbytes = (uint32_t)(fac_elems<PD>(mmax) * sizeof(P));
            mbar_init(bar, 1);
            mbar_fence_init();
            mbar_expect_tx(bar, fbytes);
            bulk_load(fm.F, v.fpad, fbytes, bar);
        }
    } else {
        stage_factors<P, PD>(v, mmax, fm);
    }
    __syncthreads();
    if (fbulk) {
        const bool ok = __syncthreads_and(mbar_wait_bounded(bar, 0, a.wait_ns));
        if (!ok) {
            mbar_drain(bar, 0);
            if (tid == 0 && v.tstatus) atomicOr(v.tstatus, 4);
            return;
        }
    }
    const P* __restrict__ pre = v.premul;
    const P* Fk = fm.F + t * mmax * NF;
    P prev[PD];
#pragma unroll
    for (int i = 0; i < PD; ++i) prev[i] = P(0);
    if (pre) {
        // right-hand side prescale (premul band (x) I) in: rows s .. s+m-1 of the product
        const P ps = v.prescale;
        for (int o = 0; o < m; ++o) {
            const int row = s + o;
            P acc = 0;
#pragma unroll
            for (int d = 0; d < W; ++d) {
                const int rr = row + d - PD;
                if (rr >= 0 && rr < N) acc += pre[(size_t)row * W + d] * v.in[(size_t)rr * pitch + line];
            }
            P x[1] = {ps * acc};
            fwd_rows<P, PD, 1>(x, Fk + o * NF, prev);
            g[o] = x[0];
        }
    } else {
        const P* __restrict__ src = v.in + (size_t)s * pitch + line;
        int o = 0;
        for (; o + B <= m; o += B) {
            P r[B];
#pragma unroll
            for (int q = 0; q < B; ++q) r[q] = src[q * pitch];
            src += B * pitch;
            fwd_rows<P, PD, B>(r, Fk + o * NF, prev);
#pragma unroll
            for (int q = 0; q < B; ++q) g[o + q] = r[q];
        }
        for (; o < m; ++o) {
            P r[1] = {*src};
            src += pitch;
            fwd_rows<P, PD, 1>(r, Fk + o * NF, prev);
            g[o] = r[0];
        }
    }
    lu_backward<P, PD>(g, m, fm.U + t * mmax * NU);
    __syncthreads();
    const P* gn = buf + (size_t)((k + 1 < C ? k + 1 : k) * G + c) * mpad;
    const P* gp = buf + (size_t)((k > 0 ? k - 1 : k) * G + c) * mpad + (base - PD);
    P tn[PD], bp[PD];
    interface_solve<P, PD>(ch, k, mmax, fm.S, fm.E, g, g + (base - PD), gn, gp, tn, bp);
    if (!valid) return;  // no barrier follows
    const P* Sk = fm.S + t * mmax * NS;
    const P* __restrict__ bs = v.base ? v.base + (size_t)s * pitch + line : nullptr;
    P* dst = v.out + (size_t)s * pitch + line;
    const P tmax = a.tmax;
    bool bad = false;
    // final rows: spike correction, increment base, store, guard
    auto finish = [&](auto nrows, int o) {
        constexpr int R = decltype(nrows)::value;
        P x[R], bv[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            x[q] = g[o + q];
            bv[q] = bs ? bs[(size_t)q * pitch] : P(0);
        }
        spike_rows<P, PD, R>(x, Sk + o * NS, tn, bp);
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const P y = x[q] + bv[q];
            dst[(size_t)q * pitch] = y;
            bad |= !(fabs(y) <= tmax);  // also catches NaN
        }
        if (bs) bs += R * pitch;
        dst += R * pitch;
    };
    int o = 0;
    for (; o + B2 <= m; o += B2) finish(std::integral_constant<int, B2>{}, o);
    for (; o < m; ++o) finish(std::integral_constant<int, 1>{}, o);
    if (bad && v.status != nullptr && arr == 0) atomicOr(v.status, 1);
}

// y pass for long lines (many chunks): CTA = 32 columns x C chunks (up to 1024 threads), thread
// tid = k*32 + c owns chunk k of column c, so a warp's loads and stores cover 32 consecutive columns
// (128-byte row pieces) whatever the chunk count.  The chunk's partial results are kept in the
// pass's input array (the right-hand side, dead after the pass: LineArgs::in_dead) instead of a
// shared-memory strip (a strip per thread of a long chunk fills the shared memory with one CTA of
// eight columns): each thread overwrites the input elements it has read and reads them back in the
// later sweeps (its own writes, in program order; the CTA's column block stays in L2); neighbouring
// chunks exchange their first and last p values through shared memory.
// Per column the operations, and their order, are those of k_ysolve_cols: the same bits.
template <typename P, int PD, int B>
__global__ void __launch_bounds__(1024) k_ysolve_long(const FastArgs<P> a) {
    constexpr int B2 = 8;
    constexpr int NF = FacW<PD>::F, NU = FacW<PD>::U, NS = FacW<PD>::S;
    if (!scene_active(a.b)) return;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x;
    const Chunks ch = a.ch;
    const int C = ch.C, base = ch.base;
    constexpr int G = 32;
    const int mmax = base + 2 * PD;
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);  // 16 bytes: the factors' mbarrier
    const FacSmem<P, PD> fm(reinterpret_cast<P*>(smem_raw + 16), mmax);
    P* xch = fm.end();  // [C][G][2p]: the first and the last p values of every chunk
    const int arr = blockIdx.y;
    const int k = tid / G, c = tid - k * G;
    const int s = k * base;
    const int m = (k < C - 1) ? base : ch.last;
    const int t = chunk_type(ch, k);
    const int line = blockIdx.x * G + c;
    const bool valid = line < a.nlines;  // threads past the last line only take part in the barriers
    const LineView<P> v = scene_line(a, arr);
    const size_t pitch = (size_t)a.pitch;
    const bool fbulk = v.fpad != nullptr;
    if (fbulk) {
        if (tid == 0) {
            const uint32_t fbytes = (uint32_t)(fac_elems<PD>(mmax) * sizeof(P));
            mbar_init(bar, 1);
            mbar_fence_init();
            mbar_expect_tx(bar, fbytes);
            bulk_load(fm.F, v.fpad, fbytes, bar);
        }
    } else {
        stage_factors<P, PD>(v, mmax, fm);
    }
    __syncthreads();
    if (fbulk) {
        const bool ok = __syncthreads_and(mbar_wait_bounded(bar, 0, a.wait_ns));
        if (!ok) {
            mbar_drain(bar, 0);
            if (tid == 0 && v.tstatus) atomicOr(v.tstatus, 4);
            return;
        }
    }
    P* g = const_cast<P*>(v.in) + (size_t)s * pitch + (valid ? line : 0);  // this chunk's input elements
    P top[PD], bot[PD];
    if (valid) {
        const P* Fk = fm.F + t * mmax * NF;
        P prev[PD];
#pragma unroll
        for (int i = 0; i < PD; ++i) prev[i] = P(0);
        const P* src = v.in + (size_t)s * pitch + line;  // the elements g overwrites, each after its read
        int o = 0;
        for (; o + B <= m; o += B) {
            P r[B];
#pragma unroll
            for (int q = 0; q < B; ++q) r[q] = src[q * pitch];
            src += B * pitch;
            fwd_rows<P, PD, B>(r, Fk + o * NF, prev);
#pragma unroll
            for (int q = 0; q < B; ++q) g[(size_t)(o + q) * pitch] = r[q];
        }
        for (; o < m; ++o) {
            P r[1] = {*src};
            src += pitch;
            fwd_rows<P, PD, 1>(r, Fk + o * NF, prev);
            g[(size_t)o * pitch] = r[0];
        }
        // backward substitution from the last row up, on the elements just written
        const P* Uk = fm.U + t * mmax * NU;
#pragma unroll
        for (int i = 0; i < PD; ++i) prev[i] = P(0);
        int top_r = m - 1;
        for (; top_r - B2 + 1 >= 0; top_r -= B2) {
            P gv[B2];
#pragma unroll
            for (int q = 0; q < B2; ++q) gv[q] = g[(size_t)(top_r - q) * pitch];
            bwd_rows<P, PD, B2>(gv, Uk + top_r * NU, prev);
#pragma unroll
            for (int q = 0; q < B2; ++q) g[(size_t)(top_r - q) * pitch] = gv[q];
        }
        for (; top_r >= 0; --top_r) {
            P gv[1] = {g[(size_t)top_r * pitch]};
            bwd_rows<P, PD, 1>(gv, Uk + top_r * NU, prev);
            g[(size_t)top_r * pitch] = gv[0];
        }
        P* mine = xch + (size_t)tid * 2 * PD;
#pragma unroll
        for (int q = 0; q < PD; ++q) {
            top[q] = g[(size_t)q * pitch];
            // the last chunk may be shorter than base (its last p values are not used)
            bot[q] = (k + 1 < C) ? g[(size_t)(base - PD + q) * pitch] : P(0);
            mine[q] = top[q];
            mine[PD + q] = bot[q];
        }
    }
    __syncthreads();
    if (!valid) return;  // no barrier follows
    const P* nx = xch + (size_t)((k + 1 < C ? k + 1 : k) * G + c) * 2 * PD;
    const P* pv = xch + (size_t)((k > 0 ? k - 1 : k) * G + c) * 2 * PD + PD;
    P nt[PD], pb[PD], tn[PD], bp[PD];
#pragma unroll
    for (int q = 0; q < PD; ++q) {
        nt[q] = nx[q];
        pb[q] = pv[q];
    }
    interface_solve<P, PD>(ch, k, mmax, fm.S, fm.E, top, bot, nt, pb, tn, bp);
    const P* Sk = fm.S + t * mmax * NS;
    const P* bs = v.base ? v.base + (size_t)s * pitch + line : nullptr;  // may be the output array
    P* dst = v.out + (size_t)s * pitch + line;
    const P tmax = a.tmax;
    bool bad = false;
    auto finish = [&](auto nrows, int o) {
        constexpr int R = decltype(nrows)::value;
        P x[R], bv[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            x[q] = g[(size_t)(o + q) * pitch];
            bv[q] = bs ? bs[(size_t)(o + q) * pitch] : P(0);
        }
        spike_rows<P, PD, R>(x, Sk + o * NS, tn, bp);
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const P y = x[q] + bv[q];
            dst[(size_t)(o + q) * pitch] = y;
            bad |= !(fabs(y) <= tmax);  // also catches NaN
        }
    };
    int o = 0;
    for (; o + B2 <= m; o += B2) finish(std::integral_constant<int, B2>{}, o);
    for (; o < m; ++o) finish(std::integral_constant<int, 1>{}, o);
    if (bad && v.status != nullptr && arr == 0) atomicOr(v.status, 1);
}

template <typename P, int PD, bool X>
cudaError_t run_fast(const LineArgs& a, cudaStream_t s) {
    const Chunks& ch = a.f[0].ch;
    if (ch.C > 32) return cudaErrorNotSupported;
    const int mmax = ch.base + 2 * PD;
    const size_t fbytes = (size_t)fac_elems<PD>(mmax) * sizeof(P);
    FastArgs<P> f;
    f.nlines = a.nlines;
    f.pitch = a.pitch;
    f.ch = ch;
    for (int q = 0; q < 2; ++q) {
        f.in[q] = (const P*)a.in[q];
        f.out[q] = (P*)a.out[q];
        f.base[q] = (const P*)a.base[q];
        f.premul[q] = (const P*)a.premul[q];
        f.prescale[q] = (P)a.prescale[q];
        f.luc[q] = (const P*)a.f[q].luc;
        f.spkc[q] = (const P*)a.f[q].spkc;
        f.Ec[q] = (const P*)a.f[q].Ec;
        f.fpad[q] = (const P*)a.f[q].fpad;
    }
    f.status = a.status;
    f.tstatus = a.tstatus;
    f.wait_ns = a.wait_ns;
    f.tmax = (P)a.tmax;
    f.b = a.b;
    f.mpad = (ch.base > ch.last ? ch.base : ch.last) | 1;
    if (X) {
        // rows per CTA: as many warps as fit 100 KB of staged rows (at least one)
        const size_t row_bytes = (size_t)a.pitch * sizeof(P);
        // lines per warp: as many as the chunks allow (C <= 8: four, C <= 16: two), or fewer
        int lsh = ch.C <= 8 ? 3 : (ch.C <= 16 ? 4 : 5);
        if (a.rpw == 1) lsh = 5;
        else if (a.rpw == 2 && lsh < 4) lsh = 4;
        const int lpw = 1 << (5 - lsh);
        // shared-memory row stride: the lines of a warp start L banks apart (L = lanes per line,
        // chunk lengths odd), so its lanes hit distinct banks; 16-byte multiple for bulk copies
        const int L = 32 >> (5 - lsh);
        const int slots = sizeof(P) == 4 ? 32 : 16;  // bank-width words per wavefront
        int sp = a.pitch;
        if (L < slots)
            while (sp % (2 * L) != L || (sp * sizeof(P)) % 16 != 0) ++sp;
        const size_t srow = (size_t)sp * sizeof(P);
        auto need = [&](int g) { return 128 + g * srow + fbytes; };
        // lines per CTA: up to 8 warps' worth, fewer when the staged rows need more than 100 KB
        int G = 8 * lpw;
        if (a.G > 0 && a.G < G) G = a.G < lpw ? lpw : a.G;
        G = (G + lpw - 1) / lpw * lpw;
        while (G > lpw && need(G) > 100 * 1024) G = ((G / 2) + lpw - 1) / lpw * lpw;
        const size_t smem = need(G);
        if (smem > 227 * 1024) return cudaErrorNotSupported;
        bool aligned = (row_bytes % 16 == 0) && (a.b.sbytes % 16 == 0);
        for (int q = 0; q < a.narr; ++q)
            aligned = aligned && ((uintptr_t)a.in[q] % 16 == 0) && ((uintptr_t)a.out[q] % 16 == 0);
        f.G = G;
        f.lsh = lsh;
        f.sp = sp;
        f.tma = aligned ? 1 : 0;
        auto kern = k_xsolve_warp<P, PD>;
        cudaError_t e = allow_dynamic_smem(kern, (size_t)smem);
        if (e != cudaSuccess) return e;
        dim3 grid((a.nlines + G - 1) / G, a.narr, a.b.S);
        kern<<<grid, 32 * (G / lpw), smem, s>>>(f);
        count_launches(1);
    } else {
        int sms = 152, dev = 0;
        if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        // long lines (more than 8 chunks) whose input is dead after the pass, no prescale band, and
        // enough 32-column blocks for half the SMs: 32 columns per CTA, partial results in the input
        bool lng = a.in_dead && ch.C > 8 && (long)((a.nlines + 31) / 32) * a.narr * a.b.S >= sms / 2;
        for (int q = 0; q < a.narr; ++q) lng = lng && a.premul[q] == nullptr;
        if (lng) {
            const int ntl = 32 * ch.C;
            const size_t smeml = 16 + fbytes + (size_t)ntl * 2 * PD * sizeof(P);
            f.G = 32;
            f.tma = 0;
            dim3 grid((a.nlines + 31) / 32, a.narr, a.b.S);
            auto kern = k_ysolve_long<P, PD, 16>;
            cudaError_t e = allow_dynamic_smem(kern, smeml);
            if (e != cudaSuccess) return e;
            kern<<<grid, ntl, smeml, s>>>(f);
            count_launches(1);
            return cudaGetLastError();
        }
        int G = a.G > 0 ? (a.G < 256 ? a.G : 256) : (sizeof(P) == 4 ? 8 : 4);
        while (G > 1 && G * ch.C > 256) G /= 2;
        const int nt = G * ch.C;
        if (nt > 256) return cudaErrorNotSupported;
        const size_t smem = 16 + fbytes + (size_t)nt * f.mpad * sizeof(P);
        if (smem > 227 * 1024) return cudaErrorNotSupported;
        f.G = G;
        f.tma = 0;
        // rows loaded per batch: 32 when the launch leaves at most two CTAs per SM (its threads then
        // wait on load latency, and more loads in flight pay), else 16 (fewer registers, more CTAs)
        dim3 grid((a.nlines + G - 1) / G, a.narr, a.b.S);
        const bool wide = (long)grid.x * grid.y * grid.z <= 2L * sms;
        auto kern = wide ? k_ysolve_cols<P, PD, 32> : k_ysolve_cols<P, PD, 16>;
        cudaError_t e = allow_dynamic_smem(kern, (size_t)smem);
        if (e != cudaSuccess) return e;
        kern<<<grid, nt, smem, s>>>(f);
        count_launches(1);
    }
    return cudaGetLastError();
}

// Padded factor block of one operator: the layout stage_factors builds in shared memory, written
// once to global memory when the operator is factored (padding entries zero).
template <typename P, int PD>
__global__ void k_pad_factors(const P* __restrict__ luc, const P* __restrict__ spkc, const P* __restrict__ Ec,
                              int mmax, P* out) {
    const FacSmem<P, PD> fm(out, mmax);
    fill_factors<P, PD>(luc, spkc, Ec, mmax, fm, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

}  // namespace

cudaError_t launch_line_fast(int prec, int p, bool xdir, const LineArgs& a, cudaStream_t s) {
    for (int q = 0; q < a.narr; ++q)
        if (!a.f[q].compact || a.f[q].ch.base != a.f[0].ch.base || a.f[q].ch.C != a.f[0].ch.C)
            return cudaErrorNotSupported;
#define WF_FAST(P, PD) return xdir ? run_fast<P, PD, true>(a, s) : run_fast<P, PD, false>(a, s)
    if (prec == 0) {
        switch (p) {
            case 1: WF_FAST(float, 1);
            case 2: WF_FAST(float, 2);
            case 3: WF_FAST(float, 3);
        }
    } else {
        switch (p) {
            case 1: WF_FAST(double, 1);
            case 2: WF_FAST(double, 2);
            case 3: WF_FAST(double, 3);
        }
    }
#undef WF_FAST
    return cudaErrorNotSupported;
}

size_t fac_pad_elems(int p, int mmax) {
    switch (p) {
        case 1: return (size_t)fac_elems<1>(mmax);
        case 2: return (size_t)fac_elems<2>(mmax);
        case 3: return (size_t)fac_elems<3>(mmax);
    }
    return 0;
}

cudaError_t launch_pad_factors(int prec, int p, int mmax, const void* luc, const void* spkc, const void* Ec,
                               void* fpad, cudaStream_t s) {
    const size_t es = prec == 0 ? sizeof(float) : sizeof(double);
    const size_t n = fac_pad_elems(p, mmax);
    if (n == 0) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(fpad, 0, n * es, s);
    if (e != cudaSuccess) return e;
#define WF_PAD(P, PD) \
    k_pad_factors<P, PD><<<4, 256, 0, s>>>((const P*)luc, (const P*)spkc, (const P*)Ec, mmax, (P*)fpad)
    if (prec == 0) {
        switch (p) {
            case 1: WF_PAD(float, 1); break;
            case 2: WF_PAD(float, 2); break;
            case 3: WF_PAD(float, 3); break;
        }
    } else {
        switch (p) {
            case 1: WF_PAD(double, 1); break;
            case 2: WF_PAD(double, 2); break;
            case 3: WF_PAD(double, 3); break;
        }
    }
#undef WF_PAD
    return cudaGetLastError();
}

}  // namespace wf
