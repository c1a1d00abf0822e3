// Kernels and launchers of the line passes of one degree (WF_LINES_P), see wf_lines.cuh.
#include "wf_lines.cuh"

namespace wf {

namespace {

// Threads of a CTA at most, and CTAs per SM the registers are budgeted for: FP32 with up to 17 values a
// thread 40 registers (three CTAs), 33 values 64 (two; one: 4099^2 cubic 611 us instead of 556); FP64 128.
// The 40 registers are for launches of many waves, and spill (uniform factors, x and y pass: p = 2 72 and 28 bytes with 9
// values, 96 and 48 with 17; p = 3 36 and 32, 96 and 236).  Step with three / two CTAs: 256 x 258^2 324 / 344 us; launches
// of one partial wave would rather have two: 1026^2 34.1 / 31.8, 130^2 13.4 / 12.4, 8 x 515^2 cubic 104.3 / 102.7.
template <typename P, int M>
struct LineOcc {
    static constexpr int threads = 512;
    static constexpr int ctas = sizeof(P) == 4 ? (M <= 17 ? 3 : 2) : 1;
};

template <typename P, int PD, int M, bool UNI, int NT, bool STAGED>
__global__ void __launch_bounds__(NT, NT > 512 ? 1 : LineOcc<P, M>::ctas) k_xlines(const __grid_constant__ PassArgs<P> a,
                                                                                   int nt) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    long long off = (long long)blockIdx.z * a.b.sbytes;
    grid_wait(off);
    if (!scene_active(a.b)) return;
    x_any<P, PD, M, UNI, STAGED>(a, off, blockIdx.y, blockIdx.x, smem_raw, threadIdx.x, nt);
}

template <typename P, int PD, int M, bool UNI, int NT>
__global__ void __launch_bounds__(NT, NT > 512 ? 1 : LineOcc<P, M>::ctas) k_ylines(const __grid_constant__ PassArgs<P> a,
                                                                                   int ntiles) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    long long off = (long long)blockIdx.z * a.b.sbytes;
    const int cg = blockIdx.x / ntiles;
    grid_wait(off);
    if (!scene_active(a.b)) return;
    y_any<P, PD, M, UNI, false>(a, off, blockIdx.y, cg, blockIdx.x - cg * ntiles, smem_raw, threadIdx.x);
}

// The middle pass holds two chunks: FP32 with 17 values 80 registers and tiles of 384 threads, two CTAs per SM, so
// that the 264 CTAs of a 1026^2 domain run at once (with 512 threads and 128 registers 198 CTAs took two turns of
// 152: step 79.1 us against 72.5; 71.7 since the explicit operator acts on differences).
template <typename P, int M>
struct MidOcc {
    static constexpr bool two = sizeof(P) == 4 && M == 17;
    static constexpr int threads = two ? 384 : 512, ctas = two ? 2 : 1;
};

template <typename P, int PD, int M, bool UNI, int NT>
__global__ void __launch_bounds__(NT, NT > 512 ? 1 : MidOcc<P, M>::ctas) k_ymid(const __grid_constant__ PassArgs<P> a,
                                                                                const P* band, int ntiles) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    long long off = (long long)blockIdx.z * a.b.sbytes;
    const int cg = blockIdx.x / ntiles;
    grid_wait(off);
    if (!scene_active(a.b)) return;
    y_mid_any<P, PD, M, UNI>(a, band, off, cg, blockIdx.x - cg * ntiles, smem_raw, threadIdx.x);
}

template <typename K, typename... A>
cudaError_t go(K kern, dim3 grid, int threads, size_t smem, cudaStream_t s, A... args) {
    if (smem > 48 * 1024) {
        cudaError_t e = allow_dynamic_smem(kern, smem);
        if (e != cudaSuccess) return e;
    }
    const cudaError_t e = launch_overlapped(kern, grid, threads, smem, s, args...);
    if (e == cudaSuccess) count_launches(1);
    return e;
}

template <typename P, int PD, int M, bool UNI>
cudaError_t run_x(const LineArgs& l, cudaStream_t s) {
    PassArgs<P> a;
    pass_args(l, l.N, a);
    int nt = 0;
    size_t smem = 0;
    // lines of more chunks than 512 threads hold (above 16384 values) take a kernel of 1024
    const bool wide = !x_geometry<P, PD, M>(l, LineOcc<P, M>::threads, 72 * 1024, a, &nt, &smem);
    if (wide && (M < 33 || !x_geometry<P, PD, M>(l, 1024, 72 * 1024, a, &nt, &smem))) return cudaErrorInvalidValue;
    bool aligned = a.staged && (a.pitch * sizeof(P)) % 16 == 0 && a.b.sbytes % 16 == 0;
    for (int q = 0; q < l.narr; ++q)
        aligned = aligned && (uintptr_t)l.in[q] % 16 == 0 && (uintptr_t)l.out[q] % 16 == 0;
    a.bulk = aligned ? 1 : 0;
    const dim3 grid((l.nlines + a.G - 1) / a.G, l.narr, l.b.S);
    if constexpr (M == 33) {
        if (wide)
            return a.staged ? go(k_xlines<P, PD, M, UNI, 1024, true>, grid, nt, smem, s, a, nt)
                            : go(k_xlines<P, PD, M, UNI, 1024, false>, grid, nt, smem, s, a, nt);
        if (!a.staged) return go(k_xlines<P, PD, M, UNI, 512, false>, grid, nt, smem, s, a, nt);
    }
    // (shorter chunks mean rows of at most 1600 values, which always fit: there is no other kernel for them)
    if (!a.staged) return cudaErrorInvalidValue;
    return go(k_xlines<P, PD, M, UNI, 512, true>, grid, nt, smem, s, a, nt);
}

template <typename P, int PD, int M, bool UNI>
cudaError_t run_y(const LineArgs& l, cudaStream_t s) {
    PassArgs<P> a;
    pass_args(l, l.N, a);
    int nt = 0;
    size_t smem = 0;
    const bool wide = !y_geometry<P, PD, M>(l, LineOcc<P, M>::threads, a, &nt, &smem);
    if (wide && (M < 33 || !y_geometry<P, PD, M>(l, 1024, a, &nt, &smem))) return cudaErrorInvalidValue;
    const int ntiles = (a.C + a.KO - 1) / a.KO;
    const dim3 grid((unsigned)((l.nlines + a.G - 1) / a.G * ntiles), l.narr, l.b.S);
    if constexpr (M == 33)
        if (wide) return go(k_ylines<P, PD, M, UNI, 1024>, grid, nt, smem, s, a, ntiles);
    return go(k_ylines<P, PD, M, UNI, 512>, grid, nt, smem, s, a, ntiles);
}

template <typename P, int PD, int M, bool UNI>
cudaError_t run_ymid(const LineArgs& l, cudaStream_t s) {
    PassArgs<P> a;
    pass_args(l, l.N, a);
    int nt = 0;
    size_t smem = 0;
    // (states that reach over more than a tile of a line of more than 512 chunks: whole columns of up to 1024)
    const bool wide = !y_geometry<P, PD, M>(l, MidOcc<P, M>::threads, a, &nt, &smem);
    if (wide && (M < 33 || !y_geometry<P, PD, M>(l, 1024, a, &nt, &smem))) return cudaErrorInvalidValue;
    const int ntiles = (a.C + a.KO - 1) / a.KO;
    const dim3 grid((unsigned)((l.nlines + a.G - 1) / a.G * ntiles), 1, l.b.S);
    if constexpr (M == 33)
        if (wide) return go(k_ymid<P, PD, M, UNI, 1024>, grid, nt, 2 * smem, s, a, (const P*)l.band, ntiles);
    return go(k_ymid<P, PD, M, UNI, MidOcc<P, M>::threads>, grid, nt, 2 * smem, s, a, (const P*)l.band, ntiles);
}

template <typename P, int PD, int M, bool UNI>
cudaError_t run_kind(int kind, const LineArgs& l, cudaStream_t s) {
    return kind == 0 ? run_x<P, PD, M, UNI>(l, s)
                     : (kind == 1 ? run_y<P, PD, M, UNI>(l, s) : run_ymid<P, PD, M, UNI>(l, s));
}

template <typename P, int PD, int M>
cudaError_t run_pass(int kind, const LineArgs& l, cudaStream_t s) {
    if constexpr (kUniformFactors<P>)
        if (l.uni) return run_kind<P, PD, M, true>(kind, l, s);
    return run_kind<P, PD, M, false>(kind, l, s);
}

template <typename P, int PD>
cudaError_t by_chunk(int kind, const LineArgs& l, cudaStream_t s) {
    switch (l.M) {
        case 9: return run_pass<P, PD, 9>(kind, l, s);
        case 17: return run_pass<P, PD, 17>(kind, l, s);
        case 33: return run_pass<P, PD, 33>(kind, l, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace
}  // namespace wf
