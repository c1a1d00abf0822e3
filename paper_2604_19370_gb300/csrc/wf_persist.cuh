// Device code and launch of the persistent line passes, included by one translation unit per degree (the
// scheme is described at the top of wf_persist.cu).
#pragma once
#include <string.h>

#include <algorithm>

#include "wf.h"
#include "wf_lines.cuh"

namespace wf {

namespace {

enum { PH_X = 0, PH_Y = 1 };

constexpr int kCntStride = 32;  // counters of a slot: arrivals of the x pass per array, items done

template <typename P>
struct PersistArgs {
    PassArgs<P> x, y;
    long long sbytes;
    int nxg, nty;  // row groups of the x pass, row tiles of a y column group
    int ntx;       // threads of an x tile
    const int4* items;
    const int* nitems;
    int* ctl;  // [0] ticket, [1] abort flag, [2] items, [3] items per slot
    int* cnt;  // slot z's counters at cnt + z * kCntStride
    long long wait_ns;
    int* status;  // slot 0's flag word (slot z: z * sbytes further)
    const int* active;  // per-slot activity flags: an inactive slot's items are skipped
    int* budget;        // per-slot step budgets (NULL: none); a spent one (0) skips the slot too
};

__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_relaxed(const int* p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Wait until *c >= target.  false: the wait gave up (limit reached: the slot's timeout bit and
// the abort flag are set) or another wait already did (abort flag seen).  Limit 0 gives up at
// once without looking, so that tests can take this path deterministically.
template <typename P>
__device__ bool wait_count(const PersistArgs<P>& A, const int* c, int target, int* slot_status) {
    if (A.wait_ns > 0) {
        if (ld_acquire(c) >= target) return true;
        const unsigned long long t0 = global_ns();
        for (unsigned it = 1;; ++it) {
            if (ld_acquire(c) >= target) return true;
            if (ld_relaxed(A.ctl + 1)) return false;
            if ((it & 7u) == 0u && (long long)(global_ns() - t0) > A.wait_ns) break;
            __nanosleep(64);
        }
    }
    atomicExch(A.ctl + 1, 1);
    if (slot_status) atomicOr(slot_status, WF_STATUS_TIMEOUT);
    return false;
}

__device__ __forceinline__ void arrive(int* c) {
    __threadfence();
    atomicAdd(c, 1);
}

// a slot takes part in this step: active and its step budget not spent
template <typename P>
__device__ __forceinline__ bool slot_live(const PersistArgs<P>& A, int z) {
    return ld_relaxed(A.active + z) != 0 && (!A.budget || ld_relaxed(A.budget + z) != 0);
}

// an item of slot z finished; the slot's last item of the step spends one step of its budget
// (every item of the slot has then started, so all of them saw the same budget)
template <typename P>
__device__ __forceinline__ void slot_done(const PersistArgs<P>& A, int* cnt, int z) {
    const int old = atomicAdd(cnt + 2, 1);
    if (old == A.ctl[3] - 1 && A.budget) {
        const int b = A.budget[z];
        if (b > 0) A.budget[z] = b - 1;
    }
}

// CTAs per SM the registers are budgeted for, by the CTA's threads.
template <typename P, int M, int NT>
struct PersistOcc {
    static constexpr int ctas = (sizeof(P) == 4 ? (M <= 17 ? 1536 : 1024) : 512) / NT;
};

template <typename P, int PD, int M, bool UNI, int NT>
__global__ void __launch_bounds__(NT, PersistOcc<P, M, NT>::ctas) k_lines_persist(const __grid_constant__ PersistArgs<P> A) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_item, s_go;
    const int tid = threadIdx.x;
    const int n = *A.nitems;
    int next = 0;
    if (tid == 0) next = atomicAdd(A.ctl, 1);
    for (;;) {
        if (tid == 0) {
            s_item = next;
            if (next < n) next = atomicAdd(A.ctl, 1);  // fetched while this item runs
        }
        __syncthreads();
        const int it = s_item;
        if (it >= n) break;
        const int4 d = A.items[it];
        const int ph = d.x & 0xff, m = d.x >> 8, z = d.y, arr = d.z;  // m: tiles of this item
        const long long off = (long long)z * A.sbytes;
        int* cnt = A.cnt + (size_t)z * kCntStride;
        if (tid == 0) {
            // bit 1: the slot takes part in this step; bit 0: go ahead (the item's inputs are ready)
            const bool live = slot_live(A, z);
            bool ok = live && !ld_relaxed(A.ctl + 1);
            if (ok && ph == PH_Y) ok = wait_count(A, cnt + arr, A.nxg, shift(A.status, off));
            s_go = (live ? 2 : 0) | (ok ? 1 : 0);
        }
        __syncthreads();
        const int go = s_go;
        if (go & 1) {
            for (int k = 0; k < m; ++k) {
                const int tile = d.w + k;
                if (ph == PH_X)
                    x_any<P, PD, M, UNI, true>(A.x, off, arr, tile, smem, tid, A.ntx);
                else
                    y_any<P, PD, M, UNI, true>(A.y, off, arr, tile / A.nty, tile % A.nty, smem, tid);
                __syncthreads();
                if (tid == 0 && ph == PH_X) arrive(cnt + arr);
            }
        }
        if (tid == 0 && (go & 2)) slot_done(A, cnt, z);
        __syncthreads();  // s_item and the shared memory are reused by the next item
    }
}

template <typename P, int PD, int M, bool UNI, int NT>
cudaError_t persist_typed(const PersistHost& h, PersistPlan* plan, bool launch, cudaStream_t s) {
    PersistArgs<P> A;
    memset(&A, 0, sizeof(A));
    pass_args(h.x, h.x.N, A.x);
    pass_args(h.y, h.y.N, A.y);
    int ntx = 0, nty = 0;
    size_t sx = 0, sy = 0;
    if (!x_geometry<P, PD, M>(h.x, NT, 72 * 1024, A.x, &ntx, &sx) ||
        !y_geometry<P, PD, M>(h.y, NT, A.y, &nty, &sy) || !A.x.staged)
        return cudaErrorNotSupported;
    A.x.bulk = 0;
    A.sbytes = h.x.b.sbytes;
    A.ntx = ntx;
    A.nxg = (h.x.nlines + A.x.G - 1) / A.x.G;
    A.nty = (A.y.C + A.y.KO - 1) / A.y.KO;
    const size_t smem = std::max(sx, sy);
    const int threads = std::max(ntx, nty);
    auto kern = k_lines_persist<P, PD, M, UNI, NT>;
    cudaError_t e = allow_dynamic_smem(kern, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0, sms = 152, dev = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorNotSupported;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    plan->nxg = A.nxg;
    plan->nyg = (h.y.nlines + A.y.G - 1) / A.y.G * A.nty;
    plan->narr = h.x.narr;
    plan->cstride = kCntStride;
    plan->ctas = per_sm * sms;
    if (!launch) return cudaSuccess;
    // the item list and counters were laid out for this plan (prepare step): never write past them
    if (!h.items || !h.ctl || !h.cnt || (size_t)h.nslots_cap * kCntStride > h.cnt_cap) return cudaErrorInvalidValue;
    A.items = h.items;
    A.nitems = h.ctl + 2;
    A.ctl = h.ctl;
    A.cnt = h.cnt;
    A.wait_ns = h.wait_ns;
    A.status = h.status;
    A.active = h.active;
    A.budget = h.budget;
    // every counter of this step starts at zero (ticket, abort flag, arrival counters)
    e = cudaMemsetAsync(h.ctl, 0, 2 * sizeof(int), s);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(h.cnt, 0, (size_t)h.nslots_cap * kCntStride * sizeof(int), s);
    if (e != cudaSuccess) return e;
    kern<<<plan->ctas, threads, smem, s>>>(A);
    count_launches(1);
    return cudaGetLastError();
}

// CTAs of 256 threads where they hold both kinds of tile: an x tile uses at most that many (128 on 258 values),
// so larger CTAs idle in the x pass (256 scenarios of
// 258^2, step: 1175 us with 512 threads, 671 with 256; one 1026^2 domain 73).
template <typename P, int PD, int M, bool UNI>
cudaError_t persist_threads(const PersistHost& h, PersistPlan* plan, bool launch, cudaStream_t s) {
    const cudaError_t e = persist_typed<P, PD, M, UNI, 256>(h, plan, launch, s);
    return e == cudaErrorNotSupported ? persist_typed<P, PD, M, UNI, 512>(h, plan, launch, s) : e;
}

template <typename P, int PD, bool UNI>
cudaError_t persist_by_chunk(const PersistHost& h, PersistPlan* plan, bool launch, cudaStream_t s) {
    switch (h.x.M) {
        case 9: return persist_threads<P, PD, 9, UNI>(h, plan, launch, s);
        case 17: return persist_threads<P, PD, 17, UNI>(h, plan, launch, s);
        case 33: return persist_threads<P, PD, 33, UNI>(h, plan, launch, s);
    }
    return cudaErrorNotSupported;
}

template <int PD>
cudaError_t persist_prec(const PersistHost& h, PersistPlan* plan, bool launch, cudaStream_t s) {
    if (h.prec == WF_FP32)
        return h.x.uni ? persist_by_chunk<float, PD, true>(h, plan, launch, s)
                       : persist_by_chunk<float, PD, false>(h, plan, launch, s);
    return persist_by_chunk<double, PD, false>(h, plan, launch, s);
}

}  // namespace
}  // namespace wf
