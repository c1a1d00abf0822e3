// Persistent line passes: after the quadrature launch of a Peaceman-Rachford step (one F per
// step), one launch runs the rest of the step for every active slot of a batch handle.
//
// Paper: Sec. 3.1 Eq. matrixPR (the two substeps, in their combined form, wf_api.cu), Sec. 4
// (every directional solve is a set of independent 1-D line solves, which is what lets one launch
// cover every pass of a whole batch).
//
// After the quadrature (R and Phi of every slot), the step of one slot is two passes, each a set
// of independent tiles:
//   X  x lines of R with X_+ and of Phi with M^x, in groups of rows
//   Y  y lines (R -> T^{n+1} with Y_+, Phi -> phi^{n+1} with M^y, increment bases added, guard),
//      in groups of columns
// The arithmetic of every tile is that of the per-pass kernels (the same device functions or
// the same operations in the same order), so both step forms give the same bits.
//
// Work items (pass, slot, tiles) are listed by the host in a wavefront over groups of slots: at
// "time" t the list holds X of group t and Y of group t-1, so the fields of about two groups are
// live at once, and consecutive items are independent.  A CTA claims the next item from a ticket
// counter (the next ticket is fetched while the current item runs); before touching its inputs a
// Y item waits for the arrival counter of the X row groups of its array.  A tile waits only for
// tiles with smaller tickets, which are running or done when it is claimed, so the launch always
// makes progress whatever the number of resident CTAs.
// Producers release (stores, barrier, fence, counter add); consumers acquire (ld.acquire on
// the counter, barrier) and read data produced in this launch through L2 (ld.global.cg),
// never through the read-only path.  Every wait is bounded by the handle's wait limit (the
// SM's global timer); a wait that gives up sets the slot's timeout bit and the launch-wide
// abort flag, after which every remaining item is skipped, so a failure costs one limit.
#include <algorithm>

#include "wf_internal.h"

namespace wf {

cudaError_t persist_step(const PersistHost& h, PersistPlan* plan, bool launch, cudaStream_t s) {
    PersistPlan dummy;
    if (!plan) plan = &dummy;
    switch (h.p) {
        case 1: return persist_p1(h, plan, launch, s);
        case 2: return persist_p2(h, plan, launch, s);
        case 3: return persist_p3(h, plan, launch, s);
    }
    return cudaErrorNotSupported;
}

// Wavefront order of the work items over groups of `gs` active slots (see the top of the file).
// An item covers several consecutive tiles of one (pass, slot, array): about two items per CTA
// in every pass over all active slots, so that a CTA stages an operator's factors once for
// several tiles and the fixed costs of an item (claim, barriers, dependency check) amortise.
// ph: 0 x, 1 y.
int persist_items(const PersistPlan& plan, const int* slots, int nslots, int gs, int4* out, int cap,
                  int* items_per_slot) {
    if (gs < 1) gs = 1;
    const int ngroups = (nslots + gs - 1) / gs;
    const long target = 2L * std::max(1, plan.ctas);
    auto per_item = [&](long tiles_all, int most) {
        return (int)std::max(1L, std::min((long)most, tiles_all / target));
    };
    const int tx = per_item((long)nslots * plan.narr * plan.nxg, plan.nxg);
    const int ty = per_item((long)nslots * plan.narr * plan.nyg, plan.nyg);
    int n = 0, per_slot = 0;
    auto put = [&](int ph, int m, int z, int a, int b) {
        if (n < cap) out[n] = make_int4(ph | (m << 8), z, a, b);
        ++n;
    };
    auto tiles = [&](int ph, int z, int arr, int count, int per) {
        for (int i = 0; i < count; i += per) put(ph, std::min(per, count - i), z, arr, i);
    };
    for (int t = 0; t < ngroups + 1; ++t)
        for (int ph = 0; ph < 2; ++ph) {
            const int g = t - ph;
            if (g < 0 || g >= ngroups) continue;
            for (int k = g * gs; k < std::min(nslots, (g + 1) * gs); ++k) {
                const int z = slots[k];
                const int n0 = n;
                for (int arr = 0; arr < plan.narr; ++arr)
                    tiles(ph, z, arr, ph == 0 ? plan.nxg : plan.nyg, ph == 0 ? tx : ty);
                if (k == 0) per_slot += n - n0;
            }
        }
    *items_per_slot = per_slot;
    return n;
}

}  // namespace wf
