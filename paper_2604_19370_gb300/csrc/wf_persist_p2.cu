// Persistent line passes of degree 2.
#include "wf_persist.cuh"

namespace wf {

cudaError_t persist_p2(const PersistHost& h, PersistPlan* plan, bool launch, cudaStream_t s) {
    return persist_prec<2>(h, plan, launch, s);
}

}  // namespace wf
