// Persistent line passes of degree 1.
#include "wf_persist.cuh"

namespace wf {

cudaError_t persist_p1(const PersistHost& h, PersistPlan* plan, bool launch, cudaStream_t s) {
    return persist_prec<1>(h, plan, launch, s);
}

}  // namespace wf
