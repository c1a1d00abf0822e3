// Persistent line passes of degree 3.
#include "wf_persist.cuh"

namespace wf {

cudaError_t persist_p3(const PersistHost& h, PersistPlan* plan, bool launch, cudaStream_t s) {
    return persist_prec<3>(h, plan, launch, s);
}

}  // namespace wf
