// Quadrature kernels of degree 1, FP64 (see wf_quad.cuh).
#include "wf_quad.cuh"

namespace wf {

cudaError_t launch_quad_p1_f64(const RhsArgs& r, cudaStream_t s) { return quad_by_rank<double, 1>(r, s); }

}  // namespace wf
