// Quadrature kernels of degree 3, FP32 (see wf_quad.cuh).
#include "wf_quad.cuh"

namespace wf {

cudaError_t launch_quad_p3_f32(const RhsArgs& r, cudaStream_t s) { return quad_by_rank<float, 3>(r, s); }

}  // namespace wf
