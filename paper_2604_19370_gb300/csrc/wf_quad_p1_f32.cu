// Quadrature kernels of degree 1, FP32 (see wf_quad.cuh).
#include "wf_quad.cuh"

namespace wf {

cudaError_t launch_quad_p1_f32(const RhsArgs& r, cudaStream_t s) { return quad_by_rank<float, 1>(r, s); }

}  // namespace wf
