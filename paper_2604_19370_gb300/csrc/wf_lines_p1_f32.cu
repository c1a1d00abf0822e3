// Line passes of degree 1, FP32.
#include "wf_lines_body.cuh"

namespace wf {

cudaError_t launch_lines_p1_f32(int kind, const LineArgs& l, cudaStream_t s) { return by_chunk<float, 1>(kind, l, s); }

}  // namespace wf
