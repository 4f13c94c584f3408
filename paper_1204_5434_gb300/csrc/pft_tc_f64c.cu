// pft_tc_f64.cu's launches for complex fields.
#include "pft_tc64_launch.cuh"

namespace pft {
cudaError_t tc_launch_f64c(const SeppGeom& g, const BatchStep* ss, int ax, int pw, int members, cudaStream_t sm) {
  return tc64_axis_k<1>(g, ss, ax, pw, members, sm);
}
}  // namespace pft
