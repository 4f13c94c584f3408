// The FP64 separable pencil march with its convolutions on the tensor cores, real fields: FP64
// fields between the launches (an axis without a table runs the FFT kernel).  A translation unit
// per field kind and layout, compiled in parallel.
#include "pft_tc64_launch.cuh"

namespace pft {

bool tc64_axis_applies(const SeppGeom& g, int ax) { return g.lv == 0 && tc64_axis_ok(g.n[ax]); }
cudaError_t tc_launch_f64(const SeppGeom& g, const BatchStep* ss, int ax, int pw, int members, cudaStream_t sm) {
  return g.kind == 0 ? tc64_axis_k<0, 0>(g, ss, ax, pw, members, sm) : tc_launch_f64c(g, ss, ax, pw, members, sm);
}
size_t tc64_axis_table_bytes(int n) { return tc64_axis_ok(n) ? tc64_table_bytes(n) : 0; }
void tc64_axis_table(int n, const long double* d, unsigned char* dst) { tc64_build_table(n, d, dst); }

}  // namespace pft
