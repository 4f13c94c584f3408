// The FP64 separable pencil march with its convolutions on the tensor cores, real fields: FP64
// fields between the launches (an axis without a table runs the FFT kernel).  A translation unit
// per field kind and layout, compiled in parallel.
#include "pft_tc64_launch.cuh"

namespace pft {

// Axes with a table, but for short launches on x (the march's serial chain of two convolutions a
// tile, and a tile holds 128 real lines against the FFT kernels' 16, so few lines leave a tile per
// SM or less and its latency counts): measured in us a contour step of both marches, FFT -> tensor
// cores, complex fields, 16x8x8 22.9 -> 24.5, 16x12x192 65.6 -> 68.6, 16x24x192 76.6 -> 75.7;
// 64x8x8 30.5 -> 35.3, 64x24x24 53.5 -> 59.3, 64x12x192 124 -> 122, 128x24x24 77.9 -> 83.1,
// 128x12x192 253 -> 194; real fields 16x8x8 21.1 -> 21.8, 16x12x192 58.9 -> 59.4, 64x8x8 30.1 ->
// 29.0.  x lines of 32 and 48 points, and y and z, gain or are level at every size measured.  The
// rule counts one member's lines: what a system computes does not depend on its neighbours in a
// batch.
bool tc64_axis_applies(const SeppGeom& g, int ax) {
  if (g.lv != 0 || !tc64_axis_ok(g.n[ax])) return false;
  if (ax != 0) return true;
  const long long lines = (long long)g.n[1] * g.n[2];
  if (g.n[0] == 16) return lines >= 4096;
  return g.kind == 0 || g.n[0] < 64 || lines >= 2048;
}
cudaError_t tc_launch_f64(const SeppGeom& g, const BatchStep* ss, int ax, int pw, int members, cudaStream_t sm) {
  return g.kind == 0 ? tc64_axis_k<0>(g, ss, ax, pw, members, sm) : tc_launch_f64c(g, ss, ax, pw, members, sm);
}
size_t tc64_axis_table_bytes(int n) { return tc64_axis_ok(n) ? tc64_table_bytes(n) : 0; }
void tc64_axis_table(int n, const long double* d, unsigned char* dst) { tc64_build_table(n, d, dst); }

}  // namespace pft
