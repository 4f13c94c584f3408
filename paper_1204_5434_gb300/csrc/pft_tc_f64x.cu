// The FP64 separable pencil march on the tensor cores with fixed-point fields and Boltzmann factors
// (every axis with a table), real fields.
#include "pft_tc64_launch.cuh"

namespace pft {

cudaError_t tc_launch_f64x(const SeppGeom& g, const BatchStep* ss, int ax, int pw, int members, cudaStream_t sm) {
  return g.kind == 0 ? tc64_axis_k<1, 0>(g, ss, ax, pw, members, sm) : tc_launch_f64xc(g, ss, ax, pw, members, sm);
}
size_t tc64_fixed_bytes(long long n) { return kTc64FixedHeader + (size_t)n * 8; }
size_t tc64_scale_bytes(int Ns) { return ((size_t)2 * Ns + 1) * sizeof(Tc64Scale); }
size_t tc64_scale_step() { return 2 * sizeof(Tc64Scale); }
cudaError_t tc64_fix(int kind, const double* a, const double* b, const double* q0, const double* qd0, long long n,
                     unsigned* mx, void* fa, void* fb, int blocks, cudaStream_t sm) {
  blocks = (int)std::min<long long>(blocks, (n / 2 + 255) / 256);
  k_tc64_max<<<blocks, 256, 0, sm>>>((const double2*)a, (const double2*)b, (const double2*)q0, (const double2*)qd0, n / 2,
                                     mx);
  if (kind == 0) k_tc64_fix<0><<<blocks, 256, 0, sm>>>(a, b, n, mx, (char*)fa, (char*)fb);
  else k_tc64_fix<1><<<blocks, 256, 0, sm>>>(a, b, n, mx, (char*)fa, (char*)fb);
  return cudaGetLastError();
}

}  // namespace pft
