// pft_tc64_launch.cuh -- launches of kb_tc64_line.
#pragma once
#include "pft_engine.h"
#include "pft_tc64.cuh"

namespace pft {

// complex fields (a translation unit of their own)
cudaError_t tc_launch_f64c(const SeppGeom& g, const BatchStep* ss, int ax, int pw, int members, cudaStream_t sm);

template <int N, int KIND, int PW, int AX>
cudaError_t tc64_launch(const BatchStep* st, long long nlines, long long cin, long long s_outer, long long s_k, int members,
                   int* err, cudaStream_t sm) {
  auto kern = kb_tc64_line<N, KIND, PW, AX>;
  constexpr size_t smem = tc64_smem<N, KIND, PW, AX>();
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  kern<<<dim3((unsigned)((nlines + 127) / 128), (unsigned)members), Tc64Cfg<N>::THREADS, smem, sm>>>(
      st, (int)nlines, (int)cin, (int)s_outer, (int)s_k, err);
  return cudaGetLastError();
}

template <int KIND, int PW, int AX>
cudaError_t tc64_launch_n(int n, const BatchStep* st, long long nlines, long long cin, long long s_outer, long long s_k,
                     int members, int* err, cudaStream_t sm) {
  switch (n) {
    case 16: return tc64_launch<16, KIND, PW, AX>(st, nlines, cin, s_outer, s_k, members, err, sm);
    case 32: return tc64_launch<32, KIND, PW, AX>(st, nlines, cin, s_outer, s_k, members, err, sm);
    case 48: return tc64_launch<48, KIND, PW, AX>(st, nlines, cin, s_outer, s_k, members, err, sm);
    case 64: return tc64_launch<64, KIND, PW, AX>(st, nlines, cin, s_outer, s_k, members, err, sm);
    case 96: return tc64_launch<96, KIND, PW, AX>(st, nlines, cin, s_outer, s_k, members, err, sm);
    case 128: return tc64_launch<128, KIND, PW, AX>(st, nlines, cin, s_outer, s_k, members, err, sm);
    default: return cudaErrorInvalidValue;
  }
}

template <int KIND>
cudaError_t tc64_axis_k(const SeppGeom& g, const BatchStep* ss, int ax, int pw, int members, cudaStream_t sm) {
  const long long nx = g.n[0], ny = g.n[1], row = (long long)g.n[2] * (KIND ? 2 : 1);  // doubles a row
  if (ax == 0) return tc64_launch_n<KIND, 2, 0>(g.n[0], ss, ny * row, ny * row, 0, ny * row, members, g.err, sm);
  if (ax == 1) return tc64_launch_n<KIND, 0, 1>(g.n[1], ss, nx * row, row, ny * row, row, members, g.err, sm);
  const long long rows = nx * ny * (KIND ? 2 : 1);
  return pw == 1 ? tc64_launch_n<KIND, 1, 2>(g.n[2], ss, rows, 0, 0, 0, members, g.err, sm)
                 : tc64_launch_n<KIND, 2, 2>(g.n[2], ss, rows, 0, 0, 0, members, g.err, sm);
}

}  // namespace pft
