// pft_tcgen05.cuh -- the tensor-core instructions of the separable march's convolutions, and the
// storage of their circulant operand.
//
// K_a = F_a^-1 d_a F_a, the periodic Gaussian convolution along axis a (pft_sep.cuh), is the
// product with a real symmetric circulant matrix of the n_a kernel values
// kern[j] = (1/n_a) sum_k d_a(k) cos(2 pi j k / n_a): one tile of 128 lines of n points is
// D[line][out] = sum_k X[line][k] kern[(out - k) mod n], one tcgen05 product with X in tensor
// memory (lane = line) and the matrix in shared memory.
//
// The matrix is stored once per diagonal of 8 x 8 blocks ("core matrices" of the unswizzled
// shared-memory layout, 128 bytes each): block (k8, n8) depends on n8 - k8 only, so both
// strides of the operand descriptor are one block and 2 n/8 - 1 blocks hold the matrix (4 KB at
// n = 128 instead of 32 KB).  A 16-wide k step takes two neighbouring k8; descending k8 is the
// ascending storage order, so the two halves of each 16 points of X are swapped in tensor
// memory to match.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "pft_batch.cuh"
#include "pft_tma.cuh"

namespace pft {

__device__ __forceinline__ void tc_alloc(uint32_t* dst_smem, unsigned cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(dst_smem)), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tc_dealloc(uint32_t base, unsigned cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols));
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}
// D (tensor memory) (+)= A (tensor memory, 128 x 16 FP16) x B (shared memory)
__device__ __forceinline__ void tc_mma_f16_ts(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t idesc, unsigned acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d), "r"(a), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
// 32 lanes x 8 columns from and into registers
__device__ __forceinline__ void tc_st4(uint32_t addr, const uint32_t (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3])
               : "memory");
}
__device__ __forceinline__ void tc_ld8(uint32_t addr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(addr)
               : "memory");
}
// Unswizzled operand of the circulant storage: both block strides are one 128-byte block.
__device__ __forceinline__ uint64_t tc_desc(unsigned saddr) {
  return (uint64_t)((saddr >> 4) & 0x3fffu) | ((uint64_t)8 << 16) | ((uint64_t)8 << 32) | ((uint64_t)1 << 46);
}
// FP16 x FP16 -> FP32, M = 128, both operands k-major
__host__ __device__ constexpr uint32_t tc_idesc(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
// true in one lane of a converged warp
__device__ __forceinline__ bool elect_one() {
  unsigned p;
  asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void named_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// An axis' table lies behind its factors sd (n values), at the next multiple of 256 bytes.
__host__ __device__ constexpr size_t tc_align(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace pft
