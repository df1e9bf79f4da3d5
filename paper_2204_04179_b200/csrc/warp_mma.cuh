// Warp-level MMA (m16n8k16, bf16 operands, fp32 accumulators) and its fragment loads, shared by the attention kernels.
#pragma once
#include "gram_internal.h"

namespace wmma16 {

__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack2(float x, float y) {
  __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float quad_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// Fragment conventions of m16n8k16 (g = lane / 4, q = lane % 4):
//   A (16 x 16, row-major source X[m][k]):  a0 = X[g][2q..], a1 = X[g+8][2q..], a2 = X[g][2q+8..], a3 = X[g+8][2q+8..]
//   B (16 x 8, source stored as Y[n][k]):   b0 = Y[g][2q..], b1 = Y[g][2q+8..]
//   C (16 x 8):                             c0,c1 = C[g][2q, 2q+1], c2,c3 = C[g+8][2q, 2q+1]
// Where the contraction index is contiguous in shared memory (Q K^T, dO V^T) fragments are plain 32-bit
// loads.  Where it is the row index (P V, dS K, dS^T Q, P^T dO) the 8 x 8 tiles are read with
// ldmatrix.trans, so every matrix is kept once, row-major, with rows padded by 8 elements (conflict-free
// for both access kinds).

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm_x4_trans(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3, const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(smem_addr(p)));
}
__device__ __forceinline__ void ldsm_x4(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3, const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(smem_addr(p)));
}
// B fragments of two adjacent n-tiles (n0, n0+8) for the k-tile k0, from Y[n][k] (contraction index contiguous):
// (b0, b1) of tile n0 and (b2, b3) of tile n0 + 8
__device__ __forceinline__ void load_b_rows(const bf16* Y, int ld, int n0, int k0, int lane, uint32_t& b0, uint32_t& b1,
                                            uint32_t& b2, uint32_t& b3) {
  const int row = n0 + (lane & 7) + (lane >> 4) * 8, col = k0 + ((lane >> 3) & 1) * 8;
  ldsm_x4(b0, b1, b2, b3, Y + row * ld + col);
}
// A fragment (rows m0.., k-tile k0) of a row-major X[m][k]
__device__ __forceinline__ void load_a_rows(const bf16* X, int ld, int m0, int k0, int lane, uint32_t& a0, uint32_t& a1,
                                            uint32_t& a2, uint32_t& a3) {
  const int row = m0 + (lane & 7) + ((lane >> 3) & 1) * 8, col = k0 + (lane >> 4) * 8;
  ldsm_x4(a0, a1, a2, a3, X + row * ld + col);
}
// B fragments of two adjacent n-tiles (n0, n0+8) for the k-tile k0, from a row-major S[k][n] with row stride ld:
// (b0, b1) of tile n0 and (b2, b3) of tile n0 + 8
__device__ __forceinline__ void load_b_trans(const bf16* S, int ld, int k0, int n0, int lane, uint32_t& b0, uint32_t& b1,
                                             uint32_t& b2, uint32_t& b3) {
  const int row = k0 + (lane & 7) + ((lane >> 3) & 1) * 8, col = n0 + (lane >> 4) * 8;
  ldsm_x4_trans(b0, b1, b2, b3, S + row * ld + col);
}
// A fragment (m-tile m0, k-tile k0) of the transpose of a row-major S[k][m] with row stride ld
__device__ __forceinline__ void load_a_trans(const bf16* S, int ld, int k0, int m0, int lane, uint32_t& a0, uint32_t& a1,
                                             uint32_t& a2, uint32_t& a3) {
  const int row = k0 + (lane & 7) + (lane >> 4) * 8, col = m0 + ((lane >> 3) & 1) * 8;
  ldsm_x4_trans(a0, a1, a2, a3, S + row * ld + col);
}

}  // namespace wmma16
