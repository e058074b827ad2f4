// Warp-level helpers shared by the GSTA and one-candidate kernels: mma.sync m16n8k16 (bf16 operands, fp32 accumulators),
// ldmatrix fragment loads, cp.async groups.  These kernels are bound by HBM / L2 traffic and instruction issue, not by
// tensor throughput; the warp-level MMA is used because its 16-row tiles fit their small per-candidate contractions.
//
// Fragment layout of m16n8k16 (g = lane / 4, t = lane % 4):
//   A (16 x 16, row major)  a[0] = (row g,     k 2t..2t+1)   a[1] = (row g + 8, k 2t..2t+1)
//                           a[2] = (row g,     k 2t+8..2t+9) a[3] = (row g + 8, k 2t+8..2t+9)
//   B (16 x 8)              b0 = (k 2t..2t+1, col g)         b1 = (k 2t+8..2t+9, col g)
//   C (16 x 8)              c[0], c[1] = (row g, cols 2t, 2t+1)   c[2], c[3] = (row g + 8, cols 2t, 2t+1)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace laser {
namespace mma {

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Four 8x8 b16 matrices; lanes 8i..8i+7 supply the row addresses of matrix i; r[i] = (row g, elements 2t, 2t+1) of it.
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
// Same, each matrix transposed on the way in.
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2(uint32_t (&r)[2], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}

// Transposes an 8x8 b16 matrix held one row per lane group: in: lane (g, t) holds row g, elements 2t, 2t+1;
// out: lane (g, t) holds column g, elements 2t, 2t+1.
__device__ __forceinline__ uint32_t movmatrix_t(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}

// Adds four floats to a 16-byte aligned place in global memory with one reduction.
__device__ __forceinline__ void red_add4(float* at, float x, float y, float z, float w) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(at), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

// Adds scale * (a 16 x 8 accumulator tile of mma16816) to the rows of C below `rows`.  Neighbouring lanes trade halves, so that
// a lane owns four columns of one row and adds them with one 16-byte reduction (C 16-byte aligned, ld a multiple of 4).
__device__ __forceinline__ void red_tile(float* C, size_t ld, const float (&v)[4], float scale, int lane, int rows = 16) {
  const int g = lane >> 2, t = lane & 3;
  const bool odd = t & 1;
  const float o0 = __shfl_xor_sync(0xffffffffu, odd ? v[0] : v[2], 1), o1 = __shfl_xor_sync(0xffffffffu, odd ? v[1] : v[3], 1);
  const int row = g + (odd ? 8 : 0);
  if (row < rows)
    red_add4(C + (size_t)row * ld + (t >> 1) * 4, scale * (odd ? o0 : v[0]), scale * (odd ? o1 : v[1]), scale * (odd ? v[2] : o0),
             scale * (odd ? v[3] : o1));
}

// 16-byte asynchronous global -> shared copy; src_bytes = 0 zero-fills the destination.
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// {lo, hi} -> packed bf16x2 (lo in bits 0-15), round to nearest even
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xFFFF0000u); }

// Reductions over the eight lane groups g = lane / 4 (lanes with the same t = lane % 4).
__device__ __forceinline__ float group_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 4));
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 8));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 16));
}
__device__ __forceinline__ float group_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 8);
  return v + __shfl_xor_sync(0xffffffffu, v, 16);
}
__device__ __forceinline__ float quad_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

}  // namespace mma
}  // namespace laser
