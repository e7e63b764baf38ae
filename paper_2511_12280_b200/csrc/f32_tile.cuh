// Building blocks of the CUDA-core (fp32 arithmetic) matrix kernels: a 16 x 32 register tile per warp over K-major
// operands in shared memory, and 16-byte asynchronous copies into rows padded by 16 bytes.
//
// Lane layout of a warp tile: ty (0..3) owns rows ty + 4 r, tx (0..7) owns columns tx + 8 j (r, j = 0..3), the bits of ty
// and tx interleaved over the lane number.  A vector read then finds equal addresses in lanes that differ in bit 0 (first
// operand) or bit 1 (second operand), and takes 2 passes over the banks instead of 4: with ty = lane / 8 the second
// operand took 4, and a 1152 x 6144 x 2048 product ran at 32 TFLOP/s instead of 35.
// Both operands are read as 16-byte vectors along K from rows whose length is a multiple of 4 floats plus 4: the eight
// rows (or four rows, for the first operand) that a warp touches then start in different bank groups, so a vector read
// costs one pass over the banks.  Per 4 of K a lane reads 8 vectors for 32 packed multiply-adds (fma.f32x2 along K).
#pragma once

#include "common.cuh"

namespace f32 {

__device__ __forceinline__ int lane_ty(int lane) { return ((lane >> 1) & 1) | ((lane >> 2) & 2); }
__device__ __forceinline__ int lane_tx(int lane) { return (lane & 1) | ((lane >> 1) & 2) | ((lane >> 2) & 4); }
// over the eight lanes of one ty, partners tx ^ 4, tx ^ 2, tx ^ 1 in this order
__device__ __forceinline__ float max_over_tx(float v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 2) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, d));
  return v;
}
__device__ __forceinline__ float sum_over_tx(float v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 2) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc, bool in_bounds) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
  const int bytes = in_bounds ? 16 : 0;              // 0: the 16 bytes are filled with zeros, the source is not read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(gsrc), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// One vector of four elements, columns [c, c + 4) of a row that has `cols` of them, into four floats of shared memory.
// `vec`: every such vector is 16-byte aligned and lies wholly inside or outside the row (fp32 only).
template <typename T>
__device__ __forceinline__ void load4(float* dst, const T* row, int c, int cols, bool row_ok, bool vec) {
  if (sizeof(T) == 4 && vec) {
    const bool in = row_ok && c < cols;
    cp_async16(dst, row + c, in);
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) dst[e] = (row_ok && c + e < cols) ? Storage<T>::to_float(row[c + e]) : 0.f;
  }
}

// acc[r][j] += a[ty + 4 r][k] * b[tx + 8 j][k] over K4 vectors of four (even and odd k in the two halves of the pair).
// The vectors of the next step are read while this step's are multiplied, and consecutive multiply-adds go to different
// accumulators: with one or two warps per scheduler it is latency that would show otherwise.
template <int LDA, int LDB, int K4>
__device__ __forceinline__ void dot_16x32(float2 (&acc)[4][4], const float* a, const float* b, int ty, int tx) {
  const float* ar = a + ty * LDA;
  const float* br = b + tx * LDB;
  static_assert(K4 % 2 == 0, "two steps per turn");
  float4 av[2][4], bv[2][4];
  auto fetch = [&](int buf, int k) {
#pragma unroll
    for (int r = 0; r < 4; ++r) av[buf][r] = *reinterpret_cast<const float4*>(ar + r * 4 * LDA + k * 4);
#pragma unroll
    for (int j = 0; j < 4; ++j) bv[buf][j] = *reinterpret_cast<const float4*>(br + j * 8 * LDB + k * 4);
  };
  auto multiply = [&](int buf) {
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        acc[r][j] = __ffma2_rn(make_float2(av[buf][r].x, av[buf][r].y), make_float2(bv[buf][j].x, bv[buf][j].y), acc[r][j]);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        acc[r][j] = __ffma2_rn(make_float2(av[buf][r].z, av[buf][r].w), make_float2(bv[buf][j].z, bv[buf][j].w), acc[r][j]);
  };
  fetch(0, 0);
#pragma unroll 4
  for (int k = 0; k < K4; k += 2) {
    fetch(1, k + 1);
    multiply(0);
    if (k + 2 < K4) fetch(0, k + 2);
    multiply(1);
  }
}

}  // namespace f32
