// Building blocks of the CUDA-core (fp32 arithmetic) matrix kernels: a 16 x 32 register tile per warp over K-major
// operands in shared memory, and 16-byte asynchronous copies into rows padded by 16 bytes.
//
// Lane layout of a warp tile: ty (0..3) owns rows ty + 4 r, tx (0..7) owns columns tx + 8 j (r, j = 0..3), the bits of ty
// and tx interleaved over the lane number, so that equal addresses lie in lanes that differ in bit 0 (first operand) or
// bit 1 (second operand).  Both operands are read as 16-byte vectors along K from rows whose length is a multiple of 4
// floats plus 4: the eight rows (or four rows, for the first operand) that a warp touches start in different bank groups.
// A vector read then takes 2 passes over the banks without conflicts (counted: 1.93 wavefronts per read); with
// ty = lane / 8 the second operand took 4, and a 1152 x 6144 x 2048 product ran at 32 TFLOP/s instead of 35.
// Per 4 of K a lane reads 8 vectors for 32 packed multiply-adds (fma.f32x2 along K).
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

// Four elements, columns [c, c + 4) of a row that has `cols` of them, as floats (zeros outside).  `vec`: vectors of four are
// aligned to their own size and lie wholly inside or outside the row.
template <typename T>
__device__ __forceinline__ float4 fetch4(const T* row, int c, int cols, bool row_ok, bool vec) {
  float v[4] = {0.f, 0.f, 0.f, 0.f};
  if (sizeof(T) == 2 && vec) {           // (fp32 vectors of four come by asynchronous copy)
    if (row_ok && c < cols) {
      const uint2 w = *reinterpret_cast<const uint2*>(row + c);
      v[0] = __uint_as_float(w.x << 16); v[1] = __uint_as_float(w.x & 0xffff0000u);
      v[2] = __uint_as_float(w.y << 16); v[3] = __uint_as_float(w.y & 0xffff0000u);
    }
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) if (row_ok && c + e < cols) v[e] = Storage<T>::to_float(row[c + e]);
  }
  return make_float4(v[0], v[1], v[2], v[3]);
}

// The vectors at column c of N rows, row(u) = {pointer, whether the row exists}, to dst + u * dst_step in shared memory: by
// asynchronous copies where the source allows it (fp32 and `vec`), otherwise through registers, four vectors requested
// before the first is stored (a store to shared memory in between holds the next load back: fp32 linear 33 x 130 x 65 with
// load and store in turn 10.0 us, now 5.2).
template <typename T, int N, typename RowFn>
__device__ __forceinline__ void load_vecs(float* dst, int dst_step, RowFn row, int c, int cols, bool vec) {
  if (sizeof(T) == 4 && vec) {
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const auto r = row(u);
      cp_async16(dst + u * dst_step, r.p + c, r.ok && c < cols);
    }
  } else {
    constexpr int kBatch = 4;
#pragma unroll
    for (int u0 = 0; u0 < N; u0 += kBatch) {
      float4 v[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        if (u0 + u >= N) continue;
        const auto r = row(u0 + u);
        v[u] = fetch4<T>(r.p, c, cols, r.ok, vec);
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) if (u0 + u < N) *reinterpret_cast<float4*>(dst + (u0 + u) * dst_step) = v[u];
    }
  }
}
template <typename T> struct RowRef { const T* p; bool ok; };

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
