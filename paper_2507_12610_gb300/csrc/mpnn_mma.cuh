// Tensor-core helpers of the surrogate's kernels: bf16 m16n8k16 products with
// fp32 accumulation, fragments loaded from shared memory by ldmatrix,
// asynchronous 16-byte copies into shared memory.
//
// Tiles in shared memory keep their rows a whole number of 16-byte pieces
// apart, an odd number modulo 8, so that the eight rows of an ldmatrix fall in
// different banks.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/dem.h"

namespace mpnn {

constexpr int kSms = 152;
constexpr int kH = 128;            // the network's width
constexpr uint32_t kRowH = 272;    // bytes of a staged row of 128 bf16 (17 pieces)
constexpr uint32_t kRow64 = 144;   // ... of 64 bf16 (9 pieces)
constexpr uint32_t kRow16 = 48;    // ... of 16 bf16 (3 pieces)

inline int launch_status() {
  return cudaGetLastError() == cudaSuccess ? DEM_OK : DEM_ERR_CUDA;
}

template <typename... P>
bool aligned16(const P*... p) {
  uintptr_t bits = 0;
  ((bits |= reinterpret_cast<uintptr_t>(p)), ...);
  return (bits & 15u) == 0;
}

// A barrier of one of a block's groups of warps.
constexpr int kGroupThreads = 256;
__device__ __forceinline__ void group_sync(int group) {
  asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(kGroupThreads) : "memory");
}

__device__ __forceinline__ uint16_t to_bf16(float x) {
  const __nv_bfloat16 b = __float2bfloat16_rn(x);
  return *reinterpret_cast<const uint16_t*>(&b);
}

// two values to a pair of bf16, the first in the low half
__device__ __forceinline__ uint32_t pack_bf16(float x, float y) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<const uint32_t*>(&b);
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

// 16 bytes from global to shared memory (zeros if !valid)
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool valid = true) {
  const int bytes = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
               "r"(bytes));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

// A lane's offset (bytes) into a 16 x 16 A tile with rows of `row` bytes, for
// ldsm4: the four 8 x 8 parts in the order of the A fragment.
__device__ __forceinline__ uint32_t a_lane(int lane, uint32_t row) {
  return (uint32_t)((lane & 7) + 8 * ((lane >> 3) & 1)) * row + 16u * (uint32_t)(lane >> 4);
}
// The same for 16 columns of B held as rows of k (B fragments of two n-tiles).
__device__ __forceinline__ uint32_t b_lane(int lane, uint32_t row) {
  return (uint32_t)((lane & 7) + 8 * (lane >> 4)) * row + 16u * (uint32_t)((lane >> 3) & 1);
}

// acc += A (32 rows) B (32 columns) over NCH chunks of 16 in ascending k.
// a, b: shared addresses of the warp's first row / column at the first chunk,
// lane offsets included.
template <int NCH>
__device__ __forceinline__ void mma_chain(float (&acc)[2][4][4], uint32_t a, uint32_t a_row,
                                          uint32_t b, uint32_t b_row) {
#pragma unroll
  for (int ch = 0; ch < NCH; ++ch) {
    uint32_t A[2][4], B[2][4];
    ldsm4(A[0], a + 32u * ch);
    ldsm4(A[1], a + 16u * a_row + 32u * ch);
    ldsm4(B[0], b + 32u * ch);
    ldsm4(B[1], b + 16u * b_row + 32u * ch);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        mma_bf16(acc[i][j], A[i][0], A[i][1], A[i][2], A[i][3], B[j >> 1][2 * (j & 1)],
                 B[j >> 1][2 * (j & 1) + 1]);
  }
}

// acc += [1, 0 x 15] B: the chunk of the constant column (rows with one[i][h]
// false contribute nothing; i: 16-row tile, h: its upper half).
__device__ __forceinline__ void mma_const(float (&acc)[2][4][4], const bool (&one)[2][2],
                                          uint32_t b, uint32_t b_row, int lane) {
  uint32_t B[2][4];
  ldsm4(B[0], b);
  ldsm4(B[1], b + 16u * b_row);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const uint32_t a0 = (lane & 3) == 0 && one[i][0] ? 0x3F80u : 0u;
    const uint32_t a1 = (lane & 3) == 0 && one[i][1] ? 0x3F80u : 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      mma_bf16(acc[i][j], a0, a1, 0u, 0u, B[j >> 1][2 * (j & 1)], B[j >> 1][2 * (j & 1) + 1]);
  }
}

__device__ __forceinline__ void zero(float (&acc)[2][4][4]) {
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.f;
}

// relu(v + 0): the epilogue of a layer whose bias is a column of its input
__device__ __forceinline__ float relu0(float v) { return fmaxf(v + 0.f, 0.f); }

}  // namespace mpnn
