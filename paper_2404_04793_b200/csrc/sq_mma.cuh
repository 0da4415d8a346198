// Shared by the grouped-head decode kernels: mma.sync / ldmatrix / cp.async wrappers, the layout of their
// shared-memory tiles (rows of D bf16 elements, 16-byte chunks XOR-swizzled by the row so that ldmatrix is
// free of bank conflicts) and the plan of H2O launches with the score update.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace sq {

constexpr int kTile = 64;  // tokens per pipeline stage
constexpr int kScoresSmem = 110 * 1024;  // dynamic shared memory of a CTA with the score update: two CTAs per SM
constexpr int kMaxPieces = 16;           // CTAs of a cluster (above 8: opt-in)
// tiles of a piece when a unit of `len` slots is cut into `pieces`
__host__ __device__ inline int piece_tiles(int len, int pieces) {
  return ((len + kTile - 1) / kTile + pieces - 1) / pieces;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
  const int sz = valid ? 16 : 0;  // 0: the 16 bytes are zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(sz));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N));
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2,
                                                  uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// two floats -> packed bf16x2 (lo in the low half), and the values the packing kept
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi, float& lo_r, float& hi_r) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  uint32_t u = *reinterpret_cast<uint32_t*>(&v);
  lo_r = __uint_as_float(u << 16);
  hi_r = __uint_as_float(u & 0xffff0000u);
  return u;
}

template <int D>
__device__ __forceinline__ uint32_t swz(int row, int chunk) {
  // byte offset of 16-byte chunk `chunk` of row `row` inside a [rows][D] bf16 tile
  return (uint32_t)(row * (D * 2) + ((chunk ^ (row & 7)) << 4));
}

// transposes the 8 x 8 matrix of 16-bit elements that a warp holds as ldmatrix leaves it
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}
}  // namespace sq
