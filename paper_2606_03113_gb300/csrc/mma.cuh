// mma.cuh -- warp-level tensor-core helpers of the attention kernels:
// swizzled shared-memory rows, cp.async, ldmatrix, mma.sync and the split of
// an fp32 operand into three bf16 parts.
#pragma once

#include "pipe.cuh"

namespace ssd {

// Byte offset of 16-byte chunk c of row `row` (256- or 128-byte rows; the
// chunk's place is swizzled by row % 8, so eight rows' chunks c lie on
// distinct banks).
__device__ __forceinline__ uint32_t sw256(int row, int c) {
  return (uint32_t)(row * 256 + ((c ^ (row & 7)) << 4));
}
__device__ __forceinline__ uint32_t sw128(int row, int c) {
  return (uint32_t)(row * 128 + ((c ^ (row & 7)) << 4));
}
// 16 bytes from src, or zeros.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// (x, y) as packed bf16 pairs of high and low parts: 16 bits of each.
__device__ __forceinline__ void split2(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  const __nv_bfloat162 l = __floats2bfloat162_rn(x - __uint_as_float(hi << 16),
                                                 y - __uint_as_float(hi & 0xffff0000u));
  lo = *reinterpret_cast<const uint32_t*>(&l);
}
// (x, y) as three packed bf16 pairs whose sum keeps 24 bits of each.
__device__ __forceinline__ void split3(float x, float y, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
  auto pack = [](float u, float w) -> uint32_t {
    const __nv_bfloat162 b = __floats2bfloat162_rn(u, w);
    return *reinterpret_cast<const uint32_t*>(&b);
  };
  auto lo = [](uint32_t p) { return __uint_as_float(p << 16); };
  auto hi = [](uint32_t p) { return __uint_as_float(p & 0xffff0000u); };
  p0 = pack(x, y);
  const float x1 = x - lo(p0), y1 = y - hi(p0);
  p1 = pack(x1, y1);
  p2 = pack(x1 - lo(p1), y1 - hi(p1));
}

}  // namespace ssd
