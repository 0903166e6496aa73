// Primitives of the summary builder's main route: packed fp32 arithmetic, ldmatrix, mma.sync, split operands.
#pragma once

#include "build_common.cuh"

namespace cobs {
namespace {

using u64 = unsigned long long;                       // two packed floats

__device__ __forceinline__ u64 pk(float lo, float hi) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float lo(u64 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi(u64 v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float rcp(float x) {       // to one unit in the last place; 0 beyond 2^126
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
struct __align__(16) U64x2 { u64 a, b; };
__device__ __forceinline__ U64x2 ld4(const float *p) { return *reinterpret_cast<const U64x2 *>(p); }

__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16_zero(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {      // c = a b
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};\n"
               : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void add4(float (&c)[4], const float (&t)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) c[i] += t[i];
}
// c += (h + l) (bh + bl) but for l bl.  The tensor core cuts what it adds to an accumulator where an addition rounds: the three
// products start from zero, the small ones first, and their sum is added.  (All in c, the largest first: the Gram matrix of
// a subspace descriptor was off by 1.2 times what the same sums by fused multiply-adds are, this way by as much; with the
// projection's sums taken the same way, 16 384 blocks of 64: 1.35 -> 1.38 ms.)
template <bool ZERO = false>                          // (c = instead of c +=)
__device__ __forceinline__ void mma_split(float (&c)[4], const uint32_t (&h)[4], const uint32_t (&l)[4], uint32_t bh0, uint32_t bh1, uint32_t bl0, uint32_t bl1) {
  float t[4] = {0.f, 0.f, 0.f, 0.f};
  mma_f16(t, h[0], h[1], h[2], h[3], bl0, bl1);
  mma_f16(t, l[0], l[1], l[2], l[3], bh0, bh1);
  mma_f16(t, h[0], h[1], h[2], h[3], bh0, bh1);
  if constexpr (ZERO) {
#pragma unroll
    for (int i = 0; i < 4; ++i) c[i] = t[i];
  } else {
    add4(c, t);
  }
}
// The same all in c, the small products first: for iterates, which the next one corrects.
__device__ __forceinline__ void mma_chain(float (&c)[4], const uint32_t (&h)[4], const uint32_t (&l)[4], uint32_t bh0, uint32_t bh1, uint32_t bl0, uint32_t bl1) {
  mma_f16(c, h[0], h[1], h[2], h[3], bl0, bl1);
  mma_f16(c, l[0], l[1], l[2], l[3], bh0, bh1);
  mma_f16(c, h[0], h[1], h[2], h[3], bh0, bh1);
}
__device__ __forceinline__ void cpa16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src));
}
// x, y -> f16x2 high parts and f16x2 remainders: 22 bits of each value together
__device__ __forceinline__ void split_f16(float x, float y, uint32_t &h, uint32_t &l) {
  const __half2 hh = __floats2half2_rn(x, y);
  const float2 hf = __half22float2(hh);
  const __half2 ll = __floats2half2_rn(x - hf.x, y - hf.y);
  h = *reinterpret_cast<const uint32_t *>(&hh);
  l = *reinterpret_cast<const uint32_t *>(&ll);
}

}  // namespace
}  // namespace cobs
