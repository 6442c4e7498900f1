// Fixed-point digits for exact products on the FP16 tensor cores (the scheme
// is described in fx_gemm.cu): 63-bit numbers as eight balanced base-256
// digits, FP32 accumulators started at 1.5 * 2^23 so that their bit patterns
// are the integer sums.
#pragma once

#include <cstdint>

#include "common.cuh"

namespace pdep {

constexpr int FX_S = 8;                     // digits per operand
constexpr uint32_t FX_MAGIC = 0x4B400000u;  // bits of 1.5 * 2^23

__device__ __forceinline__ int exp_of(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// x as a 63-bit fixed-point number scaled by its row's exponent field er
// (>= 1 and >= that of x): x = v 2^(er - 1084)
__device__ __forceinline__ long long fx_of(double x, int er) {
  const int hi = __double2hiint(x);
  const int e = (hi >> 20) & 0x7ff;
  unsigned long long m =
      ((unsigned long long)(unsigned)((hi & 0xfffff) | (e ? 0x100000 : 0)) << 32) |
      (unsigned)__double2loint(x);
  const int sh = er - (e > 1 ? e : 1);
  m = (unsigned)sh < 64u ? (m << 9) >> sh : 0ull;
  return hi < 0 ? -(long long)m : (long long)m;
}

// digit s (0 = most significant) of two biased fixed-point numbers as a pair
// of FP16 integers: the bytes go into the mantissas of 1024 + byte, then
// 1024 + 128 is subtracted (all exact)
__device__ __forceinline__ uint32_t digit_pair(uint2 u0, uint2 u1, int s) {
  const uint32_t w0 = s < 4 ? u0.y : u0.x, w1 = s < 4 ? u1.y : u1.x;
  const int j = 3 - (s & 3);
  uint32_t p = __byte_perm(w0, w1, (uint32_t)(j | (4 + j) << 8));
  p = (p & 0x00ff00ffu) | 0x64006400u;
  uint32_t r;
  asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(p), "r"(0xE480E480u));
  return r;
}
__device__ __forceinline__ uint2 biased(long long v) {
  const unsigned long long u = (unsigned long long)v + 0x8080808080808080ull;
  return make_uint2((uint32_t)u, (uint32_t)(u >> 32));
}

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                        uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}


// d = a b + c
__device__ __forceinline__ void mma_f16_from(float (&d)[4], const float (&c)[4],
                                             const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%10,%11,%12,%13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]),
        "f"(c[2]), "f"(c[3]));
}
__device__ __forceinline__ void mma_f16_k8_from(float (&d)[4], const float (&c)[4], uint32_t a0,
                                                uint32_t a1, uint32_t b0) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, "
      "{%7,%8,%9,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(b0), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}
// m16n8k8: two registers of A (rows g and g + 8), one of B
__device__ __forceinline__ void mma_f16_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(b0));
}

}  // namespace pdep
