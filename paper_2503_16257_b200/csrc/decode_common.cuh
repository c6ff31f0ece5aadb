// Device helpers shared by the decode attention kernels (decode_block.cu, decode_prep.cu,
// decode_stream.cu, decode.cu):
// mma.sync wrappers, the logic / multiply-add forms of the code expansion, and the query
// normalisation.
#pragma once

#include "common.cuh"
#include "kernels.cuh"

namespace vidkv {
namespace {

__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// d = a b + c with c given separately (no copy into the accumulator beforehand)
__device__ __forceinline__ void mma_f16_c(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1, float c0, float c1, float c2, float c3) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// q . k with the operands in the cache's element type (rows 8-15 of A unused)
template <typename T> __device__ __forceinline__ void mma_in(float (&d)[4], uint32_t a0, uint32_t a2, uint32_t b0, uint32_t b1);
template <> __device__ __forceinline__ void mma_in<__half>(float (&d)[4], uint32_t a0, uint32_t a2, uint32_t b0, uint32_t b1) {
  mma_f16(d, a0, 0u, a2, 0u, b0, b1);
}
template <> __device__ __forceinline__ void mma_in<__nv_bfloat16>(float (&d)[4], uint32_t a0, uint32_t a2, uint32_t b0,
                                                                  uint32_t b1) {
  mma_bf16(d, a0, 0u, a2, 0u, b0, b1);
}

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ uint32_t mad_u32(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// Code expansion as one three-input logic instruction.  The masks are immediates: only two registers are read, and
// register reads are what other instructions compete for with mma.sync (measured beside eight products: 64 logic
// instructions with three register operands take 152 clocks, with two 140; a decode step of 28 x 16 x 12544 tokens
// 1.4 % less).
// The two-bit field at mantissa bits 8-9 of each binary16 lane of x, joined with the bits of c.
__device__ __forceinline__ uint32_t field_or(uint32_t x, uint32_t c) {
  uint32_t d;
  asm("lop3.b32 %0, %1, 0x03000300, %2, 0xEA;" : "=r"(d) : "r"(x), "r"(c));
  return d;
}
constexpr uint32_t kFour = 0x44004400u;   // binary16 pair (4.0, 4.0)

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}

// 2^k as a float, |k| <= 126
__device__ __forceinline__ float pow2i(int k) { return __uint_as_float(static_cast<uint32_t>(127 + k) << 23); }

// Query normalisation.  The query goes to the tensor cores as binary16, its transform as a leading part and a remainder.  Every query
// head is therefore multiplied by the power of two 2^(-e - kQShift), e = floor(log2(max_c |q_c|)), which puts its largest entry into
// [1/8, 1/4) and its largest spectrum coefficient below 4 (at most 16 times the largest entry), well inside the binary16 range.  Scores
// are linear in q, so the softmax multiplies by the
// inverse power of two; both factors are exact.  head_exponent returns e (0 for a head that is all
// zero or holds no finite maximum); the NSUB lanes sub = 0..NSUB-1 share the 128 entries of the row,
// and all 32 lanes of the warp must call it.
constexpr int kQShift = 3;
template <typename T, int NSUB>
__device__ __forceinline__ int head_exponent(const T* qrow, int sub, bool live) {
  float m = 0.0f;
  if (live) {
    const uint2* p = reinterpret_cast<const uint2*>(qrow + sub * (kD / NSUB));
#pragma unroll
    for (int i = 0; i < kD / NSUB / 4; ++i) {
      const uint2 v = p[i];
      const float2 a = Elem<T>::to_float2(v.x), b = Elem<T>::to_float2(v.y);
      m = fmaxf(m, fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(b.x), fabsf(b.y))));
    }
  }
#pragma unroll
  for (int o = NSUB / 2; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (!(m > 0.0f) || m > 3.0e38f) return 0;
  const int e = static_cast<int>(__float_as_uint(m) >> 23) - 127;
  return max(-100, min(100, e));
}


}  // namespace
}  // namespace vidkv
