// Device helpers of the quantizers: 16-bit element operations and the exact decision of Eq. 4 codes
// without a division per element.
#pragma once

#include "common.cuh"

namespace vidkv {
namespace {

__device__ __forceinline__ __half2 as_h2(uint32_t v) { return *reinterpret_cast<const __half2*>(&v); }
__device__ __forceinline__ __nv_bfloat162 as_bf2(uint32_t v) { return *reinterpret_cast<const __nv_bfloat162*>(&v); }
__device__ __forceinline__ uint32_t as_u32(__nv_bfloat162 v) { return *reinterpret_cast<const uint32_t*>(&v); }
__device__ __forceinline__ uint32_t as_u32(__half2 v) { return *reinterpret_cast<const uint32_t*>(&v); }

// Element-type helpers: raw 16-bit patterns in, binary16 1.0 / 0.0 pairs out of the comparison.
template <typename T> struct Ops;
template <> struct Ops<__half> {
  static __device__ __forceinline__ float to_float(uint16_t b) { return __half2float(__ushort_as_half(b)); }
  static __device__ __forceinline__ uint16_t from_float_rn(float f) { return __half_as_ushort(__float2half_rn(f)); }
  static __device__ __forceinline__ uint32_t ge(uint32_t a, uint32_t b) { return as_u32(__hge2(as_h2(a), as_h2(b))); }
  // 0xffff per lane where a >= b
  static __device__ __forceinline__ uint32_t ge_mask(uint32_t a, uint32_t b) { return __hge2_mask(as_h2(a), as_h2(b)); }
  static __device__ __forceinline__ uint32_t min2(uint32_t a, uint32_t b) { return as_u32(__hmin2(as_h2(a), as_h2(b))); }
  static __device__ __forceinline__ uint32_t max2(uint32_t a, uint32_t b) { return as_u32(__hmax2(as_h2(a), as_h2(b))); }
  static constexpr uint16_t kInf = 0x7c00u;
};
template <> struct Ops<__nv_bfloat16> {
  static __device__ __forceinline__ float to_float(uint16_t b) { return __uint_as_float(static_cast<uint32_t>(b) << 16); }
  static __device__ __forceinline__ uint16_t from_float_rn(float f) { return __bfloat16_as_ushort(__float2bfloat16_rn(f)); }
  static __device__ __forceinline__ uint32_t ge(uint32_t a, uint32_t b) {
    const __nv_bfloat162 r = __hge2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
    return *reinterpret_cast<const uint32_t*>(&r) & 0x3c003c00u;   // bfloat16 1.0 -> binary16 1.0
  }
  static __device__ __forceinline__ uint32_t ge_mask(uint32_t a, uint32_t b) { return __hge2_mask(as_bf2(a), as_bf2(b)); }
  static __device__ __forceinline__ uint32_t min2(uint32_t a, uint32_t b) { return as_u32(__hmin2(as_bf2(a), as_bf2(b))); }
  static __device__ __forceinline__ uint32_t max2(uint32_t a, uint32_t b) { return as_u32(__hmax2(as_bf2(a), as_bf2(b))); }
  static constexpr uint16_t kInf = 0x7f80u;
};

// Value order of 16-bit sign-magnitude patterns as integers (both zeros map to 0).
__device__ __forceinline__ int ord_of(uint16_t b) { return (b & 0x8000u) ? -static_cast<int>(b & 0x7fffu) : static_cast<int>(b); }
__device__ __forceinline__ uint16_t bits_of(int o) { return o >= 0 ? static_cast<uint16_t>(o) : static_cast<uint16_t>(0x8000u | static_cast<uint32_t>(-o)); }

// Eq. 4 for one element: is clamp(rint(RN(RN(x - z) / s)), 0, 3) >= k for the element with value
// order o (k = 1..3, s > 0)?  Decided without the division.  rint(q) >= k holds from q = 0.5 + 2^-24,
// 1.5 and 2.5 + 2^-22 on (round half to even), and the rounded quotient reaches that float exactly
// when the real quotient passes the midpoint below it: d / s > 0.5 + 2^-25, >= 1.5 - 2^-24,
// > 2.5 + 2^-23 (ties go to the even neighbour 0.5, 1.5, 2.5).  With c = k - 0.5 the sign of
// d - (c + delta) s is that of u - delta s, u = fma(-c, s, d): c s is exact, u is exact whenever
// d is within a factor two of c s (the only case where delta matters), delta s is a power of two times s.
template <typename T>
__device__ __forceinline__ bool code_at_least(int o, float z, float s, int k) {
  const float d = __fsub_rn(Ops<T>::to_float(bits_of(o)), z);
  const float u = fmaf(0.5f - static_cast<float>(k), s, d);
  if (k == 1) return u > 0x1p-25f * s;
  if (k == 2) return u >= -0x1p-24f * s;
  return u > 0x1p-23f * s;
}

// Bit pattern of the smallest element value whose Eq. 4 code with (s, z) is at least k; infinity where s is 0
// (every code is 0).
//
// e = the element nearest to c = z + (k - 1/2) s.  Unless c is much smaller than |z| + 3 s, the elements next to e are
// half a step of the element type from c at least, 2^-12 |c| >= 2^-22 (|z| + 3 s): more than the roundings of c and of
// code_at_least's difference and its midpoint offset together (2^-23 (|z| + 3 s)), so the element below e does not reach
// the code and the one above does, and one evaluation decides (branch-free; the search it replaces took 40 % of the
// encoder's epilogue in divergent branches).  Otherwise the threshold is searched from e.
template <typename T>
__device__ __forceinline__ uint16_t code_cut(float z, float s, int k) {
  const float c = fmaf(static_cast<float>(k) - 0.5f, s, z);
  const uint16_t e = Ops<T>::from_float_rn(c);
  const float u = fmaf(0.5f - static_cast<float>(k), s, __fsub_rn(Ops<T>::to_float(e), z));
  const bool reached = k == 1 ? u > 0x1p-25f * s : k == 2 ? u >= -0x1p-24f * s : u > 0x1p-23f * s;
  uint16_t X = reached ? e : static_cast<uint16_t>(e + ((e & 0x8000u) ? 0xffffu : 1u));
  const bool unsafe = fabsf(c) < 0x1p-10f * fmaf(3.0f, s, fabsf(z));
  if (s == 0.0f) X = Ops<T>::kInf;
  if (unsafe && s != 0.0f) {
    int o = ord_of(e);
    if (code_at_least<T>(o, z, s, k)) {
#pragma unroll 1
      for (int it = 0; it < 6 && code_at_least<T>(o - 1, z, s, k); ++it) --o;
    } else {
      ++o;
#pragma unroll 1
      for (int it = 0; it < 5 && !code_at_least<T>(o, z, s, k); ++it) ++o;
    }
    X = bits_of(o);
  }
  return X;
}

}  // namespace
}  // namespace vidkv
