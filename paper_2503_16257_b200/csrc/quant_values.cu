// Value quantizer kernels: Algorithm 2 of the paper (1.58Quant, STPQuant), the token
// selection of Sec. 3.3(2), and the residual copies of Algorithm 1.
#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.cuh"
#include "quant_common.cuh"

namespace vidkv {

namespace cg = cooperative_groups;

__device__ __forceinline__ __half2 as_half2(uint32_t v) { return *reinterpret_cast<const __half2*>(&v); }

// ---------------------------------------------------------------------------------
// 1.58Quant (Eq. 6) of one supergroup = 5 groups x 32 stream tokens x 128 channels by a block of 320 threads.
// Stream position u of the unprotected tokens maps to token idx_rest[u] (identity when
// no token is protected).
//   stage   the 160 x 128 tile is copied to shared memory as it is (cp.async, 16 bytes a piece);
//   pass 1  s = Mean |v| per (group, channel), float32, and the threshold: thread = (group, channel pair), so nothing
//           has to meet in shared memory but the threshold;
//   pass 2  thread = two 32-bit words of the byte plane = (token pair, four channels):
//           the comparisons |v| > alpha run on two channels at a time against the smallest
//           representable number above alpha = gamma * s, the five digits of a byte are
//           summed in binary16 (exact, 1024 to 1266), and the byte code is the top byte of one multiply-add.
// What bounds it is instructions (7396 a block; SM throughput 72 %) beside the copies' latency, which the blocks that
// share a multiprocessor cover: five of them (45 KB, 32 registers; a list of token positions costs a second latency).  With 256 threads, partial sums in shared memory, a table of byte codes and four
// blocks, 64 slabs of 12544 tokens took 55.2 us and 73.1 with a fifth of the tokens protected; now 44.1 (205 MB in and
// 53 out, 5.9 TB/s) and 55.1.  The 64-bit pass 2 alone gave 51.8 and 72.0, five blocks 46.3 and 56.6, digits with their weights in one
// multiply-add a comparison and no division for full groups the rest.
// ---------------------------------------------------------------------------------
constexpr int kSGTokens = kSGGroups * kG;   // 160
constexpr int kVThreads = kSGGroups * kD / 2;  // 320: a channel pair of a group each
constexpr int kVRowBytes = 272;             // 256 bytes of data + padding: rows four apart land 16 banks apart

template <typename T> struct Simd2;
template <> struct Simd2<__half> {
  // 1.0 / 0.0 in binary16 per lane
  static __device__ __forceinline__ uint32_t ge(uint32_t a, uint32_t b) {
    const __half2 r = __hge2(*reinterpret_cast<const __half2*>(&a), *reinterpret_cast<const __half2*>(&b));
    return *reinterpret_cast<const uint32_t*>(&r);
  }
  static __device__ __forceinline__ uint32_t above_minus(uint32_t a, uint32_t b) {      // a > -b
    const __half2 r = __hgt2(*reinterpret_cast<const __half2*>(&a), __hneg2(*reinterpret_cast<const __half2*>(&b)));
    return *reinterpret_cast<const uint32_t*>(&r);
  }
  // smallest element value strictly above x >= 0
  static __device__ __forceinline__ uint16_t above(float x) {
    return static_cast<uint16_t>(__half_as_ushort(__float2half_rd(x)) + 1u);
  }
};
template <> struct Simd2<__nv_bfloat16> {
  // the comparison yields 1.0 in bfloat16 (0x3f80); keeping bits 10-13 turns it into binary16 1.0
  static __device__ __forceinline__ uint32_t ge(uint32_t a, uint32_t b) {
    const __nv_bfloat162 r = __hge2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
    return *reinterpret_cast<const uint32_t*>(&r) & 0x3c003c00u;
  }
  static __device__ __forceinline__ uint32_t above_minus(uint32_t a, uint32_t b) {
    const __nv_bfloat162 r = __hgt2(*reinterpret_cast<const __nv_bfloat162*>(&a), __hneg2(*reinterpret_cast<const __nv_bfloat162*>(&b)));
    return *reinterpret_cast<const uint32_t*>(&r) & 0x3c003c00u;
  }
  static __device__ __forceinline__ uint16_t above(float x) {
    return static_cast<uint16_t>(__bfloat16_as_ushort(__float2bfloat16_rd(x)) + 1u);
  }
};

__device__ __forceinline__ void cp_async16_v(void* smem_dst, const void* gmem_src) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}

// NZ: the stored scale is the mean of |v| over the non-zero codes instead of Mean |v| (one more
// sweep over the staged tile).
template <typename T, bool NZ>
__device__ __forceinline__ void ternary_supergroup(uint8_t* vsm, KSrc src, int64_t n_rest, CacheView cv, int layer0,
                                                   SelView sel, float gamma) {
  uint8_t* tile = vsm;                                                         // [160][kVRowBytes]
  uint32_t* thr = reinterpret_cast<uint32_t*>(tile + kSGTokens * kVRowBytes);  // [5][64] threshold pairs
  const int tid = threadIdx.x;
  const int slab = blockIdx.y;                              // over the layers of the call, then b, then h
  const int lb = slab / cv.H_kv, h = slab % cv.H_kv;
  const int b = lb % cv.B, layer = layer0 + lb / cv.B;
  const T* base = reinterpret_cast<const T*>(src.ptr) + static_cast<int64_t>(lb) * src.stride_b + h * src.stride_h;
  const int64_t u0 = static_cast<int64_t>(blockIdx.x) * kSGTokens;
  const int n_rows = static_cast<int>(min(static_cast<int64_t>(kSGTokens), n_rest - u0));
  const int32_t* idx = sel.idx_rest ? sel.idx_rest + b * sel.stride_rest : nullptr;
  // ---- stage (rows past the end of the stream are zero: their trits come out 0)
  {
    // thread = 16-byte piece (tid % 16) of rows tid / 16 + 20 k.  The stream positions of all its
    // rows are fetched first, so that the gather list costs one memory latency, not one per row.
    constexpr int kRowsPerThread = kSGTokens * 16 / kVThreads;
    const int row0 = tid >> 4, piece = tid & 15;
    int tok[kRowsPerThread];                                // positions fit 32 bits, as the index lists do
#pragma unroll
    for (int k = 0; k < kRowsPerThread; ++k) {
      const int row = row0 + kVThreads / 16 * k;
      tok[k] = row < n_rows ? (idx ? idx[u0 + row] : static_cast<int>(u0) + row) : -1;
    }
#pragma unroll
    for (int k = 0; k < kRowsPerThread; ++k) {
      uint8_t* dst = tile + (row0 + kVThreads / 16 * k) * kVRowBytes + piece * 16;
      if (tok[k] >= 0) cp_async16_v(dst, reinterpret_cast<const uint8_t*>(base + static_cast<int64_t>(tok[k]) * src.stride_t) + piece * 16);
      else *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  uint8_t* sg = cv.slab(layer, b, h) + cv.tern_offset + static_cast<int64_t>(blockIdx.x) * kSGBytes;
  // ---- pass 1: thread = (group, channel pair); the sum of 32 tokens is the sum of four sums of eight
  {
    const int g = tid >> 6, cp = tid & 63;
    const int n = max(0, min(kG, n_rows - g * kG));
    const uint8_t* rp = tile + g * (kG * kVRowBytes) + cp * 4;
    float sum[2] = {0.0f, 0.0f};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 f = Elem<T>::to_float2(*reinterpret_cast<const uint32_t*>(rp + (q * 8 + j) * kVRowBytes));
        a0 += fabsf(f.x); a1 += fabsf(f.y);
      }
      sum[0] = q ? sum[0] + a0 : a0;
      sum[1] = q ? sum[1] + a1 : a1;
    }
    uint32_t A = 0x00010001u;                          // empty group: every v is 0, nothing exceeds it
    if (n > 0) {
      // a full group's quotient by 32 is the product with 2^-5, to the bit
      const float m0 = n == kG ? sum[0] * (1.0f / kG) : __fdiv_rn(sum[0], static_cast<float>(n));
      const float m1 = n == kG ? sum[1] * (1.0f / kG) : __fdiv_rn(sum[1], static_cast<float>(n));
      const uint16_t s0 = f2h_bits(m0), s1 = f2h_bits(m1);
      if (!NZ) reinterpret_cast<uint32_t*>(sg + kSG_Scales)[tid] = s0 | static_cast<uint32_t>(s1) << 16;
      A = Simd2<T>::above(__fmul_rn(gamma, h2f(s0))) | static_cast<uint32_t>(Simd2<T>::above(__fmul_rn(gamma, h2f(s1)))) << 16;
    }
    thr[tid] = A;
    if (NZ && n > 0) {
      // ---- sums and counts of |v| over the elements whose code is not 0 (v >= A or v <= -A)
      const uint32_t one = 0x3c003c00u;
      float count[2] = {0.0f, 0.0f};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t w = *reinterpret_cast<const uint32_t*>(rp + (q * 8 + j) * kVRowBytes);
          const __half2 nz = __hsub2(__hadd2(as_half2(Simd2<T>::ge(w, A)), as_half2(one)), as_half2(Simd2<T>::above_minus(w, A)));
          const float2 m = __half22float2(nz), f = Elem<T>::to_float2(w);
          a0 = fmaf(m.x, fabsf(f.x), a0); a1 = fmaf(m.y, fabsf(f.y), a1);
          count[0] += m.x; count[1] += m.y;
        }
        sum[0] = q ? sum[0] + a0 : a0;
        sum[1] = q ? sum[1] + a1 : a1;
      }
      uint32_t sh = 0u;
#pragma unroll
      for (int j = 0; j < 2; ++j)
        if (count[j] > 0.0f) sh |= static_cast<uint32_t>(f2h_bits(__fdiv_rn(sum[j], count[j]))) << (16 * j);
      reinterpret_cast<uint32_t*>(sg + kSG_Scales)[tid] = sh;
    }
  }
  __syncthreads();
  // ---- pass 2: two words of the plane (four channels) per thread and step
#pragma unroll 1
  for (int i = tid; i < kG * kD / 8; i += kVThreads) {
    // bits 3 and 4 of the pair's index trade places: a half warp then reads 64 bytes of each of two rows that lie four rows
    // apart (conflict-free with the 272-byte row stride) and still writes whole 64-byte pieces of the plane
    const int pair = (i & ~0x18) | ((i & 0x08) << 1) | ((i & 0x10) >> 1);
    const int cp = 16 * ((pair >> 5) & 3) + 2 * (pair & 7);
    const int m = 4 * (pair >> 7) + ((pair >> 3) & 3);
    // binary16 pairs (even channel, odd channel) of tokens 2m, 2m+1; 1024 + b puts the integer b into the low mantissa bits
    uint32_t b0[2] = {0x64006400u, 0x64006400u}, b1[2] = {0x64006400u, 0x64006400u};
    constexpr uint32_t weights[kSGGroups] = {0x55105510u, 0x4ec04ec0u, 0x48804880u, 0x42004200u, 0x3c003c00u};   // 81, 27, 9, 3, 1
    const uint8_t* rp0 = tile + (2 * m) * kVRowBytes + cp * 4;
#pragma unroll
    for (int g = 0; g < kSGGroups; ++g) {
      const uint8_t* rp = rp0 + g * (kG * kVRowBytes);
      const uint2 t = *reinterpret_cast<const uint2*>(thr + g * 64 + cp);
      const uint32_t A[2] = {t.x, t.y};
      const uint2 r0 = *reinterpret_cast<const uint2*>(rp), r1 = *reinterpret_cast<const uint2*>(rp + kVRowBytes);
      const uint32_t v0[2] = {r0.x, r0.y}, v1[2] = {r1.x, r1.y};
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        // digit = [v > alpha] + [v >= -alpha] = [v >= A] + [v > -A]
        const __half2 w = as_half2(weights[g]);
        const __half2 t0 = __hfma2(as_half2(Simd2<T>::above_minus(v0[j], A[j])), w, __hfma2(as_half2(Simd2<T>::ge(v0[j], A[j])), w, as_half2(b0[j])));
        const __half2 t1 = __hfma2(as_half2(Simd2<T>::above_minus(v1[j], A[j])), w, __hfma2(as_half2(Simd2<T>::ge(v1[j], A[j])), w, as_half2(b1[j])));
        b0[j] = *reinterpret_cast<const uint32_t*>(&t0);
        b1[j] = *reinterpret_cast<const uint32_t*>(&t1);
      }
    }
    uint32_t word[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint32_t x0 = b0[j], x1 = b1[j];
      // word bytes: (even ch, tok 2m), (even ch, tok 2m+1), (odd ch, tok 2m), (odd ch, tok 2m+1)
      const uint32_t even = __byte_perm(trit_byte_top(x0 & 0xffu), trit_byte_top(x1 & 0xffu), 0x0073);
      const uint32_t odd = __byte_perm(trit_byte_top((x0 >> 16) & 0xffu), trit_byte_top((x1 >> 16) & 0xffu), 0x0073);
      word[j] = __byte_perm(even, odd, 0x5410);
    }
    reinterpret_cast<uint2*>(sg)[pair] = make_uint2(word[0], word[1]);
  }
}

// ---------------------------------------------------------------------------------
// 2-bit GQuant (Eq. 4) of groups of up to 32 protected tokens: 128 threads per group, two groups per block (its last two warps idle).
//
// code(v) = clamp(rint((v - z) / s), 0, 3) does not decrease with v, so it equals the number of
// k in {1, 2, 3} with v >= X_k, X_k the smallest value of the input type whose code reaches k (code_cut).
// The elements are compared with X_k two channels at a time; the comparisons' ones times 4^e, on top of 1024, put the
// fields of a code byte into the low bits of two binary16 lanes.  2508 protected and 10036 other tokens of 64 slabs took 78 us
// when it came in (55 now); three threshold searches with divisions per channel, conversions and float comparisons per element took 95.
// ---------------------------------------------------------------------------------
constexpr int kPRow = 144;                  // elements per staged row: rows two apart land 16 banks apart
constexpr int kProtectSmem = 2 * (kG * kPRow * 2 + 3 * kD * 2);

template <typename T>
__device__ __forceinline__ void protect_groups(uint8_t* vsm, const KSrc& src, int block, const CacheView& cv, int layer0, const SelView& sel) {
  const int half = threadIdx.x >> 7, tid = threadIdx.x & 127;                           // half 2: the block's last two warps, idle
  uint16_t* tile = reinterpret_cast<uint16_t*>(vsm) + half * kG * kPRow;                    // [32][kPRow]
  uint16_t* s_thr = reinterpret_cast<uint16_t*>(vsm + 2 * kG * kPRow * 2) + half * 3 * kD;     // [3][128]
  const int slab = blockIdx.y;
  const int lb = slab / cv.H_kv, h = slab % cv.H_kv;
  const int b = lb % cv.B, layer = layer0 + lb / cv.B;
  const T* base = reinterpret_cast<const T*>(src.ptr) + static_cast<int64_t>(lb) * src.stride_b + h * src.stride_h;
  const int64_t pgroup = 2 * static_cast<int64_t>(block) + half;
  const int64_t p0 = pgroup * kG;
  const int n_rows = half > 1 ? 0 : static_cast<int>(min(static_cast<int64_t>(kG), sel.n_prot - p0));   // <= 0: nothing left for this half
  const int32_t* idx = sel.idx_prot + b * sel.stride_prot;
  if (half <= 1) {
    const int lane16 = tid & 15, row = tid >> 4;
    int tok[kG / 8];
#pragma unroll
    for (int k = 0; k < kG / 8; ++k) tok[k] = row + 8 * k < n_rows ? idx[p0 + row + 8 * k] : -1;
    uint4 v[kG / 8];
#pragma unroll
    for (int k = 0; k < kG / 8; ++k) {
      v[k] = make_uint4(0, 0, 0, 0);
      if (tok[k] >= 0) v[k] = reinterpret_cast<const uint4*>(base + static_cast<int64_t>(tok[k]) * src.stride_t)[lane16];
    }
#pragma unroll
    for (int k = 0; k < kG / 8; ++k) reinterpret_cast<uint4*>(tile + (row + 8 * k) * kPRow)[lane16] = v[k];
  }
  __syncthreads();
  uint8_t* pg = cv.slab(layer, b, h) + cv.prot_offset + pgroup * kPGBytes;
  if (n_rows > 0) {
    const int c = tid;
    float mn = INFINITY, mx = -INFINITY;
#pragma unroll 8
    for (int j = 0; j < n_rows; ++j) {
      const float v = Elem<T>::to_float(reinterpret_cast<const T*>(tile)[j * kPRow + c]);
      mn = fminf(mn, v); mx = fmaxf(mx, v);
    }
    const uint16_t sh = f2h_bits(__fdiv_rn(__fsub_rn(mx, mn), 3.0f)), zh = f2h_bits(mn);
    reinterpret_cast<uint16_t*>(pg + kPG_S)[c] = sh;
    reinterpret_cast<uint16_t*>(pg + kPG_Z)[c] = zh;
    const float s = h2f(sh), z = h2f(zh);
#pragma unroll
    for (int k = 1; k <= 3; ++k) s_thr[(k - 1) * kD + c] = code_cut<T>(z, s, k);
  }
  __syncthreads();
  if (n_rows <= 0) return;
  for (int item = tid; item < kG * 8; item += 128) {
    // item = word index ((kt * 4 + w) * 4 + r) * 8 + rho: 4 channels x 4 tokens
    const int rho = item & 7, r = (item >> 3) & 3, w = (item >> 5) & 3, kt = item >> 7;
    const int c0 = 32 * w + 4 * rho;
    uint2 X[3];                                       // thresholds of channels c0 .. c0 + 3
#pragma unroll
    for (int k = 0; k < 3; ++k) X[k] = *reinterpret_cast<const uint2*>(s_thr + k * kD + c0);
    uint32_t word = 0;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int j = 16 * kt + 8 * u + 2 * r + hf;
        const uint2 v = *reinterpret_cast<const uint2*>(tile + j * kPRow + c0);
        // lanes: (c0, c0 + 1) with weights 1, 4, then (c0 + 2, c0 + 3) with 16, 64
        __half2 acc = as_h2(0x64006400u);
#pragma unroll
        for (int k = 0; k < 3; ++k) acc = __hfma2(as_h2(Ops<T>::ge(v.x, X[k].x)), as_h2(0x44003c00u), acc);
#pragma unroll
        for (int k = 0; k < 3; ++k) acc = __hfma2(as_h2(Ops<T>::ge(v.y, X[k].y)), as_h2(0x54004c00u), acc);
        const uint32_t a = as_u32(acc);
        const uint32_t byte = (a | (a >> 16)) & 0xffu;
        if (j < n_rows) word |= byte << (8 * u + 16 * hf);
      }
    }
    reinterpret_cast<uint32_t*>(pg)[item] = word;
  }
}

// ---------------------------------------------------------------------------------
// Algorithm 2 and the value half of Algorithm 1's residual in one launch.  grid = (supergroups of the ternary stream and
// pairs of protected groups, then one block for the n_res rows that stay as they are, if any; slabs of the call).  It lets
// the kernel behind it start only when it is done: with the next layer's range pass resident beside it four layers of 64 x
// 12544 tokens took 745 us, without 720.
// ---------------------------------------------------------------------------------
template <typename T, bool NZ>
__global__ void __launch_bounds__(kVThreads, 5) v_quantize_kernel(KSrc src, int64_t T_q, int64_t n_rest, int n_res, CacheView cv, int layer0, SelView sel,
                                                         float gamma, int ternary_blocks, int protect_blocks) {
  extern __shared__ __align__(16) uint8_t vsm[];
  pdl_wait();
  const uint32_t block = blockIdx.x;
  if (block >= static_cast<uint32_t>(ternary_blocks)) {
    const int pair = static_cast<int>(block) - ternary_blocks;
    if (pair < protect_blocks) protect_groups<T>(vsm, src, pair, cv, layer0, sel);
    else copy_residual_rows(src, T_q, n_res, cv, layer0, blockIdx.y, cv.vres_offset);
    return;
  }
  ternary_supergroup<T, NZ>(vsm, src, n_rest, cv, layer0, sel, gamma);
}

// ---------------------------------------------------------------------------------
// Residual flush, value half (Algorithm 1, Decoding): 1.58Quant of the 128 residual tokens
// of every slab, appended as 4 groups at ternary stream group index tgroup0.  The groups
// may land in a supergroup that already holds earlier groups, so bytes are updated digit
// by digit.  grid = slabs (over layers); block = 128 threads (thread = channel).
// ---------------------------------------------------------------------------------
template <typename T, bool NZ>
__global__ void __launch_bounds__(kD) v_flush_kernel(KSrc src, CacheView cv, int layer0, int slabs_per_layer,
                                                     int64_t tgroup0, float gamma) {
  const int slab = blockIdx.x;
  const int layer = layer0 + slab / slabs_per_layer;
  const int bh = slab % slabs_per_layer;
  const T* base = reinterpret_cast<const T*>(src.ptr) + (slab / src.H) * src.stride_b + (slab % src.H) * src.stride_h;
  uint8_t* tern = cv.slab(layer, bh / cv.H_kv, bh % cv.H_kv) + cv.tern_offset;
  const int c = threadIdx.x;
  const uint32_t p3[5] = {81u, 27u, 9u, 3u, 1u};
  for (int g4 = 0; g4 < kR / kG; ++g4) {
    const int64_t gi = tgroup0 + g4;
    uint8_t* sg = tern + (gi / kSGGroups) * kSGBytes;
    const int slot = static_cast<int>(gi % kSGGroups);
    float sum = 0.0f;
    for (int j = 0; j < kG; ++j) sum += fabsf(Elem<T>::to_float(base[(g4 * kG + j) * src.stride_t + c]));
    const uint16_t sh = f2h_bits(__fdiv_rn(sum, static_cast<float>(kG)));
    const float a = __fmul_rn(gamma, h2f(sh));
    float nz_sum = 0.0f, nz_cnt = 0.0f;
    for (int j = 0; j < kG; ++j) {
      const float v = Elem<T>::to_float(base[(g4 * kG + j) * src.stride_t + c]);
      const uint32_t d = v > a ? 2u : (v < -a ? 0u : 1u);
      if (NZ && d != 1u) { nz_sum += fabsf(v); nz_cnt += 1.0f; }
      const uint32_t bold = trit_byte_decode(sg[tern_byte_offset(j, c)]);
      const uint32_t dold = (bold / p3[slot]) % 3u;
      sg[tern_byte_offset(j, c)] = static_cast<uint8_t>(trit_byte_encode(bold - dold * p3[slot] + d * p3[slot]));
    }
    // the stored scale: Mean |v|, or the mean of |v| over the non-zero codes (0 where there is none)
    reinterpret_cast<uint16_t*>(sg + kSG_Scales)[slot * kD + c] =
        !NZ ? sh : (nz_cnt > 0.0f ? f2h_bits(__fdiv_rn(nz_sum, nz_cnt)) : static_cast<uint16_t>(0));
  }
}

// ---------------------------------------------------------------------------------
// Algorithm 1 for a prompt that is shorter than one group (longer ones leave it to the quantizing kernels).
// ---------------------------------------------------------------------------------
__global__ void copy_to_residual_kernel(KSrc src, int n_tok, CacheView cv, int layer0, int64_t res_offset) {
  copy_residual_rows(src, 0, n_tok, cv, layer0, blockIdx.x, res_offset);
}

// ---------------------------------------------------------------------------------
// Token selection: top n of l_v saliency scores per batch element (ties: lower index).
// One block of 1024 threads per batch element, or a cluster of kSelCluster of them where the row is long.
//   phase 1  radix select of the n-th largest key, 11 + 11 + 10 bits (11 bits of a float's pattern spread a smooth
//            distribution over some twenty bins where 8 bits have four, which the shared-memory atomics of a warp would
//            queue up on); the blocks of a cluster add their histograms up through distributed shared memory;
//   phase 2  E words, per-word prefix counts and the two gather lists.  With gt / eq the numbers of keys above / at the
//            threshold before a word, min(eq, need) + gt tokens are protected before it: one scan for both.  Token t is
//            lane t % 32 everywhere, so that scores, mask bytes and list entries move in whole lines.
// What bounds it is latency: 4 sweeps over scores that sit in L2, and a barrier after each.  4 x 196000 scores take 43
// us (298 with one block a row, 32 consecutive scores a thread and a serial walk over 256 bins), 6272 take 18 (39).
// ---------------------------------------------------------------------------------
constexpr int kSelThreads = 1024;
constexpr int kSelCluster = 8;                 // portable cluster size
// Up to 8 rows from 16384 tokens on get a cluster each.  us with one block / a cluster per row: 4 x 6272 18.8 / 20.4,
// 4 x 12544 22.7 / 22.8, 4 x 25088 28.7 / 24.7, 4 x 196000 142 / 43; 16 x 25088 28.9 / 45.5, 16 x 50176 45.6 / 53.7.
constexpr int64_t kSelClusterTokens = 16384;
constexpr int kSelClusterRows = 8;
constexpr int kSelBins = 2048;

// Exclusive prefix sum over the block; *total = the sum.  s_warp: 32 words that nothing else uses until the next barrier.
__device__ __forceinline__ int64_t block_exclusive_scan(int64_t v, int64_t* s_warp, int64_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  int64_t w = s_warp[lane];                    // every warp sums up the warps itself
  const int64_t own = w;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, w, o);
    if (lane >= o) w += y;
  }
  *total = __shfl_sync(0xffffffffu, w, 31);
  const int64_t before = __shfl_sync(0xffffffffu, w - own, warp);
  __syncthreads();
  return before + x - v;
}

// From saliency (radix select) or, where that is NULL, from a byte mask E [B][T].
__global__ void __launch_bounds__(kSelThreads) select_tokens_kernel(const float* __restrict__ saliency,
                                                                    const uint8_t* __restrict__ mask, int64_t mask_stride,
                                                                    int64_t vis_begin, int64_t l_v, int64_t n_prot,
                                                                    int64_t T_q, CacheView cv, int32_t* idx_prot,
                                                                    int32_t* idx_rest, int64_t stride_prot,
                                                                    int64_t stride_rest, int32_t* counts,
                                                                    int64_t expect_count) {
  __shared__ __align__(8) int hist[3][kSelBins];   // read two bins at a time
  __shared__ int64_t s_warp[32];
  __shared__ int64_t s_block;                  // (keys at the threshold) << 32 | (keys above it) in this block's words
  __shared__ uint32_t s_bin, s_need;
  cg::cluster_group cluster = cg::this_cluster();
  const int n_blocks = static_cast<int>(cluster.num_blocks()), rank = static_cast<int>(cluster.block_rank());
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x / n_blocks;
  const float* sal = saliency ? saliency + b * l_v : nullptr;
  const int64_t W = T_q / kG;
  const int64_t w_begin = W * rank / n_blocks, w_end = W * (rank + 1) / n_blocks;
  uint32_t thr = 0, need = 0;
  if (sal) {
    for (int i = tid; i < 3 * kSelBins; i += kSelThreads) hist[0][i] = 0;
    __syncthreads();
    const int64_t s_begin = l_v * rank / n_blocks, s_end = l_v * (rank + 1) / n_blocks;
    uint32_t pmask = 0;
    need = static_cast<uint32_t>(n_prot);
#pragma unroll
    for (int pass = 0; pass < 3; ++pass) {
      const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0);
      const uint32_t bins = pass == 2 ? 1024u : 2048u;
#pragma unroll 8
      for (int64_t i = s_begin + tid; i < s_end; i += kSelThreads) {
        const uint32_t key = float_ordered(__ldg(sal + i));
        if ((key & pmask) == thr) atomicAdd(&hist[pass][(key >> shift) & (bins - 1)], 1);
      }
      cluster.sync();
      // bins from the top: thread i has bins - 1 - 2 i and the one below it
      int c0 = 0, c1 = 0;
      const int top = kSelBins - 1 - 2 * tid;
      for (int r = 0; r < n_blocks; ++r) {
        const int2 c = *reinterpret_cast<const int2*>(cluster.map_shared_rank(&hist[pass][top - 1], r));
        c0 += c.y; c1 += c.x;
      }
      int64_t total;
      const int64_t above = block_exclusive_scan(c0 + c1, s_warp, &total);
      if (above < need && above + c0 >= need) { s_bin = top; s_need = need - static_cast<uint32_t>(above); }
      else if (above + c0 < need && above + c0 + c1 >= need) { s_bin = top - 1; s_need = need - static_cast<uint32_t>(above + c0); }
      __syncthreads();
      thr |= s_bin << shift; need = s_need;    // thr: key of the n-th largest; `need` of the keys equal to it are taken
      pmask |= (bins - 1) << shift;
    }
  }
  int stray = 0;                               // the row of a mask protects more (1) or fewer (-1) tokens than stated
  // gt / eq bits of token group w, the same in every lane
  auto word_bits = [&](int64_t w, uint32_t& gt, uint32_t& eq) {
    const int64_t t = w * kG + lane;
    bool g = false, e = false;
    if (sal) {
      if (t >= vis_begin && t < vis_begin + l_v) {
        const uint32_t key = float_ordered(__ldg(sal + (t - vis_begin)));
        g = key > thr; e = key == thr;
      }
    } else {
      const bool marked = __ldg(mask + b * mask_stride + t) != 0;
      g = marked && stray <= 0;
      e = stray > 0 ? marked : stray < 0 && !marked;
    }
    gt = __ballot_sync(0xffffffffu, g); eq = __ballot_sync(0xffffffffu, e);
  };
#pragma unroll 1
  for (bool again = true; again;) {
    int64_t carry = 0;                           // (at) << 32 | (above) before the next stretch of words
    if (n_blocks > 1) {
      int64_t mine = 0;
#pragma unroll 8
      for (int64_t w = w_begin + warp; w < w_end; w += 32) {
        uint32_t gt, eq;
        word_bits(w, gt, eq);
        mine += static_cast<int64_t>(__popc(gt)) | (static_cast<int64_t>(__popc(eq)) << 32);
      }
      if (lane == 0) s_warp[warp] = mine;
      __syncthreads();
      if (tid == 0) {
        int64_t sum = 0;
        for (int i = 0; i < 32; ++i) sum += s_warp[i];
        s_block = sum;
      }
      cluster.sync();
      for (int r = 0; r < rank; ++r) carry += *cluster.map_shared_rank(&s_block, r);
    }
    uint32_t* e_words = const_cast<uint32_t*>(cv.e_words(b));
    uint32_t* e_prefix = const_cast<uint32_t*>(cv.e_prefix(b));
    for (int64_t base = w_begin; base < w_end; base += kSelThreads) {
      // up to 1024 words at a time: every warp takes per_warp consecutive ones, lane i keeps word i
      const int n = static_cast<int>(min(static_cast<int64_t>(kSelThreads), w_end - base));
      const int per_warp = (n + 31) / 32;
      const int n_own = max(0, min(per_warp, n - warp * per_warp));
      const int64_t w0 = base + warp * per_warp;
      uint32_t gt = 0, eq = 0;
#pragma unroll 8
      for (int i = 0; i < n_own; ++i) {
        uint32_t g, e;
        word_bits(w0 + i, g, e);
        if (lane == i) { gt = g; eq = e; }
      }
      int64_t total;
      const int64_t before = carry + block_exclusive_scan(static_cast<int64_t>(__popc(gt)) | (static_cast<int64_t>(__popc(eq)) << 32), s_warp, &total);
      carry += total;
      const int64_t eq_before = before >> 32;
      int take = static_cast<int>(need) - static_cast<int>(min(eq_before, static_cast<int64_t>(need)));
      const int prot = static_cast<int>((before & 0xffffffff) + (static_cast<int64_t>(need) - take));
      uint32_t word = gt;
      for (uint32_t rem = eq; rem && take > 0; rem &= rem - 1, --take) word |= rem & (0u - rem);
      if (lane < n_own) {
        e_words[w0 + lane] = word;
        e_prefix[w0 + lane] = static_cast<uint32_t>(prot);
      }
#pragma unroll 4
      for (int i = 0; i < n_own; ++i) {
        const uint32_t bits = __shfl_sync(0xffffffffu, word, i);
        const int64_t t = (w0 + i) * kG + lane;
        const int64_t pk = __shfl_sync(0xffffffffu, prot, i) + __popc(bits & ((1u << lane) - 1u));
        if ((bits >> lane) & 1u) {
          if (pk < stride_prot) idx_prot[b * stride_prot + pk] = static_cast<int32_t>(t);
        } else {
          idx_rest[b * stride_rest + (t - pk)] = static_cast<int32_t>(t);
        }
      }
    }
    if (rank == n_blocks - 1 && tid == 0) {
      const int n = static_cast<int>((carry & 0xffffffff) + min(carry >> 32, static_cast<int64_t>(need)));
      e_prefix[W] = static_cast<uint32_t>(n);
      e_words[W] = 0;
      if (counts) counts[b] = n;
      s_block = n;
    }
    // A mask whose row does not protect the number of tokens that the caller stated: reported, and the row is done once more
    // with its first `expect_count` tokens, or with unprotected ones added in token order, so that the lists and the mask hold
    // what the quantizer and the attention kernels count on.
    again = false;
    if (expect_count >= 0 && stray == 0) {
      cluster.sync();
      const int64_t n = *cluster.map_shared_rank(&s_block, n_blocks - 1);
      cluster.sync();
      if (n != expect_count) {
        if (rank == 0 && tid == 0) atomicCAS(reinterpret_cast<int*>(cv.base + kHdrStatus), VIDKV_OK, VIDKV_ERR_INVALID_ARG);
        stray = n > expect_count ? 1 : -1;
        need = static_cast<uint32_t>(stray > 0 ? expect_count : expect_count - n);
        again = true;
      }
    }
  }
  if (n_blocks > 1) cluster.sync();            // the other blocks may still read this one's shared memory
}

// ---------------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------------
template <typename T, bool NZ>
static cudaError_t quantize_values_t(const KSrc& src, int64_t T_q, int n_res, const CacheView& cv, int layer, int n_layers,
                                     const SelView& sel, float gamma, cudaStream_t stream) {
  const int n_slabs = n_layers * cv.B * cv.H_kv;
  const int ternary_blocks = static_cast<int>((T_q - sel.n_prot + kSGTokens - 1) / kSGTokens);
  const int protect_blocks = static_cast<int>((sel.n_prot + 2 * kG - 1) / (2 * kG));
  constexpr size_t smem = kSGTokens * kVRowBytes + sizeof(uint32_t) * kSGGroups * 64;
  static_assert(smem >= kProtectSmem, "the protected groups live in the ternary tile's shared memory");
  static bool attr_set_dev[64] = {};   // function attributes are per device (and per instantiation)
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  bool& attr_set = attr_set_dev[dev];
  cudaError_t e;
  if (!attr_set) {
    if ((e = cudaFuncSetAttribute(v_quantize_kernel<T, NZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    attr_set = true;
  }
  count_launches(1);
  return launch_dependent(v_quantize_kernel<T, NZ>, dim3(static_cast<unsigned>(ternary_blocks + protect_blocks + (n_res > 0)), n_slabs),
                          dim3(kVThreads), smem, stream, src, T_q, T_q - sel.n_prot, n_res, cv, layer, sel, gamma, ternary_blocks, protect_blocks);
}

cudaError_t launch_quantize_values(int dtype, const KSrc& src, int64_t T_q, int n_res, const CacheView& cv, int layer, int n_layers,
                                   const SelView& sel, float gamma, bool nonzero_mean_scale, cudaStream_t stream) {
  if (dtype == VIDKV_F16)
    return nonzero_mean_scale ? quantize_values_t<__half, true>(src, T_q, n_res, cv, layer, n_layers, sel, gamma, stream)
                              : quantize_values_t<__half, false>(src, T_q, n_res, cv, layer, n_layers, sel, gamma, stream);
  return nonzero_mean_scale ? quantize_values_t<__nv_bfloat16, true>(src, T_q, n_res, cv, layer, n_layers, sel, gamma, stream)
                            : quantize_values_t<__nv_bfloat16, false>(src, T_q, n_res, cv, layer, n_layers, sel, gamma, stream);
}

template <typename T, bool NZ>
static void flush_values_t(const KSrc& src, const CacheView& cv, int layer0, int n_layers, int64_t tgroup0, float gamma,
                           cudaStream_t stream) {
  const int spl = cv.B * cv.H_kv;
  v_flush_kernel<T, NZ><<<spl * n_layers, kD, 0, stream>>>(src, cv, layer0, spl, tgroup0, gamma);
}

cudaError_t launch_flush_values(int dtype, const KSrc& src, const CacheView& cv, int layer0, int n_layers,
                                int64_t tgroup0, float gamma, bool nonzero_mean_scale, cudaStream_t stream) {
  if (dtype == VIDKV_F16) {
    if (nonzero_mean_scale) flush_values_t<__half, true>(src, cv, layer0, n_layers, tgroup0, gamma, stream);
    else flush_values_t<__half, false>(src, cv, layer0, n_layers, tgroup0, gamma, stream);
  } else {
    if (nonzero_mean_scale) flush_values_t<__nv_bfloat16, true>(src, cv, layer0, n_layers, tgroup0, gamma, stream);
    else flush_values_t<__nv_bfloat16, false>(src, cv, layer0, n_layers, tgroup0, gamma, stream);
  }
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_copy_to_residual(const KSrc& src, int n_tok, const CacheView& cv, int layer, int n_layers, bool is_value,
                                    cudaStream_t stream) {
  if (n_tok <= 0) return cudaSuccess;
  copy_to_residual_kernel<<<n_layers * cv.B * cv.H_kv, 256, 0, stream>>>(src, n_tok, cv, layer, is_value ? cv.vres_offset : cv.kres_offset);
  count_launches(1);
  return cudaGetLastError();
}

static cudaError_t launch_select(const float* saliency, const uint8_t* mask, int64_t mask_stride, int64_t vis_begin, int64_t l_v,
                                 int64_t n_prot, int64_t T_q, const CacheView& cv, int32_t* idx_prot, int32_t* idx_rest,
                                 int64_t stride_prot, int64_t stride_rest, int32_t* counts, int64_t expect_count, cudaStream_t stream) {
  const unsigned blocks = T_q >= kSelClusterTokens && cv.B <= kSelClusterRows ? kSelCluster : 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks * cv.B); cfg.blockDim = dim3(kSelThreads); cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = blocks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  count_launches(1);
  return cudaLaunchKernelEx(&cfg, select_tokens_kernel, saliency, mask, mask_stride, vis_begin, l_v, n_prot, T_q, cv, idx_prot, idx_rest,
                            stride_prot, stride_rest, counts, expect_count);
}

cudaError_t launch_select_tokens(const float* saliency, int64_t vis_begin, int64_t l_v, int64_t n_prot, int64_t T_q,
                                 const CacheView& cv, int32_t* idx_prot, int32_t* idx_rest, int64_t stride_prot,
                                 int64_t stride_rest, cudaStream_t stream) {
  return launch_select(saliency, nullptr, 0, vis_begin, l_v, n_prot, T_q, cv, idx_prot, idx_rest, stride_prot, stride_rest, nullptr, -1, stream);
}

cudaError_t launch_mask_to_selection(const uint8_t* E, int64_t T, int64_t T_q, const CacheView& cv, int32_t* idx_prot,
                                     int32_t* idx_rest, int64_t stride_prot, int64_t stride_rest, int32_t* counts,
                                     int64_t expect_count, cudaStream_t stream) {
  return launch_select(nullptr, E, T, 0, 0, 0, T_q, cv, idx_prot, idx_rest, stride_prot, stride_rest, counts, expect_count, stream);
}

}  // namespace vidkv
