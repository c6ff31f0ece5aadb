// Key encode pass of Algorithm 3 (MixQuant), one tile of 128 tokens x 128 channels at a time.
// The tile is the B operand of one product on the fifth-generation tensor cores (tcgen05.mma,
// operands in shared memory in the 128-byte-swizzled K-major layout, accumulators in tensor
// memory); the A operand has one row per output of the channel sort:
//   anomalous channels (Eq. 4) 64 selector rows (a single 1.0) copy the 64 anomalous channels
//                     exactly, so that accumulator row = slot, columns = tokens.  Per (slot,
//                     32-token group): min / max, s = (max - min) / 3, z = min rounded to
//                     binary16, code = clamp(rint((x - z) / s), 0, 3).  No division: code >= k
//                     is a monotone predicate of x, so the three smallest element values X_k
//                     with code(X_k) >= k are found once, with an exact test (code_at_least),
//                     and the elements are compared against them two at a time; the 2-bit
//                     fields are assembled into the cache's code words across lanes.
//   normal channels   (Eq. 5) 64 rows hold the columns of the orthonormal 64-point DFT over the
//                     channel axis, spread over the slab's normal channels and split into
//                     parts (binary16: 2, bfloat16: 3) so that products carry 22 - 24 bits;
//                     float32 accumulation.  Accumulator row = spectrum column: the sign bits
//                     and the per-group mean |.| are per-thread work, a warp-wide bit
//                     transpose gives the cache's (token, 16 columns) half-words.
// Persistent grid of two blocks per SM; block = 8 warps that load and encode and one that issues the products.
//
// What bounds it: the instructions of the epilogue (code thresholds, comparisons, bit transposes).  A tile goes through in
// two halves of 64 tokens with accumulators of their own, so that the products of one half run behind the epilogue of the
// other and the loads of the next tile behind both.  The parts of the DFT rows accumulate apart and are added at the end;
// in one accumulator the sums would take 10 us less but come out one rounding different, and a coefficient next to zero
// would change its stored sign.  64 slabs x 12544 tokens, binary16, with the range pass: 128 us, 140 before the halves,
// code_cut and the selection in here; bfloat16 145 / 159.
#include <math.h>

#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "kernels.cuh"
#include "quant_common.cuh"

namespace vidkv {

namespace {

constexpr int kEncTokens = 128;
constexpr int kDftWords = 4 * 8 * 32 * 4;      // [k step][column tile][lane][hi0, hi1, lo0, lo1]

// B fragments of the DFT matrix in the order the MMA wants them (see dft_table_kernel).
__device__ __align__(16) uint32_t g_dft_frag[kDftWords];

// The same matrix as plain 16-bit patterns [part][spectrum column f][channel position c]:
// parts 0, 1: binary16 leading part and remainder; parts 2, 3, 4: bfloat16 leading, middle and
// last part (w = sum of the parts to 22 resp. 24 bits).
constexpr int kWParts = 5;
__device__ __align__(16) uint16_t g_dft_w[kWParts * 64 * 64];

// [channel position c][spectrum column f]: the weight with which column f of a 32-point Hermitian half spectrum
// enters channel c under the inverse orthonormal transform (the query preparation of the k = 0.75 Eq. 5 format).
__device__ __align__(16) float g_dft_w32[32 * 32];

// Byte offset of element (row, k) of a K-major operand with 64 binary16 per row under the
// 128-byte swizzle: 8-row atoms of 1024 bytes, 16-byte pieces XORed with the row within the atom.
__host__ __device__ constexpr int sw128_offset(int row, int k) {
  return (row >> 3) * 1024 + (row & 7) * 128 + ((((k >> 3) ^ row) & 7) << 4) + (k & 7) * 2;
}

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}
}  // namespace

// Column f of the DFT matrix at channel position c: f = 0: 1/8; f = 1: (-1)^c / 8;
// f = 2k: cos(2 pi k c / 64) / 8; f = 2k + 1: -sin(2 pi k c / 64) / 8.
__device__ double dft_weight(int f, int c) {
  if (f == 0) return 0.125;
  if (f == 1) return (c & 1) ? -0.125 : 0.125;
  double sn, cs;
  sincospi(static_cast<double>(((f >> 1) * c) & 63) / 32.0, &sn, &cs);
  return ((f & 1) ? -sn : cs) * 0.125;
}

// One block of 256 threads.  mma.sync fragments (used by the decode path for the query): word
// layout for k step ks, column tile nt and lane (n = lane / 4, r = lane % 4): rows
// k0 = 16 ks + 2 r (and k0 + 1; k0 + 8, k0 + 9) of column f = 16 (n / 2) + 2 nt + (n % 2), so
// that after the product lane (., r) holds the spectrum columns 16 r .. 16 r + 15 of its two rows.
__global__ void dft_table_kernel() {
  for (int i = threadIdx.x; i < kDftWords / 4; i += blockDim.x) {
    const int lane = i & 31, nt = (i >> 5) & 7, ks = i >> 8;
    const int n = lane >> 2, r = lane & 3;
    const int f = 16 * (n >> 1) + 2 * nt + (n & 1);
    float w[4];
    const int rows[4] = {16 * ks + 2 * r, 16 * ks + 2 * r + 1, 16 * ks + 2 * r + 8, 16 * ks + 2 * r + 9};
    for (int j = 0; j < 4; ++j) w[j] = static_cast<float>(dft_weight(f, rows[j]));
    const __half h0 = __float2half_rn(w[0]), h1 = __float2half_rn(w[1]), h2 = __float2half_rn(w[2]), h3 = __float2half_rn(w[3]);
    g_dft_frag[i * 4 + 0] = as_u32(__halves2half2(h0, h1));
    g_dft_frag[i * 4 + 1] = as_u32(__halves2half2(h2, h3));
    g_dft_frag[i * 4 + 2] = as_u32(__floats2half2_rn(w[0] - __half2float(h0), w[1] - __half2float(h1)));
    g_dft_frag[i * 4 + 3] = as_u32(__floats2half2_rn(w[2] - __half2float(h2), w[3] - __half2float(h3)));
  }
  for (int i = threadIdx.x; i < 64 * 64; i += blockDim.x) {
    const int f = i >> 6, c = i & 63;
    const float w = static_cast<float>(dft_weight(f, c));
    const __half hi = __float2half_rn(w);
    g_dft_w[i] = __half_as_ushort(hi);
    g_dft_w[4096 + i] = __half_as_ushort(__float2half_rn(w - __half2float(hi)));
    const __nv_bfloat16 b0 = __float2bfloat16_rn(w);
    const float r1 = w - __bfloat162float(b0);
    const __nv_bfloat16 b1 = __float2bfloat16_rn(r1);
    const float r2 = r1 - __bfloat162float(b1);
    g_dft_w[2 * 4096 + i] = __bfloat16_as_ushort(b0);
    g_dft_w[3 * 4096 + i] = __bfloat16_as_ushort(b1);
    g_dft_w[4 * 4096 + i] = __bfloat16_as_ushort(__float2bfloat16_rn(r2));
  }
  for (int i = threadIdx.x; i < 32 * 32; i += blockDim.x) {
    const int c = i >> 5, f = i & 31, k = f < 2 ? 16 * f : f >> 1;
    double sn, cs;
    sincospi(static_cast<double>((k * c) & 31) / 16.0, &sn, &cs);
    g_dft_w32[i] = static_cast<float>((f < 2 ? cs : 2.0 * ((f & 1) ? -sn : cs)) / sqrt(32.0));
  }
}

// ---- tcgen05 helpers -------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// Shared-memory matrix descriptor of a K-major operand with one 128-byte swizzle atom along K:
// start address / 16, 8-row groups 1024 bytes apart, descriptor version 1, 128-byte swizzle.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t smem_addr) {
  return static_cast<uint64_t>((smem_addr >> 4) & 0x3fffu) | (static_cast<uint64_t>(1u) << 16) |
         (static_cast<uint64_t>(1024u >> 4) << 32) | (static_cast<uint64_t>(1u) << 46) | (static_cast<uint64_t>(2u) << 61);
}
constexpr int kTmemCols = 256;        // two halves of a tile, each with two float32 accumulators of 128 x 64
constexpr int kWaitLimit = 1 << 14;

// One lane of a converged warp.  Issued behind this in a warp-uniform branch an MMA takes the tensor pipe's own time
// (35 clocks at N = 64); behind "if (threadIdx.x == 0)" its operands take a slower way: 49 clocks and more for any N.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{ .reg .pred q; elect.sync _|q, 0xffffffff; selp.u32 %0, 1, 0, q; }" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5}, p;\n\t}"
      ::"r"(tmem_d), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(0u)
      : "memory");
}
// 32 consecutive accumulator columns of the calling warp's 32 lanes of tensor memory.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}

// Per element type: how the DFT matrix is split (binary16: 2 parts, bfloat16: 3 parts), the
// operand format code of the instruction descriptor, and 1.0.
template <typename T> struct Enc;
template <> struct Enc<__half> {
  static constexpr int kParts = 2, kFmt = 0, kTab = 0;
  static constexpr uint16_t kOne = 0x3c00u;
  static __device__ __forceinline__ uint32_t pack(float a, float b) { return as_u32(__floats2half2_rn(a, b)); }
};
template <> struct Enc<__nv_bfloat16> {
  static constexpr int kParts = 3, kFmt = 1, kTab = 2;
  static constexpr uint16_t kOne = 0x3f80u;
  static __device__ __forceinline__ uint32_t pack(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
  }
};

// Shared memory of one block, from a 1024-byte boundary.  All operands are K-major with the
// 128-byte swizzle, one 64-channel block of K after the other.
//   [0, 32768)     the tile as the B operand: [2 K blocks][128 tokens][64 channels]
//   then           X: the remaining parts of the DFT rows, per part [2 K blocks][64 rows][64 channels]
//                  A: the leading part, [2 K blocks][128 rows][64 channels].  Arrangement 0: row
//                  m < 64 selects the anomalous channel of slot m, row 64 + f holds column f of the
//                  DFT matrix spread over the normal channels (zero elsewhere); arrangement 1 swaps
//                  the two halves.
//                  The products of X use M = 128 too: in arrangement 0 the descriptor starts 64
//                  rows early, in arrangement 1 it runs 64 rows long; the extra rows read
//                  neighbouring shared memory and land in accumulator rows that nobody reads.
//   then the channel order [128], the five mbarriers, the tensor-memory address, the fault flag (64 bytes), and the channel
//   selection's work area: float range [128], int rank of two halves [2][128], mask words [4]
constexpr int kEncSelect = kD * 4 + 2 * kD * 4 + 16;
constexpr int kEncThreads = 288;       // eight warps that load and encode, one that issues the products
constexpr int kSmTile = 0, kSmAex = 32768;
template <typename T> __host__ __device__ constexpr int enc_sm_ahi() { return kSmAex + 16384 * (Enc<T>::kParts - 1); }
template <typename T> __host__ __device__ constexpr int enc_sm_perm() { return enc_sm_ahi<T>() + 32768; }
template <typename T> __host__ __device__ constexpr int enc_sm_bytes() { return enc_sm_perm<T>() + kD + 64 + kEncSelect + 1024; }

size_t k_encode_smem_bytes(int dtype) { return dtype == VIDKV_F16 ? enc_sm_bytes<__half>() : enc_sm_bytes<__nv_bfloat16>(); }

// Persistent blocks, two per SM: block b encodes the tiles [n b / G, n (b + 1) / G) of the
// launch's n = slabs x tiles-per-slab tiles.  Warp w works on tensor-memory lanes 32 (w % 4):
// warps with w % 4 < 2 own 32 anomalous slots each, the others 32 spectrum columns each (and
// issue the tile loads); w / 4 picks the first or second of the two 32-token groups of each half tile.
template <typename T>
__global__ void __launch_bounds__(kEncThreads, 2) k_encode_kernel(KSrc src, int64_t T_tokens, CacheView cv, int layer0,
                                                          int slabs_per_layer, int chunk, int64_t kgroup0, MinMaxBuffers mm,
                                                          int tiles_per_slab, int total_tiles, int withhold_first) {
  extern __shared__ uint8_t esm_raw[];
  uint8_t* esm = esm_raw + ((1024u - (smem_u32(esm_raw) & 1023u)) & 1023u);
  uint8_t* tile = esm + kSmTile;
  uint8_t* a_hi = esm + enc_sm_ahi<T>();
  uint8_t* a_ex = esm + kSmAex;
  uint8_t* perm = esm + enc_sm_perm<T>();
  uint64_t* mbar = reinterpret_cast<uint64_t*>(perm + kD);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(perm + kD + 40);
  volatile uint32_t* fault = reinterpret_cast<volatile uint32_t*>(perm + kD + 44);
  float* sel_range = reinterpret_cast<float*>(perm + kD + 64);
  int* sel_rank = reinterpret_cast<int*>(sel_range + kD);
  uint32_t* sel_mask = reinterpret_cast<uint32_t*>(sel_rank + 2 * kD);

  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int quad = warp & 3, half = warp >> 2;
  // Row arrangement of the A operand: 0 puts the anomalous slots in rows 0 .. 63 and the DFT
  // columns in rows 64 .. 127, 1 the other way round.  The two blocks that share an SM (b and
  // b + G / 2 when blocks are handed out breadth first) take different arrangements so that the
  // heavier anomalous warps of one block sit on the schedulers of the lighter warps of the other.
  const int arr = (2 * blockIdx.x >= gridDim.x) ? 1 : 0;
  const bool loader = (quad >= 2) != (arr == 1);        // the spectrum warps also move the tiles
  const int lt = half * 64 + (quad & 1) * 32 + lane;    // 0 .. 127 among the loading threads

  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < 5; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar + i)), "r"(i < 3 ? 1 : 8) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *fault = 0u;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  const int tile_begin = static_cast<int>(static_cast<int64_t>(total_tiles) * blockIdx.x / gridDim.x);
  const int tile_end = static_cast<int>(static_cast<int64_t>(total_tiles) * (blockIdx.x + 1) / gridDim.x);

  // Tiles are walked as (slab, tile of the slab) pairs so that divisions happen once per block,
  // once for the tile being encoded and once for the tile being fetched.
  int slab = tile_begin / tiles_per_slab, ti = tile_begin - slab * tiles_per_slab;
  int lslab = slab, lti = ti, lbase_slab = -1;
  const T* lbase = nullptr;

  // Half hs of the next tile in 16-byte pieces: thread lt moves piece lt % 16 of the rows 64 hs + lt / 16 + 8 i
  auto load_next = [&](int hs) {
    if (lslab != lbase_slab) {
      lbase_slab = lslab;
      lbase = reinterpret_cast<const T*>(src.ptr) + (lslab / src.H) * src.stride_b + (lslab % src.H) * src.stride_h;
    }
    const int64_t t0 = static_cast<int64_t>(lti) * kEncTokens;
    const int n_tok = static_cast<int>(min(static_cast<int64_t>(kEncTokens), T_tokens - t0));
    const int row0 = 64 * hs + (lt >> 4), piece = lt & 15;
    const uint8_t* srow = reinterpret_cast<const uint8_t*>(lbase + (t0 + row0) * src.stride_t) + piece * 16;
    uint8_t* drow = tile + (piece >> 3) * 16384 + row0 * 128 + (((piece ^ row0) & 7) << 4);
    const int64_t sstep = 8 * src.stride_t * static_cast<int64_t>(sizeof(T));
#pragma unroll
    for (int i = 0; i < kEncTokens / 16; ++i)
      if (row0 + 8 * i < n_tok) cp_async16(drow + i * 1024, srow + i * sstep);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (hs == 1 && ++lti == tiles_per_slab) { lti = 0; ++lslab; }
  };

  // ---- D[128 rows x 64 tokens] = A (leading) x tile^T; D'[.. x ..] = A (remaining parts) x tile^T, for tokens 64 hs .. 64 hs + 63
  // Products issued so far arrive at mbarrier i when they are done.
  auto commit = [&](int i) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar + i)) : "memory");
  };
  auto issue = [&](int hs) {
    if (elect_one()) {
      constexpr uint32_t idesc = (1u << 4) | (static_cast<uint32_t>(Enc<T>::kFmt) << 7) | (static_cast<uint32_t>(Enc<T>::kFmt) << 10) |
                                 ((64u >> 3) << 17) | ((128u >> 4) << 24);
      const uint32_t d = tmem + static_cast<uint32_t>(hs * 128);
      const uint32_t b0 = smem_u32(tile) + static_cast<uint32_t>(hs * 8192);
#pragma unroll
      for (int kb = 0; kb < 2; ++kb) {
        const uint64_t da = umma_desc_sw128(smem_u32(a_hi + kb * 16384)), db = umma_desc_sw128(b0 + static_cast<uint32_t>(kb * 16384));
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)   // 16 elements = 32 bytes along K per step; the address field counts 16 bytes
          umma_f16(d, da + static_cast<uint64_t>(2 * ks), db + static_cast<uint64_t>(2 * ks), idesc, (kb | ks) != 0 ? 1u : 0u);
      }
#pragma unroll
      for (int part = 1; part < Enc<T>::kParts; ++part) {
#pragma unroll
        for (int kb = 0; kb < 2; ++kb) {
          // the part's 64 rows are rows 64 .. 127 of arrangement 0 (start 8192 bytes early), rows 0 .. 63 of arrangement 1
          const uint64_t da = umma_desc_sw128(smem_u32(a_ex + (part - 1) * 16384 + kb * 8192 - (arr ? 0 : 8192)));
          const uint64_t db = umma_desc_sw128(b0 + static_cast<uint32_t>(kb * 16384));
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)
            umma_f16(d + 64u, da + static_cast<uint64_t>(2 * ks), db + static_cast<uint64_t>(2 * ks), idesc,
                     (part - 1) | kb | ks ? 1u : 0u);
        }
      }
      commit(hs);
    }
    __syncwarp();
  };
  auto wait_for = [&](int i, uint32_t parity) -> bool {
    uint32_t done = 0;
    for (int it = 0; it < kWaitLimit && !done; ++it) {
      asm volatile(
          "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(done) : "r"(smem_u32(mbar + i)), "r"(parity) : "memory");
    }
    return __all_sync(0xffffffffu, done != 0);
  };

  // mbarriers: hs, the products of half hs are done; 2, all products are done; 3 + hs, half hs of the tile is in shared
  // memory, operand A is built and the half's accumulators of the tile before have been read (one arrival per warp).
  // Every wait is bounded; whoever runs out of patience sets the fault flag and waits and arrives no more.
  if (loader && tile_begin < tile_end) { load_next(0); load_next(1); }   // the keys are complete: the range pass has waited for them
  constexpr int kAVec = (32768 + 16384 * (Enc<T>::kParts - 1)) / 16;
  auto clear_operand = [&]() {
#pragma unroll 4
    for (int i = tid; i < kAVec; i += 256) reinterpret_cast<uint4*>(a_ex)[i] = make_uint4(0u, 0u, 0u, 0u);
  };
  bool cleared = true;                                       // operand A, for the block's first slab while the ranges still come in
  if (warp != 8) clear_operand();
  pdl_wait();                                                // the ranges
  if (warp == 8) {
    uint32_t parity = 0;
    bool lost = false;
    for (int t = tile_begin; t < tile_end && !lost; ++t, parity ^= 1u) {
#pragma unroll
      for (int hs = 0; hs < 2; ++hs) {
        lost = lost || !wait_for(3 + hs, parity) || __any_sync(0xffffffffu, *fault != 0u);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // (withhold_first, a test hook: the block's first tile gets neither products nor a commit, so the
        // waits for them run out with nothing outstanding)
        if (!lost && !(withhold_first && t == tile_begin)) issue(hs);
      }
    }
    if (elect_one()) commit(2);
    __syncwarp();
    wait_for(2, 0u);                                           // nothing is under way when the tensor memory is given back
    if (lost && lane == 0) {
      *fault = 1u;
      atomicCAS(reinterpret_cast<int*>(cv.base + kHdrStatus), 0, static_cast<int>(VIDKV_ERR_TIMEOUT));
    }
    __syncthreads();
    return;
  }
  bool lost = false;                                         // a wait ran out: nothing more is encoded
  auto arrive = [&](int hs) {
    __syncwarp();
    if (lane == 0 && !lost) asm volatile("{ .reg .b64 s; mbarrier.arrive.shared::cta.b64 s, [%0]; }" ::"r"(smem_u32(mbar + 3 + hs)) : "memory");
  };

  int cur_slab = -1;
  uint32_t phase = 0;
  bool ahead = false;                                        // this tile's arrivals have happened already
  uint8_t* slab_ptr = nullptr;
  // Re-arm the buffer the next call accumulates into (min half all ones, max half zero).  Nobody reads it now: its last
  // readers ran before this call's range pass in stream order.
  for (int i = blockIdx.x * 256 + tid; i < mm.next_dirty_words; i += gridDim.x * 256)
    mm.next[i] = (i & (2 * kD - 1)) < kD ? 0xffffffffu : 0u;
  for (int t = tile_begin; t < tile_end; ++t, ti = (ti + 1 == tiles_per_slab) ? 0 : ti + 1, slab += (ti == 0) ? 1 : 0) {
    if (slab != cur_slab) {
      const int layer = layer0 + slab / slabs_per_layer;
      const int bh = slab % slabs_per_layer;
      slab_ptr = cv.slab(layer, bh / cv.H_kv, bh % cv.H_kv);
    }
    const int64_t t0 = static_cast<int64_t>(ti) * kEncTokens;
    const int n_tok = static_cast<int>(min(static_cast<int64_t>(kEncTokens), T_tokens - t0));   // multiple of 32
    const int n_groups = n_tok / kG;
    uint8_t* kg_base = slab_ptr + cv.kgroup_offset + (kgroup0 + t0 / kG) * kKGroupBytes;

    // ---- a new slab: its channel order and the A operand built from it
    if (slab != cur_slab) {
      cur_slab = slab;
      // eight entries of the matrix per load, all in flight before anything else (one by one they cost the block 16 memory
      // latencies, as long as a tile)
      uint4 wv[Enc<T>::kParts][2];
#pragma unroll
      for (int part = 0; part < Enc<T>::kParts; ++part)
#pragma unroll
        for (int j = 0; j < 2; ++j)
          wv[part][j] = reinterpret_cast<const uint4*>(g_dft_w + (Enc<T>::kTab + part) * 4096)[tid + 256 * j];
      // TopK (Algorithm 3): rank(c) = channels before c in (range descending, index ascending) order, two threads per
      // channel; the first 64 are the anomalous ones.  Every block does it for the slabs it meets, about 0.5 us, where a
      // kernel of its own took 3 us and a launch gap per call.
      {
        const int c = tid & (kD - 1), side = tid >> 7;
        const uint32_t* mmw = mm.cur + static_cast<int64_t>(slab) * 2 * kD;
        if (side == 0) sel_range[c] = __fsub_rn(ordered_float(mmw[kD + c]), ordered_float(mmw[c]));
        asm volatile("bar.sync 1, 256;" ::: "memory");
        const float rg = sel_range[c];
        int rank = 0;
#pragma unroll 16
        for (int o = side * (kD / 2); o < (side + 1) * (kD / 2); o += 4) {
          const float4 v = *reinterpret_cast<const float4*>(sel_range + o);
          rank += (v.x > rg) || (v.x == rg && o < c);
          rank += (v.y > rg) || (v.y == rg && o + 1 < c);
          rank += (v.z > rg) || (v.z == rg && o + 2 < c);
          rank += (v.w > rg) || (v.w == rg && o + 3 < c);
        }
        sel_rank[tid] = rank;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        const bool abn = sel_rank[c] + sel_rank[kD + c] < kNA;
        const uint32_t word = __ballot_sync(0xffffffffu, abn);
        if (lane == 0 && side == 0) sel_mask[warp] = word;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (side == 0) {
          int before = __popc(word & ((1u << lane) - 1u));
          for (int i = 0; i < warp; ++i) before += __popc(sel_mask[i]);
          const int at = abn ? before : kNA + c - before;
          perm[at] = static_cast<uint8_t>(c);
          if (ti == 0) slab_ptr[cv.chunk_table_offset + static_cast<int64_t>(chunk) * kChunkBytes + at] = static_cast<uint8_t>(c);
        }
      }
      if (!cleared) clear_operand();
      cleared = false;
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (tid < kNA) {
        const int c = perm[tid];
        *reinterpret_cast<uint16_t*>(a_hi + (c >> 6) * 16384 + sw128_offset(64 * arr + tid, c & 63)) = Enc<T>::kOne;
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int v = tid + 256 * j, f = v >> 3;               // entries 8 (v % 8) .. + 7 of column f
        const uint2 pc = *reinterpret_cast<const uint2*>(perm + kNA + 8 * (v & 7));
#pragma unroll
        for (int x = 0; x < 8; ++x) {
          const int c = ((x < 4 ? pc.x : pc.y) >> (8 * (x & 3))) & 0xff;
          const int hi_at = (c >> 6) * 16384 + sw128_offset(64 - 64 * arr + f, c & 63), ex_at = (c >> 6) * 8192 + sw128_offset(f, c & 63);
#pragma unroll
          for (int part = 0; part < Enc<T>::kParts; ++part) {
            const uint4& q = wv[part][j];
            const uint32_t word = x < 2 ? q.x : x < 4 ? q.y : x < 6 ? q.z : q.w;
            const uint16_t val = static_cast<uint16_t>((x & 1) ? word >> 16 : word);
            if (part == 0) *reinterpret_cast<uint16_t*>(a_hi + hi_at) = val;
            else *reinterpret_cast<uint16_t*>(a_ex + (part - 1) * 16384 + ex_at) = val;
          }
        }
      }
    }

    // ---- unless operand A is new, the products were ordered behind the epilogue of the tile before
    if (!ahead) {
      if (loader) asm volatile("cp.async.wait_group 0;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      arrive(0);
      arrive(1);
    }
    const bool more = t + 1 < tile_end;
    ahead = more && ti + 1 < tiles_per_slab;                   // the next tile has the same operand A
#pragma unroll 1
    for (int hs = 0; hs < 2; ++hs) {
      // every warp waits for the half's accumulators; a timeout is reported in the status word, and the warp goes on to the
      // end without waiting or writing
      if (!lost) {
        lost = !wait_for(hs, phase) || __any_sync(0xffffffffu, *fault != 0u);
        if (lost && lane == 0) {
          *fault = 1u;
          atomicCAS(reinterpret_cast<int*>(cv.base + kHdrStatus), 0, static_cast<int>(VIDKV_ERR_TIMEOUT));
        }
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // the products are done with this half of the tile: fetch the next tile's
      if (loader && more) load_next(hs);
      const int g = 2 * hs + half;
      const uint32_t acc = tmem + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(hs * 128 + half * 32);
      if (lost || g >= n_groups) {
        // nothing to encode; the warps still meet
      } else
      if (!loader) {
        // ---- Eq. 4: lane = anomalous slot j, the accumulator row holds its 64 tokens (exact values)
        const int j = (quad & 1) * 32 + lane, wg = j >> 4;
        const int pos = (lane >> 1) & 3;                            // field of the slot inside its code byte
        const bool pb0 = (lane & 2) != 0, pb1 = (lane & 4) != 0;    // bits of pos
        const bool bb0 = (lane & 8) != 0, bb1 = (lane & 1) != 0;    // bits of the slot's byte index 2 (e % 2) + e / 8
        const uint32_t wgt = pos == 0 ? 0x3c003c00u : pos == 1 ? 0x44004400u : pos == 2 ? 0x4c004c00u : 0x54005400u;   // 4^pos
        uint32_t x[32];
        tmem_ld32(acc, x);
        float fmn = __uint_as_float(x[0]), fmx = fmn;
#pragma unroll
        for (int i = 1; i < 32; ++i) { fmn = fminf(fmn, __uint_as_float(x[i])); fmx = fmaxf(fmx, __uint_as_float(x[i])); }
        const uint16_t sh = f2h_bits(__fdiv_rn(__fsub_rn(fmx, fmn), 3.0f));
        const uint16_t zh = f2h_bits(fmn);
        uint8_t* kg = kg_base + g * kKGroupBytes;
        reinterpret_cast<uint16_t*>(kg + kKG_S2)[j] = sh;
        reinterpret_cast<uint16_t*>(kg + kKG_Z2)[j] = zh;
        const float sc = h2f(sh), z = h2f(zh);
        uint32_t thr[3];
#pragma unroll
        for (int k = 1; k <= 3; ++k) {
          const uint16_t X = code_cut<T>(z, sc, k);
          thr[k - 1] = static_cast<uint32_t>(X) * 0x10001u;
        }
        // codes of token pairs as 1024 + code * 4^pos per 16-bit lane: the low byte of a lane is the
        // slot's contribution to the code byte of that token
        uint32_t w[8];   // w[tl]: bytes nt = 0..3 for the tokens tl + 8 nt
#pragma unroll
        for (int sp = 0; sp < 4; ++sp) {
          uint32_t h[4];
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) {
            const int tp = sp + 4 * nt;   // tokens 2 sp + 8 nt and the next one
            const uint32_t v = Enc<T>::pack(__uint_as_float(x[2 * tp]), __uint_as_float(x[2 * tp + 1]));
            __half2 acc = __hfma2(as_h2(Ops<T>::ge(v, thr[0])), as_h2(wgt), as_h2(0x64006400u));
            acc = __hfma2(as_h2(Ops<T>::ge(v, thr[1])), as_h2(wgt), acc);
            acc = __hfma2(as_h2(Ops<T>::ge(v, thr[2])), as_h2(wgt), acc);
            h[nt] = as_u32(acc);
          }
          const uint32_t p01 = prmt(h[0], h[1], 0x6240u), p23 = prmt(h[2], h[3], 0x6240u);
          w[2 * sp] = prmt(p01, p23, 0x5410u);
          w[2 * sp + 1] = prmt(p01, p23, 0x7632u);
        }
        // OR over the four slots of a byte (lanes ^ 4, ^ 2), each lane keeping the token sets tl = 2 pos, 2 pos + 1
        uint32_t w1[4], w2[2];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t keep = pb1 ? w[4 + i] : w[i], send = pb1 ? w[i] : w[4 + i];
          w1[i] = keep | __shfl_xor_sync(0xffffffffu, send, 4);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const uint32_t keep = pb0 ? w1[2 + i] : w1[i], send = pb0 ? w1[i] : w1[2 + i];
          w2[i] = keep | __shfl_xor_sync(0xffffffffu, send, 2);
        }
        // gather the four bytes of a word from the four lanes that hold them (lanes ^ 8, ^ 1); the
        // lane ends with the words of token nt = 2 bb0 + bb1 of both of its token sets
        uint32_t u0, u1;
        {
          const uint32_t lo = prmt(w2[0], w2[1], 0x5410u), hi = prmt(w2[0], w2[1], 0x7632u);
          const uint32_t keep = bb0 ? hi : lo, recv = __shfl_xor_sync(0xffffffffu, bb0 ? lo : hi, 8);
          const uint32_t a = bb0 ? recv : keep, b = bb0 ? keep : recv;   // a: even byte of the pair, b: odd byte
          u0 = prmt(a, b, 0x5140u);
          u1 = prmt(a, b, 0x7362u);
        }
        {
          const uint32_t first = prmt(u0, u1, 0x5410u), second = prmt(u0, u1, 0x7632u);
          const uint32_t keep = bb1 ? second : first, recv = __shfl_xor_sync(0xffffffffu, bb1 ? first : second, 1);
          const uint32_t lowpair = bb1 ? recv : keep, highpair = bb1 ? keep : recv;
          const int nt = (bb0 ? 2 : 0) + (bb1 ? 1 : 0);
          uint32_t* codes = reinterpret_cast<uint32_t*>(kg + kKG_Codes2);
          codes[((2 * pos) * 4 + wg) * 4 + nt] = prmt(lowpair, highpair, 0x5410u);
          codes[((2 * pos + 1) * 4 + wg) * 4 + nt] = prmt(lowpair, highpair, 0x7632u);
        }
      } else {
        // ---- Eq. 5: lane = spectrum column f, the two accumulators' rows 64 + f hold its 64 tokens
        const int hq = quad & 1, f = hq * 32 + lane;
        uint32_t xa[32], xb[32];
        tmem_ld32(acc, xa);
        tmem_ld32(acc + 64u, xb);
        float sum = 0.0f;
        uint32_t bits = 0u;   // bit i = sign bit of the column's coefficient of token i
#pragma unroll
        for (int i = 31; i >= 0; --i) {
          const float X = __uint_as_float(xa[i]) + __uint_as_float(xb[i]);
          sum += fabsf(X);
          bits = __funnelshift_l(__float_as_uint(X), bits, 1);
        }
        uint8_t* kg = kg_base + g * kKGroupBytes;
        reinterpret_cast<uint16_t*>(kg + kKG_S1)[f] = f2h_bits(sum * (1.0f / 32.0f));
        // 32 x 32 bit transpose over the warp: afterwards lane = token, bit l = column 32 hq + l
#pragma unroll
        for (int jb = 4; jb >= 0; --jb) {
          const int js = 1 << jb;
          const uint32_t m = jb == 4 ? 0x0000ffffu : jb == 3 ? 0x00ff00ffu : jb == 2 ? 0x0f0f0f0fu : jb == 1 ? 0x33333333u : 0x55555555u;
          const uint32_t y = __shfl_xor_sync(0xffffffffu, bits, js);
          const bool up = (lane & js) != 0;
          const uint32_t keep = up ? ~m : m;
          const uint32_t ysh = up ? (y >> js) : (y << js);
          bits = (bits & keep) | (ysh & ~keep);
        }
        // column e of a 16-column block goes to bit 15 - e of the block's half-word, 1 = coefficient >= 0
        const uint32_t mine = ~__brev(bits);
        uint16_t* hw = reinterpret_cast<uint16_t*>(kg + kKG_Bits1);
        const int hidx = ((lane & 7) * 4 + 2 * hq) * 4 + (lane >> 3);
        hw[hidx] = static_cast<uint16_t>(mine >> 16);
        hw[hidx + 4] = static_cast<uint16_t>(mine);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      if (ahead && !loader) arrive(hs);
    }
    phase ^= 1u;
    if (ahead && loader) {
      // the products of the next tile's first half run while the anomalous warps are still at this tile's codes
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      arrive(0);
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      arrive(1);
    }
  }
  if (loader) asm volatile("cp.async.wait_group 0;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------------------------
// Host launcher of the encode pass
// ---------------------------------------------------------------------------------
// The DFT tables are written once per device by a small kernel on the stream of the first
// call that needs them, followed by an event; every call makes its stream wait for that event
// (free once it has completed), so uses on other streams are ordered after the fill without a
// host-side synchronisation.
cudaError_t dft_tables(DftTables* tables, cudaStream_t stream) {
  static bool done[64] = {}, complete[64] = {};
  static DftTables addr[64] = {};
  static cudaEvent_t ready[64] = {};
  cudaError_t e;
  int dev = 0;
  if ((e = cudaGetDevice(&dev))) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!done[dev]) {
    void *p = nullptr, *p32 = nullptr;
    if ((e = cudaGetSymbolAddress(&p, g_dft_frag))) return e;
    if ((e = cudaGetSymbolAddress(&p32, g_dft_w32))) return e;
    if ((e = cudaEventCreateWithFlags(&ready[dev], cudaEventDisableTiming))) return e;
    dft_table_kernel<<<1, 256, 0, stream>>>();
    if ((e = cudaGetLastError())) return e;
    if ((e = cudaEventRecord(ready[dev], stream))) return e;
    addr[dev].frag = static_cast<const uint32_t*>(p);
    addr[dev].w32 = static_cast<const float*>(p32);
    done[dev] = true;
    count_launches(1);
  } else if (!complete[dev]) {
    // once the fill is known to have completed, no stream has to be ordered after it any more (the wait costs 2 us of host
    // time per call); relaxed mode, so that the query leaves another thread's stream capture alone
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    if ((e = cudaThreadExchangeStreamCaptureMode(&mode))) return e;
    const cudaError_t state = cudaEventQuery(ready[dev]);
    if ((e = cudaThreadExchangeStreamCaptureMode(&mode))) return e;
    if (state == cudaSuccess) complete[dev] = true;
    else if (state != cudaErrorNotReady) return state;
    else if ((e = cudaStreamWaitEvent(stream, ready[dev], 0))) return e;
  }
  *tables = addr[dev];
  return cudaSuccess;
}

template <typename T>
static cudaError_t launch_encode_t(const KSrc& src, int64_t T_tokens, const CacheView& cv, int layer0, int n_slabs,
                                   int slabs_per_layer, int chunk, int64_t kgroup0, const MinMaxBuffers& mm, cudaStream_t stream) {
  cudaError_t e;
  DftTables tables;
  if ((e = dft_tables(&tables, stream))) return e;
  static int n_sms[64] = {};   // per device; 0 = the kernel's attributes are not set there yet
  constexpr int smem = enc_sm_bytes<T>();
  int dev = 0;
  if ((e = cudaGetDevice(&dev))) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (n_sms[dev] == 0) {
    if ((e = cudaFuncSetAttribute(k_encode_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem))) return e;
    if ((e = cudaDeviceGetAttribute(&n_sms[dev], cudaDevAttrMultiProcessorCount, dev))) return e;
  }
  const int64_t tiles_per_slab = (T_tokens + kEncTokens - 1) / kEncTokens;
  const int64_t total = tiles_per_slab * n_slabs;
  if (total <= 0) return cudaSuccess;
  if (total > INT32_MAX) return cudaErrorInvalidValue;
  const int blocks = static_cast<int>(std::min<int64_t>(total, 2 * n_sms[dev]));
  const int withhold = (g_debug_withhold == 1) ? 1 : 0;
  if (withhold) g_debug_withhold = 0;
  count_launches(1);
  return launch_dependent(k_encode_kernel<T>, dim3(blocks), dim3(kEncThreads), smem, stream, src, T_tokens, cv, layer0, slabs_per_layer, chunk,
                          kgroup0, mm, static_cast<int>(tiles_per_slab), static_cast<int>(total), withhold);
}

cudaError_t launch_encode_keys(int dtype, const KSrc& src, int64_t T_tokens, const CacheView& cv, int layer0, int n_slabs,
                               int slabs_per_layer, int chunk, int64_t kgroup0, const MinMaxBuffers& mm, cudaStream_t stream) {
  if (dtype == VIDKV_F16) return launch_encode_t<__half>(src, T_tokens, cv, layer0, n_slabs, slabs_per_layer, chunk, kgroup0, mm, stream);
  return launch_encode_t<__nv_bfloat16>(src, T_tokens, cv, layer0, n_slabs, slabs_per_layer, chunk, kgroup0, mm, stream);
}

}  // namespace vidkv
