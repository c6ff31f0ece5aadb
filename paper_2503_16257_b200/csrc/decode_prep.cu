// Query preparation of the decode attention (Algorithm 1 "Decoding", Eq. 3): per (slab, chunk)
// the register images of the query that the stream kernels (decode_stream.cu) multiply with the
// packed key codes.  Everything that depends on the query alone is done here, once per chunk:
//   anomalous channels  sum_j q_j (s_j code_j + z_j): the kernels need q at the chunk's 2-bit
//       channels, in the order of the MMA fragments;
//   normal channels     K' = IDFT(+-s), so q . K'_t = sum_f Q_f s_f (+-1) with Q the weighted
//       forward transform of the permuted query, computed here on the tensor cores against the
//       split-precision DFT matrix the encoder uses.
// The step's append of k_new / v_new to the residual rides on this kernel.
#include "decode_common.cuh"

namespace vidkv {

constexpr int kPrepThreads = 128;

size_t decode_prep_bytes(int64_t n_slabs, int64_t n_chunks) {
  return static_cast<size_t>(n_slabs) * n_chunks * kPrepWords * 32 * sizeof(uint32_t);
}

// ---------------------------------------------------------------------------------
// Query preparation: one block of four warps per (chunk, slab), each a quarter of the words.  Writes, per lane, the 24 register images the
// attention kernel needs for this chunk's channel split:
//   words  j < 8  binary16 pairs of q at the anomalous slots (8 j + 2 r, 8 j + 2 r + 1)
//   words  8 + j  leading binary16 part of the transformed query Q at the spectrum
//                 columns (c, c + 1), c = 16 (j / 2) + 14 - 8 (j % 2) - 2 r
//   words 16 + j  binary16 remainder Q - leading part
//   word  24      float: softmax scale * log2 e * 2^(e + kQShift), which turns a score of this
//                 normalised query into a base-2 logit
// for head lane / 4 (zero when that head does not exist) and r = lane % 4, all of the query
// normalised by its head's power of two (head_exponent).
// Q_f = sum_c q_c W[c, f] with W the weights with which spectrum column f enters channel c of
// the inverse orthonormal 64-point transform of a Hermitian half spectrum: the forward DFT
// matrix, doubled for the columns f >= 2 that stand for a conjugate pair.  The product runs
// on the tensor cores against the same split-precision matrix fragments the encoder uses.
// What bounds it is latency (the stream kernel behind it waits for it): all loads that depend on nothing are under way before the
// first is used.
// ---------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(kPrepThreads) decode_prep_kernel(DecodeArgs a, int n_chunks) {
  const CacheView& cv = a.cv;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  pdl_release();                                           // the attention kernel may start its first copies now
  const int chunk = blockIdx.x % n_chunks, slab = blockIdx.x / n_chunks;
  const int hd = lane >> 2, r = lane & 3;
  const int h = slab % cv.H_kv, lb = slab / cv.H_kv;
  const int rep = cv.rep;
  uint8_t* sp = cv.slab(a.layer0 + lb / cv.B, lb % cv.B, h);
  const uint8_t* perm = sp + cv.chunk_table_offset + static_cast<int64_t>(chunk) * kChunkBytes;
  const T* qrow = reinterpret_cast<const T*>(a.q) + (static_cast<int64_t>(lb) * cv.H_q + h * rep + hd) * kD;
  const bool live = hd < rep;
  // the channel order of this warp's words and of the product's operand, the matrix fragments of its columns
  uint32_t two[2], pa[4], pb[4];
  uint4 bw[2][4];
#pragma unroll
  for (int x = 0; x < 2; ++x) two[x] = __ldg(reinterpret_cast<const uint16_t*>(perm + 8 * (2 * warp + x) + 2 * r));
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    pa[ks] = __ldg(reinterpret_cast<const uint16_t*>(perm + kNA + 16 * ks + 2 * r));
    pb[ks] = __ldg(reinterpret_cast<const uint16_t*>(perm + kNA + 16 * ks + 2 * r + 8));
#pragma unroll
    for (int x = 0; x < 2; ++x) bw[x][ks] = __ldg(reinterpret_cast<const uint4*>(a.dft.frag + ((ks * 8 + 2 * warp + x) * 32 + lane) * 4));
  }
  if (warp == 0 && chunk == 0 && a.append_row >= 0) {
    // Algorithm 1, Decoding: the step's new key / value row joins the residual (lanes 0-15 copy
    // the key row, 16-31 the value row); the attention kernel that follows reads it there.
    const uint4* srcp = reinterpret_cast<const uint4*>(lane < 16 ? a.k_new : a.v_new) + static_cast<int64_t>(slab) * 16 + (lane & 15);
    reinterpret_cast<uint4*>(sp + (lane < 16 ? cv.kres_offset : cv.vres_offset))[a.append_row * 16 + (lane & 15)] = __ldg(srcp);
  }
  const int qe = head_exponent<T, 4>(qrow, r, live);
  const float qf = pow2i(-qe - kQShift);                                   // normalised query, see head_exponent
  auto q_at = [&](uint32_t c) -> float { return live ? Elem<T>::to_float(qrow[c]) * qf : 0.0f; };
  uint32_t* out = a.prep + (static_cast<int64_t>(slab) * n_chunks + chunk) * (kPrepWords * 32) + lane;
  // anomalous slots
#pragma unroll
  for (int x = 0; x < 2; ++x) out[(2 * warp + x) * 32] = pack_half2(q_at(two[x] & 0xffu), q_at(two[x] >> 8));
  // transformed query: A = q at the normal channels (rows 8-15 unused), B = matrix fragments
  uint32_t af[4][2];
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    af[ks][0] = pack_half2(q_at(pa[ks] & 0xffu), q_at(pa[ks] >> 8));
    af[ks][1] = pack_half2(q_at(pb[ks] & 0xffu), q_at(pb[ks] >> 8));
  }
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const int nt = 2 * warp + x;
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      mma_f16(acc, af[ks][0], 0u, af[ks][1], 0u, bw[x][ks].x, bw[x][ks].y);
      mma_f16(acc, af[ks][0], 0u, af[ks][1], 0u, bw[x][ks].z, bw[x][ks].w);
    }
    // lane (hd, r) now holds Q of head hd at columns 16 r + 2 nt + {0, 1}: word 2 r + (nt < 4) of lane (hd, 3 - nt % 4)
    const float w0 = (r == 0 && nt == 0) ? 1.0f : 2.0f;            // columns 0 and 1 are not doubled
    const float x0 = acc[0] * w0, x1 = acc[1] * w0;
    const __half h0 = __float2half_rn(x0), h1 = __float2half_rn(x1);
    uint32_t* o = out + (8 + 2 * r + (nt < 4 ? 1 : 0)) * 32 + 3 - r - (nt & 3);
    o[0] = pack_half2(__half2float(h0), __half2float(h1));
    o[8 * 32] = pack_half2(x0 - __half2float(h0), x1 - __half2float(h1));
  }
  // factor that turns a score in the normalised units into a base-2 logit
  if (warp == 0) out[24 * 32] = __float_as_uint(a.scale * 1.4426950408889634f * pow2i(qe + kQShift));
}

// ---------------------------------------------------------------------------------
// The same for the general key formats (KeyFmt): a block of four warps per (chunk, slab), each a quarter of the pair words and of the sums
// over the normal channels, which meet in shared memory; per lane (head hd = lane / 4, r = lane % 4), all of the normalised query:
//   words w < n2/8              binary16 pairs of q at the two-bit slots 8 w + 2 r, + 1
//   then n1/8 words             plain mode: pairs of q at the one-bit channels 8 w + 6 - 2 r, + 1;
//                               Eq. 5: leading binary16 part of the transformed query Q at those columns,
//   then (Eq. 5) n1/8 words     binary16 remainder Q - leading part
//   word 24                     the factor that turns a score into a base-2 logit
// Q_f = sum_c q_c W[c, f], W = the weights with which column f of the Hermitian half spectrum enters
// normal channel c under the inverse orthonormal n1-point transform (columns >= 2 count twice), read from a
// table: computing sines and cosines here took 49 us of a decode step of 224 slabs, the table takes 13.
// ---------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(kPrepThreads) decode_prep_general_kernel(DecodeArgs a, int n_chunks) {
  __shared__ float part[3][8][32];                         // Eq. 5: the sums of warps 1-3, [column of the lane][lane]
  const CacheView& cv = a.cv;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  pdl_release();                                           // the attention kernel may start its first copies now
  const int chunk = blockIdx.x % n_chunks, slab = blockIdx.x / n_chunks;
  const int hd = lane >> 2, r = lane & 3;
  const int h = slab % cv.H_kv, lb = slab / cv.H_kv;
  const int rep = cv.rep;
  const int n2 = cv.kf.n2, n1 = kD - n2, w1 = n2 / 8;
  uint8_t* sp = cv.slab(a.layer0 + lb / cv.B, lb % cv.B, h);
  const uint8_t* perm = sp + cv.chunk_table_offset + static_cast<int64_t>(chunk) * kChunkBytes;
  const T* qrow = reinterpret_cast<const T*>(a.q) + (static_cast<int64_t>(lb) * cv.H_q + h * rep + hd) * kD;
  const bool live = hd < rep;
  // channels of this warp's words 4 i + warp: two-bit slots 8 w + 2 r, + 1, then (plain mode) one-bit channels 8 (w - w1) + 6 - 2 r, + 1
  const int n_pairs = cv.kf.plain ? kD / 8 : w1;
  uint32_t two[4], mine[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int w = 4 * i + warp;
    two[i] = w < n_pairs ? __ldg(reinterpret_cast<const uint16_t*>(perm + (w < w1 ? 8 * w + 2 * r : 8 * w + 6 - 2 * r))) : 0u;
  }
  // Eq. 5 (n1 = 32): the warp sums over the normal channels 8 warp .. + 7
  const bool fft = !cv.kf.plain && n1 > 0;
#pragma unroll
  for (int i = 0; i < 2; ++i) mine[i] = fft ? __ldg(reinterpret_cast<const uint32_t*>(perm + n2 + 8 * warp) + i) : 0u;
  if (warp == 0 && chunk == 0 && a.append_row >= 0) {
    const uint4* srcp = reinterpret_cast<const uint4*>(lane < 16 ? a.k_new : a.v_new) + static_cast<int64_t>(slab) * 16 + (lane & 15);
    reinterpret_cast<uint4*>(sp + (lane < 16 ? cv.kres_offset : cv.vres_offset))[a.append_row * 16 + (lane & 15)] = __ldg(srcp);
  }
  const int qe = head_exponent<T, 4>(qrow, r, live);
  const float qf = pow2i(-qe - kQShift);
  auto q_at = [&](uint32_t c) -> float { return live ? Elem<T>::to_float(qrow[c]) * qf : 0.0f; };
  uint32_t* out = a.prep + (static_cast<int64_t>(slab) * n_chunks + chunk) * (kPrepWords * 32) + lane;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int w = 4 * i + warp;
    if (w < n_pairs) out[w * 32] = pack_half2(q_at(two[i] & 0xffu), q_at(two[i] >> 8));
  }
  if (fft) {
    // lane r owns the columns 8 r .. 8 r + 7; the weights (norm and doubling included) come from the table
    float x[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    const float4* wt = reinterpret_cast<const float4*>(a.dft.w32) + 2 * r + 8 * (8 * warp);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const float qv = q_at((mine[c >> 2] >> (8 * (c & 3))) & 0xffu);
      const float4 wa = __ldg(wt + 8 * c), wb = __ldg(wt + 8 * c + 1);
      x[0] = fmaf(qv, wa.x, x[0]); x[1] = fmaf(qv, wa.y, x[1]); x[2] = fmaf(qv, wa.z, x[2]); x[3] = fmaf(qv, wa.w, x[3]);
      x[4] = fmaf(qv, wb.x, x[4]); x[5] = fmaf(qv, wb.y, x[5]); x[6] = fmaf(qv, wb.z, x[6]); x[7] = fmaf(qv, wb.w, x[7]);
    }
    if (warp > 0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) part[warp - 1][i][lane] = x[i];
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = ((x[i] + part[0][i][lane]) + part[1][i][lane]) + part[2][i][lane];
      uint32_t* outQ = out + (w1 + r) * 32 + 3 - r;            // columns 8 r + 2 w, + 1: word r of lane (hd, 3 - w)
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const __half h0 = __float2half_rn(x[2 * w]), h1 = __float2half_rn(x[2 * w + 1]);
        outQ[-w] = pack_half2(__half2float(h0), __half2float(h1));
        outQ[4 * 32 - w] = pack_half2(x[2 * w] - __half2float(h0), x[2 * w + 1] - __half2float(h1));
      }
    }
  }
  if (warp == 0) out[24 * 32] = __float_as_uint(a.scale * 1.4426950408889634f * pow2i(qe + kQShift));
}

cudaError_t launch_decode_prep(const DecodeArgs& a, cudaStream_t stream) {
  const int n_slabs = a.n_layers * a.cv.B * a.cv.H_kv;
  const int n_chunks = a.plan.n_chunks;
  if (n_chunks < 1) return cudaSuccess;
  const int n_items = n_slabs * n_chunks;
  if (a.cv.kf.general) {
    if (a.in_dtype == VIDKV_F16) decode_prep_general_kernel<__half><<<n_items, kPrepThreads, 0, stream>>>(a, n_chunks);
    else decode_prep_general_kernel<__nv_bfloat16><<<n_items, kPrepThreads, 0, stream>>>(a, n_chunks);
    count_launches(1);
    return cudaGetLastError();
  }
  if (a.in_dtype == VIDKV_F16) decode_prep_kernel<__half><<<n_items, kPrepThreads, 0, stream>>>(a, n_chunks);
  else decode_prep_kernel<__nv_bfloat16><<<n_items, kPrepThreads, 0, stream>>>(a, n_chunks);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace vidkv
