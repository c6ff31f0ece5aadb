// Key encode pass of Algorithm 3 (MixQuant) for the general key formats: k other than 0.5, and the
// plain min/max 1-bit code of 1BitQuant's other branch at any k.  The default format (k = 0.5 with
// Eq. 5) has its own tensor-core encoder and never comes here.
//   anomalous slot j   (Eq. 4, n = 2)  s = (max - min) / 3, z = min, both rounded to binary16;
//                      code = clamp(rint((x - z) / s), 0, 3) with the float32 division as written.
//   normal channel i, plain mode (Eq. 4, n = 1)  s = max - min, z = min; code in {0, 1}.
//   spectrum column f, Eq. 5  X = orthonormal n1-point DFT of the token's normal channels (ascending
//                      channel order), Hermitian half: column 0 = Re X[0], 1 = Re X[n1 / 2],
//                      2 k = Re X[k], 2 k + 1 = Im X[k]; bit = [X >= 0], s = mean |X| over the group.
//                      The sums run in float64 (the scale then rounds once).
//
// What bounds it: the second read of the keys (256 bytes per token-head) plus about 250 warp instructions per
// 8 tokens; the kernel it replaces, one block per group with a thread per channel walking the tokens one by one,
// was bound by its serial per-thread loops.  Measured at 28 layers x 4 heads: k = 0.75 with Eq. 5, batch 2 x 6400
// tokens (binary16) 1382 -> 219 us; k = 0.25 plain, 12800 tokens (bfloat16) 498 -> 146 us.  Blocks are persistent and walk a contiguous range of 32-token
// groups, the next group's tile arriving (cp.async) while this one is coded.  Inside a block:
//   * warps 0-3 work on the channels in their own order, two at a time (thread = channel pair and half of the
//     tokens): min / max and the comparisons against the code thresholds (code_cut, no division per element)
//     take two channels per instruction, and a channel's codes end up as two 32-bit planes over the tokens;
//   * only those planes are gathered into slot order, one slot per lane, and turned into the layout's bytes by
//     a reduce-scatter (two-bit codes) or a bit transpose (one-bit codes) over the warp;
//   * in Eq. 5 mode a fifth warp owns the transform, one token per lane: a 32-point real FFT in registers (about
//     300 float64 operations a token instead of the 1024 of the matrix form).
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "quant_common.cuh"

namespace vidkv {

namespace {

constexpr int kGenRow = kD * 2 + 16;            // bytes of a staged token row: 16-byte pieces, rows four banks apart
constexpr int kFftChannels = 32;                // Eq. 5 comes here for k = 0.75 only
constexpr int kGenBlocksPlain = 8, kGenBlocksFft = 4;   // resident blocks per SM (register bound: 64 / 102 a thread)

__device__ __forceinline__ void gen_cp16(void* smem_dst, const void* gmem_src) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ uint32_t gen_prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}

// cos(2 pi j / 32), j = 0 .. 8
__device__ constexpr double kCos32[9] = {1.0, 0.98078528040323044913, 0.92387953251128675613, 0.83146961230254523708,
                                         0.70710678118654752440, 0.55557023301960222474, 0.38268343236508977173,
                                         0.19509032201612826785, 0.0};
__device__ constexpr double cos32(int j) {      // j in 0 .. 31
  return j <= 8 ? kCos32[j] : j <= 16 ? -kCos32[16 - j] : j <= 24 ? -kCos32[j - 16] : kCos32[32 - j];
}
__device__ constexpr double sin32(int j) { return cos32((j + 24) & 31); }

// In-place radix-2 decimation in frequency over 16 complex values (bit-reversed output order).
__device__ __forceinline__ void fft16(double (&re)[16], double (&im)[16]) {
#pragma unroll
  for (int half = 8; half >= 1; half >>= 1) {
#pragma unroll
    for (int base = 0; base < 16; base += 2 * half) {
#pragma unroll
      for (int i = 0; i < half; ++i) {
        const int a = base + i, b = a + half, tw = i * (16 / half);   // twiddle e^(-2 pi i tw / 32)
        const double ur = re[a], ui = im[a], vr = re[b], vi = im[b];
        re[a] = ur + vr; im[a] = ui + vi;
        const double dr = ur - vr, di = ui - vi;
        if (tw == 0) { re[b] = dr; im[b] = di; }
        else if (tw == 8) { re[b] = di; im[b] = -dr; }
        else {
          const double c = cos32(tw), s = sin32(tw);
          re[b] = dr * c + di * s;
          im[b] = di * c - dr * s;
        }
      }
    }
  }
}
__device__ constexpr int rev4(int k) { return ((k & 1) << 3) | ((k & 2) << 1) | ((k & 4) >> 1) | ((k & 8) >> 3); }

template <bool FFT> struct GenShared {
  alignas(16) uint8_t tile[2][kG * kGenRow];
  uint32_t mm[2][2][kD / 2];            // [token half][min, max][channel pair]
  uint16_t cut[3][kD];                  // code thresholds per channel
  uint16_t plane[2][kD][2];             // [bit of the code][channel][token half]: one bit per token
  uint8_t perm[kD], slot_of[kD];        // slot -> channel, channel -> slot
  double mag[FFT ? kFftChannels : 1][kG + 1];   // |X| per (spectrum column, token)
};

template <typename T, bool FFT>
__global__ void __launch_bounds__(FFT ? 160 : 128, FFT ? kGenBlocksFft : kGenBlocksPlain)
    k_encode_general_kernel(KSrc src, int groups_per_slab, int64_t total_groups, CacheView cv, int layer0, int slabs_per_layer,
                            int chunk, int64_t kgroup0) {
  __shared__ GenShared<FFT> sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const KeyFmt kf = cv.kf;
  const int n2 = kf.n2;
  const int64_t g_begin = total_groups * blockIdx.x / gridDim.x, g_end = total_groups * (blockIdx.x + 1) / gridDim.x;
  if (g_begin >= g_end) return;
  int slab = static_cast<int>(g_begin / groups_per_slab), g = static_cast<int>(g_begin - static_cast<int64_t>(slab) * groups_per_slab);
  int lslab = slab, lg = g;
  auto load_next = [&](int buf) {
    if (tid < 128) {
      const T* base = reinterpret_cast<const T*>(src.ptr) + (lslab / src.H) * src.stride_b + (lslab % src.H) * src.stride_h +
                      static_cast<int64_t>(lg) * kG * src.stride_t;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = (tid >> 4) + 8 * i, piece = tid & 15;
        gen_cp16(sh.tile[buf] + row * kGenRow + piece * 16, reinterpret_cast<const uint8_t*>(base + row * src.stride_t) + piece * 16);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (++lg == groups_per_slab) { lg = 0; ++lslab; }
  };
  load_next(0);
  int cur_slab = -1, buf = 0;
  uint8_t* slab_ptr = nullptr;
#pragma unroll 1
  for (int64_t gi = g_begin; gi < g_end; ++gi, buf ^= 1) {
    if (slab != cur_slab) {
      cur_slab = slab;
      const int layer = layer0 + slab / slabs_per_layer, bh = slab % slabs_per_layer;
      slab_ptr = cv.slab(layer, bh / cv.H_kv, bh % cv.H_kv);
      __syncthreads();                                     // the last group's readers of the channel order are done
      if (tid < kD) {
        const uint8_t c = slab_ptr[cv.chunk_table_offset + static_cast<int64_t>(chunk) * kChunkBytes + tid];
        sh.perm[tid] = c;
        sh.slot_of[c] = static_cast<uint8_t>(tid);
      }
    }
    uint8_t* kg = slab_ptr + cv.kgroup_offset + (kgroup0 + g) * kf.group_bytes;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                       // tile and channel order are there; the other buffer is free
    if (gi + 1 < g_end) load_next(buf ^ 1);
    const uint8_t* tile = sh.tile[buf];

    if (!FFT || warp < 4) {
      // ---- min / max of a channel pair over half of the tokens
      const int cp = tid & 63, half = (tid >> 6) & 1;
      uint32_t v[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = *reinterpret_cast<const uint32_t*>(tile + (16 * half + i) * kGenRow + cp * 4);
      uint32_t mn = v[0], mx = v[0];
#pragma unroll
      for (int i = 1; i < 16; ++i) { mn = Ops<T>::min2(mn, v[i]); mx = Ops<T>::max2(mx, v[i]); }
      sh.mm[half][0][cp] = mn;
      sh.mm[half][1][cp] = mx;
      asm volatile("bar.sync 1, 128;" ::: "memory");
      // ---- scale, zero point and thresholds of one channel
      {
        const int c = tid, slot = sh.slot_of[c];
        const bool two = slot < n2;
        if (two || !FFT) {
          const uint16_t* lo = reinterpret_cast<const uint16_t*>(sh.mm[0][0]);
          const float fmn = fminf(Ops<T>::to_float(lo[c]), Ops<T>::to_float(lo[2 * kD + c]));
          const float fmx = fmaxf(Ops<T>::to_float(lo[kD + c]), Ops<T>::to_float(lo[3 * kD + c]));
          const uint16_t sb = f2h_bits(__fdiv_rn(__fsub_rn(fmx, fmn), two ? 3.0f : 1.0f)), zb = f2h_bits(fmn);
          const float s = h2f(sb), z = h2f(zb);
          if (two) {
            reinterpret_cast<uint16_t*>(kg + kf.off_s2)[slot] = sb;
            reinterpret_cast<uint16_t*>(kg + kf.off_z2)[slot] = zb;
          } else {
            reinterpret_cast<uint16_t*>(kg + kf.off_s1)[slot - n2] = sb;
            reinterpret_cast<uint16_t*>(kg + kf.off_z1)[slot - n2] = zb;
          }
          sh.cut[0][c] = code_cut<T>(z, s, 1);
          if (two) {
            sh.cut[1][c] = code_cut<T>(z, s, 2);
            sh.cut[2][c] = code_cut<T>(z, s, 3);
          } else {                                         // one bit: no value reaches a second level
            sh.cut[1][c] = 0x7fffu;
            sh.cut[2][c] = 0x7fffu;
          }
        }
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      // ---- codes as bit planes over the tokens, two channels at a time (16 tokens in each half-word)
      {
        const uint32_t c1 = reinterpret_cast<const uint32_t*>(sh.cut[0])[cp], c2 = reinterpret_cast<const uint32_t*>(sh.cut[1])[cp],
                       c3 = reinterpret_cast<const uint32_t*>(sh.cut[2])[cp];
        uint32_t lo = 0u, hi = 0u;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const uint32_t m1 = Ops<T>::ge_mask(v[i], c1), m2 = Ops<T>::ge_mask(v[i], c2), m3 = Ops<T>::ge_mask(v[i], c3);
          lo |= (m1 ^ m2 ^ m3) & (0x00010001u << i);
          hi |= m2 & (0x00010001u << i);
        }
        sh.plane[0][2 * cp][half] = static_cast<uint16_t>(lo);
        sh.plane[0][2 * cp + 1][half] = static_cast<uint16_t>(lo >> 16);
        sh.plane[1][2 * cp][half] = static_cast<uint16_t>(hi);
        sh.plane[1][2 * cp + 1][half] = static_cast<uint16_t>(hi >> 16);
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (32 * warp < n2) {
        // ---- two-bit slots 32 warp + lane: contributions of the slot to its code bytes, then an OR over the four
        // slots of a byte (lanes ^ 4, ^ 2; each lane keeps two token sets), then the two parities join (lane ^ 1)
        const int c = sh.perm[32 * warp + lane];
        const uint32_t lo = *reinterpret_cast<const uint32_t*>(sh.plane[0][c]), hi = *reinterpret_cast<const uint32_t*>(sh.plane[1][c]);
        const int pos = (lane >> 1) & 3;
        const bool pb0 = (lane & 2) != 0, pb1 = (lane & 4) != 0, par = (lane & 1) != 0;
        uint32_t w[8], w1[4], w2[2];
#pragma unroll
        for (int tl = 0; tl < 8; ++tl)
          w[tl] = (((lo >> tl) & 0x01010101u) + 2u * ((hi >> tl) & 0x01010101u)) << (2 * pos);   // byte nt: token 8 nt + tl
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
        const uint32_t keep = par ? w2[1] : w2[0], recv = __shfl_xor_sync(0xffffffffu, par ? w2[0] : w2[1], 1);
        const uint32_t even = par ? recv : keep, odd = par ? keep : recv;       // bytes nt of the even / odd slots
        const int tl = 2 * pos + (par ? 1 : 0), r = lane >> 3;
        *reinterpret_cast<uint2*>(kg + 256 * warp + (4 * tl + r) * 8) = make_uint2(gen_prmt(even, odd, 0x5140u), gen_prmt(even, odd, 0x7362u));
      }
    }
    if (FFT ? warp == 4 : 32 * warp >= n2) {
      // ---- one-bit columns 32 blk + i: a word per token (bit i = column i) ...
      const int blk = FFT ? 0 : warp - (n2 >> 5);
      uint32_t bits;
      if (FFT) {
        double re[16], im[16];
        const uint8_t* row = tile + lane * kGenRow;
        const uint32_t* pw = reinterpret_cast<const uint32_t*>(sh.perm + n2);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint32_t four = pw[i];
          auto at = [&](int k) { return static_cast<double>(Ops<T>::to_float(*reinterpret_cast<const uint16_t*>(row + ((four >> (8 * k)) & 0xffu) * 2))); };
          re[2 * i] = at(0); im[2 * i] = at(1); re[2 * i + 1] = at(2); im[2 * i + 1] = at(3);
        }
        // 32 real values as 16 complex ones (even + i odd); X[k] = E[k] + e^(-2 pi i k / 32) O[k] from Z[k], Z[16 - k]
        fft16(re, im);
        bits = 0u;
        auto put = [&](int f, double x) {
          sh.mag[f][lane] = fabs(x);
          bits |= x >= 0.0 ? 1u << f : 0u;
        };
        put(0, re[0] + im[0]);
        put(1, re[0] - im[0]);
#pragma unroll
        for (int k = 1; k <= 8; ++k) {
          const int a = rev4(k), b = rev4(16 - k);
          const double er = 0.5 * (re[a] + re[b]), ei = 0.5 * (im[a] - im[b]);          // E[k]
          const double orr = 0.5 * (im[a] + im[b]), oi = -0.5 * (re[a] - re[b]);        // O[k]
          const double c = cos32(k), s = sin32(k);
          const double tr = orr * c + oi * s, ti = oi * c - orr * s;
          put(2 * k, er + tr);
          put(2 * k + 1, ei + ti);
          if (k < 8) {                                     // X[16 - k] = conj(E[k] - e^(-2 pi i k / 32) O[k])
            put(2 * (16 - k), er - tr);
            put(2 * (16 - k) + 1, ti - ei);
          }
        }
        __syncwarp();
        double sum = 0.0;                                  // lane = column: magnitudes in token order
#pragma unroll
        for (int t = 0; t < kG; ++t) sum += sh.mag[lane][t];
        const double mean = sum * (1.0 / kG) * 0.17677669529663688110;   // 1 / sqrt(32)
        reinterpret_cast<uint16_t*>(kg + kf.off_s1)[lane] = __half_as_ushort(__double2half(mean));
      } else {
        bits = *reinterpret_cast<const uint32_t*>(sh.plane[0][sh.perm[n2 + 32 * blk + lane]]);
        // 32 x 32 bit transpose over the warp: column words over tokens become token words over columns
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
      }
      // ... then byte r (columns 8 r .. 8 r + 7, first column in the highest bit) of the four tokens 8 nt + tl goes to
      // byte nt of word 4 tl + r: a 4 x 4 byte transpose over the lanes ^ 8, ^ 16
      uint32_t w = __brev(bits);
      w = gen_prmt(w, w, 0x0123u);                         // bit order turned within each byte
      {
        const bool up = (lane & 8) != 0;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, w, 8);
        w = up ? gen_prmt(y, w, 0x7351u) : gen_prmt(w, y, 0x6240u);   // lanes nt even: bytes (0, 2 of both), odd: (1, 3 of both)
      }
      {
        const bool up = (lane & 16) != 0;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, w, 16);
        w = up ? gen_prmt(y, w, 0x7632u) : gen_prmt(w, y, 0x5410u);
      }
      reinterpret_cast<uint32_t*>(kg + kf.off_bits1 + 128 * blk)[(lane & 7) * 4 + (lane >> 3)] = w;
    }
    if (++g == groups_per_slab) { g = 0; ++slab; }
  }
}

template <typename T, bool FFT>
cudaError_t launch_general_t(const KSrc& src, int64_t groups, int n_slabs, const CacheView& cv, int layer0, int slabs_per_layer,
                             int chunk, int64_t kgroup0, cudaStream_t stream) {
  const int64_t total = groups * n_slabs;
  const int sms = device_sm_count();
  if (sms < 1) return cudaErrorInvalidDevice;
  const int blocks = static_cast<int>(std::min<int64_t>(total, static_cast<int64_t>(sms) * (FFT ? kGenBlocksFft : kGenBlocksPlain)));
  k_encode_general_kernel<T, FFT><<<blocks, FFT ? 160 : 128, 0, stream>>>(src, static_cast<int>(groups), total, cv, layer0, slabs_per_layer,
                                                                          chunk, kgroup0);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_encode_keys_general(int dtype, const KSrc& src, int64_t T_tokens, const CacheView& cv, int layer0,
                                       int n_slabs, int slabs_per_layer, int chunk, int64_t kgroup0, cudaStream_t stream) {
  const int64_t groups = T_tokens / kG;
  if (groups <= 0 || n_slabs <= 0) return cudaSuccess;
  if (groups > INT32_MAX || n_slabs > 65535) return cudaErrorInvalidValue;
  const bool fft = !cv.kf.plain && cv.kf.n2 < kD;
  if (fft && kD - cv.kf.n2 != kFftChannels) return cudaErrorInvalidValue;
  if (dtype == VIDKV_F16)
    return fft ? launch_general_t<__half, true>(src, groups, n_slabs, cv, layer0, slabs_per_layer, chunk, kgroup0, stream)
               : launch_general_t<__half, false>(src, groups, n_slabs, cv, layer0, slabs_per_layer, chunk, kgroup0, stream);
  return fft ? launch_general_t<__nv_bfloat16, true>(src, groups, n_slabs, cv, layer0, slabs_per_layer, chunk, kgroup0, stream)
             : launch_general_t<__nv_bfloat16, false>(src, groups, n_slabs, cv, layer0, slabs_per_layer, chunk, kgroup0, stream);
}

}  // namespace vidkv
