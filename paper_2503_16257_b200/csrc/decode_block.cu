// Decode attention over the packed cache (Algorithm 1 "Decoding", Eq. 3) in one launch, for calls of a few thousand
// 160-token units (five 32-token key groups) at most; plan_decode holds the rule.
//
// What bounds such a call is latency: launches, dependent loads, a unit's serial work and the merge of the partial
// results.  Against the stream kernel with its query preparation and merge kernels (one warp per unit), measured per call:
// one layer of 1632 tokens 20.7 -> 12.3 us, 6400 tokens 26.0 -> 15.7 us, 47000 tokens (1176 units) 133 -> 25 us.
//
// A block of five warps owns a contiguous stretch of units and walks it slab by slab:
//   query     the register images of the query for the slab's channel split (normalised query at
//             the 2-bit channels, its transform at the spectrum columns) are computed by the block
//             itself and kept in shared memory; a flushed chunk's images replace them when the walk
//             reaches it;
//   scores    warp g scores key group g of the unit: mma.sync.m16n8k16 with rows = query heads
//             (exact binary16 pair hi + lo), columns = tokens, the codes expanded in registers;
//   softmax   the unit's maxima per head meet in shared memory; the probabilities against them go to shared memory as
//             binary16, and the running output is brought to the unit's maximum before its P V joins;
//   P V       warps 0-3 own 32 channels each: the ternary plane is peeled digit by digit into
//             5 + trit and multiplied with the probabilities, the per-(group, channel) scales fold
//             the group accumulators into the warp's running output, eight registers a lane.
// The stages are pipelined over one block barrier per unit: after the barrier of unit i its
// probabilities are formed and P V of unit i - 1 runs, while the keys of unit i + 2 and the values
// of unit i + 1 arrive by bulk copies (cp.async.bulk + mbarrier).
//
// Caches with protected tokens (STPQuant, Algorithm 2): the values of a unit's tokens sit in two
// streams whose order differs from the key order (unprotected tokens: position = token - protected
// tokens before it, flushed tokens from the next group boundary on; protected ones in 2-bit groups of
// 32).  The probabilities are then scattered into two rings in stream order, one row per head, and a
// ternary supergroup (160 positions) or protected group (32) is multiplied once all of its positions
// are written.  Positions that belong to a neighbouring block stay zero; the neighbour multiplies the
// same bytes with its own probabilities.  The running maximum is kept integral (base-2) there, so that
// probabilities waiting in the rings are rescaled exactly when it moves.
//
// The FP16 / BF16 residual (and the step's append) belongs to the block that owns the slab's last
// unit, or to a block of its own where blocks own one unit each.  Blocks that share a slab leave
// records (maximum, sum, out[128] per head); whoever arrives last at a node of a tree of eight-way
// joins merges its children, and the root writes the output.
#include <type_traits>

#include "decode_device.cuh"

namespace vidkv {

namespace {

constexpr int kUnitWarps = 5;
constexpr int kUnitThreads = kUnitWarps * 32;
constexpr int kImgBytes = 32 * 32 * 4;                        // query images of one chunk
constexpr int kPRowBytes = kStreamUnitTokens * 2 + 16;        // a head's probabilities of one unit; rows in different banks
constexpr int kTRing = 512, kPRing = 512;                     // ring positions: an unfinished supergroup (group), two units and the gap
constexpr int kRingRow = (kTRing + kPRing) * 2 + 16;          // before the flushed tokens; rows in different banks
constexpr int kPBufs = 6;                                     // staged protected groups
constexpr int kResS = 132, kResP = 136;                       // row lengths of the residual's scores and probabilities
constexpr int kResScratch = 8 * kResS * 4 + 8 * kResP * 2;    // 6400

// Dynamic shared memory of a block, in bytes from a 128-byte boundary.
template <bool GEN, bool STP> struct Smem {
  static constexpr int kKBuf = GEN ? kGenKBufBytes : kKBufBytes;
  static constexpr int k_at = 0;                                       // two key buffers
  static constexpr int v_at = k_at + 2 * kKBuf;                        // two ternary buffers
  static constexpr int p_at = v_at + 2 * kVBufBytes;                   // protected groups (STP)
  static constexpr int img_at = p_at + (STP ? kPBufs * kPGBytes : 0);  // images of two chunks
  static constexpr int prob_at = img_at + 2 * kImgBytes;               // probabilities (STP: the rings); the residual's scratch
  static constexpr int prob_bytes = STP ? 8 * kRingRow : (2 * 8 * kPRowBytes > kResScratch ? 2 * 8 * kPRowBytes : kResScratch);
  static constexpr int bytes = prob_at + prob_bytes;
};

// Raw scores of one 32-token key group: sc[nt][0..1] = q . K' of head hd and tokens 8 nt + 2 r, + 1
// without the group's constant, which is returned in cst (the same for the 32 tokens), all in the
// units of the normalised query.  Consecutive products go to different accumulators (the four
// 8-token tiles, and the chain of the constants in between), so that no product waits for the
// one issued just before it.
__device__ __forceinline__ void score_group(const uint8_t* kg, int lane, int hd, int r, const uint4* img, float (&sc)[4][2], float& cst) {
  uint32_t s2[8], z2[8], s1[8];
  {
    const uint4 x0 = *reinterpret_cast<const uint4*>(kg + kKG_S2 + 32 * r);
    const uint4 x1 = *reinterpret_cast<const uint4*>(kg + kKG_S2 + 32 * r + 16);
    s2[0] = x0.x; s2[1] = x0.y; s2[2] = x0.z; s2[3] = x0.w; s2[4] = x1.x; s2[5] = x1.y; s2[6] = x1.z; s2[7] = x1.w;
    const uint8_t* zs = kg + ((hd & 1) ? kKG_S2 : kKG_Z2) + 32 * r;   // B operand of the constants: z for even columns, s for odd
    const uint4 y0 = *reinterpret_cast<const uint4*>(zs);
    const uint4 y1 = *reinterpret_cast<const uint4*>(zs + 16);
    z2[0] = y0.x; z2[1] = y0.y; z2[2] = y0.z; z2[3] = y0.w; z2[4] = y1.x; z2[5] = y1.y; z2[6] = y1.z; z2[7] = y1.w;
    const uint4 w0 = *reinterpret_cast<const uint4*>(kg + kKG_S1 + 32 * r);
    const uint4 w1 = *reinterpret_cast<const uint4*>(kg + kKG_S1 + 32 * r + 16);
    s1[0] = w0.x; s1[1] = w0.y; s1[2] = w0.z; s1[3] = w0.w; s1[4] = w1.x; s1[5] = w1.y; s1[6] = w1.z; s1[7] = w1.w;
  }
  const uint4 c2 = *reinterpret_cast<const uint4*>(kg + kKG_Codes2 + lane * 16);
  const uint2 c1 = *reinterpret_cast<const uint2*>(kg + kKG_Bits1 + lane * 8);
  const uint32_t w2[4] = {c2.x, c2.y, c2.z, c2.w};
  const uint32_t wh[4] = {c2.x >> 6, c2.y >> 6, c2.z >> 6, c2.w >> 6};   // fields 5-7 come from one right shift
  // sign bits: low lane <- bit 15 - 2 m, high lane <- bit 14 - 2 m of the token's half-word
  const uint32_t X[4] = {(c1.x & 0xffffu) * 0x00020001u, (c1.x >> 16) * 0x00020001u, (c1.y & 0xffffu) * 0x00020001u,
                         (c1.y >> 16) * 0x00020001u};
  float acc[4][4];
#pragma unroll
  for (int nt = 0; nt < 4; ++nt) { acc[nt][0] = 0.0f; acc[nt][1] = 0.0f; acc[nt][2] = 0.0f; acc[nt][3] = 0.0f; }
  // constants of the group: column 2 r of the result = sum q z, column 2 r + 1 = sum q s
  float cz[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  // anomalous channels: q s as exact binary16 pairs hi + lo against 4 + code
  {
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const uint4 qv = img[ks * 32];                       // (pair, 0, pair, 0): the operand as it stands
      mma_f16(cz, qv.x, qv.y, qv.z, qv.w, z2[2 * ks], z2[2 * ks + 1]);
      const uint32_t h0 = hmul2_u(qv.x, s2[2 * ks]), h1 = hmul2_u(qv.z, s2[2 * ks + 1]);
      const uint32_t l0 = hfms2_u(qv.x, s2[2 * ks], h0), l1 = hfms2_u(qv.z, s2[2 * ks + 1], h1);
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) {
        // fields 2 ks and 2 ks + 1 of the word: shifts by 8 - 4 ks and 6 - 4 ks bits
        const uint32_t f0 = ks == 0 ? w2[nt] << 8 : ks == 1 ? w2[nt] << 4 : ks == 2 ? w2[nt] : wh[nt] << 2;
        const uint32_t f1 = ks == 0 ? w2[nt] << 6 : ks == 1 ? w2[nt] << 2 : ks == 2 ? wh[nt] << 4 : wh[nt];
        mma_f16(acc[nt], h0, l0, h1, l1, field_or(f0, kFour),
                field_or(f1, kFour));
      }
    }
  }
  // normal channels in the frequency domain: Q (leading part + remainder, rows hd and hd + 8) against
  // +-s: the scale takes the sign inside the one logic instruction that used to make +-1, and the
  // products Q s are formed exactly by the tensor core
  {
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const uint4 qv = img[(4 + ks) * 32];
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
        mma_f16(acc[nt], qv.x, qv.y, qv.z, qv.w,
                signed_by(X[nt] << (4 * ks), s1[2 * ks]), signed_by(X[nt] << (4 * ks + 2), s1[2 * ks + 1]));
    }
  }
  cst = cz[0] - 4.0f * cz[1];
#pragma unroll
  for (int nt = 0; nt < 4; ++nt) {
    sc[nt][0] = acc[nt][0] + acc[nt][2];
    sc[nt][1] = acc[nt][1] + acc[nt][3];
  }
}

// The same for a key group in the general layout (KeyFmt): blocks of 32 two-bit slots, then blocks of
// 32 one-bit columns.  img points at this lane's query words of the group's chunk (four words, 32 uint4
// apart).  Two-bit slots as above (q s as hi + lo against 4 + code).  One-bit columns: Eq. 5 as above
// with the transformed query; in plain mode the value is code s + z = (+-1) s / 2 + (z + s / 2), so q s
// (hi + lo) meets +-1, the products are halved at the end and the constant takes sum q z + sum q s / 2.
__device__ __forceinline__ void score_group_general(const uint8_t* kg, const KeyFmt& kf, int lane, int hd, int r,
                                                    const uint4* img, float (&sc)[4][2], float& cst) {
  float acc[4][4], acc1[4][4];
#pragma unroll
  for (int nt = 0; nt < 4; ++nt) {
#pragma unroll
    for (int i = 0; i < 4; ++i) { acc[nt][i] = 0.0f; acc1[nt][i] = 0.0f; }
  }
  float cz[4] = {0.0f, 0.0f, 0.0f, 0.0f}, cz1[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  const int n2b = kf.n2 >> 5, n1b = (kD - kf.n2) >> 5;
#pragma unroll 1
  for (int b = 0; b < n2b; ++b) {
    uint32_t hi[4], lo[4];
    const uint4 qv = img[b * 32];
    const uint32_t qa[4] = {qv.x, qv.y, qv.z, qv.w};
    const uint4 sv = *reinterpret_cast<const uint4*>(kg + kf.off_s2 + 64 * b + 16 * r);
    const uint4 zv = *reinterpret_cast<const uint4*>(kg + ((hd & 1) ? kf.off_s2 : kf.off_z2) + 64 * b + 16 * r);
    const uint32_t sw[4] = {sv.x, sv.y, sv.z, sv.w}, zw[4] = {zv.x, zv.y, zv.z, zv.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      hi[j] = hmul2_u(qa[j], sw[j]);
      lo[j] = hfms2_u(qa[j], sw[j], hi[j]);
    }
    const uint2 cw = *reinterpret_cast<const uint2*>(kg + 256 * b + lane * 8);
    uint32_t W[4];
    W[0] = prmt(cw.x, 0u, 0x1404u); W[1] = prmt(cw.x, 0u, 0x3424u);
    W[2] = prmt(cw.y, 0u, 0x1404u); W[3] = prmt(cw.y, 0u, 0x3424u);
#pragma unroll
    for (int kp = 0; kp < 2; ++kp) {
      mma_f16(cz, qa[2 * kp], 0u, qa[2 * kp + 1], 0u, zw[2 * kp], zw[2 * kp + 1]);
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
        mma_f16(acc[nt], hi[2 * kp], lo[2 * kp], hi[2 * kp + 1], lo[2 * kp + 1], field_or(W[nt] >> (4 * kp), kFour),
                field_or(W[nt] >> (4 * kp + 2), kFour));
    }
  }
  const uint4* img1 = img + n2b * 32;
#pragma unroll 1
  for (int b = 0; b < n1b; ++b) {
    // the stored scale takes the sign of the code bit and goes to the tensor core as it is; the other
    // operand is the transformed query as hi + lo (Eq. 5) or the query itself (plain mode, exact in one piece)
    const uint4 hv = img1[b * 32];
    const uint32_t ah[4] = {hv.x, hv.y, hv.z, hv.w};
    uint32_t al[4] = {0u, 0u, 0u, 0u};
    const uint4 sv = *reinterpret_cast<const uint4*>(kg + kf.off_s1 + 64 * b + 16 * r);
    const uint32_t sw[4] = {sv.x, sv.y, sv.z, sv.w};
    if (kf.plain) {
      const uint4 zv = *reinterpret_cast<const uint4*>(kg + ((hd & 1) ? kf.off_s1 : kf.off_z1) + 64 * b + 16 * r);
      const uint32_t zw[4] = {zv.x, zv.y, zv.z, zv.w};
      mma_f16(cz1, ah[0], 0u, ah[1], 0u, zw[0], zw[1]);
      mma_f16(cz1, ah[2], 0u, ah[3], 0u, zw[2], zw[3]);
    } else {
      const uint4 lv = img1[(n1b + b) * 32];
      al[0] = lv.x; al[1] = lv.y; al[2] = lv.z; al[3] = lv.w;
    }
    const uint32_t cw = *reinterpret_cast<const uint32_t*>(kg + kf.off_bits1 + 128 * b + lane * 4);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      const uint32_t X = ((cw >> (8 * nt)) & 0xffu) * 0x02000100u;   // low lane: bit 7 at the sign, high lane: bit 6
#pragma unroll
      for (int kp = 0; kp < 2; ++kp)
        mma_f16(acc1[nt], ah[2 * kp], al[2 * kp], ah[2 * kp + 1], al[2 * kp + 1], signed_by(X << (4 * kp), sw[2 * kp]),
                signed_by(X << (4 * kp + 2), sw[2 * kp + 1]));
    }
  }
  const float f1 = kf.plain ? 0.5f : 1.0f;
  cst = cz[0] - 4.0f * cz[1] + (kf.plain ? cz1[0] + 0.5f * cz1[1] : 0.0f);
#pragma unroll
  for (int nt = 0; nt < 4; ++nt) {
    sc[nt][0] = acc[nt][0] + acc[nt][2] + f1 * (acc1[nt][0] + acc1[nt][2]);
    sc[nt][1] = acc[nt][1] + acc[nt][3] + f1 * (acc1[nt][1] + acc1[nt][3]);
  }
}

// ---------------------------------------------------------------------------------------------
// Query images of one chunk's channel split, by the whole block: word i of lane (head hd = lane / 4,
// r = lane % 4) at ((i / 4) * 32 + lane) * 4 + i % 4, so that four words are one 16-byte load:
//   words  2 i, i < 8       binary16 pair of q at the anomalous slots (16 r + 2 i, 16 r + 2 i + 1); 2 i + 1: zero
//   words 16 + 2 i          leading binary16 part of the transformed query Q at the spectrum columns
//                           (16 r + 2 i, 16 r + 2 i + 1)
//   words 16 + 2 i + 1      binary16 remainder Q - leading part
// so that the four words of a 16-byte load are the A operand of one k step as it stands; zero for heads that do not
// exist, all of the query normalised by its head's power of two (head_exponent).  Q_f = sum_c q_c W[c, f] with W the
// weights with which spectrum column f enters channel c of the inverse orthonormal 64-point transform of a Hermitian
// half spectrum: the forward DFT matrix, doubled for the columns f >= 2 that stand for a conjugate pair, on the tensor
// cores against the split-precision matrix fragments.  General key formats (KeyFmt):
//   words 0 .. n2/8 - 1         pairs of q at the two-bit slots 32 (w / 4) + 8 r + 2 (w % 4), + 1
//   then n1/8 words             plain mode: pairs of q at the one-bit channels with the same index rule;
//                               Eq. 5: leading binary16 part of Q at those columns,
//   then (Eq. 5) n1/8 words     the remainder (Q from the table of the 32-point transform)
// A block computes them once per slab it walks (and once per flushed chunk): about 1.5 us of latency
// behind the first bulk copies, where a kernel of its own takes 5-8 us of a step.
// ---------------------------------------------------------------------------------------------
template <bool GEN, typename T>
__device__ __forceinline__ void make_images(uint32_t* img, const KeyFmt& kf, const DftTables& dft, const uint8_t* perm, const T* qrow,
                                            bool live, float qf, int warp, int lane) {
  const int r = lane & 3;
  auto q_at = [&](uint32_t c) -> float { return live ? Elem<T>::to_float(qrow[c]) * qf : 0.0f; };
  auto put = [&](int i, uint32_t v) { img[((i >> 2) * 32 + lane) * 4 + (i & 3)] = v; };
  if (!GEN) {
    // transformed query: A = q at the normal channels (rows 8-15 unused), B = matrix fragments
    uint32_t af[4][2];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const uint32_t pa = __ldg(reinterpret_cast<const uint16_t*>(perm + kNA + 16 * ks + 2 * r));
      const uint32_t pb = __ldg(reinterpret_cast<const uint16_t*>(perm + kNA + 16 * ks + 2 * r + 8));
      af[ks][0] = pack_half2(q_at(pa & 0xffu), q_at(pa >> 8));
      af[ks][1] = pack_half2(q_at(pb & 0xffu), q_at(pb >> 8));
    }
#pragma unroll 1
    for (int nt = warp; nt < 8; nt += kUnitWarps) {
      const uint32_t two = __ldg(reinterpret_cast<const uint16_t*>(perm + 16 * r + 2 * nt));
      float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        const uint4 bw = __ldg(reinterpret_cast<const uint4*>(dft.frag + ((ks * 8 + nt) * 32 + lane) * 4));
        mma_f16(acc, af[ks][0], 0u, af[ks][1], 0u, bw.x, bw.y);
        mma_f16(acc, af[ks][0], 0u, af[ks][1], 0u, bw.z, bw.w);
      }
      // lane (hd, r) now holds Q of head hd at columns 16 r + 2 nt + {0, 1}
      const float w0 = (r == 0 && nt == 0) ? 1.0f : 2.0f;            // columns 0 and 1 are not doubled
      const float x0 = acc[0] * w0, x1 = acc[1] * w0;
      const __half h0 = __float2half_rn(x0), h1 = __float2half_rn(x1);
      put(2 * nt, pack_half2(q_at(two & 0xffu), q_at(two >> 8)));
      put(2 * nt + 1, 0u);
      put(16 + 2 * nt, pack_half2(__half2float(h0), __half2float(h1)));
      put(17 + 2 * nt, pack_half2(x0 - __half2float(h0), x1 - __half2float(h1)));
    }
  } else {
    const int n2 = kf.n2, n1 = kD - n2, w1 = n2 / 8, n_pairs = kf.plain ? kD / 8 : w1;
#pragma unroll 1
    for (int w = warp; w < n_pairs; w += kUnitWarps) {
      const int j = (w < w1 ? 0 : n2) + 32 * ((w < w1 ? w : w - w1) >> 2) + 8 * r + 2 * (w & 3);
      put(w, pack_half2(q_at(perm[j]), q_at(perm[j + 1])));
    }
    if (!kf.plain && n1 > 0 && warp == kUnitWarps - 1) {
      // n1 = 32: lane r owns the columns 8 r .. 8 r + 7
      float x[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
      const float4* wt = reinterpret_cast<const float4*>(dft.w32) + 2 * r;
#pragma unroll 4
      for (int c = 0; c < 32; ++c) {
        const float qv = q_at(perm[n2 + c]);
        const float4 wa = __ldg(wt + 8 * c), wb = __ldg(wt + 8 * c + 1);
        x[0] = fmaf(qv, wa.x, x[0]); x[1] = fmaf(qv, wa.y, x[1]); x[2] = fmaf(qv, wa.z, x[2]); x[3] = fmaf(qv, wa.w, x[3]);
        x[4] = fmaf(qv, wb.x, x[4]); x[5] = fmaf(qv, wb.y, x[5]); x[6] = fmaf(qv, wb.z, x[6]); x[7] = fmaf(qv, wb.w, x[7]);
      }
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const __half h0 = __float2half_rn(x[2 * w]), h1 = __float2half_rn(x[2 * w + 1]);
        put(w1 + w, pack_half2(__half2float(h0), __half2float(h1)));
        put(w1 + 4 + w, pack_half2(x[2 * w] - __half2float(h0), x[2 * w + 1] - __half2float(h1)));
      }
    }
  }
}

// Running softmax of the block's part of one slab.  m (head lane / 4) is the same in every warp; o and l belong
// to warps 0-3: o[4 i + c] = channel 32 w + 4 (lane / 4) + 2 i + c / 2, head 2 (lane % 4) + c % 2.
struct Running {
  float m;             // reference: o and l are in units of 2^m
  float exact;         // the largest unit maximum so far
  float l[2];
  float o[8];
  __device__ __forceinline__ void reset() {
    m = -INFINITY; exact = -INFINITY; l[0] = 0.0f; l[1] = 0.0f;
#pragma unroll
    for (int j = 0; j < 8; ++j) o[j] = 0.0f;
  }
  __device__ __forceinline__ void scale(float fa, float fb) {
    l[0] *= fa; l[1] *= fb;
#pragma unroll
    for (int j = 0; j < 8; j += 2) { o[j] *= fa; o[j + 1] *= fb; }
  }
  // Reference of tokens whose largest base-2 logit is mu: their own maximum (kRefLag: see there).  Returns the factor that
  // brings the sums so far to it.
  __device__ __forceinline__ float refer_to(float mu) {
    exact = fmaxf(exact, mu);
    const float ref = fmaxf(mu, exact - kRefLag), f = ex2_approx(m - ref);    // 0 at the start of a slab (m = -inf)
    m = ref;
    return f;
  }
};

// P V of one staged ternary supergroup for the 32 channels of warp w (two MMA row blocks: fragment i covers channels
// 32 w + 4 hd + 2 i + {0, 1} in rows hd, hd + 8).  P(g, nt) = probabilities of head hd at the supergroup's tokens
// 32 g + 8 nt + 2 r, + 1 (binary16 pair); ps[g] = -5 * (sum of the group's probabilities) of heads 2 r, 2 r + 1, twice:
// the accumulator fragment P V starts from.
template <typename PFrag>
__device__ __forceinline__ void pv_ternary(const uint8_t* vbuf, int w, PFrag P, const float4 (&ps)[kSGGroups], Running& run, int hd,
                                           int r) {
  uint32_t W[2][8];
#pragma unroll
  for (int kt = 0; kt < 2; ++kt) {
    const uint2 wa = *reinterpret_cast<const uint2*>(vbuf + ((((kt * 2 + 0) * 4 + w) * 4 + r) * 8 + hd) * 8);
    const uint2 wb = *reinterpret_cast<const uint2*>(vbuf + ((((kt * 2 + 1) * 4 + w) * 4 + r) * 8 + hd) * 8);
    W[kt][0] = prmt(wa.x, 0u, 0x4140u); W[kt][1] = prmt(wa.x, 0u, 0x4342u);
    W[kt][2] = prmt(wb.x, 0u, 0x4140u); W[kt][3] = prmt(wb.x, 0u, 0x4342u);
    W[kt][4] = prmt(wa.y, 0u, 0x4140u); W[kt][5] = prmt(wa.y, 0u, 0x4342u);
    W[kt][6] = prmt(wb.y, 0u, 0x4140u); W[kt][7] = prmt(wb.y, 0u, 0x4342u);
#pragma unroll
    for (int k = 0; k < 8; ++k) W[kt][k] = mad_u32(W[kt][k], 3u, 0u);          // 3 * byte per 16-bit lane
  }
#pragma unroll
  for (int g = 0; g < kSGGroups; ++g) {
    float acc[2][4];
#pragma unroll
    for (int kt = 0; kt < 2; ++kt) {
      uint32_t A[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        // W holds 3 * (remaining byte) per 16-bit lane; the digit sits at bits 8-9.
        // Next W = 3 * (W - digit << 8) = 3 W - 3 A + 3 * 0x4400 (no lane ever borrows).
        // Half of the lanes take that route (two multiply-adds), the other half mask the digit
        // away and multiply (one logic, one multiply-add): the two pipes share the work.
        A[k] = field_or(W[kt][k], kFour);
        if (g + 1 < kSGGroups) {
          if (k & 1) W[kt][k] = mad_u32(A[k], 0xfffffffdu, mad_u32(W[kt][k], 3u, 0xcc00cc00u));
          else W[kt][k] = mad_u32(W[kt][k] & 0x00ff00ffu, 3u, 0u);
        }
      }
      const uint32_t b0 = P(g, 2 * kt), b1 = P(g, 2 * kt + 1);
      if (kt == 0) {
        mma_f16_c(acc[0], A[0], A[1], A[2], A[3], b0, b1, ps[g].x, ps[g].y, ps[g].z, ps[g].w);
        mma_f16_c(acc[1], A[4], A[5], A[6], A[7], b0, b1, ps[g].x, ps[g].y, ps[g].z, ps[g].w);
      } else {
        mma_f16(acc[0], A[0], A[1], A[2], A[3], b0, b1);
        mma_f16(acc[1], A[4], A[5], A[6], A[7], b0, b1);
      }
    }
    const uint2 sc2 = *reinterpret_cast<const uint2*>(vbuf + kSG_Scales + g * (kD * 2) + (32 * w + 4 * hd) * 2);
    const float2 sa = __half22float2(*reinterpret_cast<const __half2*>(&sc2.x));
    const float2 sb = __half22float2(*reinterpret_cast<const __half2*>(&sc2.y));
    run.o[0] = fmaf(sa.x, acc[0][0], run.o[0]); run.o[1] = fmaf(sa.x, acc[0][1], run.o[1]);
    run.o[2] = fmaf(sa.y, acc[0][2], run.o[2]); run.o[3] = fmaf(sa.y, acc[0][3], run.o[3]);
    run.o[4] = fmaf(sb.x, acc[1][0], run.o[4]); run.o[5] = fmaf(sb.x, acc[1][1], run.o[5]);
    run.o[6] = fmaf(sb.y, acc[1][2], run.o[6]); run.o[7] = fmaf(sb.y, acc[1][3], run.o[7]);
    run.l[0] = fmaf(-0.2f, ps[g].x, run.l[0]);
    run.l[1] = fmaf(-0.2f, ps[g].y, run.l[1]);
  }
}

// P V of one protected group (Eq. 4 codes as 4 + code) for the 32 channels of warp w: P4[nt] = probabilities of
// head hd at the group's tokens 8 nt + 2 r, + 1.  out += s * (sum (4 + code) p - 4 sum p) + z * sum p.
__device__ __forceinline__ void pv_protected(const uint8_t* pg, int w, const uint32_t (&P4)[4], Running& run, int hd, int r) {
  float cq[4] = {0.0f, 0.0f, 0.0f, 0.0f};               // -4 * (sum of the probabilities) of heads 2 r, 2 r + 1
  mma_f16(cq, kMinus4, kMinus4, kMinus4, kMinus4, P4[0], P4[1]);
  mma_f16(cq, kMinus4, kMinus4, kMinus4, kMinus4, P4[2], P4[3]);
  const float sp0 = -0.25f * cq[0], sp1 = -0.25f * cq[1];
  run.l[0] += sp0; run.l[1] += sp1;
  const int w_off = (((w * 4) + r) * 8 + hd) * 4, m_off = (32 * w + 4 * hd) * 2;
  const uint32_t wk[2] = {*reinterpret_cast<const uint32_t*>(pg + w_off), *reinterpret_cast<const uint32_t*>(pg + 512 + w_off)};
  const uint2 sc = *reinterpret_cast<const uint2*>(pg + kPG_S + m_off);
  const uint2 zc = *reinterpret_cast<const uint2*>(pg + kPG_Z + m_off);
  float acc[2][4];
#pragma unroll
  for (int kt = 0; kt < 2; ++kt) {
    const uint32_t wd = wk[kt], wh = wd >> 6;
    uint32_t x[8];
    x[0] = field_or(wd << 8, kFour);
    x[1] = field_or(wd << 6, kFour);
    x[2] = field_or(wd << 4, kFour);
    x[3] = field_or(wd << 2, kFour);
    x[4] = field_or(wd, kFour);
    x[5] = field_or(wh << 4, kFour);
    x[6] = field_or(wh << 2, kFour);
    x[7] = field_or(wh, kFour);
    const uint32_t b0 = P4[2 * kt], b1 = P4[2 * kt + 1];
    if (kt == 0) {
      mma_f16_c(acc[0], x[0], x[1], x[4], x[5], b0, b1, cq[0], cq[1], cq[2], cq[3]);
      mma_f16_c(acc[1], x[2], x[3], x[6], x[7], b0, b1, cq[0], cq[1], cq[2], cq[3]);
    } else {
      mma_f16(acc[0], x[0], x[1], x[4], x[5], b0, b1);
      mma_f16(acc[1], x[2], x[3], x[6], x[7], b0, b1);
    }
  }
  const float2 sa = __half22float2(*reinterpret_cast<const __half2*>(&sc.x));
  const float2 sb = __half22float2(*reinterpret_cast<const __half2*>(&sc.y));
  const float2 za = __half22float2(*reinterpret_cast<const __half2*>(&zc.x));
  const float2 zb = __half22float2(*reinterpret_cast<const __half2*>(&zc.y));
  run.o[0] += sa.x * acc[0][0] + za.x * sp0; run.o[1] += sa.x * acc[0][1] + za.x * sp1;
  run.o[2] += sa.y * acc[0][2] + za.y * sp0; run.o[3] += sa.y * acc[0][3] + za.y * sp1;
  run.o[4] += sb.x * acc[1][0] + zb.x * sp0; run.o[5] += sb.x * acc[1][1] + zb.x * sp1;
  run.o[6] += sb.y * acc[1][2] + zb.y * sp0; run.o[7] += sb.y * acc[1][3] + zb.y * sp1;
}

// The integral running maximum follows a maximum `mu` (base-2 logit of head lane / 4) that exceeds it by more than
// kStaleLog2: true if some head's moved, with the factors of heads 2 r, 2 r + 1 and of the lane's own head.
__device__ __forceinline__ bool move_maximum(float mu, int r, float& m, float& fa, float& fb, float& f) {
  const bool up = mu > m + kStaleLog2;                      // always true at the start of a slab (m = -inf)
  if (!__any_sync(0xffffffffu, up)) return false;
  const float m_new = up ? ceilf(mu) : m;
  f = ex2_approx(m - m_new);                                // 1 for heads whose maximum stays
  m = m_new;
  fa = __shfl_sync(0xffffffffu, f, 8 * r);
  fb = __shfl_sync(0xffffffffu, f, 8 * r + 4);
  return true;
}

// Algorithm 1, Decoding: the step's new key / value row joins the residual (lanes 0-15 copy the key row, 16-31 the value
// row).  One warp.
__device__ __forceinline__ void append_row(const DecodeArgs& a, int slab, uint8_t* slab_ptr, int lane) {
  if (a.append_row < 0) return;
  const uint4* srcp = reinterpret_cast<const uint4*>(lane < 16 ? a.k_new : a.v_new) + static_cast<int64_t>(slab) * 16 + (lane & 15);
  reinterpret_cast<uint4*>(slab_ptr + (lane < 16 ? a.cv.kres_offset : a.cv.vres_offset))[a.append_row * 16 + (lane & 15)] = __ldg(srcp);
}

// The slab's residual rows (n_res of them, the step's new row among them: append_row by warp 0 first) in the input type: scores on the tensor
// cores straight from global memory (the contraction may take the channels in any order: lane (token hd, r) reads
// 16-byte pieces, two k steps each), probabilities through `scratch`, P V with the two tokens of an operand register
// brought together from two rows.  Whole block; scratch as large as kResScratch.
template <typename T>
__device__ __forceinline__ void add_residual(const DecodeArgs& a, const uint8_t* slab_ptr, const T* qrow, bool live, uint8_t* scratch, int warp,
                                             int lane, Running& run) {
  const CacheView& cv = a.cv;
  const int hd = lane >> 2, r = lane & 3, n_res = a.st.n_res;
  float* Sx = reinterpret_cast<float*>(scratch);
  __half* Px = reinterpret_cast<__half*>(scratch + 8 * kResS * 4);
  uint4 qn[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) qn[j] = live ? __ldg(reinterpret_cast<const uint4*>(qrow + 32 * j + 8 * r)) : make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();                                         // the row is there, and nobody uses the scratch memory any more
  const uint8_t* kr = slab_ptr + cv.kres_offset;
  const float sl2 = a.scale * 1.4426950408889634f;
  for (int tile = warp; tile * 8 < n_res; tile += kUnitWarps) {
    const int row = min(tile * 8 + hd, n_res - 1);
    uint4 kv[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) kv[j] = *reinterpret_cast<const uint4*>(kr + row * (kD * 2) + 64 * j + 16 * r);
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      mma_in<T>(acc, qn[j].x, qn[j].y, kv[j].x, kv[j].y);
      mma_in<T>(acc, qn[j].z, qn[j].w, kv[j].z, kv[j].w);
    }
    *reinterpret_cast<float2*>(Sx + hd * kResS + tile * 8 + 2 * r) = make_float2(acc[0] * sl2, acc[1] * sl2);
  }
  __syncthreads();
  float mu = -INFINITY;
  for (int t = r; t < n_res; t += 4) mu = fmaxf(mu, Sx[hd * kResS + t]);
  mu = fmaxf(mu, __shfl_xor_sync(0xffffffffu, mu, 1));
  mu = fmaxf(mu, __shfl_xor_sync(0xffffffffu, mu, 2));
  const float f = run.refer_to(mu);
  run.scale(__shfl_sync(0xffffffffu, f, 8 * r), __shfl_sync(0xffffffffu, f, 8 * r + 4));
  const int n_pad = (n_res + 15) & ~15;
  for (int t = 8 * r + 32 * warp; warp < 4 && t < n_pad; t += kR) {
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int t0 = t + 2 * j;
      w[j] = pack_half2(t0 < n_res ? ex2_approx(Sx[hd * kResS + t0] - run.m) : 0.0f, t0 + 1 < n_res ? ex2_approx(Sx[hd * kResS + t0 + 1] - run.m) : 0.0f);
    }
    *reinterpret_cast<uint4*>(Px + hd * kResP + t) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  __syncthreads();
  if (warp < 4) {
    const uint8_t* vr = slab_ptr + cv.vres_offset + (32 * warp + 4 * hd) * 2;
    float acc[2][4] = {{0.0f, 0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f, 0.0f}}, ps[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int t = 0; t < n_pad; t += 16) {
      const uint32_t b0 = *reinterpret_cast<const uint32_t*>(Px + hd * kResP + t + 2 * r);
      const uint32_t b1 = *reinterpret_cast<const uint32_t*>(Px + hd * kResP + t + 2 * r + 8);
      uint2 v[4];                                          // tokens 2 r, 2 r + 1, 2 r + 8, 2 r + 9
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        v[j] = *reinterpret_cast<const uint2*>(vr + (t + 2 * r + (j & 1) + 8 * (j >> 1)) * (kD * 2));
        if (!std::is_same<T, __half>::value) {             // bfloat16 values -> binary16 (exact for the admitted inputs)
          const float2 x = Elem<T>::to_float2(v[j].x), y = Elem<T>::to_float2(v[j].y);
          v[j] = make_uint2(pack_half2(x.x, x.y), pack_half2(y.x, y.y));
        }
        // rows past the residual's end hold whatever the ring held before: their probabilities are zero, but a
        // value that is not a finite binary16 would still poison the product
        if (t + 2 * r + (j & 1) + 8 * (j >> 1) >= n_res) v[j] = make_uint2(0u, 0u);
      }
      mma_f16(ps, kMinus5, kMinus5, kMinus5, kMinus5, b0, b1);
      mma_f16(acc[0], prmt(v[0].x, v[1].x, 0x5410u), prmt(v[0].x, v[1].x, 0x7632u), prmt(v[2].x, v[3].x, 0x5410u),
              prmt(v[2].x, v[3].x, 0x7632u), b0, b1);
      mma_f16(acc[1], prmt(v[0].y, v[1].y, 0x5410u), prmt(v[0].y, v[1].y, 0x7632u), prmt(v[2].y, v[3].y, 0x5410u),
              prmt(v[2].y, v[3].y, 0x7632u), b0, b1);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) run.o[j] += acc[j >> 2][j & 3];
    run.l[0] = fmaf(-0.2f, ps[0], run.l[0]);
    run.l[1] = fmaf(-0.2f, ps[1], run.l[1]);
  }
}

// ---- records and their joins.  A record: m [8], l [8], o [8][128]; lane (hd, r) of warp w < 4 moves heads 2 r, 2 r + 1,
// channels 32 w + 4 hd .. + 3.
struct Part {
  float m[2], l[2], o[8];       // o[4 i + c] as in Running
};
__device__ __forceinline__ void store_record(float* rec, const Part& p, int w, int hd, int r) {
  if (w == 0 && hd == 0) {
    *reinterpret_cast<float2*>(rec + 2 * r) = make_float2(p.m[0], p.m[1]);
    *reinterpret_cast<float2*>(rec + 8 + 2 * r) = make_float2(p.l[0], p.l[1]);
  }
  float* o = rec + 16 + 2 * r * kD + 32 * w + 4 * hd;
  *reinterpret_cast<float4*>(o) = make_float4(p.o[0], p.o[2], p.o[4], p.o[6]);
  *reinterpret_cast<float4*>(o + kD) = make_float4(p.o[1], p.o[3], p.o[5], p.o[7]);
}
// Join of n <= kJoin records `stride` floats apart.
__device__ __forceinline__ void join_records(const float* rec, int64_t stride, int n, Part& p, int w, int hd, int r) {
  float2 m[kJoin];
#pragma unroll
  for (int j = 0; j < kJoin; ++j) m[j] = j < n ? __ldcg(reinterpret_cast<const float2*>(rec + j * stride + 2 * r)) : make_float2(-INFINITY, -INFINITY);
  p.m[0] = m[0].x; p.m[1] = m[0].y;
#pragma unroll
  for (int j = 1; j < kJoin; ++j) { p.m[0] = fmaxf(p.m[0], m[j].x); p.m[1] = fmaxf(p.m[1], m[j].y); }
  p.l[0] = 0.0f; p.l[1] = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) p.o[i] = 0.0f;
#pragma unroll
  for (int j0 = 0; j0 < kJoin; j0 += 4) {
    if (j0 >= n) break;
    float2 l[4];
    float4 oa[4], ob[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float* q = rec + (j0 + j < n ? j0 + j : 0) * stride;
      l[j] = __ldcg(reinterpret_cast<const float2*>(q + 8 + 2 * r));
      oa[j] = __ldcg(reinterpret_cast<const float4*>(q + 16 + 2 * r * kD + 32 * w + 4 * hd));
      ob[j] = __ldcg(reinterpret_cast<const float4*>(q + 16 + (2 * r + 1) * kD + 32 * w + 4 * hd));
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float wa = exp2f(m[j0 + j].x - p.m[0]), wb = exp2f(m[j0 + j].y - p.m[1]);   // 0 for a record that does not exist
      p.l[0] = fmaf(wa, l[j].x, p.l[0]); p.l[1] = fmaf(wb, l[j].y, p.l[1]);
      p.o[0] = fmaf(wa, oa[j].x, p.o[0]); p.o[2] = fmaf(wa, oa[j].y, p.o[2]); p.o[4] = fmaf(wa, oa[j].z, p.o[4]); p.o[6] = fmaf(wa, oa[j].w, p.o[6]);
      p.o[1] = fmaf(wb, ob[j].x, p.o[1]); p.o[3] = fmaf(wb, ob[j].y, p.o[3]); p.o[5] = fmaf(wb, ob[j].z, p.o[5]); p.o[7] = fmaf(wb, ob[j].w, p.o[7]);
    }
  }
}
// The slab's result: the normalised output, or (token shards) maximum, sum and unnormalised output.
__device__ __forceinline__ void store_result(const DecodeArgs& a, int slab, const Part& p, int w, int hd, int r) {
  const CacheView& cv = a.cv;
  const int64_t row0 = static_cast<int64_t>(slab / cv.H_kv) * cv.H_q + (slab % cv.H_kv) * cv.rep;
  const int c0 = 32 * w + 4 * hd;
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const int head = 2 * r + x;
    if (head >= cv.rep) continue;
    if (a.partial_out) {
      float* pr = a.partial_out + (row0 + head) * kRecordFloats;
      if (w == 0 && hd == 0) *reinterpret_cast<float2*>(pr) = make_float2(p.m[x], p.l[x]);
      *reinterpret_cast<float2*>(pr + 2 + c0) = make_float2(p.o[x], p.o[2 + x]);
      *reinterpret_cast<float2*>(pr + 4 + c0) = make_float2(p.o[4 + x], p.o[6 + x]);
      continue;
    }
    const float inv = 1.0f / p.l[x];
    const float v0 = p.o[x] * inv, v1 = p.o[2 + x] * inv, v2 = p.o[4 + x] * inv, v3 = p.o[6 + x] * inv;
    const int64_t i = (row0 + head) * kD + c0;
    if (a.out_dtype == VIDKV_F32) *reinterpret_cast<float4*>(reinterpret_cast<float*>(a.out) + i) = make_float4(v0, v1, v2, v3);
    else if (a.out_dtype == VIDKV_F16) *reinterpret_cast<uint2*>(reinterpret_cast<__half*>(a.out) + i) = make_uint2(pack_half2(v0, v1), pack_half2(v2, v3));
    else {
      __nv_bfloat162 b[2] = {__floats2bfloat162_rn(v0, v1), __floats2bfloat162_rn(v2, v3)};
      *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(a.out) + i) = *reinterpret_cast<const uint2*>(b);
    }
  }
}
// Part `part` of a slab is done; block `first` has part 0.  The only part writes the result; otherwise it leaves its record and arrives at its
// node of the join tree, and the last to arrive goes on with the joined record.  Whole block; `flag` is a shared word.
// The counters are zero between calls (the last arrival clears its node's).
__device__ __forceinline__ void finish_part(const DecodeArgs& a, int slab, int first, int part, int n_parts, Running& run, volatile int* flag,
                                            int warp, int lane) {
  const int hd = lane >> 2, r = lane & 3;
  if (a.partial_out) {
    const float f = exp2f(run.m - run.exact);
    run.scale(__shfl_sync(0xffffffffu, f, 8 * r), __shfl_sync(0xffffffffu, f, 8 * r + 4));
    run.m = run.exact;
  }
  Part p;
  p.m[0] = __shfl_sync(0xffffffffu, run.m, 8 * r);
  p.m[1] = __shfl_sync(0xffffffffu, run.m, 8 * r + 4);
  p.l[0] = run.l[0]; p.l[1] = run.l[1];
#pragma unroll
  for (int j = 0; j < 8; ++j) p.o[j] = run.o[j];
  float* rec = a.partials + static_cast<int64_t>(slab + first) * kPartFloats;
  int32_t* cnt = a.counters + static_cast<int64_t>(slab) * a.plan.counters_per_slab;
  int64_t stride = kPartFloats;
  while (n_parts > 1) {
    if (warp < 4) store_record(rec + part * stride, p, warp, hd, r);
    __threadfence();
    __syncthreads();
    const int node = part / kJoin, n = min(kJoin, n_parts - node * kJoin);
    if (threadIdx.x == 0) {
      const bool last = atomicAdd(cnt + node, 1) == n - 1;
      if (last) { cnt[node] = 0; __threadfence(); }
      *flag = last;
    }
    __syncthreads();
    if (!*flag) return;
    if (warp < 4) join_records(rec + node * kJoin * stride, stride, n, p, warp, hd, r);
    __syncthreads();                                       // everyone has read the flag
    n_parts = (n_parts + kJoin - 1) / kJoin;
    cnt += n_parts;
    stride *= kJoin;
    part = node;
  }
  if (warp < 4) store_result(a, slab, p, warp, hd, r);
}

// Zero the ring entries of stream positions [pos_begin, pos_end) in every head's row; `ring` points at entry 0 of
// the stream's part of row 0.  Whole block.
__device__ __forceinline__ void zero_ring(uint8_t* ring, int ring_len, int pos_begin, int pos_end) {
  for (int i = threadIdx.x; i < 8 * (pos_end - pos_begin); i += kUnitThreads)
    *reinterpret_cast<uint16_t*>(ring + (i & 7) * kRingRow + ((pos_begin + (i >> 3)) & (ring_len - 1)) * 2) = 0;
}

}  // namespace

template <bool GEN, bool STP, typename T>
__global__ void __launch_bounds__(kUnitThreads, GEN && STP ? kBlockGenStpPerSM : kBlocksPerSM) decode_block_kernel(DecodeArgs a) {
  using S = Smem<GEN, STP>;
  extern __shared__ __align__(128) uint8_t sm[];
  __shared__ __align__(8) uint64_t kbar[2], vbar[2], pbar[kPBufs];
  __shared__ __align__(16) float gmax[2][8][8];              // [unit parity][head][group]: maxima of the groups' scores
  __shared__ float4 psum[2][kSGGroups][4];                   // [unit parity][group][r]: accumulator fragment -5 * sum of the probabilities
  __shared__ int flag;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, hd = lane >> 2, r = lane & 3;
  const DecodePlan& pl = a.plan;
  const CacheView& cv = a.cv;
  const KeyFmt& kf = cv.kf;
  const int kgb = GEN ? kf.group_bytes : kKGroupBytes;
  const int n_slab_units = pl.units_per_slab;
  uint8_t* const slab0 = cv.base + cv.slab_offset + static_cast<int64_t>(a.layer0) * cv.B * cv.H_kv * cv.slab_stride;
  const bool live = hd < cv.rep;
  auto query_row = [&](int slab) { return reinterpret_cast<const T*>(a.q) + (static_cast<int64_t>(slab / cv.H_kv) * cv.H_q + (slab % cv.H_kv) * cv.rep + hd) * kD; };
  // block b owns the units [b * units / blocks, (b + 1) * units / blocks)
  const uint32_t n_units = static_cast<uint32_t>(pl.n_units), n_blocks = static_cast<uint32_t>(pl.n_blocks);
  auto block_of = [&](uint32_t u) { return static_cast<int>(((u + 1u) * n_blocks - 1u) / n_units); };
  Running run;
  // everything below may depend on the kernel before this one in the stream
  pdl_wait();
  pdl_release();
  if (static_cast<int>(blockIdx.x) >= pl.n_blocks) {
    // a residual of its own (blocks that own one unit each, or nothing quantized yet)
    const int slab = blockIdx.x - pl.n_blocks, first = slab * n_slab_units;   // one unit per block
    uint8_t* const slab_ptr = slab0 + static_cast<int64_t>(slab) * cv.slab_stride;
    run.reset();
    if (warp == 0) append_row(a, slab, slab_ptr, lane);
    add_residual<T>(a, slab_ptr, query_row(slab), live, sm + S::prob_at, warp, lane, run);
    finish_part(a, slab, first, n_slab_units, n_slab_units + 1, run, &flag, warp, lane);
    return;
  }
  const int u_begin = static_cast<int>(blockIdx.x * n_units / n_blocks);
  const int n_local = static_cast<int>((blockIdx.x + 1u) * n_units / n_blocks) - u_begin;
  // token and stream positions fit 32 bits (the layout's group counts do)
  const int T_q0 = static_cast<int>(a.st.T_q0), T_qt = T_q0 + static_cast<int>(a.st.n_flush) * kR;
  const int n_groups = T_qt / kG, g0n = T_q0 / kG;
  const int n_prot = static_cast<int>(a.n_prot), n_rest = T_q0 - n_prot;
  const int u_fl0 = (n_rest + kG - 1) / kG * kG;             // stream position where the flushed tokens start
  int slab = u_begin / n_slab_units, k = u_begin - slab * n_slab_units;
  auto chunk_of = [&](int g) { return g < g0n ? 0 : 1 + (g - g0n) / (kR / kG); };

  // ---- bulk copies, issued by one lane of warp 4 (it has no part in P V): keys of local unit ks and values of local
  // unit vs, two buffers each
  const bool producer = tid == 4 * 32;
  if (producer) {
    for (int j = 0; j < 2; ++j) { mbar_init(kbar + j, 1); mbar_init(vbar + j, 1); }
    for (int j = 0; j < kPBufs; ++j) mbar_init(pbar + j, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 128) (&gmax[0][0][0])[tid] = -INFINITY;
  int ks = 0, ks_k = k, vs = 0, vs_k = k;
  const uint8_t* key_src = slab0 + static_cast<int64_t>(slab) * cv.slab_stride + cv.kgroup_offset;
  const uint8_t* val_src = slab0 + static_cast<int64_t>(slab) * cv.slab_stride + cv.tern_offset;
  auto issue_keys = [&]() {
    const int groups = min(kSGGroups, n_groups - ks_k * kSGGroups);
    bulk_load(sm + S::k_at + (ks & 1) * S::kKBuf, key_src + static_cast<uint32_t>(ks_k) * static_cast<uint32_t>(kSGGroups * kgb),
              static_cast<uint32_t>(groups * kgb), kbar + (ks & 1));
    ++ks;
    if (++ks_k == n_slab_units) { ks_k = 0; key_src += cv.slab_stride; }
  };
  auto issue_values = [&]() {
    if (!(a.withhold && vs == 0))                            // (test hook: see DecodeArgs::withhold)
      bulk_load(sm + S::v_at + (vs & 1) * kVBufBytes, val_src + static_cast<uint32_t>(vs_k) * kVBufBytes, kVBufBytes, vbar + (vs & 1));
    ++vs;
    if (++vs_k == n_slab_units) { vs_k = 0; val_src += cv.slab_stride; }
  };
  if (producer) {
    issue_keys();
    if (!STP) issue_values();
    if (n_local > 1) {
      issue_keys();
      if (!STP) issue_values();
    }
  }
  __syncthreads();
  // STP: supergroups (groups) of the current slab that are multiplied (next), requested (req) and needed (end);
  // vcnt / vreq count supergroups over the whole walk (buffer and phase), pslot / prslot / pphase the same for groups
  int sg_next = 0, sg_req = 0, sg_end = 0, pg_next = 0, pg_req = 0, pg_end = 0, vcnt = 0, vreq = 0;
  int pslot = 0, prslot = 0;
  uint32_t pphase = 0u;
  bool fault = false, dead = false;                          // a copy never arrived: seen by this thread / by the block
  int i = 0;                                                 // local unit
#pragma unroll 1
  while (i < n_local) {
    const int k_end = min(n_slab_units, k + n_local - i);
    uint8_t* const slab_ptr = slab0 + static_cast<int64_t>(slab) * cv.slab_stride;
    const T* const qrow = query_row(slab);
    run.reset();
    if (!dead) {
      const int qe = head_exponent<T, 4>(qrow, r, live);
      const float qf = pow2i(-qe - kQShift);                                       // normalised query, see head_exponent
      const float sl2 = a.scale * 1.4426950408889634f * pow2i(qe + kQShift);       // its scores as base-2 logits
      int img_chunk[2] = {-1, -1};                           // chunk c's images are in slot c % 2
      const uint32_t *ew = nullptr, *ep = nullptr;
      int u_hi = 0, p_hi = 0;                                // STP: stream positions written so far
      float unit_factor = 0.0f;                              // otherwise: brings the sums to the reference of the unit whose P V is due
      auto request = [&]() {                                 // copies whose buffers are free (after a barrier; whole block)
        if (producer) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        while (sg_req < sg_end && sg_req < sg_next + 2) {
          if (producer) bulk_load(sm + S::v_at + (vreq & 1) * kVBufBytes, slab_ptr + cv.tern_offset + static_cast<int64_t>(sg_req) * kVBufBytes,
                                  kVBufBytes, vbar + (vreq & 1));
          ++sg_req; ++vreq;
        }
        while (pg_req < pg_end && pg_req < pg_next + kPBufs) {
          if (producer) bulk_load(sm + S::p_at + prslot * kPGBytes, slab_ptr + cv.prot_offset + static_cast<int64_t>(pg_req) * kPGBytes, kPGBytes,
                                  pbar + prslot);
          ++pg_req;
          if (++prslot == kPBufs) prslot = 0;
        }
      };
      if (STP) {
        const int b = (slab / cv.H_kv) % cv.B;
        ew = cv.e_words(b);
        ep = cv.e_prefix(b);
        // where this block enters and leaves the two value streams
        auto stream_at = [&](int t, int& u, int& p) {
          if (t <= T_q0) { p = static_cast<int>(__ldg(ep + t / kG)); u = t - p; }
          else { p = n_prot; u = u_fl0 + (t - T_q0); }
        };
        int ue, pe;
        stream_at(k * kStreamUnitTokens, u_hi, p_hi);
        stream_at(min(k_end * kStreamUnitTokens, T_qt), ue, pe);
        sg_next = u_hi / kStreamUnitTokens; sg_req = sg_next; sg_end = (ue + kStreamUnitTokens - 1) / kStreamUnitTokens;
        pg_next = p_hi / kG; pg_req = pg_next; pg_end = (pe + kG - 1) / kG;
        __syncthreads();                                     // the last slab's readers of rings and value buffers are done
        request();
      }
      // ---- P V of what is complete: the unit before (its probabilities are in buffer (i - 1) % 2), or the
      // supergroups and protected groups that have been requested and whose positions are all written
      auto multiply = [&](int unit) {                        // caches without protected tokens: local unit `unit`
        if (warp >= 4) return;
        if (!mbar_wait(vbar + (unit & 1), (unit >> 1) & 1)) { fault = true; return; }
        const uint8_t* prow = sm + S::prob_at + ((unit & 1) * 8 + hd) * kPRowBytes + 4 * r;
        float4 ps[kSGGroups];
#pragma unroll
        for (int g = 0; g < kSGGroups; ++g) ps[g] = psum[unit & 1][g][r];
        run.scale(__shfl_sync(0xffffffffu, unit_factor, 8 * r), __shfl_sync(0xffffffffu, unit_factor, 8 * r + 4));
        pv_ternary(sm + S::v_at + (unit & 1) * kVBufBytes, warp,
                   [&](int g, int nt) { return *reinterpret_cast<const uint32_t*>(prow + g * (kG * 2) + nt * 16); }, ps, run, hd, r);
      };
      auto multiply_streams = [&](int u_done, int p_done) {
        const uint8_t* trow = sm + S::prob_at + hd * kRingRow + 4 * r;
#pragma unroll 1
        while (sg_next < sg_req && (sg_next + 1) * kStreamUnitTokens <= u_done) {
          if (warp < 4) {
            if (!mbar_wait(vbar + (vcnt & 1), (vcnt >> 1) & 1)) fault = true;
            else {
              const int base = sg_next * kStreamUnitTokens;
              auto P = [&](int g, int nt) { return *reinterpret_cast<const uint32_t*>(trow + ((base + g * kG) & (kTRing - 1)) * 2 + nt * 16); };
              float4 ps[kSGGroups];
#pragma unroll
              for (int g = 0; g < kSGGroups; ++g) {
                float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                mma_f16(c, kMinus5, kMinus5, kMinus5, kMinus5, P(g, 0), P(g, 1));
                mma_f16(c, kMinus5, kMinus5, kMinus5, kMinus5, P(g, 2), P(g, 3));
                ps[g] = make_float4(c[0], c[1], c[2], c[3]);
              }
              pv_ternary(sm + S::v_at + (vcnt & 1) * kVBufBytes, warp, P, ps, run, hd, r);
            }
          }
          ++sg_next; ++vcnt;
        }
#pragma unroll 1
        while (pg_next < pg_req && (pg_next + 1) * kG <= p_done) {
          if (warp < 4) {
            if (!mbar_wait(pbar + pslot, pphase)) fault = true;
            else {
              uint32_t P4[4];
#pragma unroll
              for (int nt = 0; nt < 4; ++nt)
                P4[nt] = *reinterpret_cast<const uint32_t*>(trow + (kTRing + ((pg_next * kG) & (kPRing - 1))) * 2 + nt * 16);
              pv_protected(sm + S::p_at + pslot * kPGBytes, warp, P4, run, hd, r);
            }
          }
          ++pg_next;
          if (++pslot == kPBufs) { pslot = 0; pphase ^= 1u; }
        }
      };

      const int k_begin = k;
#pragma unroll 1
      for (; k < k_end; ++k, ++i) {
        const int g_first = k * kSGGroups, ng = min(kSGGroups, n_groups - g_first);
        // ---- images of the chunks this unit touches (two at most; what they replace was last read before a barrier)
        {
          const int c_lo = chunk_of(g_first), c_hi = chunk_of(g_first + ng - 1);
          bool made = false;
#pragma unroll 1
          for (int c = c_lo; c <= c_hi; ++c) {
            if (((c & 1) ? img_chunk[1] : img_chunk[0]) == c) continue;
            make_images<GEN, T>(reinterpret_cast<uint32_t*>(sm + S::img_at + (c & 1) * kImgBytes), kf, a.dft,
                                slab_ptr + cv.chunk_table_offset + static_cast<int64_t>(c) * kChunkBytes, qrow, live, qf, warp, lane);
            if (c & 1) img_chunk[1] = c; else img_chunk[0] = c;
            made = true;
          }
          if (made) __syncthreads();
        }
        // STP: protection mask and prefix count of this warp's group, stream position of the unit's end
        uint32_t e_word = 0u;
        int e_base = 0, p_new = 0;
        const int tg = (g_first + warp) * kG;                // first token of the warp's group
        const int t_end = (g_first + ng) * kG;
        if (STP) {
          if (warp < ng && tg < T_q0) { e_word = __ldg(ew + g_first + warp); e_base = static_cast<int>(__ldg(ep + g_first + warp)); }
          p_new = t_end <= T_q0 ? static_cast<int>(__ldg(ep + t_end / kG)) : n_prot;
        }
        // ---- scores of group `warp`
        float sc[4][2], cst = 0.0f;
        {
          if (!mbar_wait(kbar + (i & 1), (i >> 1) & 1)) fault = true;
          float gm = -INFINITY;
          if (warp < ng) {
            const uint8_t* kg = sm + S::k_at + (i & 1) * S::kKBuf + warp * kgb;
            const uint4* img = reinterpret_cast<const uint4*>(sm + S::img_at + (chunk_of(g_first + warp) & 1) * kImgBytes) + lane;
            if (GEN) score_group_general(kg, kf, lane, hd, r, img, sc, cst);
            else score_group(kg, lane, hd, r, img, sc, cst);
            gm = fmaxf(fmaxf(fmaxf(sc[0][0], sc[0][1]), fmaxf(sc[1][0], sc[1][1])), fmaxf(fmaxf(sc[2][0], sc[2][1]), fmaxf(sc[3][0], sc[3][1])));
            gm = fmaxf(gm, __shfl_xor_sync(0xffffffffu, gm, 1));
            gm = fmaxf(gm, __shfl_xor_sync(0xffffffffu, gm, 2)) + cst;
          }
          if (r == 0) gmax[i & 1][hd][warp] = gm;
        }
        dead = __syncthreads_or(fault) != 0;
        if (dead) { i += k_end - k; k = k_end; break; }
        if (producer) {
          // the buffers were read through ordinary loads; order them before the bulk copies' writes
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          if (ks < n_local) issue_keys();                    // into the buffer of this unit's keys
          if (!STP && i >= 2) issue_values();                // this unit's, into the buffer of unit i - 2
        }
        if (STP) request();
        // ---- probabilities against the running maximum
        float fa, fb, f;
        bool moved = false;
        const float4 ga = *reinterpret_cast<const float4*>(&gmax[i & 1][hd][0]);
        const float mu = fmaxf(fmaxf(fmaxf(ga.x, ga.y), fmaxf(ga.z, ga.w)), gmax[i & 1][hd][4]) * sl2;   // sl2 > 0
        if (STP) {
          run.exact = fmaxf(run.exact, ceilf(mu));
          moved = move_maximum(mu, r, run.m, fa, fb, f);
        } else {
          f = run.refer_to(mu);
        }
        const float off = fmaf(cst, sl2, -run.m);
        if (!STP) {
          uint8_t* prow = sm + S::prob_at + ((i & 1) * 8 + hd) * kPRowBytes + warp * (kG * 2) + 4 * r;
          uint32_t P[4] = {0u, 0u, 0u, 0u};
          if (warp < ng) {
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) P[nt] = pack_half2(ex2_approx(fmaf(sc[nt][0], sl2, off)), ex2_approx(fmaf(sc[nt][1], sl2, off)));
          }
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) *reinterpret_cast<uint32_t*>(prow + nt * 16) = P[nt];
          // -5 * (sums of the rounded probabilities) of heads 2 r, 2 r + 1: a product with a matrix of -5
          float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
          mma_f16(c, kMinus5, kMinus5, kMinus5, kMinus5, P[0], P[1]);
          mma_f16(c, kMinus5, kMinus5, kMinus5, kMinus5, P[2], P[3]);
          if (hd == 0) psum[i & 1][warp][r] = make_float4(c[0], c[1], c[2], c[3]);
          if (k > k_begin) multiply(i - 1);
          unit_factor = f;
        } else {
          const int u_old = u_hi, p_old = p_hi;
          p_hi = p_new;
          u_hi = t_end <= T_q0 ? t_end - p_new : u_fl0 + (t_end - T_q0);
          if (moved) {
            // what waits in the rings is in the old units: multiply what is complete, then rescale the rest
            multiply_streams(u_old, p_old);
            run.scale(fa, fb);
            __syncthreads();
            const __half2 f2 = __float2half2_rn(f);          // a power of two; at the start of a slab everything is cleared
            uint8_t* row = sm + S::prob_at + hd * kRingRow;
            for (int j = r + 4 * warp; j < (kTRing + kPRing) / 2; j += 4 * kUnitWarps) {
              __half2* q = reinterpret_cast<__half2*>(row) + j;
              *q = k > k_begin ? __hmul2(*q, f2) : __half2half2(__ushort_as_half(0));
            }
            __syncthreads();
          }
          // scattered into stream order.  Where a token goes depends on the token alone, so lane j works out the
          // destination of the group's token j (byte offset inside a head's row) and the lanes pick up the
          // destinations of their own token pairs with shuffles.
          uint8_t* row = sm + S::prob_at + hd * kRingRow;
          if (warp < ng) {
            if (tg < T_q0) {
              const int below = __popc(e_word & ((1u << lane) - 1u));
              const bool prot = (e_word >> lane) & 1u;
              uint32_t dst = 2u * static_cast<uint32_t>(prot ? kTRing + ((e_base + below) & (kPRing - 1)) : (tg - e_base + lane - below) & (kTRing - 1));
              dst |= __shfl_down_sync(0xffffffffu, dst, 1) << 16;   // even lanes: this token and the next
#pragma unroll
              for (int nt = 0; nt < 4; ++nt) {
                const __half2 ph = __floats2half2_rn(ex2_approx(fmaf(sc[nt][0], sl2, off)), ex2_approx(fmaf(sc[nt][1], sl2, off)));
                const uint32_t d = __shfl_sync(0xffffffffu, dst, 8 * nt + 2 * r);
                *reinterpret_cast<__half*>(row + (d & 0xffffu)) = __low2half(ph);
                *reinterpret_cast<__half*>(row + (d >> 16)) = __high2half(ph);
              }
            } else {
              const int tmod = (u_fl0 + (tg - T_q0)) & (kTRing - 1);
#pragma unroll
              for (int nt = 0; nt < 4; ++nt)
                *reinterpret_cast<__half2*>(row + (tmod + 8 * nt + 2 * r) * 2) =
                    __floats2half2_rn(ex2_approx(fmaf(sc[nt][0], sl2, off)), ex2_approx(fmaf(sc[nt][1], sl2, off)));
            }
          }
          if (g_first * kG <= T_q0 && t_end > T_q0) zero_ring(sm + S::prob_at, kTRing, n_rest, u_fl0);   // nobody writes the gap
          if (!moved) multiply_streams(u_old, p_old);
        }
      }
      if (!dead) {
        dead = __syncthreads_or(fault) != 0;
        if (!dead) {
          if (!STP) multiply(i - 1);
          else {
            request();
            multiply_streams(u_hi, p_hi);
            __syncthreads();
            request();
            multiply_streams(u_hi, p_hi);                    // at most three supergroups and ten groups were complete
            __syncthreads();
            // the positions of the last supergroup and group that nobody here writes belong to a neighbour
            request();
            zero_ring(sm + S::prob_at, kTRing, u_hi, sg_end * kStreamUnitTokens);
            zero_ring(sm + S::prob_at + kTRing * 2, kPRing, p_hi, pg_end * kG);
            __syncthreads();
            multiply_streams(sg_end * kStreamUnitTokens, pg_end * kG);
          }
        }
      }
    } else {
      i += k_end - k;
    }
    if (k_end == n_slab_units && a.st.n_res > 0 && pl.res_blocks == 0) {
      if (warp == 0) append_row(a, slab, slab_ptr, lane);    // also where a copy never arrived: later calls find the row
      if (!dead) add_residual<T>(a, slab_ptr, qrow, live, sm + S::prob_at, warp, lane, run);
    }
    const int first = block_of(static_cast<uint32_t>(slab) * n_slab_units), last = block_of((slab + 1u) * n_slab_units - 1u);
    finish_part(a, slab, first, static_cast<int>(blockIdx.x) - first, last - first + 1 + (pl.res_blocks ? 1 : 0), run, &flag, warp, lane);
    k = 0;
    ++slab;
  }
  if (__syncthreads_or(fault) && producer) {
    // a copy never arrived: report it, and let the others that are in flight land before the block leaves
    atomicCAS(reinterpret_cast<int*>(cv.base + kHdrStatus), VIDKV_OK, VIDKV_ERR_TIMEOUT);
    for (int j = max(0, ks - 2); j < ks; ++j) mbar_wait_lane(kbar + (j & 1), (j >> 1) & 1);
    if (STP) {
      for (int j = max(0, vreq - 2); j < vreq; ++j) mbar_wait_lane(vbar + (j & 1), (j >> 1) & 1);
      for (; pg_next < pg_req; ++pg_next) {
        mbar_wait_lane(pbar + pslot, pphase);
        if (++pslot == kPBufs) { pslot = 0; pphase ^= 1u; }
      }
    } else {
      for (int j = max(a.withhold ? 1 : 0, vs - 2); j < vs; ++j) mbar_wait_lane(vbar + (j & 1), (j >> 1) & 1);
    }
  }
}

template <bool GEN, bool STP, typename T>
static cudaError_t launch_block_t(const DecodeArgs& a, cudaStream_t stream) {
  constexpr int smem = Smem<GEN, STP>::bytes;
  static bool attr_set[64] = {};
  int dev = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev))) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr_set[dev]) {
    if ((e = cudaFuncSetAttribute(decode_block_kernel<GEN, STP, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem))) return e;
    attr_set[dev] = true;
  }
  count_launches(1);
  return launch_dependent(decode_block_kernel<GEN, STP, T>, dim3(a.plan.n_blocks + a.plan.res_blocks), dim3(kUnitThreads), smem, stream, a);
}

cudaError_t launch_decode_block(const DecodeArgs& a_in, cudaStream_t stream) {
  DecodeArgs a = a_in;
  const bool gen = a.cv.kf.general != 0, stp = a.n_prot > 0, half = a.in_dtype == VIDKV_F16;
  if (g_debug_withhold == 2) { a.withhold = stp ? 0 : 1; g_debug_withhold = 0; }
  if (gen) {
    if (stp) return half ? launch_block_t<true, true, __half>(a, stream) : launch_block_t<true, true, __nv_bfloat16>(a, stream);
    return half ? launch_block_t<true, false, __half>(a, stream) : launch_block_t<true, false, __nv_bfloat16>(a, stream);
  }
  if (stp) return half ? launch_block_t<false, true, __half>(a, stream) : launch_block_t<false, true, __nv_bfloat16>(a, stream);
  return half ? launch_block_t<false, false, __half>(a, stream) : launch_block_t<false, false, __nv_bfloat16>(a, stream);
}

}  // namespace vidkv
