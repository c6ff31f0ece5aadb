// Decode attention over the packed cache (Algorithm 1 "Decoding", Eq. 3) in one launch, for small calls (up to some 10000
// 160-token units of five 32-token key groups where the slabs are few and long); plan_decode has the rule.
//
// What bounds such a call is latency: launches, dependent loads, a unit's serial work and the merge of the partial
// results.  6400 tokens, a unit a block (11.4 us from the first block's start to the last one's end): query images 2.2,
// keys, scores and probabilities 1.5, P V 0.7, record and arrival 1.1-1.4 and its join 1.1 at each of the two levels, output 0.4.
//
// A block of five warps owns a contiguous stretch of units and walks it slab by slab:
//   query     the register images of the query for the slab's channel split (normalised query at
//             the 2-bit channels, its transform at the spectrum columns) are computed by the block
//             itself and kept in shared memory; a flushed chunk's images replace them when the walk
//             reaches it;
//   scores    warp g scores key group g of the unit (decode_score.cuh): rows = tokens, columns = query heads;
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
// 32).  The probabilities are then scattered into two rings in stream order, 16 bytes a position, and a
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

#include "decode_score.cuh"

namespace vidkv {

namespace {

constexpr int kUnitWarps = 5;
constexpr int kUnitThreads = kUnitWarps * 32;
constexpr int kImgBytes = 40 * 32 * 4;                        // query images of one chunk
constexpr int kTRing = 512, kPRing = 512;                     // ring positions: an unfinished supergroup (group), two units and the gap
                                                              // before the flushed tokens
constexpr int kPBufs = 5;                                     // staged protected groups: as many as a unit can fill, or the rings would run
                                                              // over; four blocks share a multiprocessor's memory with them
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
  static constexpr int prob_bytes = STP ? (kTRing + kPRing) * kEntry : (2 * kStreamUnitTokens * kEntry > kResScratch ? 2 * kStreamUnitTokens * kEntry : kResScratch);
  static constexpr int bytes = prob_at + prob_bytes;
};

// The query as score_blocks takes it, from the images in shared memory, four words a load.
struct ImageQuery {
  const uint32_t* img;
  __device__ __forceinline__ uint4 words(int j) const { return *reinterpret_cast<const uint4*>(img + 128 * j); }
  __device__ __forceinline__ uint4 pairs(int f) const { return words(f); }
  __device__ __forceinline__ void spectrum(int f, int par, uint32_t (&h)[4], uint32_t (&l)[4]) const {
    const uint4 a = words(2 + 2 * f + par), b = words(6 + 2 * f + par);
    h[0] = a.x; h[1] = a.y; h[2] = a.z; h[3] = a.w;
    l[0] = b.x; l[1] = b.y; l[2] = b.z; l[3] = b.w;
  }
};

struct ImageWords {                                          // the same for the general formats
  const uint32_t* img;
  __device__ __forceinline__ uint32_t operator()(int j) const { return img[(j >> 2) * 128 + (j & 3)]; }
  __device__ __forceinline__ uint4 four(int j) const { return *reinterpret_cast<const uint4*>(img + 32 * j); }
};

// Scores of one key group (t as in score_group) and the group's constants of heads 2 r, 2 r + 1.  img: this lane's query words of the
// group's chunk, four words a 16-byte load, 32 loads apart.
template <bool GEN>
__device__ __forceinline__ void score(uint8_t* kg, const KeyFmt& kf, int lane, int g, int r, const uint32_t* img, float (&t)[2][4], float (&cst)[2]) {
  if constexpr (GEN) {
    const ImageWords word{img};
    group_constants_general(kg, kf, 1, g, r, word, cst);
    score_group_general(kg, kf, lane, r, word, t);
  } else {
    GroupBytes gb;
    gb.fetch(kg, lane);
    const ImageQuery q{img};
    group_constants(kg, 1, g, r, q, cst);
    __syncwarp();
    put_scales(gb, gb, kg, lane);
    __syncwarp();
    score_group(gb, kg, r, q, t);
  }
}

// ---------------------------------------------------------------------------------------------
// Query images of one chunk's channel split, by the whole block: word i of lane (head hd = lane / 4,
// r = lane % 4) at ((i / 4) * 32 + lane) * 4 + i % 4, so that four words are one 16-byte load:
//   words  j < 8            binary16 pair of q at the anomalous slots 8 j + 2 r, + 1
//   words  8 + 4 (2 f + par) + i   (-Q, Q), leading binary16 part of the transformed query Q at the spectrum column
//                           32 f + 16 (i / 2) + 15 - 8 (i % 2) - 2 r - par
//   words 24 + 4 (2 f + par) + i   the same of the binary16 remainder Q - leading part;
// zero for heads that do not
// exist, all of the query normalised by its head's power of two (head_exponent).  Q_f = sum_c q_c W[c, f] with W the
// weights with which spectrum column f enters channel c of the inverse orthonormal 64-point transform of a Hermitian
// half spectrum: the forward DFT matrix, doubled for the columns f >= 2 that stand for a conjugate pair, on the tensor
// cores against the split-precision matrix fragments.  General key formats (KeyFmt):
//   words w < n2/8              pairs of q at the two-bit slots 8 w + 2 r, + 1
//   then n1/8 words             plain mode: pairs of q at the one-bit channels 8 w + 6 - 2 r, + 1;
//                               Eq. 5: leading binary16 part of Q at those columns,
//   then (Eq. 5) n1/8 words     the remainder (Q from the table of the 32-point transform)
// A block computes them once per slab it walks (and once per flushed chunk): about 2 us of latency (3 where the matrix
// fragments were fetched behind the channel order and the query instead of beside them)
// behind the first bulk copies, where a kernel of its own takes 5-8 us of a step.
// ---------------------------------------------------------------------------------------------
// What make_images reads besides the query (default format), fetched ahead: the channel order, and the matrix fragments of the warp's
// columns nt = warp and warp + 5.
struct ImageSource {
  static constexpr int kTurns = (8 + kUnitWarps - 1) / kUnitWarps;
  uint4 bw[kTurns][4];
  uint32_t two[kTurns], pa[4], pb[4];
  __device__ __forceinline__ void fetch(const DftTables& dft, const uint8_t* perm, int warp, int lane) {
    const int r = lane & 3;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      pa[ks] = *reinterpret_cast<const uint16_t*>(perm + kNA + 16 * ks + 2 * r);
      pb[ks] = *reinterpret_cast<const uint16_t*>(perm + kNA + 16 * ks + 2 * r + 8);
    }
#pragma unroll
    for (int turn = 0; turn < kTurns; ++turn) {
      const int nt = min(warp + turn * kUnitWarps, 7);
      two[turn] = *reinterpret_cast<const uint16_t*>(perm + 8 * nt + 2 * r);
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) bw[turn][ks] = *reinterpret_cast<const uint4*>(dft.frag + ((ks * 8 + nt) * 32 + lane) * 4);
    }
  }
};

template <bool GEN, typename T>
__device__ __forceinline__ void make_images(uint32_t* img, const ImageSource& src, const KeyFmt& kf, const DftTables& dft, const uint8_t* perm,
                                            const T* qrow, bool live, float qf, int warp, int lane) {
  const int r = lane & 3;
  auto q_at = [&](uint32_t c) -> float { return live ? Elem<T>::to_float(qrow[c]) * qf : 0.0f; };
  auto put = [&](int i, int to, uint32_t v) { img[((i >> 2) * 32 + to) * 4 + (i & 3)] = v; };
  if (!GEN) {
    // transformed query: A = q at the normal channels (rows 8-15 unused), B = matrix fragments
    uint32_t af[4][2];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      af[ks][0] = pack_half2(q_at(src.pa[ks] & 0xffu), q_at(src.pa[ks] >> 8));
      af[ks][1] = pack_half2(q_at(src.pb[ks] & 0xffu), q_at(src.pb[ks] >> 8));
    }
#pragma unroll
    for (int turn = 0; turn < ImageSource::kTurns; ++turn) {
      const int nt = warp + turn * kUnitWarps;
      if (nt >= 8) break;
      float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        const uint4 bw = src.bw[turn][ks];
        mma_f16(acc, af[ks][0], 0u, af[ks][1], 0u, bw.x, bw.y);
        mma_f16(acc, af[ks][0], 0u, af[ks][1], 0u, bw.z, bw.w);
      }
      // lane (hd, r) now holds Q of head hd at columns 16 r + 2 nt + {0, 1}, which belong to lane (hd, 3 - nt % 4)
      const float w0 = (r == 0 && nt == 0) ? 1.0f : 2.0f;            // columns 0 and 1 are not doubled
      const float x0 = acc[0] * w0, x1 = acc[1] * w0;
      const __half h0 = __float2half_rn(x0), h1 = __float2half_rn(x1);
      const int at = 8 + (r >> 1) * 8 + 2 * (r & 1) + (nt < 4 ? 1 : 0), to = lane - r + 3 - (nt & 3);   // f = r / 2, i = 2 (r % 2) + (nt < 4)
      put(nt, lane, pack_half2(q_at(src.two[turn] & 0xffu), q_at(src.two[turn] >> 8)));
      const uint32_t hi = pack_half2(__half2float(h0), __half2float(h1)), lo = pack_half2(x0 - __half2float(h0), x1 - __half2float(h1));
      put(at, to, sign_pair_hi(hi));                                 // par = 0: the odd column of the pair
      put(at + 4, to, sign_pair_lo(hi));
      put(at + 16, to, sign_pair_hi(lo));
      put(at + 20, to, sign_pair_lo(lo));
    }
  } else {
    const int n2 = kf.n2, n1 = kD - n2, w1 = n2 / 8, n_pairs = kf.plain ? kD / 8 : w1;
    constexpr int kTurns = (16 + kUnitWarps - 1) / kUnitWarps;
    uint32_t two[kTurns];
#pragma unroll
    for (int turn = 0; turn < kTurns; ++turn) {
      const int w = warp + turn * kUnitWarps;
      two[turn] = w < n_pairs ? *reinterpret_cast<const uint16_t*>(perm + (w < w1 ? 8 * w + 2 * r : 8 * w + 6 - 2 * r)) : 0u;
    }
#pragma unroll
    for (int turn = 0; turn < kTurns; ++turn) {
      const int w = warp + turn * kUnitWarps;
      if (w < n_pairs) put(w, lane, pack_half2(q_at(two[turn] & 0xffu), q_at(two[turn] >> 8)));
    }
    if (!kf.plain && n1 > 0 && warp == kUnitWarps - 1) {
      // n1 = 32: lane r owns the columns 8 r .. 8 r + 7; sums of eight channels each, added in the order of decode_prep_general_kernel
      float x[8];
      const float4* wt = reinterpret_cast<const float4*>(dft.w32) + 2 * r;
#pragma unroll 1
      for (int part = 0; part < 4; ++part) {
        float y[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int c = 8 * part, i = 0; i < 8; ++c, ++i) {
          const float qv = q_at(perm[n2 + c]);
          const float4 wa = wt[8 * c], wb = wt[8 * c + 1];
          y[0] = fmaf(qv, wa.x, y[0]); y[1] = fmaf(qv, wa.y, y[1]); y[2] = fmaf(qv, wa.z, y[2]); y[3] = fmaf(qv, wa.w, y[3]);
          y[4] = fmaf(qv, wb.x, y[4]); y[5] = fmaf(qv, wb.y, y[5]); y[6] = fmaf(qv, wb.z, y[6]); y[7] = fmaf(qv, wb.w, y[7]);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = part == 0 ? y[i] : x[i] + y[i];
      }
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const __half h0 = __float2half_rn(x[2 * w]), h1 = __float2half_rn(x[2 * w + 1]);
        put(w1 + r, lane - r + 3 - w, pack_half2(__half2float(h0), __half2float(h1)));      // columns 8 r + 2 w, + 1
        put(w1 + 4 + r, lane - r + 3 - w, pack_half2(x[2 * w] - __half2float(h0), x[2 * w + 1] - __half2float(h1)));
      }
    }
  }
}

// Running softmax of the block's part of one slab, heads 2 r and 2 r + 1 (r = lane % 4).  m and exact are the same in every warp; o and l
// belong to warps 0-3: o[4 i + c] = channel 32 w + 4 (lane / 4) + 2 i + c / 2, head 2 r + c % 2.
struct Running {
  float m[2];          // reference: o and l are in units of 2^m
  float exact[2];      // the largest unit maximum so far
  float l[2];
  float o[8];
  __device__ __forceinline__ void reset() {
#pragma unroll
    for (int x = 0; x < 2; ++x) { m[x] = -INFINITY; exact[x] = -INFINITY; l[x] = 0.0f; }
#pragma unroll
    for (int j = 0; j < 8; ++j) o[j] = 0.0f;
  }
  __device__ __forceinline__ void scale(const float (&f)[2]) {
    l[0] *= f[0]; l[1] *= f[1];
#pragma unroll
    for (int j = 0; j < 8; ++j) o[j] *= f[j & 1];
  }
  // Reference of tokens whose largest base-2 logits are mu: their own maximum (kRefLag: see there).  f: the factors that
  // bring the sums so far to it.
  __device__ __forceinline__ void refer_to(const float (&mu)[2], float (&f)[2]) {
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      exact[x] = fmaxf(exact[x], mu[x]);
      const float ref = fmaxf(mu[x], exact[x] - kRefLag);
      f[x] = ex2_approx(m[x] - ref);                        // 0 at the start of a slab (m = -inf)
      m[x] = ref;
    }
  }
};

// P V of one staged ternary supergroup for the 32 channels of warp w (two MMA row blocks: fragment i covers channels
// 32 w + 4 hd + 2 i + {0, 1} in rows hd, hd + 8).  P(g, x): x[nt] = probabilities of head hd at the supergroup's tokens
// 32 g + 8 nt + 2 r, + 1 (binary16 pair); ps[g] = -5 * (sum of the group's probabilities) of heads 2 r, 2 r + 1, twice:
// the accumulator fragment P V starts from (ps(g)).  Groups from ng on do not exist: their probabilities are zero, their scales unwritten.
template <typename PFrag, typename PSum>
__device__ __forceinline__ void pv_ternary(const uint8_t* vbuf, int w, int ng, PFrag P, PSum ps, Running& run, int hd, int r) {
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
    uint32_t p[4];
    P(g, p);
    const float4 c = ps(g);
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
      const uint32_t b0 = p[2 * kt], b1 = p[2 * kt + 1];
      if (kt == 0) {
        mma_f16_c(acc[0], A[0], A[1], A[2], A[3], b0, b1, c.x, c.y, c.z, c.w);
        mma_f16_c(acc[1], A[4], A[5], A[6], A[7], b0, b1, c.x, c.y, c.z, c.w);
      } else {
        mma_f16(acc[0], A[0], A[1], A[2], A[3], b0, b1);
        mma_f16(acc[1], A[4], A[5], A[6], A[7], b0, b1);
      }
    }
    uint2 sc2 = *reinterpret_cast<const uint2*>(vbuf + kSG_Scales + g * (kD * 2) + (32 * w + 4 * hd) * 2);
    if (g >= ng) sc2 = make_uint2(0u, 0u);
    const float2 sa = __half22float2(*reinterpret_cast<const __half2*>(&sc2.x));
    const float2 sb = __half22float2(*reinterpret_cast<const __half2*>(&sc2.y));
    run.o[0] = fmaf(sa.x, acc[0][0], run.o[0]); run.o[1] = fmaf(sa.x, acc[0][1], run.o[1]);
    run.o[2] = fmaf(sa.y, acc[0][2], run.o[2]); run.o[3] = fmaf(sa.y, acc[0][3], run.o[3]);
    run.o[4] = fmaf(sb.x, acc[1][0], run.o[4]); run.o[5] = fmaf(sb.x, acc[1][1], run.o[5]);
    run.o[6] = fmaf(sb.y, acc[1][2], run.o[6]); run.o[7] = fmaf(sb.y, acc[1][3], run.o[7]);
    run.l[0] = fmaf(-0.2f, c.x, run.l[0]);
    run.l[1] = fmaf(-0.2f, c.y, run.l[1]);
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

// The integral running maxima follow maxima `mu` (base-2 logits of heads 2 r, 2 r + 1) that exceed them by more than
// kStaleLog2: true if some head's moved, with the factors of the lane's heads.
__device__ __forceinline__ bool move_maximum(const float (&mu)[2], float (&m)[2], float (&f)[2]) {
  const bool up0 = mu[0] > m[0] + kStaleLog2, up1 = mu[1] > m[1] + kStaleLog2;   // always true at the start of a slab (m = -inf)
  if (!__any_sync(0xffffffffu, up0 || up1)) return false;
  const float m0 = up0 ? ceilf(mu[0]) : m[0], m1 = up1 ? ceilf(mu[1]) : m[1];
  f[0] = ex2_approx(m[0] - m0); f[1] = ex2_approx(m[1] - m1);                     // 1 for heads whose maximum stays
  m[0] = m0; m[1] = m1;
  return true;
}

// Algorithm 1, Decoding: the step's new key / value row joins the residual (lanes 0-15 copy the key row, 16-31 the value
// row).  One warp.
__device__ __forceinline__ void append_row(const DecodeArgs& a, int slab, uint8_t* slab_ptr, int lane) {
  if (a.append_row < 0) return;
  const uint4* srcp = reinterpret_cast<const uint4*>(lane < 16 ? a.k_new : a.v_new) + static_cast<int64_t>(slab) * 16 + (lane & 15);
  reinterpret_cast<uint4*>(slab_ptr + (lane < 16 ? a.cv.kres_offset : a.cv.vres_offset))[a.append_row * 16 + (lane & 15)] = *srcp;
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
  for (int j = 0; j < 4; ++j) qn[j] = live ? *reinterpret_cast<const uint4*>(qrow + 32 * j + 8 * r) : make_uint4(0u, 0u, 0u, 0u);
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
  const float mu2[2] = {__shfl_sync(0xffffffffu, mu, 8 * r), __shfl_sync(0xffffffffu, mu, 8 * r + 4)};
  float f[2];
  run.refer_to(mu2, f);
  run.scale(f);
  const float m0 = __shfl_sync(0xffffffffu, run.m[0], hd >> 1), m1 = __shfl_sync(0xffffffffu, run.m[1], hd >> 1);
  const float m_hd = (hd & 1) ? m1 : m0;
  const int n_pad = (n_res + 15) & ~15;
  for (int t = 8 * r + 32 * warp; warp < 4 && t < n_pad; t += kR) {
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int t0 = t + 2 * j;
      w[j] = pack_half2(t0 < n_res ? ex2_approx(Sx[hd * kResS + t0] - m_hd) : 0.0f, t0 + 1 < n_res ? ex2_approx(Sx[hd * kResS + t0 + 1] - m_hd) : 0.0f);
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
// Join of n <= kJoin records `stride` floats apart, by warps 0-3.  All loads are under way at once: lane (j, r) fetches record j's maxima and
// sums of heads 2 r, 2 r + 1, and every lane its outputs of all records (two rounds of four records behind the maxima took 2.2 us
// of a call with two levels of joins, this one 1.1).
__device__ __forceinline__ void join_records(const float* rec, int64_t stride, int n, Part& p, int w, int lane) {
  static_assert(kJoin == 8, "");
  const int hd = lane >> 2, r = lane & 3;
  const float* mine = rec + (hd < n ? hd : 0) * stride;
  const float2 m = __ldcg(reinterpret_cast<const float2*>(mine + 2 * r)), l = __ldcg(reinterpret_cast<const float2*>(mine + 8 + 2 * r));
  float4 oa[kJoin], ob[kJoin];
#pragma unroll
  for (int j = 0; j < kJoin; ++j) {
    oa[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    ob[j] = oa[j];
    if (j >= n) continue;
    const float* q = rec + j * stride + 16 + 2 * r * kD + 32 * w + 4 * hd;
    oa[j] = __ldcg(reinterpret_cast<const float4*>(q));
    ob[j] = __ldcg(reinterpret_cast<const float4*>(q + kD));
  }
  const float ma = hd < n ? m.x : -INFINITY, mb = hd < n ? m.y : -INFINITY;
  p.m[0] = ma; p.m[1] = mb;
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    p.m[0] = fmaxf(p.m[0], __shfl_xor_sync(0xffffffffu, p.m[0], o));
    p.m[1] = fmaxf(p.m[1], __shfl_xor_sync(0xffffffffu, p.m[1], o));
  }
  const float wa = exp2f(ma - p.m[0]), wb = exp2f(mb - p.m[1]);       // 0 for a record that does not exist
  p.l[0] = wa * l.x; p.l[1] = wb * l.y;
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    p.l[0] += __shfl_xor_sync(0xffffffffu, p.l[0], o);
    p.l[1] += __shfl_xor_sync(0xffffffffu, p.l[1], o);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) p.o[i] = 0.0f;
#pragma unroll
  for (int j = 0; j < kJoin; ++j) {
    const float a = __shfl_sync(0xffffffffu, wa, 4 * j + r), b = __shfl_sync(0xffffffffu, wb, 4 * j + r);
    p.o[0] = fmaf(a, oa[j].x, p.o[0]); p.o[2] = fmaf(a, oa[j].y, p.o[2]); p.o[4] = fmaf(a, oa[j].z, p.o[4]); p.o[6] = fmaf(a, oa[j].w, p.o[6]);
    p.o[1] = fmaf(b, ob[j].x, p.o[1]); p.o[3] = fmaf(b, ob[j].y, p.o[3]); p.o[5] = fmaf(b, ob[j].z, p.o[5]); p.o[7] = fmaf(b, ob[j].w, p.o[7]);
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
    const float f[2] = {exp2f(run.m[0] - run.exact[0]), exp2f(run.m[1] - run.exact[1])};
    run.scale(f);
    run.m[0] = run.exact[0]; run.m[1] = run.exact[1];
  }
  Part p;
  p.m[0] = run.m[0]; p.m[1] = run.m[1];
  p.l[0] = run.l[0]; p.l[1] = run.l[1];
#pragma unroll
  for (int j = 0; j < 8; ++j) p.o[j] = run.o[j];
  float* rec = a.partials + static_cast<int64_t>(slab + first) * kPartFloats;
  int32_t* cnt = a.counters + static_cast<int64_t>(slab) * a.plan.counters_per_slab;
  int64_t stride = kPartFloats;
  while (n_parts > 1) {
    if (warp < 4) store_record(rec + part * stride, p, warp, hd, r);
    __syncthreads();
    const int node = part / kJoin, n = min(kJoin, n_parts - node * kJoin);
    if (threadIdx.x == 0) {
      // releases the whole block's record (the barrier orders the other threads' stores before it) and acquires the others'
      int before;
      asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(before) : "l"(cnt + node) : "memory");
      const bool last = before == n - 1;
      if (last) cnt[node] = 0;
      *flag = last;
    }
    __syncthreads();
    if (!*flag) return;
    if (warp < 4) join_records(rec + node * kJoin * stride, stride, n, p, warp, lane);
    __syncthreads();                                       // everyone has read the flag
    n_parts = (n_parts + kJoin - 1) / kJoin;
    cnt += n_parts;
    stride *= kJoin;
    part = node;
  }
  if (warp < 4) store_result(a, slab, p, warp, hd, r);
}

// Zero the ring entries of stream positions [pos_begin, pos_end); `ring` points at entry 0 of the stream's part.  Whole block.
__device__ __forceinline__ void zero_ring(uint8_t* ring, int ring_len, int pos_begin, int pos_end) {
  for (int pos = pos_begin + threadIdx.x; pos < pos_end; pos += kUnitThreads)
    *reinterpret_cast<uint4*>(ring + (pos & (ring_len - 1)) * kEntry) = make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace

template <bool GEN, bool STP, int kPerSM, typename T>
__global__ void __launch_bounds__(kUnitThreads, kPerSM) decode_block_kernel(DecodeArgs a) {
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
  if (static_cast<int>(blockIdx.x) >= pl.n_blocks) {
    // a residual of its own (blocks that own one unit each, or nothing quantized yet)
    const int slab = blockIdx.x - pl.n_blocks, first = slab * n_slab_units;   // one unit per block
    uint8_t* const slab_ptr = slab0 + static_cast<int64_t>(slab) * cv.slab_stride;
    run.reset();
    pdl_wait();
    pdl_release();
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
  const int tg_total = u_fl0 / kG + (kR / kG) * static_cast<int>(a.st.n_flush);   // ternary groups that exist
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
  __syncthreads();
  auto perm_of = [&](const uint8_t* slab_ptr, int chunk) { return slab_ptr + cv.chunk_table_offset + static_cast<int64_t>(chunk) * kChunkBytes; };
  // everything below may depend on the kernel before this one in the stream
  pdl_wait();
  pdl_release();
  if (producer) {
    issue_keys();
    if (!STP) issue_values();
    if (n_local > 1) {
      issue_keys();
      if (!STP) issue_values();
    }
  }
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
      const int c_first = chunk_of(k * kSGGroups);
      auto images_at = [&](int c) { return reinterpret_cast<uint32_t*>(sm + S::img_at + (c & 1) * kImgBytes); };
      // all of a slab's first loads are under way before the first is waited for
      ImageSource src;
      if (!GEN) src.fetch(a.dft, perm_of(slab_ptr, c_first), warp, lane);
      const int qe = head_exponent<T, 4>(qrow, r, live);
      const float qf = pow2i(-qe - kQShift);                                       // normalised query, see head_exponent
      const float to_log2 = a.scale * 1.4426950408889634f * pow2i(qe + kQShift);   // its scores as base-2 logits
      const float sl2[2] = {__shfl_sync(0xffffffffu, to_log2, 8 * r), __shfl_sync(0xffffffffu, to_log2, 8 * r + 4)};
      int img_chunk[2] = {(c_first & 1) ? -1 : c_first, (c_first & 1) ? c_first : -1};   // chunk c's images are in slot c % 2
      make_images<GEN, T>(images_at(c_first), src, kf, a.dft, perm_of(slab_ptr, c_first), qrow, live, qf, warp, lane);
      bool made = true;
      const uint32_t *ew = nullptr, *ep = nullptr;
      int u_hi = 0, p_hi = 0;                                // STP: stream positions written so far
      float unit_factor[2] = {0.0f, 0.0f};                   // otherwise: bring the sums to the reference of the unit whose P V is due
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
          if (t <= T_q0) { p = static_cast<int>(ep[t / kG]); u = t - p; }
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
      const int k_begin = k, i_begin = i;
      // ---- P V of what is complete: the unit before (its probabilities are in buffer (i - 1) % 2), or the
      // supergroups and protected groups that have been requested and whose positions are all written
      auto multiply = [&](int unit) {                        // caches without protected tokens: local unit `unit`
        if (warp >= 4) return;
        if (!mbar_wait(vbar + (unit & 1), (unit >> 1) & 1)) { fault = true; return; }
        const uint32_t row = smem_u32(sm + S::prob_at) + ((unit & 1) * kStreamUnitTokens + lane) * kEntry;
        run.scale(unit_factor);
        pv_ternary(sm + S::v_at + (unit & 1) * kVBufBytes, warp, min(kSGGroups, n_groups - (k_begin + unit - i_begin) * kSGGroups),
                   [&](int g, uint32_t (&x)[4]) { load_entries(row + g * (kG * kEntry), x); }, [&](int g) { return psum[unit & 1][g][r]; }, run, hd, r);
      };
      auto multiply_streams = [&](int u_done, int p_done) {
        const uint32_t ring = smem_u32(sm + S::prob_at) + lane * kEntry;
#pragma unroll 1
        while (sg_next < sg_req && (sg_next + 1) * kStreamUnitTokens <= u_done) {
          if (warp < 4) {
            if (!mbar_wait(vbar + (vcnt & 1), (vcnt >> 1) & 1)) fault = true;
            else {
              const int base = sg_next * kStreamUnitTokens;
              auto P = [&](int g, uint32_t (&x)[4]) { load_entries(ring + ((base + g * kG) & (kTRing - 1)) * kEntry, x); };
              float4 sums[kSGGroups];
#pragma unroll
              for (int g = 0; g < kSGGroups; ++g) {
                float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                uint32_t x[4];
                P(g, x);
                mma_f16(c, kMinus5, kMinus5, kMinus5, kMinus5, x[0], x[1]);
                mma_f16(c, kMinus5, kMinus5, kMinus5, kMinus5, x[2], x[3]);
                sums[g] = make_float4(c[0], c[1], c[2], c[3]);
              }
              auto ps = [&](int g) { return sums[g]; };
              pv_ternary(sm + S::v_at + (vcnt & 1) * kVBufBytes, warp, tg_total - sg_next * kSGGroups, P, ps, run, hd, r);
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
              load_entries(ring + (kTRing + ((pg_next * kG) & (kPRing - 1))) * kEntry, P4);
              pv_protected(sm + S::p_at + pslot * kPGBytes, warp, P4, run, hd, r);
            }
          }
          ++pg_next;
          if (++pslot == kPBufs) { pslot = 0; pphase ^= 1u; }
        }
      };

#pragma unroll 1
      for (; k < k_end; ++k, ++i) {
        const int g_first = k * kSGGroups, ng = min(kSGGroups, n_groups - g_first);
        // STP: protection mask and prefix count of this warp's group, stream position of the unit's end
        uint32_t e_word = 0u;
        int e_base = 0, p_new = 0;
        const int tg = (g_first + warp) * kG;                // first token of the warp's group
        const int t_end = (g_first + ng) * kG;
        if (STP) {
          if (warp < ng && tg < T_q0) { e_word = ew[g_first + warp]; e_base = static_cast<int>(ep[g_first + warp]); }
          p_new = t_end <= T_q0 ? static_cast<int>(ep[t_end / kG]) : n_prot;
        }
        // ---- images of the chunks this unit touches (two at most; what they replace was last read before a barrier)
        {
          const int c_lo = chunk_of(g_first), c_hi = chunk_of(g_first + ng - 1);
#pragma unroll 1
          for (int c = c_lo; c <= c_hi; ++c) {
            if (((c & 1) ? img_chunk[1] : img_chunk[0]) == c) continue;
            ImageSource next;
            if (!GEN) next.fetch(a.dft, perm_of(slab_ptr, c), warp, lane);
            make_images<GEN, T>(images_at(c), next, kf, a.dft, perm_of(slab_ptr, c), qrow, live, qf, warp, lane);
            if (c & 1) img_chunk[1] = c; else img_chunk[0] = c;
            made = true;
          }
          if (made) __syncthreads();
          made = false;
        }
        // ---- scores of group `warp`
        float t[2][4], cst[2] = {0.0f, 0.0f};
        {
          if (!mbar_wait(kbar + (i & 1), (i >> 1) & 1)) fault = true;
          float g0 = -INFINITY, g1 = -INFINITY;
          if (warp < ng) {
            uint8_t* kg = sm + S::k_at + (i & 1) * S::kKBuf + warp * kgb;
            score<GEN>(kg, kf, lane, hd, r, reinterpret_cast<const uint32_t*>(sm + S::img_at + (chunk_of(g_first + warp) & 1) * kImgBytes) + lane * 4, t, cst);
            g0 = fmaxf(fmaxf(t[0][0], t[0][2]), fmaxf(t[1][0], t[1][2]));
            g1 = fmaxf(fmaxf(t[0][1], t[0][3]), fmaxf(t[1][1], t[1][3]));
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) {
              g0 = fmaxf(g0, __shfl_xor_sync(0xffffffffu, g0, o));
              g1 = fmaxf(g1, __shfl_xor_sync(0xffffffffu, g1, o));
            }
            g0 += cst[0]; g1 += cst[1];
          }
          if (hd == 0) { gmax[i & 1][2 * r][warp] = g0; gmax[i & 1][2 * r + 1][warp] = g1; }
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
        float f[2], mu[2], off[2];
        bool moved = false;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const float4 ga = *reinterpret_cast<const float4*>(&gmax[i & 1][2 * r + x][0]);
          mu[x] = fmaxf(fmaxf(fmaxf(ga.x, ga.y), fmaxf(ga.z, ga.w)), gmax[i & 1][2 * r + x][4]) * sl2[x];   // sl2 > 0
        }
        if (STP) {
          run.exact[0] = fmaxf(run.exact[0], ceilf(mu[0])); run.exact[1] = fmaxf(run.exact[1], ceilf(mu[1]));
          moved = move_maximum(mu, run.m, f);
        } else {
          run.refer_to(mu, f);
        }
        off[0] = fmaf(cst[0], sl2[0], -run.m[0]); off[1] = fmaf(cst[1], sl2[1], -run.m[1]);
        // P[nt]: token 8 nt + hd of the warp's group, heads 2 r, 2 r + 1
        uint32_t P[4] = {0u, 0u, 0u, 0u};
        auto probabilities = [&]() {
#pragma unroll
          for (int nt = 0; nt < 4; ++nt)
            P[nt] = pack_half2(ex2_approx(fmaf(t[nt >> 1][2 * (nt & 1)], sl2[0], off[0])), ex2_approx(fmaf(t[nt >> 1][2 * (nt & 1) + 1], sl2[1], off[1])));
        };
        if (!STP) {
          if (warp < ng) probabilities();
          uint8_t* row = sm + S::prob_at + ((i & 1) * kStreamUnitTokens + warp * kG + hd) * kEntry + 4 * r;
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) *reinterpret_cast<uint32_t*>(row + 8 * nt * kEntry) = P[nt];
          // -5 * (sums of the rounded probabilities) of heads 2 r, 2 r + 1: a product with a matrix of -5
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) P[nt] = transpose_tile(P[nt]);
          float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
          mma_f16(c, kMinus5, kMinus5, kMinus5, kMinus5, P[0], P[1]);
          mma_f16(c, kMinus5, kMinus5, kMinus5, kMinus5, P[2], P[3]);
          if (hd == 0) psum[i & 1][warp][r] = make_float4(c[0], c[1], c[2], c[3]);
          if (k > k_begin) multiply(i - 1);
          unit_factor[0] = f[0]; unit_factor[1] = f[1];
        } else {
          const int u_old = u_hi, p_old = p_hi;
          p_hi = p_new;
          u_hi = t_end <= T_q0 ? t_end - p_new : u_fl0 + (t_end - T_q0);
          if (moved) {
            // what waits in the rings is in the old units: multiply what is complete, then rescale the rest
            multiply_streams(u_old, p_old);
            run.scale(f);
            __syncthreads();
            const __half2 f2 = __floats2half2_rn(f[0], f[1]);   // powers of two; at the start of a slab everything is cleared
            for (int j = tid; j < (kTRing + kPRing) * 4; j += kUnitThreads) {   // word j belongs to heads 2 (j % 4), + 1: this lane's
              __half2* q = reinterpret_cast<__half2*>(sm + S::prob_at) + j;
              *q = k > k_begin ? __hmul2(*q, f2) : __half2half2(__ushort_as_half(0));
            }
            __syncthreads();
          }
          // scattered into stream order.  Where a token goes depends on the token alone, so lane j works out the entry of the group's
          // token j and the lanes pick up the entries of their own four tokens with shuffles.
          if (warp < ng) {
            uint8_t* const ring = sm + S::prob_at + 4 * r;
            probabilities();
            if (tg < T_q0) {
              const int below = __popc(e_word & ((1u << lane) - 1u));
              const bool prot = (e_word >> lane) & 1u;
              const int dst = kEntry * (prot ? kTRing + ((e_base + below) & (kPRing - 1)) : (tg - e_base + lane - below) & (kTRing - 1));
#pragma unroll
              for (int nt = 0; nt < 4; ++nt) *reinterpret_cast<uint32_t*>(ring + __shfl_sync(0xffffffffu, dst, 8 * nt + hd)) = P[nt];
            } else {
              const int tmod = (u_fl0 + (tg - T_q0)) & (kTRing - 1);
#pragma unroll
              for (int nt = 0; nt < 4; ++nt) *reinterpret_cast<uint32_t*>(ring + (tmod + 8 * nt + hd) * kEntry) = P[nt];
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
            zero_ring(sm + S::prob_at + kTRing * kEntry, kPRing, p_hi, pg_end * kG);
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

template <bool GEN, bool STP, int kPerSM, typename T>
static cudaError_t launch_block_t(const DecodeArgs& a, cudaStream_t stream) {
  constexpr int smem = Smem<GEN, STP>::bytes;
  static bool attr_set[64] = {};
  int dev = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev))) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr_set[dev]) {
    if ((e = cudaFuncSetAttribute(decode_block_kernel<GEN, STP, kPerSM, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem))) return e;
    attr_set[dev] = true;
  }
  count_launches(1);
  return launch_dependent(decode_block_kernel<GEN, STP, kPerSM, T>, dim3(a.plan.n_blocks + a.plan.res_blocks), dim3(kUnitThreads), smem, stream, a);
}

template <bool GEN, typename T>
static cudaError_t launch_block_as(const DecodeArgs& a, bool stp, bool more, cudaStream_t stream) {
  if constexpr (!GEN) {
    if (stp && more) return launch_block_t<GEN, true, kMoreBlocksPerSM, T>(a, stream);
  }
  if (stp) return launch_block_t<GEN, true, kBlocksPerSM, T>(a, stream);
  return more ? launch_block_t<GEN, false, kMoreBlocksPerSM, T>(a, stream) : launch_block_t<GEN, false, kBlocksPerSM, T>(a, stream);
}

cudaError_t launch_decode_block(const DecodeArgs& a_in, cudaStream_t stream) {
  DecodeArgs a = a_in;
  const bool gen = a.cv.kf.general != 0, stp = a.n_prot > 0, half = a.in_dtype == VIDKV_F16;
  if (g_debug_withhold == 2) { a.withhold = stp ? 0 : 1; g_debug_withhold = 0; }
  const bool more = a.plan.blocks_per_sm == kMoreBlocksPerSM;
  if (gen) return half ? launch_block_as<true, __half>(a, stp, more, stream) : launch_block_as<true, __nv_bfloat16>(a, stp, more, stream);
  return half ? launch_block_as<false, __half>(a, stp, more, stream) : launch_block_as<false, __nv_bfloat16>(a, stp, more, stream);
}

}  // namespace vidkv
