// Scores q . K' of a 32-token key group, shared by the decode attention kernels.
//
// A code bit picks a row of the query operand: mma.sp (2:4 structured sparsity) multiplies every stored entry of A with the
// row of B that its two metadata bits name, so the codes are the metadata as they are packed (one mask and one OR for 16
// of them), A is the group's stored scales and B a pair of rows per channel, one for bit 0 and one for bit 1:
//   two-bit codes  c = b0 + 2 b1: rows (0, q), once with the b0 bits and once with the b1 bits, added with weight 2;
//   Eq. 5 columns  +-s: rows (-Q, Q) with Q as leading binary16 part + remainder;
//   plain one-bit  rows (0, q).
// Rows of the result = tokens, columns = query heads; the products s q are exact inside the tensor core, sums in float32.
// What bounds it is the quarter's issue port: fetching a product's operand registers blocks it as well (measured beside 8-12 FFMA, slots
// per product: dense m16n8k16 6.7, with the A of the product before 5.6; m16n8k32 with metadata 11, with A and B of the product before
// 9.3, of the three before 8.0, of the fifteen before 4.9).  So two groups go through together: rows 0-7 of every product are tokens of
// one, rows 8-15 of the other, and the products that share their scales and query rows come one behind the other.  Clocks per unit of
// five groups, 12 warps a multiprocessor: one group at a time 2109, pairs 1858; expanding the codes to binary16 operands (eight
// instructions a product, and q s split into hi + lo for every group) 2150.
#pragma once

#include "decode_device.cuh"

namespace vidkv {
namespace {

// Product with metadata e.  F: which lanes of a quad hold the metadata (r = 2 F: k 0-15, r = 2 F + 1: k 16-31; low half-word row g,
// high half-word row g + 8).
template <int F>
__device__ __forceinline__ void mma_sp(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1, uint32_t b2, uint32_t b3, uint32_t e) {
  asm volatile(
      "mma.sp::ordered_metadata.sync.aligned.m16n8k32.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9,%10,%11}, "
      "{%0,%1,%2,%3}, %12, %13;"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1), "r"(b2), "r"(b3), "r"(e), "n"(F));
}
// Metadata of the code bits at even positions of x: entry 2 j of a row names row 4 j or 4 j + 1, entry 2 j + 1 row 4 j + 2 or 4 j + 3.
__device__ __forceinline__ uint32_t bits_meta(uint32_t x) {
  uint32_t d;
  asm("lop3.b32 %0, %1, 0x55555555, 0x88888888, 0xEA;" : "=r"(d) : "r"(x));
  return d;
}
__device__ __forceinline__ uint32_t row_pair_lo(uint32_t w) { return w << 16; }              // (0, low half of w)
__device__ __forceinline__ uint32_t row_pair_hi(uint32_t w) { return w & 0xffff0000u; }      // (0, high half of w)
__device__ __forceinline__ uint32_t sign_pair_lo(uint32_t w) { return prmt(w, w, 0x1010u) ^ 0x00008000u; }   // (-x, x), x = low half
__device__ __forceinline__ uint32_t sign_pair_hi(uint32_t w) { return prmt(w, w, 0x3232u) ^ 0x00008000u; }

// Default format.  The A operands are the group's scales in the order of the codes, the same for every row of a product: the warp
// makes them once (a lane four scales of each group) and leaves them in the first group's own first 512 bytes, whose codes its lanes hold by then.
struct GroupBytes {
  uint4 c2;        // the lane's 2-bit codes
  uint2 c1;        // its 1-bit codes
  uint2 s;         // four scales: lanes 0-15 slots 16 b + 4 r .. + 3, lanes 16-31 columns 16 b + 12 - 4 r .. + 3 (b = lane / 4 % 4)
  __device__ __forceinline__ void fetch(const uint8_t* kg, int lane) {
    c2 = *reinterpret_cast<const uint4*>(kg + kKG_Codes2 + lane * 16);
    c1 = *reinterpret_cast<const uint2*>(kg + kKG_Bits1 + lane * 8);
    const int b = (lane >> 2) & 3, r = lane & 3;
    s = *reinterpret_cast<const uint2*>(kg + (lane < 16 ? kKG_S2 + 32 * b + 8 * r : kKG_S1 + 32 * b + 24 - 8 * r));
  }
};
// The A operands of two groups (rows 0-7: a's, 8-15: b's) into kg's first 512 bytes: operand (kind, f, par) of lane r has 16 bytes at
// kind 256 + f 128 + par 64 + r 16 (kind 0: two-bit slots, 1: spectrum columns).
__device__ __forceinline__ void put_scales(const GroupBytes& a, const GroupBytes& b, uint8_t* kg, int lane) {
  const int blk = (lane >> 2) & 3, r = lane & 3;
  const uint32_t s0 = lane < 16 ? 0x5410u : 0x3276u, s1 = lane < 16 ? 0x7632u : 0x1054u;
  uint8_t* o = kg + (lane < 16 ? 0 : 256) + (blk >> 1) * 128 + r * 16 + (blk & 1) * 8;
  *reinterpret_cast<uint2*>(o) = make_uint2(prmt(a.s.x, a.s.y, s0), prmt(b.s.x, b.s.y, s0));
  *reinterpret_cast<uint2*>(o + 64) = make_uint2(prmt(a.s.x, a.s.y, s1), prmt(b.s.x, b.s.y, s1));
}

// Products of NT row blocks: block m's codes are we[m] (even slots: the low half-words' tokens in rows 0-7, the high ones' in rows 8-15),
// odd slots wo[m], signs bits[m]; kg: where put_scales left the operands.  t = a0 + 2 a1.
// The query: q.pairs(f)[i] = binary16 pair of q at slots 8 (4 f + i) + 2 r, + 1 of head g (lane = 4 g + r); q.spectrum(f, par, h, l): (-Q, Q) at
// spectrum column 32 f + 16 (i / 2) + 15 - 8 (i % 2) - 2 r - par, leading part h[i] and remainder l[i].
template <int NT, typename Q>
__device__ __forceinline__ void score_blocks(const uint32_t (&we)[NT], const uint32_t (&wo)[NT], const uint32_t (&bits)[NT], const uint8_t* kg, int r,
                                             const Q& q, float (&t)[NT][4]) {
  const uint8_t* ap = kg + 16 * r;
  float a0[NT][4], a1[NT][4];       // weight 1, weight 2
#pragma unroll
  for (int m = 0; m < NT; ++m)
#pragma unroll
    for (int i = 0; i < 4; ++i) { a0[m][i] = 0.0f; a1[m][i] = 0.0f; }
#pragma unroll
  for (int par = 0; par < 2; ++par) {
    uint32_t lo[NT], hi[NT], sg[NT];
#pragma unroll
    for (int m = 0; m < NT; ++m) {
      const uint32_t w = par ? wo[m] : we[m];
      lo[m] = bits_meta(w); hi[m] = bits_meta(w >> 1); sg[m] = bits_meta(par ? bits[m] >> 1 : bits[m]);
    }
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      uint32_t b[4], h[4], l[4];
      const uint4 qp = q.pairs(f);
      b[0] = par ? row_pair_hi(qp.x) : row_pair_lo(qp.x); b[1] = par ? row_pair_hi(qp.y) : row_pair_lo(qp.y);
      b[2] = par ? row_pair_hi(qp.z) : row_pair_lo(qp.z); b[3] = par ? row_pair_hi(qp.w) : row_pair_lo(qp.w);
      q.spectrum(f, par, h, l);
      const uint4 s2 = *reinterpret_cast<const uint4*>(ap + 128 * f + 64 * par), s1 = *reinterpret_cast<const uint4*>(ap + 256 + 128 * f + 64 * par);
#pragma unroll
      for (int m = 0; m < NT; ++m) {
        if (f == 0) mma_sp<0>(a0[m], s2, b[0], b[1], b[2], b[3], lo[m]);
        else mma_sp<1>(a0[m], s2, b[0], b[1], b[2], b[3], lo[m]);
      }
#pragma unroll
      for (int m = 0; m < NT; ++m) {
        if (f == 0) mma_sp<0>(a1[m], s2, b[0], b[1], b[2], b[3], hi[m]);
        else mma_sp<1>(a1[m], s2, b[0], b[1], b[2], b[3], hi[m]);
      }
#pragma unroll
      for (int m = 0; m < NT; ++m) {
        if (f == 0) mma_sp<0>(a0[m], s1, h[0], h[1], h[2], h[3], sg[m]);
        else mma_sp<1>(a0[m], s1, h[0], h[1], h[2], h[3], sg[m]);
      }
#pragma unroll
      for (int m = 0; m < NT; ++m) {
        if (f == 0) mma_sp<0>(a0[m], s1, l[0], l[1], l[2], l[3], sg[m]);
        else mma_sp<1>(a0[m], s1, l[0], l[1], l[2], l[3], sg[m]);
      }
    }
  }
#pragma unroll
  for (int m = 0; m < NT; ++m)
#pragma unroll
    for (int i = 0; i < 4; ++i) t[m][i] = fmaf(2.0f, a1[m][i], a0[m][i]);
}
// Scores without their group's constant, in the units of the normalised query: t[m] = tokens 16 m + g (heads 2 r, 2 r + 1) and
// 16 m + 8 + g of one group ...
template <typename Q>
__device__ __forceinline__ void score_group(const GroupBytes& a, const uint8_t* kg, int r, const Q& q, float (&t)[2][4]) {
  const uint32_t we[2] = {prmt(a.c2.x, a.c2.y, 0x5410u), prmt(a.c2.z, a.c2.w, 0x5410u)}, wo[2] = {prmt(a.c2.x, a.c2.y, 0x7632u), prmt(a.c2.z, a.c2.w, 0x7632u)};
  const uint32_t bits[2] = {a.c1.x, a.c1.y};
  score_blocks<2>(we, wo, bits, kg, r, q, t);
}
// ... and of two.
template <typename Q>
__device__ __forceinline__ void score_groups(const GroupBytes& a, const GroupBytes& b, const uint8_t* kg, int r, const Q& q, float (&ta)[2][4],
                                             float (&tb)[2][4]) {
  const uint32_t wa[4] = {a.c2.x, a.c2.y, a.c2.z, a.c2.w}, wb[4] = {b.c2.x, b.c2.y, b.c2.z, b.c2.w};
  uint32_t we[4], wo[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) { we[m] = prmt(wa[m], wb[m], 0x5410u); wo[m] = prmt(wa[m], wb[m], 0x7632u); }
  const uint32_t bits[4] = {prmt(a.c1.x, b.c1.x, 0x5410u), prmt(a.c1.x, b.c1.x, 0x7632u), prmt(a.c1.y, b.c1.y, 0x5410u), prmt(a.c1.y, b.c1.y, 0x7632u)};
  float t[4][4];
  score_blocks<4>(we, wo, bits, kg, r, q, t);
#pragma unroll
  for (int m = 0; m < 4; ++m)
#pragma unroll
    for (int x = 0; x < 2; ++x) { ta[m >> 1][2 * (m & 1) + x] = t[m][x]; tb[m >> 1][2 * (m & 1) + x] = t[m][2 + x]; }
}

// The constants sum q z of up to eight groups at once: c[0], c[1] = those of group min(g, n - 1) and heads 2 r, 2 r + 1.
template <typename Q>
__device__ __forceinline__ void group_constants(const uint8_t* kbuf, int n, int g, int r, const Q& q, float (&c)[2]) {
  const uint8_t* z = kbuf + min(g, n - 1) * kKGroupBytes + kKG_Z2 + 4 * r;
  float d[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  auto word = [&](int at) { return *reinterpret_cast<const uint32_t*>(z + at); };
#pragma unroll
  for (int f = 0; f < 2; ++f) {
    const uint4 qp = q.pairs(f);
    mma_f16(d, word(64 * f), 0u, word(64 * f + 16), 0u, qp.x, qp.y);
    mma_f16(d, word(64 * f + 32), 0u, word(64 * f + 48), 0u, qp.z, qp.w);
  }
  c[0] = d[0]; c[1] = d[1];
}

// The same for the general layout (KeyFmt), one group (ga) or two.  word(j): this lane's query words of the groups' chunk, word.four(j)
// four of them from a multiple of four on: n2 / 8 pairs of q at slots 8 j + 2 r, + 1; then pairs at the one-bit columns 8 j + 6 - 2 r, + 1:
// of q in plain mode, of Q's leading part and then of its remainder for Eq. 5.
template <bool TWO, typename Word>
__device__ __forceinline__ void score_general(const uint8_t* ga, const uint8_t* gb, const KeyFmt& kf, int lane, int r, Word word, float (&t)[TWO ? 4 : 2][4]) {
  constexpr int NT = TWO ? 4 : 2;
  float a0[NT][4], a1[NT][4];
#pragma unroll
  for (int m = 0; m < NT; ++m)
#pragma unroll
    for (int i = 0; i < 4; ++i) { a0[m][i] = 0.0f; a1[m][i] = 0.0f; }
  const int n2b = kf.n2 >> 5, n1b = (kD - kf.n2) >> 5;
  const uint32_t sel2 = r < 2 ? 0x5410u : 0x7632u, sel1 = r < 2 ? 0x3276u : 0x1054u;
  // scales of eight channels in the order of the codes' entries, at byte offset `at` of the groups: the operand registers of rows 0-7 and 8-15
  auto scales = [&](int at, uint32_t sel, uint32_t& x, uint32_t& y) {
    const uint2 va = *reinterpret_cast<const uint2*>(ga + at);
    x = prmt(va.x, va.y, sel);
    if (TWO) {
      const uint2 vb = *reinterpret_cast<const uint2*>(gb + at);
      y = prmt(vb.x, vb.y, sel);
    } else {
      y = x;
    }
  };
#pragma unroll 1
  for (int b = 0; b < n2b; ++b) {
    uint4 q;
    uint32_t lo[NT], hi[NT];
    uint4 sa, sb;
    const int at = kf.off_s2 + 64 * b + 8 * (r & 1);
    scales(at, sel2, sa.x, sa.y); scales(at + 16, sel2, sa.z, sa.w); scales(at + 32, sel2, sb.x, sb.y); scales(at + 48, sel2, sb.z, sb.w);
    q = word.four(4 * b);
    const uint2 ca = *reinterpret_cast<const uint2*>(ga + 256 * b + lane * 8);
    uint32_t w[NT];
    if constexpr (TWO) {
      const uint2 cb = *reinterpret_cast<const uint2*>(gb + 256 * b + lane * 8);
      w[0] = prmt(ca.x, cb.x, 0x5410u); w[1] = prmt(ca.x, cb.x, 0x7632u); w[2] = prmt(ca.y, cb.y, 0x5410u); w[3] = prmt(ca.y, cb.y, 0x7632u);
    } else {
      w[0] = ca.x; w[1] = ca.y;
    }
#pragma unroll
    for (int m = 0; m < NT; ++m) { lo[m] = bits_meta(w[m]); hi[m] = bits_meta(w[m] >> 1); }
#pragma unroll
    for (int m = 0; m < NT; ++m) mma_sp<0>(a0[m], sa, row_pair_lo(q.x), row_pair_hi(q.x), row_pair_lo(q.y), row_pair_hi(q.y), lo[m]);
#pragma unroll
    for (int m = 0; m < NT; ++m) mma_sp<0>(a1[m], sa, row_pair_lo(q.x), row_pair_hi(q.x), row_pair_lo(q.y), row_pair_hi(q.y), hi[m]);
#pragma unroll
    for (int m = 0; m < NT; ++m) mma_sp<1>(a0[m], sb, row_pair_lo(q.z), row_pair_hi(q.z), row_pair_lo(q.w), row_pair_hi(q.w), lo[m]);
#pragma unroll
    for (int m = 0; m < NT; ++m) mma_sp<1>(a1[m], sb, row_pair_lo(q.z), row_pair_hi(q.z), row_pair_lo(q.w), row_pair_hi(q.w), hi[m]);
  }
  const int w1 = kf.n2 >> 3, nw1 = (kD - kf.n2) >> 3;
#pragma unroll 1
  for (int b = 0; b < n1b; ++b) {
    uint4 q;
    uint32_t e[NT];
    uint4 sa, sb;
    const int at = kf.off_s1 + 64 * b + 8 - 8 * (r & 1);
    scales(at, sel1, sa.x, sa.y); scales(at + 16, sel1, sa.z, sa.w); scales(at + 32, sel1, sb.x, sb.y); scales(at + 48, sel1, sb.z, sb.w);
    q = word.four(w1 + 4 * b);
    const uint32_t ca = *reinterpret_cast<const uint32_t*>(ga + kf.off_bits1 + 128 * b + lane * 4);
    const uint32_t cb = TWO ? *reinterpret_cast<const uint32_t*>(gb + kf.off_bits1 + 128 * b + lane * 4) : 0u;
#pragma unroll
    for (int m = 0; m < NT; ++m) {
      // a token's byte twice in its half-word: the even bits stay in the low byte, the odd ones move down one in the high byte
      const uint32_t u = TWO ? prmt(ca, cb, 0x4400u + 0x1111u * m) : prmt(ca, 0u, m ? 0x3322u : 0x1100u);
      e[m] = bits_meta((u & 0x00ff00ffu) | ((u >> 1) & 0xff00ff00u));
    }
    if (kf.plain) {
#pragma unroll
      for (int m = 0; m < NT; ++m) mma_sp<0>(a0[m], sa, row_pair_hi(q.x), row_pair_lo(q.x), row_pair_hi(q.y), row_pair_lo(q.y), e[m]);
#pragma unroll
      for (int m = 0; m < NT; ++m) mma_sp<1>(a0[m], sb, row_pair_hi(q.z), row_pair_lo(q.z), row_pair_hi(q.w), row_pair_lo(q.w), e[m]);
    } else {
#pragma unroll
      for (int piece = 0; piece < 2; ++piece) {
#pragma unroll
        for (int m = 0; m < NT; ++m) mma_sp<0>(a0[m], sa, sign_pair_hi(q.x), sign_pair_lo(q.x), sign_pair_hi(q.y), sign_pair_lo(q.y), e[m]);
#pragma unroll
        for (int m = 0; m < NT; ++m) mma_sp<1>(a0[m], sb, sign_pair_hi(q.z), sign_pair_lo(q.z), sign_pair_hi(q.w), sign_pair_lo(q.w), e[m]);
        if (piece == 0) q = word.four(w1 + nw1 + 4 * b);
      }
    }
  }
#pragma unroll
  for (int m = 0; m < NT; ++m)
#pragma unroll
    for (int i = 0; i < 4; ++i) t[m][i] = fmaf(2.0f, a1[m][i], a0[m][i]);
}
template <typename Word>
__device__ __forceinline__ void score_group_general(const uint8_t* ga, const KeyFmt& kf, int lane, int r, Word word, float (&t)[2][4]) {
  score_general<false>(ga, ga, kf, lane, r, word, t);
}
template <typename Word>
__device__ __forceinline__ void score_groups_general(const uint8_t* ga, const uint8_t* gb, const KeyFmt& kf, int lane, int r, Word word, float (&ta)[2][4],
                                                     float (&tb)[2][4]) {
  float t[4][4];
  score_general<true>(ga, gb, kf, lane, r, word, t);
#pragma unroll
  for (int m = 0; m < 4; ++m)
#pragma unroll
    for (int x = 0; x < 2; ++x) { ta[m >> 1][2 * (m & 1) + x] = t[m][x]; tb[m >> 1][2 * (m & 1) + x] = t[m][2 + x]; }
}

template <typename Word>
__device__ __forceinline__ void group_constants_general(const uint8_t* kbuf, const KeyFmt& kf, int n, int g, int r, Word word, float (&c)[2]) {
  const uint8_t* kg = kbuf + min(g, n - 1) * kf.group_bytes;
  float d[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
  for (int j = 0; j < kf.n2 >> 3; j += 2)
    mma_f16(d, *reinterpret_cast<const uint32_t*>(kg + kf.off_z2 + 16 * j + 4 * r), 0u, *reinterpret_cast<const uint32_t*>(kg + kf.off_z2 + 16 * j + 16 + 4 * r),
            0u, word(j), word(j + 1));
  if (kf.plain) {
    const int w1 = kf.n2 >> 3;
#pragma unroll 1
    for (int j = 0; j < (kD - kf.n2) >> 3; j += 2)
      mma_f16(d, *reinterpret_cast<const uint32_t*>(kg + kf.off_z1 + 16 * j + 12 - 4 * r), 0u,
              *reinterpret_cast<const uint32_t*>(kg + kf.off_z1 + 16 * j + 28 - 4 * r), 0u, word(w1 + j), word(w1 + j + 1));
  }
  c[0] = d[0]; c[1] = d[1];
}

// Entries of 32 positions as the B operand of P V: P[nt] = head lane / 4 at positions 8 nt + 2 (lane % 4), + 1.  An entry is a
// position's binary16 probabilities of the eight heads, 16 bytes; `row` is the shared-memory address of the lane's own position.
constexpr int kEntry = 16;
// The same within registers for an 8-token tile: lane (token g, heads 2 r, 2 r + 1) -> lane (head g, tokens 2 r, 2 r + 1).
__device__ __forceinline__ uint32_t transpose_tile(uint32_t x) {
  uint32_t d;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(x));
  return d;
}
__device__ __forceinline__ void load_entries(uint32_t row, uint32_t (&P)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(P[0]), "=r"(P[1]), "=r"(P[2]), "=r"(P[3]) : "r"(row) : "memory");
}

}  // namespace
}  // namespace vidkv
