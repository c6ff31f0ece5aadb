// Decode attention over the packed cache for caches without protected tokens (Algorithm 1
// "Decoding", Eq. 3): the stream kernel.
//
// The quantized tokens of all slabs of a call form one sequence of 160-token units (five
// 32-token key groups and the ternary supergroup that holds the same tokens' values).  Every
// warp of the launch owns a contiguous run of units and works through it alone, the way a
// streaming softmax does:
//   1. the unit's key groups arrive in the warp's key buffer by one bulk copy
//      (cp.async.bulk + mbarrier); the scores q . K' of its 160 tokens come out of products whose
//      sparsity metadata are the codes (decode_score.cuh), rows = tokens, columns = query heads;
//   2. the probabilities 2^(logit - reference), binary16, are transposed in registers (movmatrix) into the
//      B fragment of the next product;
//   3. the unit's ternary supergroup (second bulk copy, in flight during step 1) is peeled digit
//      by digit into 5 + trit, multiplied with the probabilities into per-group accumulators
//      that start at -5 sum p (the sums come from a product with a constant matrix, which also
//      yields the softmax denominator), and the per-(group, channel) scales fold the group
//      accumulators into the warp's running output for all 128 channels x 8 heads.
// While a unit is being worked on, the next unit's keys and values are already on their way
// into the two buffers (a buffer is refilled as soon as its reader is done).  A warp leaves one
// partial record (maximum, sum, out[128]) per query head for every slab its run touches; the
// merge kernel combines them and attends to the FP16 / BF16 residual.
//
// Nothing is shared between warps: no block-wide barrier, no shared score matrix.
#include "decode_score.cuh"

namespace vidkv {

namespace {

constexpr int kTotBytes = 4 * 2 * 32 * 16;             // 4096: the warp's running output (128 channels x 8 heads, float)
constexpr int kWarpBufBytes = kKBufBytes + kVBufBytes + kTotBytes;   // 15232 per warp

// Per-lane state of the running softmax of one slab, heads 2 r and 2 r + 1 (the running output itself is in shared memory).
struct Running {
  float m[2];           // reference that the running sums are in units of (base-2 logit)
  float top[2];         // the largest unit maximum so far
  float l[2];           // sums of the probabilities
  __device__ __forceinline__ void reset() {
    m[0] = -INFINITY; m[1] = -INFINITY; top[0] = -INFINITY; top[1] = -INFINITY; l[0] = 0.0f; l[1] = 0.0f;
  }
};

// What a lane keeps of one chunk's prepared query.
template <bool GEN> struct Query;
template <> struct Query<false> {
  uint32_t q[8], qh[16], ql[16];      // as score_blocks takes them: words 4 f + i and (2 f + par) 4 + i
  __device__ __forceinline__ uint4 pairs(int f) const { return make_uint4(q[4 * f], q[4 * f + 1], q[4 * f + 2], q[4 * f + 3]); }
  __device__ __forceinline__ void spectrum(int f, int par, uint32_t (&h)[4], uint32_t (&l)[4]) const {
#pragma unroll
    for (int i = 0; i < 4; ++i) { h[i] = qh[(2 * f + par) * 4 + i]; l[i] = ql[(2 * f + par) * 4 + i]; }
  }
  __device__ __forceinline__ void load(const uint32_t* pp) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      q[j] = pp[j * 32];
      const uint32_t h = pp[(8 + j) * 32], l = pp[(16 + j) * 32];
      const int at = (j >> 2) * 8 + (j & 3);
      qh[at] = (h & 0xffff0000u) | ((h >> 16) ^ 0x8000u); qh[at + 4] = (h << 16) | ((h & 0xffffu) ^ 0x8000u);   // (-x, x) of either half
      ql[at] = (l & 0xffff0000u) | ((l >> 16) ^ 0x8000u); ql[at + 4] = (l << 16) | ((l & 0xffffu) ^ 0x8000u);
    }
  }
  __device__ __forceinline__ void constants(const uint8_t* kbuf, const KeyFmt&, int n, int g, int r, float (&c)[2]) const {
    group_constants(kbuf, n, g, r, *this, c);
  }
  __device__ __forceinline__ void score(uint8_t* ga, uint8_t* gb, const KeyFmt&, int lane, int r, float (&ta)[2][4], float (&tb)[2][4]) const {
    GroupBytes a, b;
    a.fetch(ga, lane);
    b.fetch(gb, lane);
    __syncwarp();
    put_scales(a, b, ga, lane);
    __syncwarp();
    score_groups(a, b, ga, r, *this, ta, tb);
  }
  __device__ __forceinline__ void score(uint8_t* ga, const KeyFmt&, int lane, int r, float (&t)[2][4]) const {
    GroupBytes a;
    a.fetch(ga, lane);
    __syncwarp();
    put_scales(a, a, ga, lane);
    __syncwarp();
    score_group(a, ga, r, *this, t);
  }
};
template <> struct Query<true> {
  struct Words {
    const uint32_t* p;
    __device__ __forceinline__ uint32_t operator()(int j) const { return p[j * 32]; }
    __device__ __forceinline__ uint4 four(int j) const { return make_uint4((*this)(j), (*this)(j + 1), (*this)(j + 2), (*this)(j + 3)); }
  };
  const uint32_t* p;                  // the words stay in global memory (L1): five formats share one instantiation
  __device__ __forceinline__ void load(const uint32_t* pp) { p = pp; }
  __device__ __forceinline__ void constants(const uint8_t* kbuf, const KeyFmt& kf, int n, int g, int r, float (&c)[2]) const {
    group_constants_general(kbuf, kf, n, g, r, Words{p}, c);
  }
  __device__ __forceinline__ void score(uint8_t* ga, uint8_t* gb, const KeyFmt& kf, int lane, int r, float (&ta)[2][4], float (&tb)[2][4]) const {
    score_groups_general(ga, gb, kf, lane, r, Words{p}, ta, tb);
  }
  __device__ __forceinline__ void score(uint8_t* ga, const KeyFmt& kf, int lane, int r, float (&t)[2][4]) const {
    score_group_general(ga, kf, lane, r, Words{p}, t);
  }
};

// The lane's words of the prepared query of a slab's first chunk.
__device__ __forceinline__ const uint32_t* prep_words(const DecodeArgs& a, int slab, int lane) {
  return a.prep + static_cast<int64_t>(slab) * a.plan.n_chunks * (kPrepWords * 32) + lane;
}

// A group's scores, without its constant, replace its (spent) bytes in the key buffer: 16 bytes of tokens 16 m + g and + 8 at
// (m * 32 + lane) * 16; the lane's maxima follow.
__device__ __forceinline__ void park(uint8_t* kg, const float (&t)[2][4], int gi, const float (&cst)[2], float (&mx)[2], int lane, int r) {
#pragma unroll
  for (int m = 0; m < 2; ++m) reinterpret_cast<float4*>(kg)[m * 32 + lane] = make_float4(t[m][0], t[m][1], t[m][2], t[m][3]);
  const float c0 = __shfl_sync(0xffffffffu, cst[0], 4 * gi + r), c1 = __shfl_sync(0xffffffffu, cst[1], 4 * gi + r);
  mx[0] = fmaxf(mx[0], fmaxf(fmaxf(t[0][0], t[0][2]), fmaxf(t[1][0], t[1][2])) + c0);
  mx[1] = fmaxf(mx[1], fmaxf(fmaxf(t[0][1], t[0][3]), fmaxf(t[1][1], t[1][3])) + c1);
}

// Scores of the unit's ng groups, the first of which is key group g_first of its slab, two at a time; cur_chunk is the chunk whose query
// is in qy.  cst: lane (g, r)'s are the constants of group g and heads 2 r, 2 r + 1; mx: the unit's maxima of these heads.
template <bool GEN>
__device__ __forceinline__ void score_unit(const DecodeArgs& a, int slab, uint8_t* kbuf, int kgb, int ng, int g_first, int& cur_chunk, Query<GEN>& qy,
                                           int lane, int g, int r, float (&cst)[2], float (&mx)[2]) {
  const KeyFmt& kf = a.cv.kf;
  const int g0n = static_cast<int>(a.st.T_q0 / kG);
  mx[0] = -INFINITY; mx[1] = -INFINITY;
  auto chunk_of = [&](int gidx) { return gidx < g0n ? 0 : 1 + static_cast<int>(static_cast<unsigned>(gidx - g0n) / (kR / kG)); };
  int gi = 0;
#pragma unroll 1
  while (gi < ng) {
    const int chunk = chunk_of(g_first + gi);
    const bool fresh = chunk != cur_chunk, two = gi + 1 < ng && chunk_of(g_first + gi + 1) == chunk;
    if (__builtin_expect(fresh, 0)) {
      cur_chunk = chunk;
      qy.load(prep_words(a, slab, lane) + static_cast<int64_t>(chunk) * (kPrepWords * 32));
    }
    if (fresh || gi == 0) {
      // constants of this group and those behind it, lane g's for group g (the bytes of the groups before are spent)
      float c[2];
      qy.constants(kbuf, kf, ng, g, r, c);
      if (g >= gi) { cst[0] = c[0]; cst[1] = c[1]; }
    }
    uint8_t* kg = kbuf + gi * kgb;
    float ta[2][4], tb[2][4];
    if (two) {
      qy.score(kg, kg + kgb, kf, lane, r, ta, tb);
      __syncwarp();                                         // every lane has read the groups' bytes
      park(kg, ta, gi, cst, mx, lane, r);
      park(kg + kgb, tb, gi + 1, cst, mx, lane, r);
      gi += 2;
    } else {
      qy.score(kg, kf, lane, r, ta);
      __syncwarp();
      park(kg, ta, gi, cst, mx, lane, r);
      ++gi;
    }
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    mx[0] = fmaxf(mx[0], __shfl_xor_sync(0xffffffffu, mx[0], o));
    mx[1] = fmaxf(mx[1], __shfl_xor_sync(0xffffffffu, mx[1], o));
  }
}

// A load that stays where it stands.  What a warp reads once a slab is kept out of the compiler's reach (these factors, the pairs made of the
// query words, the branch that takes a new chunk's): read as any other word it gave the loop for protected tokens other registers, 32
// slabs of 1225 units 253.8 us against 249.6 so, 448 of 79 229.8 against 226.5.
__device__ __forceinline__ float load_here(const uint32_t* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
// The factors of heads 2 r, 2 r + 1 that turn a score in the units of the normalised query into a base-2 logit (word 24 of lane 4 h
// holds head h's; prep_slab points at the lane's own words).
__device__ __forceinline__ void head_factors(const uint32_t* prep_slab, int lane, int r, float (&sl2)[2]) {
  sl2[0] = load_here(prep_slab + 24 * 32 - lane + 8 * r);
  sl2[1] = load_here(prep_slab + 24 * 32 - lane + 8 * r + 4);
}

// Probabilities of group gi: P[nt] = binary16 pair of heads 2 r, 2 r + 1 and token 8 nt + g.
__device__ __forceinline__ void probabilities(const uint8_t* kg, int gi, int lane, int r, const float (&cst)[2], const float (&sl2)[2], const float (&m)[2],
                                              uint32_t (&P)[4]) {
  const float off0 = fmaf(__shfl_sync(0xffffffffu, cst[0], 4 * gi + r), sl2[0], -m[0]);
  const float off1 = fmaf(__shfl_sync(0xffffffffu, cst[1], 4 * gi + r), sl2[1], -m[1]);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float4 v = reinterpret_cast<const float4*>(kg)[i * 32 + lane];
    P[2 * i] = pack_half2(ex2_approx(fmaf(v.x, sl2[0], off0)), ex2_approx(fmaf(v.y, sl2[1], off1)));
    P[2 * i + 1] = pack_half2(ex2_approx(fmaf(v.z, sl2[0], off0)), ex2_approx(fmaf(v.w, sl2[1], off1)));
  }
}

// Running output of the warp, kept in shared memory: float4 tot[j][lane], j = 2 w + i, holds the
// accumulator fragment of channels 32 w + 4 hd + 2 i + (e >> 1) and heads 2 r + (e & 1), e = 0..3.

__device__ __forceinline__ void scale_output(float* totbuf, float fa, float fb, int lane) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    float4* t = reinterpret_cast<float4*>(totbuf) + j * 32 + lane;
    float4 v = *t;
    v.x *= fa; v.y *= fb; v.z *= fa; v.w *= fb;
    *t = v;
  }
}

// P V of one staged ternary supergroup, its first ng groups (FULL: five; the others' probabilities are zero): P[g][nt] holds the probabilities of
// head hd at stream tokens 32 g + 8 nt + 2 r, + 1 (binary16 pairs) and ps[g] the accumulator
// fragment -5 * (sum of those probabilities) of heads 2 r, 2 r + 1.  32 channels (two MMA row
// blocks) at a time: fragment i of block w covers channels 32 w + 4 hd + 2 i + {0, 1} in rows hd,
// hd + 8.  Adds into the warp's running output, which RESCALE multiplies by fa (heads 2 r) and fb (heads 2 r + 1) first.
template <bool FULL, bool RESCALE>
__device__ __forceinline__ void pv_ternary(const uint8_t* vbuf, float* totbuf, int ng, const uint32_t (&P)[kSGGroups][4],
                                           const float (&ps)[kSGGroups][4], float fa, float fb, int lane, int hd, int r) {
#pragma unroll 1
  for (int w = 0; w < 4; ++w) {
    float4* tp = reinterpret_cast<float4*>(totbuf) + (2 * w) * 32 + lane;
    float4 t0 = tp[0], t1 = tp[32];
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
    if (RESCALE) {
      t0.x *= fa; t0.y *= fb; t0.z *= fa; t0.w *= fb;
      t1.x *= fa; t1.y *= fb; t1.z *= fa; t1.w *= fb;
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
        const uint32_t b0 = P[g][2 * kt], b1 = P[g][2 * kt + 1];
        if (kt == 0) {
          mma_f16_c(acc[0], A[0], A[1], A[2], A[3], b0, b1, ps[g][0], ps[g][1], ps[g][2], ps[g][3]);
          mma_f16_c(acc[1], A[4], A[5], A[6], A[7], b0, b1, ps[g][0], ps[g][1], ps[g][2], ps[g][3]);
        } else {
          mma_f16(acc[0], A[0], A[1], A[2], A[3], b0, b1);
          mma_f16(acc[1], A[4], A[5], A[6], A[7], b0, b1);
        }
      }
      uint2 sc2 = *reinterpret_cast<const uint2*>(vbuf + kSG_Scales + g * (kD * 2) + (32 * w + 4 * hd) * 2);
      if (!FULL && g >= ng) sc2 = make_uint2(0u, 0u);       // nobody has written the scales of a group that does not exist
      const float2 sa = __half22float2(*reinterpret_cast<const __half2*>(&sc2.x));
      const float2 sb = __half22float2(*reinterpret_cast<const __half2*>(&sc2.y));
      t0.x += sa.x * acc[0][0]; t0.y += sa.x * acc[0][1];
      t0.z += sa.y * acc[0][2]; t0.w += sa.y * acc[0][3];
      t1.x += sb.x * acc[1][0]; t1.y += sb.x * acc[1][1];
      t1.z += sb.y * acc[1][2]; t1.w += sb.y * acc[1][3];
    }
    tp[0] = t0;
    tp[32] = t1;
  }
}

// One unit of ng groups (FULL: five): scores, probabilities, P V into the running state.
// Returns false if a copy never arrived.
// SHARD (the call leaves triples): the probabilities are taken against the running maximum, which is part of the result
// and fixes the cut.  Otherwise against the unit's own maximum: where their binary16 rounding falls depends on the unit
// alone, not on where the warp's run began, and the largest one is exact; the running sums are brought to the unit's
// reference first.  Off by 3.3e-5 of the outputs' norm on 64 slabs x 12544 tokens, where the running maximum gives
// 1.14e-4 and another cut moves the outputs by 1.5e-4; 32 steps of 1792 slabs x 79 units take 25.89 ms that way, 25.61 ms
// against the running maximum.
template <bool FULL, bool GEN, bool SHARD>
__device__ __forceinline__ bool process_unit(const DecodeArgs& a, int slab, int k, bool more, const uint8_t* slab_ptr, Query<GEN>& qy, uint8_t* kbuf,
                                             uint8_t* vbuf, float* totbuf, uint64_t* kbar, uint64_t* vbar, uint32_t& kpar, uint32_t& vpar, int lane, int hd,
                                             int r, int& cur_chunk, const float (&sl2)[2], Running& run) {
  const CacheView& cv = a.cv;
  const int kgb = GEN ? cv.kf.group_bytes : kKGroupBytes;   // bytes of one key group
  const int n_groups = static_cast<int>((a.st.T_q0 + a.st.n_flush * kR) / kG), ng = FULL ? kSGGroups : n_groups - k * kSGGroups;
  if (!mbar_wait(kbar, kpar)) {
    mbar_wait(vbar, vpar);                                  // the unit's value copy is under way: let it land before leaving
    return false;
  }
  kpar ^= 1u;
  float cst[2], mx[2];
  score_unit<GEN>(a, slab, kbuf, kgb, ng, k * kSGGroups, cur_chunk, qy, lane, hd, r, cst, mx);
  // ---- maximum of the unit, reference, probabilities
  const float mu[2] = {mx[0] * sl2[0], mx[1] * sl2[1]};     // sl2 > 0
  float fa = 1.0f, fb = 1.0f;
  if (!SHARD) {
    float f[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      run.top[x] = fmaxf(run.top[x], mu[x]);
      const float ref = fmaxf(mu[x], run.top[x] - kRefLag);
      f[x] = ex2_approx(run.m[x] - ref);                    // 0 for the first unit (run.m = -inf)
      run.m[x] = ref;
      run.l[x] *= f[x];
    }
    fa = f[0]; fb = f[1];
  } else {
    const bool up0 = mu[0] > run.m[0] + kStaleLog2, up1 = mu[1] > run.m[1] + kStaleLog2;   // always true for the first unit (run.m = -inf)
    if (__any_sync(0xffffffffu, up0 || up1)) {
      const float m0 = up0 ? mu[0] : run.m[0], m1 = up1 ? mu[1] : run.m[1];
      const float ga = ex2_approx(run.m[0] - m0), gb = ex2_approx(run.m[1] - m1);          // 1 for heads whose maximum stays
      run.m[0] = m0; run.m[1] = m1;
      scale_output(totbuf, ga, gb, lane);
      run.l[0] *= ga; run.l[1] *= gb;
    }
  }
  uint32_t P[kSGGroups][4];
  float ps[kSGGroups][4];
#pragma unroll
  for (int g = 0; g < kSGGroups; ++g) {
    probabilities(kbuf + g * kgb, g, lane, r, cst, sl2, run.m, P[g]);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      P[g][nt] = transpose_tile(P[g][nt]);
      if (!FULL && g >= ng) P[g][nt] = 0u;                  // what lies behind the unit's last group is not a score
    }
    // -5 * (sums of the rounded probabilities) of heads 2 r, 2 r + 1, for rows hd and hd + 8 alike:
    // a product with a matrix of -5, whose accumulator fragment is the initial value of every
    // P V accumulator of the group as it stands
    ps[g][0] = 0.0f; ps[g][1] = 0.0f; ps[g][2] = 0.0f; ps[g][3] = 0.0f;
    mma_f16(ps[g], kMinus5, kMinus5, kMinus5, kMinus5, P[g][0], P[g][1]);
    mma_f16(ps[g], kMinus5, kMinus5, kMinus5, kMinus5, P[g][2], P[g][3]);
    run.l[0] = fmaf(-0.2f, ps[g][0], run.l[0]);
    run.l[1] = fmaf(-0.2f, ps[g][1], run.l[1]);
  }
  __syncwarp();                                             // the scores are in registers: the key buffer is free
  // the unit behind this one: the slab's next, or the next slab's first
  const bool last = k + 1 == a.plan.units_per_slab;
  const int nk = last ? 0 : k + 1;
  const uint8_t* next = slab_ptr + (last ? cv.slab_stride : 0);
  if (more && lane == 0) {
    // the buffer was used through ordinary loads and stores; order them before the bulk copy's writes
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    bulk_load(kbuf, next + cv.kgroup_offset + static_cast<int64_t>(nk) * (kSGGroups * kgb), min(kSGGroups, n_groups - nk * kSGGroups) * kgb, kbar);
  }
  // ---- P V over the ternary supergroup
  if (!mbar_wait(vbar, vpar)) {
    if (more) mbar_wait(kbar, kpar);                        // let the key copy issued above land before leaving
    return false;
  }
  vpar ^= 1u;
  pv_ternary<FULL, !SHARD>(vbuf, totbuf, ng, P, ps, fa, fb, lane, hd, r);
  __syncwarp();
  if (more && lane == 0) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    bulk_load(vbuf, next + cv.tern_offset + static_cast<int64_t>(nk) * kVBufBytes, kVBufBytes, vbar);
  }
  return true;
}

__device__ __forceinline__ void write_record(const DecodeArgs& a, int slab, int run_id, int lane, int hd, int r,
                                             const Running& run, const float* totbuf) {
  const int rep = a.cv.rep;
  float* rec = a.partials + static_cast<int64_t>(slab + run_id) * (kMaxRep * kRecordFloats);
#pragma unroll
  for (int w = 0; w < 4; ++w)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float4 t = reinterpret_cast<const float4*>(totbuf)[(w * 2 + i) * 32 + lane];
      const int c = 32 * w + 4 * hd + 2 * i;
      if (2 * r < rep) {
        rec[(2 * r) * kRecordFloats + 2 + c] = t.x;
        rec[(2 * r) * kRecordFloats + 2 + c + 1] = t.z;
      }
      if (2 * r + 1 < rep) {
        rec[(2 * r + 1) * kRecordFloats + 2 + c] = t.y;
        rec[(2 * r + 1) * kRecordFloats + 2 + c + 1] = t.w;
      }
    }
  if (hd == 0) {
#pragma unroll
    for (int x = 0; x < 2; ++x)
      if (2 * r + x < rep) { rec[(2 * r + x) * kRecordFloats] = run.m[x]; rec[(2 * r + x) * kRecordFloats + 1] = run.l[x]; }
  }
}

}  // namespace

template <bool GEN, bool SHARD>
__global__ void __launch_bounds__(kStreamWarps * 32, kStreamCtasPerSM) decode_stream_kernel(DecodeArgs a) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[kStreamWarps][2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, hd = lane >> 2, r = lane & 3;
  const DecodePlan& pl = a.plan;
  const CacheView& cv = a.cv;
  const int run_id = blockIdx.x * kStreamWarps + warp;
  const int64_t u_begin = pl.run_begin(run_id);
  const int64_t u_end = run_id < pl.n_runs ? pl.run_begin(run_id + 1) : u_begin;
  if (u_begin >= u_end) return;                            // warps do not wait on one another
  const int kgb = GEN ? cv.kf.group_bytes : kKGroupBytes;
  constexpr int kbuf_bytes = GEN ? kGenKBufBytes : kKBufBytes;
  uint8_t* kbuf = smem_raw + warp * (kbuf_bytes + kVBufBytes + kTotBytes);
  uint8_t* vbuf = kbuf + kbuf_bytes;
  float* totbuf = reinterpret_cast<float*>(vbuf + kVBufBytes);
  uint64_t* kbar = &bars[warp][0];
  uint64_t* vbar = &bars[warp][1];
  if (lane == 0) {
    mbar_init(kbar, 1);
    mbar_init(vbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  const int S = pl.units_per_slab;
  const int n_groups = static_cast<int>((a.st.T_q0 + a.st.n_flush * kR) / kG);   // key groups = ternary groups per slab
  int slab = static_cast<int>(u_begin / S);
  int k = static_cast<int>(u_begin - static_cast<int64_t>(slab) * S);
  const uint8_t* slab_ptr = cv.base + cv.slab_offset + (static_cast<int64_t>(a.layer0) * cv.B * cv.H_kv + slab) * cv.slab_stride;
  if (lane == 0) {
    bulk_load(kbuf, slab_ptr + cv.kgroup_offset + static_cast<int64_t>(k) * (kSGGroups * kgb), min(kSGGroups, n_groups - k * kSGGroups) * kgb, kbar);
    if (!a.withhold) bulk_load(vbuf, slab_ptr + cv.tern_offset + static_cast<int64_t>(k) * kVBufBytes, kVBufBytes, vbar);   // (test hook: see DecodeArgs::withhold)
  }
  // the packed cache is not written by the query preparation, so the copies above may start while
  // it still runs; the prepared query is read from here on
  pdl_wait();
  pdl_release();
  uint32_t kpar = 0u, vpar = 0u;
  Running run;
  Query<GEN> qy;
  int cur_chunk = -1;
  float sl2[2] = {0.0f, 0.0f};
  bool ok = true, entering = true;
#pragma unroll 1
  for (int left = static_cast<int>(u_end - u_begin); left > 0; --left) {
    if (entering) {
      cur_chunk = -1;
#pragma unroll
      for (int j = 0; j < 8; ++j) reinterpret_cast<float4*>(totbuf)[j * 32 + lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      run.reset();
      head_factors(prep_words(a, slab, lane), lane, r, sl2);
    }
    ok = n_groups - k * kSGGroups >= kSGGroups
             ? process_unit<true, GEN, SHARD>(a, slab, k, left > 1, slab_ptr, qy, kbuf, vbuf, totbuf, kbar, vbar, kpar, vpar, lane, hd, r, cur_chunk, sl2, run)
             : process_unit<false, GEN, SHARD>(a, slab, k, left > 1, slab_ptr, qy, kbuf, vbuf, totbuf, kbar, vbar, kpar, vpar, lane, hd, r, cur_chunk, sl2, run);
    if (!ok) break;
    entering = ++k == S;
    if (entering || left == 1) write_record(a, slab, run_id, lane, hd, r, run, totbuf);
    if (entering) {
      k = 0;
      ++slab;
      slab_ptr += cv.slab_stride;
    }
  }
  if (!ok) {
    // a copy never arrived: report it and leave (process_unit has waited for the other one that was in flight)
    if (lane == 0) atomicCAS(reinterpret_cast<int*>(cv.base + kHdrStatus), VIDKV_OK, VIDKV_ERR_TIMEOUT);
  }
}

// ---------------------------------------------------------------------------------
// Caches with protected tokens (STPQuant, Algorithm 2): the same walk over 160-token key units,
// but the values of a unit's tokens sit in two streams whose order differs from the key order:
// unprotected tokens in the ternary stream (position = token - protected tokens before it;
// flushed tokens follow from the next group boundary), protected ones in 2-bit groups of 32.
// The probabilities of a unit are therefore scattered (as binary16) into two per-warp rings in
// stream order, 16 bytes a position, and a ternary supergroup (160 stream positions) or protected
// group (32) is multiplied as soon as all of its positions have been written.  Positions of a
// supergroup or group that belong to a neighbouring run stay zero; the neighbour multiplies the
// same bytes with its own probabilities.  The running maximum is kept integral (base-2), so that
// probabilities waiting in the rings are rescaled exactly when it moves.
// Per-warp shared memory: key buffer, ternary supergroup buffer, protected group buffer, running
// output, and the rings: 320 ternary and 192 protected positions.
// ---------------------------------------------------------------------------------
namespace {

constexpr int kTRing = 2 * kStreamUnitTokens;          // ternary ring: an unfinished supergroup plus one unit
constexpr int kPRing = 6 * kG;                         // protected ring: an unfinished group plus one unit
constexpr int kRingBytes = (kTRing + kPRing) * kEntry;   // the ternary positions, then the protected ones
constexpr int kStpWarpBytes = kKBufBytes + kVBufBytes + kPGBytes + kTotBytes + kRingBytes;

// P V of one protected group (Eq. 4 codes as 4 + code): P4[nt] = probabilities of head hd at
// the group's tokens 8 nt + 2 r, + 1.  out += s * (sum (4 + code) p - 4 sum p) + z * sum p.
__device__ __forceinline__ void pv_protected(const uint8_t* pg, float* totbuf, const uint32_t (&P4)[4], float (&l)[2],
                                             int lane, int hd, int r) {
  float cq[4] = {0.0f, 0.0f, 0.0f, 0.0f};               // -4 * (sum of the probabilities) of heads 2 r, 2 r + 1
  mma_f16(cq, kMinus4, kMinus4, kMinus4, kMinus4, P4[0], P4[1]);
  mma_f16(cq, kMinus4, kMinus4, kMinus4, kMinus4, P4[2], P4[3]);
  const float sp0 = -0.25f * cq[0], sp1 = -0.25f * cq[1];
  l[0] += sp0; l[1] += sp1;
#pragma unroll 1
  for (int w = 0; w < 4; ++w) {
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
    float4* tp = reinterpret_cast<float4*>(totbuf) + (2 * w) * 32 + lane;
    float4 t0 = tp[0], t1 = tp[32];
    t0.x += sa.x * acc[0][0] + za.x * sp0; t0.y += sa.x * acc[0][1] + za.x * sp1;
    t0.z += sa.y * acc[0][2] + za.y * sp0; t0.w += sa.y * acc[0][3] + za.y * sp1;
    t1.x += sb.x * acc[1][0] + zb.x * sp0; t1.y += sb.x * acc[1][1] + zb.x * sp1;
    t1.z += sb.y * acc[1][2] + zb.y * sp0; t1.w += sb.y * acc[1][3] + zb.y * sp1;
    tp[0] = t0;
    tp[32] = t1;
  }
}

// Zero the entries of stream positions [pos_begin, pos_end); `ring` points at entry 0 of the stream's part.
__device__ __forceinline__ void zero_ring_range(uint8_t* ring, int ring_len, int pos_begin, int pos_end, int lane) {
  for (int pos = pos_begin + lane; pos < pos_end; pos += 32) *reinterpret_cast<uint4*>(ring + (pos % ring_len) * kEntry) = make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace

template <bool GEN>
__global__ void __launch_bounds__(kStreamWarps * 32, kStreamStpCtasPerSM) decode_stream_stp_kernel(DecodeArgs a) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[kStreamWarps][3];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, hd = lane >> 2, r = lane & 3;
  const DecodePlan& pl = a.plan;
  const CacheView& cv = a.cv;
  const int run_id = blockIdx.x * kStreamWarps + warp;
  const int64_t u_begin = pl.run_begin(run_id);
  const int64_t u_end = run_id < pl.n_runs ? pl.run_begin(run_id + 1) : u_begin;
  if (u_begin >= u_end) return;
  const int kgb = GEN ? cv.kf.group_bytes : kKGroupBytes;
  constexpr int kbuf_bytes = GEN ? kGenKBufBytes : kKBufBytes;
  uint8_t* kbuf = smem_raw + warp * (kStpWarpBytes - kKBufBytes + kbuf_bytes);
  uint8_t* vbuf = kbuf + kbuf_bytes;
  uint8_t* pbuf = vbuf + kVBufBytes;
  float* totbuf = reinterpret_cast<float*>(pbuf + kPGBytes);
  uint8_t* rings = reinterpret_cast<uint8_t*>(totbuf) + kTotBytes;
  const uint32_t ring_addr = smem_u32(rings) + lane * kEntry;
  uint64_t* kbar = &bars[warp][0];
  uint64_t* vbar = &bars[warp][1];
  uint64_t* pbar = &bars[warp][2];
  if (lane == 0) {
    mbar_init(kbar, 1);
    mbar_init(vbar, 1);
    mbar_init(pbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  const int S = pl.units_per_slab;
  // token and stream positions fit 32 bits (the layout's group counts do)
  const int T_q0 = static_cast<int>(a.st.T_q0), T_qt = T_q0 + static_cast<int>(a.st.n_flush) * kR;
  const int n_groups = T_qt / kG;
  const int n_prot = static_cast<int>(a.n_prot), n_rest = T_q0 - n_prot;
  const int u_fl0 = (n_rest + kG - 1) / kG * kG;            // stream position where the flushed tokens start
  int slab = static_cast<int>(u_begin / S);
  int k = static_cast<int>(u_begin - static_cast<int64_t>(slab) * S);
  const uint8_t* slab_ptr = cv.base + cv.slab_offset + (static_cast<int64_t>(a.layer0) * cv.B * cv.H_kv + slab) * cv.slab_stride;
  auto load_keys = [&](const uint8_t* slab_at, int kk) {    // one lane
    bulk_load(kbuf, slab_at + cv.kgroup_offset + static_cast<int64_t>(kk) * (kSGGroups * kgb), min(kSGGroups, n_groups - kk * kSGGroups) * kgb, kbar);
  };
  auto load_supergroup = [&](int sg) { bulk_load(vbuf, slab_ptr + cv.tern_offset + static_cast<int64_t>(sg) * kVBufBytes, kVBufBytes, vbar); };
  auto load_protected = [&](int pg) { bulk_load(pbuf, slab_ptr + cv.prot_offset + static_cast<int64_t>(pg) * kPGBytes, kPGBytes, pbar); };
  if (lane == 0) load_keys(slab_ptr, k);
  pdl_wait();                                              // the prepared query (and nothing else so far) comes from the kernel before
  pdl_release();
  const uint32_t lt_mask = (1u << lane) - 1u;              // lanes (= tokens of a group) before this one
  uint32_t kpar = 0u, vpar = 0u, ppar = 0u;
  bool k_pending = true, v_pending = false, p_pending = false;   // a copy into kbuf / vbuf / pbuf has been issued and not yet waited for
  Running run;
  run.reset();
  Query<GEN> qy;
  int cur_chunk = -1;
  const uint32_t* ew = nullptr;
  const uint32_t* ep = nullptr;
  // the part of the slab's value streams that the run's units fill ends before supergroup sg_end and protected group pg_end: nothing is
  // fetched for a neighbour
  int sg_next = 0, pg_next = 0, sg_end = 0, pg_end = 0;
  float sl2[2] = {0.0f, 0.0f};
  bool ok = true, entering = true;
#pragma unroll 1
  for (int left = static_cast<int>(u_end - u_begin); left > 0; --left) {
    const int t_unit = k * kStreamUnitTokens;
    if (entering) {
      cur_chunk = -1;
      const int b = (slab / cv.H_kv) % cv.B;
      ew = cv.e_words(b);
      ep = cv.e_prefix(b);
      // where the run enters and leaves the two value streams
      auto streams_at = [&](int t, int& u, int& p) {
        if (t <= T_q0) { p = static_cast<int>(ep[t / kG]); u = t - p; }
        else { p = n_prot; u = u_fl0 + (t - T_q0); }
      };
      int t_begin, p_begin, t_stop, p_stop;
      streams_at(t_unit, t_begin, p_begin);
      streams_at(left < S - k ? (k + left) * kStreamUnitTokens : T_qt, t_stop, p_stop);
      sg_next = t_begin / kStreamUnitTokens; sg_end = (t_stop + kStreamUnitTokens - 1) / kStreamUnitTokens;
      pg_next = p_begin / kG; pg_end = (p_stop + kG - 1) / kG;
      // zero the running output and both rings
      for (int i = lane; i < (kTotBytes + kRingBytes) / 16; i += 32)
        reinterpret_cast<uint4*>(totbuf)[i] = make_uint4(0u, 0u, 0u, 0u);
      run.reset();
      head_factors(prep_words(a, slab, lane), lane, r, sl2);
      __syncwarp();
      v_pending = sg_next < sg_end;
      p_pending = pg_next < pg_end;
      if (lane == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (v_pending) load_supergroup(sg_next);
        if (p_pending) load_protected(pg_next);
      }
    }
    const int ng = min(kSGGroups, n_groups - k * kSGGroups);
    const bool last = k + 1 == S, more = left > 1, last_of_slab = !more || last;   // the run leaves this slab after this unit
    // the E words and prefix counts of the unit's groups (lane g: group g; lane ng: the prefix count at the
    // unit's end) are fetched now and picked up with shuffles after the scores, their latency hidden behind them
    uint32_t e_word_l = 0u;
    int e_base_l = 0;
    {
      const int gl = t_unit / kG + lane;
      if (lane <= ng && gl * kG <= T_q0) {
        e_base_l = static_cast<int>(ep[gl]);
        if (lane < ng && gl * kG < T_q0) e_word_l = ew[gl];
      }
    }
    // ---- scores of the unit's groups into the key buffer (raw scores, then the group's constant)
    if (!mbar_wait(kbar, kpar)) { ok = false; break; }
    kpar ^= 1u;
    k_pending = more;                                       // the next unit's is issued below, before anything else can fail
    float cst[2], mx[2];
    score_unit<GEN>(a, slab, kbuf, kgb, ng, k * kSGGroups, cur_chunk, qy, lane, hd, r, cst, mx);
    // ---- running maximum (integral), exact rescale of everything that is kept in its units
    {
      const float mu[2] = {mx[0] * sl2[0], mx[1] * sl2[1]};
      const bool up0 = mu[0] > run.m[0] + kStaleLog2, up1 = mu[1] > run.m[1] + kStaleLog2;
      if (__any_sync(0xffffffffu, up0 || up1)) {
        const float m0 = up0 ? ceilf(mu[0]) : run.m[0], m1 = up1 ? ceilf(mu[1]) : run.m[1];
        const float fa = ex2_approx(run.m[0] - m0), fb = ex2_approx(run.m[1] - m1);   // powers of two (0 on the first unit)
        run.m[0] = m0; run.m[1] = m1;
        scale_output(totbuf, fa, fb, lane);
        run.l[0] *= fa; run.l[1] *= fb;
        // probabilities waiting in the rings: every fourth word belongs to heads 2 r, 2 r + 1
        const __half2 f2 = __floats2half2_rn(fa, fb);
#pragma unroll 4
        for (int i = lane; i < (kTRing + kPRing) * 4; i += 32) {
          __half2* q = reinterpret_cast<__half2*>(rings) + i;
          *q = __hmul2(*q, f2);
        }
        __syncwarp();
      }
    }
    // ---- probabilities, scattered into stream order.  Where a token goes depends on the token
    // alone, so lane j works out the entry of the group's token j and the lanes pick up the entries of
    // their own four tokens with shuffles.
    const int base0 = __shfl_sync(0xffffffffu, e_base_l, 0);   // protected tokens before the unit
    const int t_at = (t_unit - base0) % kTRing, p_at = base0 % kPRing;
#pragma unroll 1
    for (int g = 0; g < ng; ++g) {
      uint32_t P[4];
      probabilities(kbuf + g * kgb, g, lane, r, cst, sl2, run.m, P);
      const int tg = t_unit + g * kG;
      const uint32_t word = __shfl_sync(0xffffffffu, e_word_l, g);
      const int base = __shfl_sync(0xffffffffu, e_base_l, g);   // protected tokens before the group
      if (tg < T_q0) {
        const int below = __popc(word & lt_mask);
        const bool prot = (word >> lane) & 1u;
        int at = prot ? p_at + (base - base0) + below : t_at + g * kG - (base - base0) + lane - below;   // less than one turn ahead
        const int turn = prot ? kPRing : kTRing;
        at -= at >= turn ? turn : 0;
        const int dst = (prot ? kTRing + at : at) * kEntry;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) *reinterpret_cast<uint32_t*>(rings + __shfl_sync(0xffffffffu, dst, 8 * nt + hd) + 4 * r) = P[nt];
      } else {
        if (tg == T_q0 && u_fl0 > n_rest) zero_ring_range(rings, kTRing, n_rest, u_fl0, lane);   // the gap before the flushed tokens
        uint8_t* row = rings + ((u_fl0 + (tg - T_q0)) % kTRing + hd) * kEntry + 4 * r;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) *reinterpret_cast<uint32_t*>(row + 8 * nt * kEntry) = P[nt];
      }
    }
    __syncwarp();
    if (more && lane == 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      load_keys(slab_ptr + (last ? cv.slab_stride : 0), last ? 0 : k + 1);
    }
    // ---- how far the two streams are complete now
    const int t_end = t_unit + ng * kG;
    int pp_hi, u_hi;
    if (t_end <= T_q0) { pp_hi = __shfl_sync(0xffffffffu, e_base_l, ng); u_hi = t_end - pp_hi; }
    else { pp_hi = n_prot; u_hi = u_fl0 + (t_end - T_q0); }
    if (last_of_slab) {
      // what is left of the last supergroup / group belongs to a neighbour (or to nobody): zeros
      zero_ring_range(rings, kTRing, u_hi, sg_end * kStreamUnitTokens, lane);
      zero_ring_range(rings + kTRing * kEntry, kPRing, pp_hi, pg_end * kG, lane);
      __syncwarp();
    }
    // ---- ternary supergroups whose positions are all written
    while (last_of_slab ? sg_next < sg_end : (sg_next + 1) * kStreamUnitTokens <= u_hi) {
      if (!mbar_wait(vbar, vpar)) { ok = false; break; }
      vpar ^= 1u;
      v_pending = false;
      uint32_t P[kSGGroups][4];
      float ps[kSGGroups][4];
      const uint32_t rp = ring_addr + (sg_next & 1) * (kStreamUnitTokens * kEntry);
#pragma unroll
      for (int g = 0; g < kSGGroups; ++g) {
        load_entries(rp + g * (kG * kEntry), P[g]);
        ps[g][0] = 0.0f; ps[g][1] = 0.0f; ps[g][2] = 0.0f; ps[g][3] = 0.0f;
        mma_f16(ps[g], kMinus5, kMinus5, kMinus5, kMinus5, P[g][0], P[g][1]);
        mma_f16(ps[g], kMinus5, kMinus5, kMinus5, kMinus5, P[g][2], P[g][3]);
        run.l[0] = fmaf(-0.2f, ps[g][0], run.l[0]);
        run.l[1] = fmaf(-0.2f, ps[g][1], run.l[1]);
      }
      // groups without positions of this run may not exist.  (Leaving their products out, and those before the run's first position, takes
      // branches between the groups: 848 -> 926 us a step of 16 users, 47.3 -> 49.4 of one clip.)
      const int n_used = last_of_slab ? (u_hi - sg_next * kStreamUnitTokens + kG - 1) / kG : kSGGroups;
      pv_ternary<false, false>(vbuf, totbuf, n_used, P, ps, 1.0f, 1.0f, lane, hd, r);
      ++sg_next;
      __syncwarp();
      v_pending = sg_next < sg_end;
      if (v_pending && lane == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        load_supergroup(sg_next);
      }
    }
    // ---- protected groups whose positions are all written
    while (ok && (last_of_slab ? pg_next < pg_end : (pg_next + 1) * kG <= pp_hi)) {
      if (!mbar_wait(pbar, ppar)) { ok = false; break; }
      ppar ^= 1u;
      p_pending = false;
      uint32_t P4[4];
      load_entries(ring_addr + (kTRing + (pg_next % (kPRing / kG)) * kG) * kEntry, P4);
      pv_protected(pbuf, totbuf, P4, run.l, lane, hd, r);
      ++pg_next;
      __syncwarp();
      p_pending = pg_next < pg_end;
      if (p_pending && lane == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        load_protected(pg_next);
      }
    }
    if (!ok) break;
    entering = last;
    if (last_of_slab) write_record(a, slab, run_id, lane, hd, r, run, totbuf);
    ++k;
    if (last) {
      k = 0;
      ++slab;
      slab_ptr += cv.slab_stride;
    }
  }
  if (!ok) {
    // a copy never arrived: report it, and let the others that are in flight land before the warp leaves
    if (lane == 0) atomicCAS(reinterpret_cast<int*>(cv.base + kHdrStatus), VIDKV_OK, VIDKV_ERR_TIMEOUT);
    if (k_pending) mbar_wait(kbar, kpar);
    if (v_pending) mbar_wait(vbar, vpar);
    if (p_pending) mbar_wait(pbar, ppar);
  }
}

cudaError_t launch_decode_stream_stp(const DecodeArgs& a, cudaStream_t stream) {
  const bool gen = a.cv.kf.general != 0;
  const size_t smem = static_cast<size_t>(kStreamWarps) * (kStpWarpBytes + (gen ? kGenKBufBytes - kKBufBytes : 0));
  static bool attr_set[64][2] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr_set[dev][gen]) {
    const cudaError_t e = gen ? cudaFuncSetAttribute(decode_stream_stp_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                              : cudaFuncSetAttribute(decode_stream_stp_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_set[dev][gen] = true;
  }
  const int grid = (a.plan.n_runs + kStreamWarps - 1) / kStreamWarps;
  if (grid < 1) return cudaSuccess;
  // with profiling events around the launch the kernel starts after the event, as an ordinary launch
  cudaError_t le;
  if (a.ev_begin) {
    if (gen) decode_stream_stp_kernel<true><<<grid, kStreamWarps * 32, smem, stream>>>(a);
    else decode_stream_stp_kernel<false><<<grid, kStreamWarps * 32, smem, stream>>>(a);
    le = cudaGetLastError();
  } else {
    le = gen ? launch_dependent(decode_stream_stp_kernel<true>, dim3(grid), dim3(kStreamWarps * 32), smem, stream, a)
             : launch_dependent(decode_stream_stp_kernel<false>, dim3(grid), dim3(kStreamWarps * 32), smem, stream, a);
  }
  count_launches(1);
  return le;
}

template <bool GEN, bool SHARD>
static cudaError_t launch_stream_t(const DecodeArgs& a, cudaStream_t stream) {
  constexpr int smem = kStreamWarps * (kWarpBufBytes + (GEN ? kGenKBufBytes - kKBufBytes : 0));
  static bool attr_set[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr_set[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(decode_stream_kernel<GEN, SHARD>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  const int grid = (a.plan.n_runs + kStreamWarps - 1) / kStreamWarps;
  if (grid < 1) return cudaSuccess;
  count_launches(1);
  if (!a.ev_begin) return launch_dependent(decode_stream_kernel<GEN, SHARD>, dim3(grid), dim3(kStreamWarps * 32), smem, stream, a);
  decode_stream_kernel<GEN, SHARD><<<grid, kStreamWarps * 32, smem, stream>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_decode_stream(const DecodeArgs& a_in, cudaStream_t stream) {
  DecodeArgs a = a_in;
  if (g_debug_withhold == 2) { a.withhold = 1; g_debug_withhold = 0; }
  if (a.cv.kf.general) return a.partial_out ? launch_stream_t<true, true>(a, stream) : launch_stream_t<true, false>(a, stream);
  return a.partial_out ? launch_stream_t<false, true>(a, stream) : launch_stream_t<false, false>(a, stream);
}

}  // namespace vidkv
