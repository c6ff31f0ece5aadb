// Decode attention over the packed cache (Algorithm 1 "Decoding", Eq. 3): how a call is cut into
// work (plan_decode), the launch sequence, and the last kernel of a step, which merges the
// partial records of the attention kernels by log-sum-exp and, for caches without protected
// tokens, attends to the FP16 / BF16 residual itself.
#include <cmath>
#include <numeric>
#include <type_traits>

#include "decode_common.cuh"

namespace vidkv {

namespace {

constexpr int kMaxSMs = 256;        // multiprocessor count the sizing formulas assume at most
constexpr int64_t kMostForcedUnits = 1 << 21;   // the block kernel multiplies units by blocks in 32 bits
// What the choice between the attention kernels goes by: estimated microseconds of a call, linear in what it is made of.  The block
// kernel has one launch and a parallel merge; the stream kernel has three launches, a merge block per slab that reads the slab's records one
// behind the other, and a third fewer instructions per unit.  The block kernel comes with three blocks on a multiprocessor and 128 registers
// a thread, or with four and 96 (which keep some of the loop's state in local memory); not for general key formats with protected tokens,
// where four are slower throughout.  The coefficients are least-squares fits to 648 measured calls of 4 to 1120 slabs and 1 to 1800 units a
// slab, the ones near the line weighted most, and moved within a few percent so that the choice is the faster kernel there: over those
// calls it costs 0.2 % more than the fastest of the three, 6.4 % at most.  us, three blocks / four / stream:
//   half of the channels two-bit (slabs of units): 112 of 2 10.9 / 13.1 / 15.5, 448 of 3 26.1 / 22.3 / 25.1, 448 of 4 29.0 / 26.5 / 26.3,
//     448 of 8 40.9 / 43.4 / 35.1, 224 of 8 28.3 / 28.1 / 24.6, 112 of 20 29.5 / 27.9 / 28.6, 192 of 13 32.3 / 31.6 / 29.0,
//     176 of 13 31.1 / 32.8 / 28.7, 128 of 18 28.7 / 32.6 / 29.2, 32 of 140 44.7 / 44.2 / 43.5, 16 of 79 20.9 / 24.4 / 30.9,
//     16 of 400 56.5 / 56.6 / 59.9, 4 of 1225 48.1 / 49.0 / 104.0
//   k = 0.75, plain one-bit code: 112 of 2 10.4 / 12.9 / 18.4, 448 of 2 22.5 / 19.6 / 24.2, 448 of 3 26.2 / 25.3 / 25.3,
//     112 of 10 22.9 / 21.4 / 24.6, 112 of 20 30.6 / 32.1 / 32.1, 96 of 24 31.5 / 32.2 / 32.7, 192 of 13 34.1 / 36.9 / 32.8,
//     16 of 200 39.5 / 42.7 / 48.4, 16 of 400 66.0 / 70.6 / 68.6
//   k = 0.75, Eq. 5 (longer preparation in every block): 112 of 2 13.2 / 15.7 / 18.5, 448 of 3 31.5 / 27.9 / 26.4,
//     112 of 14 31.8 / 29.3 / 26.7, 32 of 40 31.4 / 29.4 / 28.8
//   a fifth of the tokens protected, half of the channels two-bit: 112 of 4 22.3 / 21.8 / 24.6, 224 of 4 27.1 / 29.7 / 25.1,
//     448 of 2 - / 26.3 / 26.6, 560 of 3 - / 33.0 / 37.1, 592 of 4 - / 40.1 / 34.9, 64 of 14 27.2 / 32.1 / 26.6, 32 of 40 32.6 / - / 33.7,
//     16 of 300 64.7 / - / 61.5, 8 of 600 61.8 / - / 71.9
//   the same with k = 0.75, plain, three blocks / stream: 224 of 4 29.0 / 27.5, 64 of 14 27.8 / 28.6, 16 of 200 55.7 / 55.3,
//     16 of 300 74.0 / 69.7
struct BlockCost {
  double base;
  double unit;      // a unit of the longest stretch
  double load;      // a unit per multiprocessor
  double entry;     // a slab that a block enters behind its first
  double join;      // a level of the merge tree
  double slab;      // a hundred slabs
};
struct StreamCost {
  double base;
  double unit;      // a unit of the longest run
  double load;      // a unit per warp of the device
  double record;    // a record of a slab
  double slab;      // a hundred slabs
};
struct CallCost { BlockCost three, four; StreamCost stream; };
// [protected tokens][format: default, general without Eq. 5, general with it]
constexpr CallCost kCallCost[2][3] = {
    {{{7.83, 2.16, 0.30, 3.49, 1.91, 0.46}, {9.93, 3.38, 0.16, 4.53, 1.36, 0.29}, {12.76, 2.28, 6.67, 0.16, 0.97}},
     {{6.02, 2.42, 0.45, 2.74, 2.27, 0.71}, {8.08, 4.67, 0.20, 3.74, 1.12, 0.40}, {12.88, 5.17, 4.26, 0.18, 0.90}},
     {{9.28, 2.47, 0.45, 4.72, 1.96, 0.43}, {10.88, 4.62, 0.23, 4.61, 1.25, 0.36}, {13.47, 5.41, 4.23, 0.20, 0.95}}},
    {{{12.20, 3.77, 0.15, 0.0, 2.02, -0.38}, {17.03, 4.68, 0.31, 0.0, 1.66, -0.28}, {15.93, 5.20, 2.22, 0.18, 0.86}},
     {{9.81, 4.83, 0.10, 0.0, 2.54, -0.25}, {}, {16.80, 7.04, 2.08, 0.18, 0.65}},
     {{12.74, 4.63, 0.18, 0.0, 2.33, -0.29}, {}, {17.19, 7.43, 1.84, 0.19, 0.82}}}};

}  // namespace

int device_sm_count() {
  static int sm_of_device[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (sm_of_device[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 0;
    sm_of_device[dev] = n;
  }
  return sm_of_device[dev];
}

// Levels of eight-way joins over n parts: how many counters they take.
static int64_t join_counters(int64_t n) {
  int64_t c = 0;
  while (n > 1) { n = (n + kJoin - 1) / kJoin; c += n; }
  return c;
}

DecodePlan plan_decode(const LayerState& st, int64_t n_slabs, bool stp, const KeyFmt& kf, int sm_count, int force_run_units, bool partial) {
  DecodePlan p = {};
  const int64_t T_qt = st.T_q0 + st.n_flush * kR;
  p.n_chunks = T_qt > 0 ? 1 + static_cast<int32_t>(st.n_flush) : 0;
  p.units_per_slab = static_cast<int32_t>((T_qt + kStreamUnitTokens - 1) / kStreamUnitTokens);
  p.n_units = n_slabs * p.units_per_slab;
  const int sms = sm_count < 1 ? 1 : (sm_count > kMaxSMs ? kMaxSMs : sm_count);
  const int64_t warps = static_cast<int64_t>(sms) * (stp ? kStreamStpCtasPerSM : kStreamCtasPerSM) * kStreamWarps;
  int64_t run = (p.n_units + warps - 1) / warps;
  if (run < 1) run = 1;                                    // nothing quantized
  if (force_run_units > 0) run = force_run_units;
  p.run_units = static_cast<int32_t>(run);
  if (partial) p.equal_units = p.run_units;
  int64_t runs = p.n_units < warps ? p.n_units : warps;
  if (force_run_units > 0 || partial) {
    runs = (p.n_units + run - 1) / run;
  } else if (stp && n_slabs > 0 && warps >= n_slabs) {
    // With protected tokens a run pays for every slab that it enters and for the supergroup and the protected group that it
    // shares with its neighbour at a cut inside a slab.  Where a slab divides evenly into its share of the warps (at most half
    // a key group per run left over), every slab gets that many runs and none straddles two.  us per step, all warps /
    // evenly: 112 slabs of 6400 tokens 53.1 / 53.1, of 16000 101.0 / 101.2, 168 of 9000 93.3 / 87.0, 224 of 6400 (k = 0.75)
    // 111.3 / 107.8; uneven shares lose (measured before the merge blocks spread, which takes 5 us off either): 64 slabs of
    // 12544 (4.4 units a run) 64.8 / 69.2, 112 of 12544 (7.8) 90.4 / 92.9, without protected tokens 112 of 12819 70.3 / 77.0.
    const int64_t share = warps / n_slabs, groups = T_qt / kG;
    if (groups >= share * kSGGroups && groups % (share * kSGGroups) <= share / 2 && n_slabs * share * run >= p.n_units)
      runs = n_slabs * share;
  }
  p.n_runs = static_cast<int32_t>(runs);
  // a run is n_units / n_runs units long or one more
  const auto most_parts = [&](int64_t n) -> int64_t {
    const int64_t shortest = p.equal_units > 0 ? p.equal_units : n > 0 ? p.n_units / n : 1;
    return p.units_per_slab > 0 ? (p.units_per_slab + shortest - 1) / shortest + 1 : 1;
  };
  p.slab_parts = static_cast<int32_t>(most_parts(p.n_runs));
  p.records = (p.n_runs + n_slabs) * kMaxRep;
  // The block kernel's cut for `per_sm` blocks on each multiprocessor, and its estimated time.
  struct BlockCut { int64_t blocks, longest, even; bool straddles; double us; };
  const CallCost& cost = kCallCost[stp][kf.general == 0 ? 0 : kf.plain || kf.n1() == 0 ? 1 : 2];
  const auto cut_for = [&](int per_sm, const BlockCost& c) -> BlockCut {
    BlockCut cut = {static_cast<int64_t>(sms) * per_sm, 0, 0, false, 0.0};
    cut.longest = (p.n_units + cut.blocks - 1) / cut.blocks;
    // A block that goes on in the next slab pays for query images, rings and join twice: where the proportional cut makes such
    // blocks (slab s then begins d units * slabs / blocks after a block does, d running through the multiples of
    // gcd(blocks, slabs)), every slab gets its own blocks, if it can without a longer stretch.  us, straddling / not: 64 slabs
    // of 14 units 28.9 / 21.8, 448 of 3 28.2 / 21.0; with protected tokens 42.3 / 31.7 and 45.2 / 30.0.
    cut.straddles = p.n_units > 0 && p.n_units - std::gcd(cut.blocks, n_slabs) * p.units_per_slab >= cut.blocks;
    bool apart = true;                                     // with protected tokens blocks never share slabs' ends
    if (cut.straddles) {
      const int64_t share = cut.blocks / n_slabs, even = share > 0 ? (p.units_per_slab + share - 1) / share : 0;
      apart = share > 0;
      if (share > 0 && (stp || even <= cut.longest)) {
        cut.longest = even;
        cut.even = n_slabs * (share < p.units_per_slab ? share : p.units_per_slab);
        cut.straddles = false;
      }
    }
    if (p.n_units == 0) return cut;
    const int64_t entered = cut.straddles ? (cut.longest - 1 + p.units_per_slab - 1) / p.units_per_slab : 0;
    int levels = 0;
    for (int64_t parts = (p.units_per_slab + cut.longest - 1) / cut.longest; parts > 1; parts = (parts + kJoin - 1) / kJoin) ++levels;
    cut.us = c.base + c.unit * cut.longest + c.load * p.n_units / sms + c.entry * entered + c.join * levels + c.slab * 0.01 * n_slabs;
    if (stp && !apart) cut.us = INFINITY;
    return cut;
  };
  BlockCut cut = cut_for(kBlocksPerSM, cost.three);
  p.blocks_per_sm = kBlocksPerSM;
  if (!stp || !kf.general) {
    const BlockCut more = cut_for(kMoreBlocksPerSM, cost.four);
    if (more.us < cut.us) { cut = more; p.blocks_per_sm = kMoreBlocksPerSM; }
  }
  const StreamCost& sc = cost.stream;
  const double stream_us = sc.base + sc.unit * run + sc.load * p.n_units / warps + sc.record * p.units_per_slab / run + sc.slab * 0.01 * n_slabs;
  const bool block = cut.us < stream_us;
  if (p.n_units == 0 || ((block || (force_run_units < 0 && p.n_units < kMostForcedUnits)) && force_run_units <= 0 && (!partial || run == 1))) {
    p.n_blocks = static_cast<int32_t>(cut.even > 0 ? cut.even : p.n_units < cut.blocks ? p.n_units : cut.blocks);
    p.records = (p.n_blocks + n_slabs) * kMaxRep;
    p.res_blocks = st.n_res > 0 && cut.longest <= 1 ? static_cast<int32_t>(n_slabs) : 0;
    p.counters_per_slab = static_cast<int32_t>(join_counters(most_parts(p.n_blocks) + (p.res_blocks > 0)));
  }
  return p;
}

int64_t max_decode_counters(int64_t max_slabs, int64_t records) {
  // the levels over n parts have at most n / 7 nodes and one more per level; ten levels cover 2^30 parts
  return records / kMaxRep / 7 + 12 * max_slabs + 64;
}

int64_t max_decode_records(int64_t max_slabs, int64_t max_tokens) {
  if (max_tokens < 1) max_tokens = 1;
  // a call has at most min(units, warps) runs (the test hook may force one unit per run) and leaves fewer than
  // runs + slabs records; units <= slabs * S.
  const int64_t S = (max_tokens + kStreamUnitTokens - 1) / kStreamUnitTokens;
  const int64_t warps = static_cast<int64_t>(kMaxSMs) * kStreamCtasPerSM * kStreamWarps;
  int64_t parts = max_slabs * S;
  if (parts > warps + max_slabs) parts = warps + max_slabs;
  parts += max_slabs;
  return parts * kMaxRep;
}

// ---------------------------------------------------------------------------------
// One block of 4 warps per slab = (layer, batch element, KV head), serving its query heads.
// Residual tokens: the FP16 / BF16 rows K_r, V_r are staged in shared memory (V_r as
// binary16; the inputs are representable there), q K_r^T runs on the tensor cores in the input
// type (rows = heads, columns = tokens; products of two 16-bit values are exact), a warp per head
// turns the scores and the records' maxima into probabilities (binary16, as in the attention
// kernels), P V_r runs on the tensor cores with V_r read through transposing matrix loads, and the
// records join with their weights 2^(m_record - M).  Scores and maxima are base-2 logits.
// Shared memory for n_pad staged rows (n_res rounded up to 16):
//   Ks, Vs  n_pad rows of 272 bytes (256 + 16 of padding: conflict-free fragment loads)
//   S       [8][n_pad] float scores        Ph  [8][n_pad + 8] binary16 probabilities
//   Mh, Lh, Wh  [8] maxima, denominators and the weight of the residual's sums, whose probabilities are
//           taken against the residual's own maximum
// ---------------------------------------------------------------------------------
constexpr int kMergeRow = kD * 2 + 16;
size_t merge_smem_bytes(int n_pad) {
  return static_cast<size_t>(2) * n_pad * kMergeRow + sizeof(float) * 8 * n_pad + sizeof(__half) * 8 * (n_pad + 8) + 3 * 8 * sizeof(float);
}

// Shared memory asked for so that no multiprocessor takes more than its share of the n_slabs merge blocks: left alone they
// gather on the multiprocessors that the stream kernel frees first and share one path to L2 while others idle.  us a call,
// gathered / spread: triples of 4 slabs x 600 units 125.8 / 79.8, protected 16 x 74 54.5 / 41.4, 112 x 40 57.9 / 53.7; asking
// for 100 KB or 56 KB at most instead: 4 x 600 94.6 / 175.7.
constexpr size_t kMaxSmem = 226 * 1024;       // a block's largest, less the kilobyte that every block costs besides
static size_t spread_smem(size_t needed, int n_slabs) {
  const int sms = device_sm_count();
  if (sms < 1) return needed;
  const size_t share = (kMaxSmem + 1024) / static_cast<size_t>((n_slabs + sms - 1) / sms);
  const size_t smem = share > 2048 ? (share - 1024) / 1024 * 1024 : 0;
  return smem > needed ? smem : needed;
}

template <typename T>
__global__ void __launch_bounds__(kD) decode_merge_kernel(DecodeArgs a, int n_res, int n_pad) {
  extern __shared__ __align__(16) uint8_t msm[];
  uint8_t* Ks = msm;
  uint8_t* Vs = Ks + n_pad * kMergeRow;
  float* S = reinterpret_cast<float*>(Vs + n_pad * kMergeRow);
  __half* Ph = reinterpret_cast<__half*>(S + 8 * n_pad);
  const int PS = n_pad + 8;
  float* Mh = reinterpret_cast<float*>(Ph + 8 * PS);
  float* Lh = Mh + 8;
  float* Wh = Lh + 8;
  const CacheView& cv = a.cv;
  const int slab = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, hd = lane >> 2, r = lane & 3;
  const int h = slab % cv.H_kv, lb = slab / cv.H_kv, rep = cv.rep;
  const uint8_t* slab_ptr = cv.base + cv.slab_offset + (static_cast<int64_t>(a.layer0) * cv.B * cv.H_kv + slab) * cv.slab_stride;
  int n_parts;
  int64_t first_run = 0;
  {
    const DecodePlan& pl = a.plan;
    if (pl.units_per_slab == 0) n_parts = 0;
    else {
      const int64_t u0 = static_cast<int64_t>(slab) * pl.units_per_slab;
      first_run = pl.run_of(u0);
      n_parts = static_cast<int>(pl.run_of(u0 + pl.units_per_slab - 1) - first_run) + 1;
    }
  }
  const float* rec = a.partials + (slab + first_run) * (kMaxRep * kRecordFloats);
  const int64_t q0 = (static_cast<int64_t>(lb) * cv.H_q + h * rep) * kD;
  if (n_pad > 0) {
    // ---- stage the residual rows (16-byte pieces, all loads of a thread independent).  Up to the records nothing here comes from the
    // attention kernel before, so it goes on while that kernel's last blocks still run: the rows, the appended one among them, are
    // older than the preparation kernel, for which that kernel waited before it let this one start.  (Behind the wait the residual took
    // 3-5 us of a step.)
    const uint4* ksrc = reinterpret_cast<const uint4*>(slab_ptr + cv.kres_offset);
    const uint4* vsrc = reinterpret_cast<const uint4*>(slab_ptr + cv.vres_offset);
    constexpr bool kConvert = !std::is_same<T, __half>::value;          // bfloat16 values -> binary16 (exact for the admitted inputs)
    for (int i = tid; i < n_pad * 16; i += kD) {
      const int row = i >> 4, col = i & 15;
      uint8_t* kd = Ks + row * kMergeRow + col * 16;
      uint8_t* vd = Vs + row * kMergeRow + col * 16;
      if (row < n_res) {
        cp_async16(kd, ksrc + i);
        if (!kConvert) cp_async16(vd, vsrc + i);
      } else {
        *reinterpret_cast<uint4*>(kd) = make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(vd) = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    cp_async_commit();
    if (kConvert) {
#pragma unroll 4
      for (int i = tid; i < n_res * 16; i += kD) {
        uint4 vv = __ldg(vsrc + i);
        uint32_t* w = &vv.x;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 f = Elem<T>::to_float2(w[j]);
          const __half2 hh = __floats2half2_rn(f.x, f.y);
          w[j] = *reinterpret_cast<const uint32_t*>(&hh);
        }
        *reinterpret_cast<uint4*>(Vs + (i >> 4) * kMergeRow + (i & 15) * 16) = vv;
      }
    }
    // ---- q fragments: rows 0-7 = this slab's heads (zero beyond rep), rows 8-15 unused
    const T* qp = reinterpret_cast<const T*>(a.q) + q0;
    uint32_t qn[16];
#pragma unroll
    for (int i = 0; i < 16; ++i)
      qn[i] = hd < rep ? __ldg(reinterpret_cast<const uint32_t*>(qp + hd * kD + 8 * i + 2 * r)) : 0u;
    cp_async_wait<0>();
    __syncthreads();
    const float sl2 = a.scale * 1.4426950408889634f;
    for (int tile = warp; tile < n_pad / 8; tile += kD / 32) {
      const uint32_t* kr = reinterpret_cast<const uint32_t*>(Ks + (tile * 8 + hd) * kMergeRow) + r;
      float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) mma_in<T>(acc, qn[2 * ks], qn[2 * ks + 1], kr[ks * 8], kr[ks * 8 + 4]);
      *reinterpret_cast<float2*>(S + hd * n_pad + tile * 8 + 2 * r) = make_float2(acc[0] * sl2, acc[1] * sl2);
    }
    __syncthreads();
  }
  // ---- the residual's maxima and probabilities: warp w takes heads w and w + 4
  float m_res[2], l_res[2];
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const int k = warp + 4 * x;
    m_res[x] = -INFINITY;
    if (k < rep)
      for (int t = lane; t < n_res; t += 32) m_res[x] = fmaxf(m_res[x], S[k * n_pad + t]);
#pragma unroll
    for (int o = 16; o; o >>= 1) m_res[x] = fmaxf(m_res[x], __shfl_xor_sync(0xffffffffu, m_res[x], o));
    l_res[x] = 0.0f;                                       // this lane's tokens
    for (int t = lane; t < n_pad; t += 32) {
      __half ph = __float2half_rn(0.0f);
      if (k < rep && t < n_res) ph = __float2half_rn(exp2f(S[k * n_pad + t] - m_res[x]));
      Ph[k * PS + t] = ph;
      l_res[x] += __half2float(ph);
    }
  }
  __syncthreads();
  // ---- P V_r: warp w owns channels 32 w .. 32 w + 31 as four 8-channel tiles
  float acc[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j) { acc[j][0] = 0.0f; acc[j][1] = 0.0f; acc[j][2] = 0.0f; acc[j][3] = 0.0f; }
  for (int kt = 0; kt < n_pad / 16; ++kt) {
    const uint32_t a0 = *reinterpret_cast<const uint32_t*>(Ph + hd * PS + 16 * kt + 2 * r);
    const uint32_t a2 = *reinterpret_cast<const uint32_t*>(Ph + hd * PS + 16 * kt + 2 * r + 8);
    const uint32_t vrow = static_cast<uint32_t>(__cvta_generic_to_shared(Vs + (16 * kt + (lane & 15)) * kMergeRow + 64 * warp));
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t b0, b1;
      asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(b0), "=r"(b1) : "r"(vrow + 16 * j));
      mma_f16(acc[j], a0, 0u, a2, 0u, b0, b1);
    }
  }
  // ---- the records: maxima and sums (lane j: record j, for the heads warp and warp + 4) and this lane's output fragments
  // of the first kRecAhead of them in one round of loads
  pdl_wait();
  rec = behind_wait(rec);
  float2 head_ml[2];
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const int k = warp + 4 * x;
    head_ml[x] = make_float2(-INFINITY, 0.0f);
    if (k < rep && lane < n_parts) head_ml[x] = *reinterpret_cast<const float2*>(rec + (lane * kMaxRep + k) * kRecordFloats);
  }
  constexpr int kRecAhead = 3;
  float rec_m[kRecAhead];
  float2 rec_o[kRecAhead][4];
#pragma unroll
  for (int jp = 0; jp < kRecAhead; ++jp) {
    rec_m[jp] = -INFINITY;
#pragma unroll
    for (int j = 0; j < 4; ++j) rec_o[jp][j] = make_float2(0.0f, 0.0f);
    if (jp < n_parts && hd < rep) {
      const float* pr = rec + (jp * kMaxRep + hd) * kRecordFloats;
      rec_m[jp] = *pr;
#pragma unroll
      for (int j = 0; j < 4; ++j) rec_o[jp][j] = *reinterpret_cast<const float2*>(pr + 2 + 32 * warp + 8 * j + 2 * r);
    }
  }
  // ---- maxima and denominators over all parts
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const int k = warp + 4 * x;
    float m = head_ml[x].x;
    if (k < rep)
      for (int j = lane + 32; j < n_parts; j += 32) m = fmaxf(m, load_settled(rec + (j * kMaxRep + k) * kRecordFloats));
#pragma unroll
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    m = fmaxf(m, m_res[x]);
    const float w_res = k < rep && n_res > 0 ? exp2f(m_res[x] - m) : 0.0f;
    float l = l_res[x] * w_res;
    if (k < rep) {
      l += head_ml[x].y * exp2f(head_ml[x].x - m);          // 0 for a record that does not exist
      for (int j = lane + 32; j < n_parts; j += 32) {
        const float* pr = rec + (j * kMaxRep + k) * kRecordFloats;
        l += pr[1] * exp2f(pr[0] - m);
      }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) { Mh[k] = m; Lh[k] = l; Wh[k] = w_res; }
  }
  __syncthreads();
  // ---- join the records: lane (hd, r) holds head hd, channels 32 w + 8 j + 2 r, + 1
  if (hd < rep) {
    const float M = Mh[hd], inv = 1.0f / Lh[hd], w_res = Wh[hd];
#pragma unroll
    for (int j = 0; j < 4; ++j) { acc[j][0] *= w_res; acc[j][1] *= w_res; }
#pragma unroll
    for (int jp = 0; jp < kRecAhead; ++jp) {
      const float wgt = exp2f(rec_m[jp] - M);                // 0 for a record that does not exist
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[j][0] += wgt * rec_o[jp][j].x;
        acc[j][1] += wgt * rec_o[jp][j].y;
      }
    }
    for (int jp = kRecAhead; jp < n_parts; ++jp) {
      const float* pr = rec + (jp * kMaxRep + hd) * kRecordFloats;
      const float wgt = exp2f(pr[0] - M);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 o = *reinterpret_cast<const float2*>(pr + 2 + 32 * warp + 8 * j + 2 * r);
        acc[j][0] += wgt * o.x;
        acc[j][1] += wgt * o.y;
      }
    }
    if (a.partial_out) {
      // a token shard of a longer sequence: leave (maximum, sum, unnormalised out) for the caller's exchange
      float* pr = a.partial_out + (q0 / kD + hd) * kRecordFloats;
      if (warp == 0 && r == 0) { pr[0] = M; pr[1] = Lh[hd]; }
#pragma unroll
      for (int j = 0; j < 4; ++j) *reinterpret_cast<float2*>(pr + 2 + 32 * warp + 8 * j + 2 * r) = make_float2(acc[j][0], acc[j][1]);
      return;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float v0 = acc[j][0] * inv, v1 = acc[j][1] * inv;
      const int64_t i = q0 + hd * kD + 32 * warp + 8 * j + 2 * r;
      if (a.out_dtype == VIDKV_F32) *reinterpret_cast<float2*>(reinterpret_cast<float*>(a.out) + i) = make_float2(v0, v1);
      else if (a.out_dtype == VIDKV_F16) *reinterpret_cast<__half2*>(reinterpret_cast<__half*>(a.out) + i) = __floats2half2_rn(v0, v1);
      else *reinterpret_cast<__nv_bfloat162*>(reinterpret_cast<__nv_bfloat16*>(a.out) + i) = __floats2bfloat162_rn(v0, v1);
    }
  }
}

// out[row][c] = sum_p 2^(m_p - M) o_p[c] / sum_p 2^(m_p - M) l_p over n_parts partial sets of n_rows rows each
// (M = max_p m_p); a set that saw no token has l = 0 and m = -inf.
__global__ void __launch_bounds__(kD) merge_partials_kernel(const float* __restrict__ parts, int64_t n_parts, int64_t n_rows,
                                                           void* __restrict__ out, int out_dtype) {
  const int64_t row = blockIdx.x;
  const int c = threadIdx.x;
  float M = -INFINITY;
  for (int64_t p = 0; p < n_parts; ++p) M = fmaxf(M, parts[(p * n_rows + row) * kRecordFloats]);
  float num = 0.0f, den = 0.0f;
  for (int64_t p = 0; p < n_parts; ++p) {
    const float* pr = parts + (p * n_rows + row) * kRecordFloats;
    const float w = pr[1] > 0.0f ? exp2f(pr[0] - M) : 0.0f;
    num += w * pr[2 + c];
    den += w * pr[1];
  }
  const float v = num / den;
  if (out_dtype == VIDKV_F32) reinterpret_cast<float*>(out)[row * kD + c] = v;
  else if (out_dtype == VIDKV_F16) reinterpret_cast<__half*>(out)[row * kD + c] = __float2half_rn(v);
  else reinterpret_cast<__nv_bfloat16*>(out)[row * kD + c] = __float2bfloat16_rn(v);
}

cudaError_t launch_merge_partials(const float* parts, int64_t n_parts, int64_t n_rows, void* out, int out_dtype,
                                  cudaStream_t stream) {
  merge_partials_kernel<<<static_cast<unsigned>(n_rows), kD, 0, stream>>>(parts, n_parts, n_rows, out, out_dtype);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_decode(const DecodeArgs& a_in, cudaStream_t stream) {
  DecodeArgs a = a_in;
  cudaError_t e;
  if ((e = dft_tables(&a.dft, stream))) return e;
  if (a.plan.n_blocks + a.plan.res_blocks > 0) {
    if (a.ev_begin) cudaEventRecord(a.ev_begin, stream);
    e = launch_decode_block(a, stream);
    if (a.ev_end) cudaEventRecord(a.ev_end, stream);
    return e;
  }
  const int n_slabs = a.n_layers * a.cv.B * a.cv.H_kv;
  if (a.plan.n_chunks > 0) {
    if ((e = launch_decode_prep(a, stream)) != cudaSuccess) return e;
    if (a.ev_begin) cudaEventRecord(a.ev_begin, stream);
    e = a.n_prot > 0 ? launch_decode_stream_stp(a, stream) : launch_decode_stream(a, stream);
    if (a.ev_end) cudaEventRecord(a.ev_end, stream);
    if (e != cudaSuccess) return e;
  }
  count_launches(1);
  const int n_res = a.st.n_res;
  const int n_pad = (n_res + 15) / 16 * 16;
  const size_t smem = spread_smem(merge_smem_bytes(n_pad), n_slabs);
  static bool attr_set[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr_set[dev]) {
    const int most = static_cast<int>(kMaxSmem);
    if ((e = cudaFuncSetAttribute(decode_merge_kernel<__half>, cudaFuncAttributeMaxDynamicSharedMemorySize, most))) return e;
    if ((e = cudaFuncSetAttribute(decode_merge_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, most))) return e;
    attr_set[dev] = true;
  }
  if (a.ev_end) {                                          // profiling events sit between the launches: ordinary launch
    if (a.in_dtype == VIDKV_F16) decode_merge_kernel<__half><<<n_slabs, kD, smem, stream>>>(a, n_res, n_pad);
    else decode_merge_kernel<__nv_bfloat16><<<n_slabs, kD, smem, stream>>>(a, n_res, n_pad);
    return cudaGetLastError();
  }
  return a.in_dtype == VIDKV_F16
             ? launch_dependent(decode_merge_kernel<__half>, dim3(n_slabs), dim3(kD), smem, stream, a, n_res, n_pad)
             : launch_dependent(decode_merge_kernel<__nv_bfloat16>, dim3(n_slabs), dim3(kD), smem, stream, a, n_res, n_pad);
}

}  // namespace vidkv
