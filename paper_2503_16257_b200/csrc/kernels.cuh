// Internal launcher interface between the host API and the kernel files.
#pragma once

#include "common.cuh"

namespace vidkv {

// Programmatic dependent launch: a kernel launched with the stream-serialization attribute may start
// while the kernel before it still runs; pdl_wait() returns once that kernel has completed and its
// writes are visible (a no-op for an ordinary launch), pdl_release() lets the kernel after this one start.
// Behind the wait, global memory is read through ordinary loads.  A read-only load (__ldg) is for data that nobody writes while
// the kernel runs, which what the kernel before leaves is not, and nothing but its address keeps the compiler from moving it ahead of the wait.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// For a chain of such loads that should all be under way at once: a pointer that is known from here (behind the wait) on, and a load
// through it that the compiler may schedule as freely as a read-only one (nobody writes the data any more until the kernel ends).
__device__ __forceinline__ const float* behind_wait(const float* p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}
__device__ __forceinline__ float load_settled(const float* p) {
  float v;
  asm("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
// Launch `kernel` so that it may overlap the tail of the previous kernel on `stream` (it must call pdl_wait()
// before touching anything that kernel writes).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// A [slabs, tokens, 128] source of keys or values.  Source slab i (= b * H + h, running
// over layers first when several layers are processed) starts at
// ptr + (i / H) * stride_b + (i % H) * stride_h elements; token t at + t * stride_t.
struct KSrc {
  const void* ptr;
  int64_t stride_b, stride_h, stride_t;
  int32_t H;
};

// Algorithm 1: X_r = X[l - r:].  Rows t_begin .. t_begin + n_tok - 1 of source slab `slab` into the residual ring at
// res_offset of its cache slab, rows 0 on; called by a whole block (16-bit elements either way: the copy is type-agnostic).
__device__ __forceinline__ void copy_residual_rows(const KSrc& src, int64_t t_begin, int n_tok, const CacheView& cv, int layer0, int slab,
                                                   int64_t res_offset) {
  const int lb = slab / cv.H_kv, h = slab % cv.H_kv;
  const uint16_t* base = static_cast<const uint16_t*>(src.ptr) + static_cast<int64_t>(lb) * src.stride_b + h * src.stride_h;
  uint4* dst = reinterpret_cast<uint4*>(cv.slab(layer0 + lb / cv.B, lb % cv.B, h) + res_offset);
  auto piece = [&](int i) { return reinterpret_cast<const uint4*>(base + (t_begin + (i >> 4)) * src.stride_t)[i & 15]; };
  const int n = n_tok * 16, step = blockDim.x;
  for (int i = threadIdx.x; i < n; i += 2 * step) {         // two loads under way per thread
    const bool two = i + step < n;
    const uint4 a = piece(i), b = two ? piece(i + step) : a;
    dst[i] = a;
    if (two) dst[i + step] = b;
  }
}

// Token-selection data handed to the value quantizer (NULL lists = no protection).
struct SelView {
  const int32_t* idx_prot;   // [B][n_prot]       ascending protected token ids
  const int32_t* idx_rest;   // [B][T - n_prot]   ascending unprotected token ids
  int64_t stride_prot, stride_rest;
  int64_t n_prot;
};

// Channel min / max accumulators of the range pass: 256 ordered-integer words per slab (128
// minima that start at all ones, 128 maxima that start at zero).  Two buffers alternate: a call
// accumulates into `cur`, which the call before it re-armed, and re-arms the first
// `next_dirty_words` words of `next` for the call after it, so no call spends a launch on it.
struct MinMaxBuffers {
  uint32_t* cur;
  uint32_t* next;
  int next_dirty_words;
};
// Arms both buffers, clears the decode counters and writes the cache header (magic, version, cleared status word).
cudaError_t launch_init_workspace(uint32_t* minmax, int64_t n_words, int32_t* counters, int64_t n_counters, uint32_t* header,
                                  uint32_t version, cudaStream_t stream);

// Algorithm 3 on `T_tokens` tokens (a multiple of 32) of every slab of layers
// [layer0, layer0 + n_layers): writes chunk `chunk` of the chunk table and the key groups
// starting at group index kgroup0.
// n_res rows that follow (0..31) are copied to the residual.  n_counters > 0: clears the decode kernel's arrival counters on
// the way.
cudaError_t launch_quantize_keys(int dtype, const KSrc& src, int64_t T_tokens, int n_res, const CacheView& cv, int layer0,
                                 int n_layers, int chunk, int64_t kgroup0, const MinMaxBuffers& mm, int32_t* counters, int64_t n_counters,
                                 cudaStream_t stream);

// Channel split and encode pass of Algorithm 3 for `n_slabs` slabs whose channel ranges are in mm.cur; launched behind the
// range pass.  Writes the chunk table entry `chunk` too, and re-arms mm.next.
cudaError_t launch_encode_keys(int dtype, const KSrc& src, int64_t T_tokens, const CacheView& cv, int layer0, int n_slabs,
                               int slabs_per_layer, int chunk, int64_t kgroup0, const MinMaxBuffers& mm, cudaStream_t stream);

// Encode pass for the general key formats (other k, plain 1-bit code), whose channel split (chunk table entry `chunk`) is
// already written.
cudaError_t launch_encode_keys_general(int dtype, const KSrc& src, int64_t T_tokens, const CacheView& cv, int layer0,
                                       int n_slabs, int slabs_per_layer, int chunk, int64_t kgroup0, cudaStream_t stream);

// Device addresses of the DFT tables.  frag: the 64-point matrix in MMA B-fragment order: word
// ((ks * 8 + nt) * 32 + lane) * 4 + {0, 1} = leading binary16 pairs, + {2, 3} = remainders, for
// rows 16 ks + 2 r (+1; +8, +9) and column 16 (n / 2) + 2 nt + (n % 2), lane = 4 n + r; column f
// holds 1/8, (-1)^c / 8, cos(2 pi k c / 64) / 8 (f = 2k) or -sin(2 pi k c / 64) / 8 (f = 2k + 1).
// w32: the 32-point matrix [channel][column] in float32, orthonormal, columns from 2 on doubled.
// Filled on first use on each device by one small kernel; later calls order their stream after it with an event.
struct DftTables {
  const uint32_t* frag;
  const float* w32;
};
cudaError_t dft_tables(DftTables* tables, cudaStream_t stream);

// Algorithm 2 on the prefill tokens of n_layers layers (source slabs run over layers, then b, then h).  T_q (multiple of 32) tokens; the
// unprotected ones go to ternary stream positions 0.., the protected ones to 2-bit groups.
// n_res rows that follow the T_q are copied to the residual.
cudaError_t launch_quantize_values(int dtype, const KSrc& src, int64_t T_q, int n_res, const CacheView& cv, int layer, int n_layers,
                                   const SelView& sel, float gamma, bool nonzero_mean_scale, cudaStream_t stream);

// 1.58Quant of a full 128-token residual of every slab of the given layers, appended at
// ternary stream group index tgroup0 (read-modify-write of shared supergroup bytes).
cudaError_t launch_flush_values(int dtype, const KSrc& src, const CacheView& cv, int layer0, int n_layers,
                                int64_t tgroup0, float gamma, bool nonzero_mean_scale, cudaStream_t stream);

// A prompt shorter than one group: all of its n_tok tokens into the residual rings.
cudaError_t launch_copy_to_residual(const KSrc& src, int n_tok, const CacheView& cv, int layer, int n_layers, bool is_value,
                                    cudaStream_t stream);

// Token selection (Sec. 3.3(2)): top-n by saliency, E words + prefix counts into the cache,
// gather lists into the workspace.
cudaError_t launch_select_tokens(const float* saliency, int64_t vis_begin, int64_t l_v, int64_t n_prot, int64_t T_q,
                                 const CacheView& cv, int32_t* idx_prot, int32_t* idx_rest, int64_t stride_prot,
                                 int64_t stride_rest, cudaStream_t stream);
cudaError_t launch_mask_to_selection(const uint8_t* E, int64_t T, int64_t T_q, const CacheView& cv, int32_t* idx_prot,
                                     int32_t* idx_rest, int64_t stride_prot, int64_t stride_rest, int32_t* counts,
                                     int64_t expect_count, cudaStream_t stream);

// Token counts the decode kernels need (the same for every layer of one call).
struct LayerState {
  int64_t T_q0;        // prefill tokens quantized (multiple of 32)
  int64_t n_flush;     // flushed 128-token chunks
  int32_t n_res;       // residual tokens (after the append of this step)
};

constexpr int kStreamUnitTokens = 160;  // one unit of the stream kernel: 5 key groups = 1 ternary supergroup
constexpr int kStreamWarps = 4;         // warps per CTA of the stream kernel
constexpr int kStreamCtasPerSM = 3;     // its CTAs per multiprocessor (register bound)
constexpr int kStreamStpCtasPerSM = 2;  // the same for the variant with protected tokens (shared-memory bound)
constexpr int kPrepWords = 25;          // 32-bit words per lane per (slab, chunk) of prepared query
constexpr int kBlocksPerSM = 3;         // blocks of the block kernel per multiprocessor: 128 registers x 160 threads
constexpr int kMoreBlocksPerSM = 4;     // its variant for calls that are better off with more blocks (96 registers)
constexpr int kRecordFloats = 130; // one partial record: running maximum (base-2 logits), sum, out[128]
constexpr int kPartFloats = kMaxRep * kRecordFloats;   // the block kernel's record of a part of a slab: m [8], l [8], out [8][128]
constexpr int kJoin = 8;           // records joined at a node of the block kernel's merge tree

// How one attention call over n_slabs slabs is cut into work (host side, decode.cu): the
// quantized tokens of all slabs form one sequence of 160-token units (units_per_slab each).
//   stream kernel  warp number w of the launch walks the units [w * units / runs, (w + 1) * units / runs), all
//                  warps that fit the device taking part: runs of equal length, rounded up, left some multiprocessors a
//                  whole block short (8960 units on 1776 warps as 1494 runs of 6: 76.5 us a step, now 70).  It leaves
//                  one partial record per slab it touches, record slab + w: from one record to the next the slab or
//                  the warp number goes up, so the records need no more room than there are runs and slabs.
//   block kernel   (small calls: n_blocks > 0 or res_blocks > 0) the same with blocks in place of warps; the records
//                  of a slab are joined by a tree of eight-way nodes.
struct DecodePlan {
  int32_t units_per_slab;
  int32_t run_units;       // units of the longest run
  int32_t n_runs;
  int64_t n_units;
  int32_t slab_parts;      // most runs that can touch one slab
  int32_t n_chunks;        // chunk-table entries the query preparation covers (0: nothing quantized)
  int64_t records;         // records of one query head: (n_runs + n_slabs) * 8, or (n_blocks + n_slabs) * 8 in the block kernel
  int32_t n_blocks;
  int32_t blocks_per_sm;   // the block kernel's variant: kBlocksPerSM or kMoreBlocksPerSM
  int32_t res_blocks;      // blocks that attend to a slab's residual alone: n_slabs or 0 (the slab's last block does it)
  int32_t counters_per_slab;   // arrival counters of the merge tree
  int32_t equal_units;     // > 0: runs of exactly this many units (the last one shorter) instead of a proportional share
  __host__ __device__ int64_t run_begin(int64_t w) const {
    if (equal_units > 0) return w * equal_units < n_units ? w * equal_units : n_units;
    return w * n_units / n_runs;
  }
  __host__ __device__ int64_t run_of(int64_t u) const { return equal_units > 0 ? u / equal_units : ((u + 1) * n_runs - 1) / n_units; }
};
// stp: the cache holds protected tokens (the stream kernel for them keeps fewer warps per multiprocessor).
// force_run_units: 0 = choose; otherwise the test hook's value: > 0 the stream kernel with runs of that many units, -1 the block kernel.
// partial: the call leaves (maximum, sum, unnormalised output) triples.  Their maximum is the one the walk has kept, which
// need not be the largest logit, so it depends on how the units are cut: such calls keep runs of equal length, and take the
// block kernel only where every run is one unit (its maximum is then exact however blocks share the units).
DecodePlan plan_decode(const LayerState& st, int64_t n_slabs, bool stp, const KeyFmt& kf, int sm_count, int force_run_units,
                       bool partial = false);
// Arrival counters any call that needs at most `records` records on at most max_slabs slabs uses.
int64_t max_decode_counters(int64_t max_slabs, int64_t records);
// Largest `records` any call on at most max_slabs slabs and max_tokens tokens can plan.
int64_t max_decode_records(int64_t max_slabs, int64_t max_tokens);
// Multiprocessors of the current device (cached per device); 0 on error.
int device_sm_count();

struct DecodeArgs {
  CacheView cv;
  const void* q;
  const void* k_new;
  const void* v_new;
  void* out;
  float* partials;     // [n_runs + n_slabs][8 heads][kRecordFloats]
  uint32_t* prep;      // stream kernel: per (slab, chunk) query images (decode_prep_bytes)
  int32_t* counters;   // block kernel: [n_slabs][counters_per_slab], zero between calls
  DftTables dft;       // set by launch_decode
  int32_t append_row;  // >= 0: k_new / v_new are written into this residual row first
  int32_t layer0, n_layers;
  int32_t in_dtype, out_dtype;
  DecodePlan plan;
  int64_t n_prot;      // protected tokens per batch element (0 = no STP)
  float scale;
  LayerState st;
  cudaEvent_t ev_begin, ev_end;   // optional: recorded around the attention kernel (profiling)
  int32_t withhold;    // test hook: the stream kernel does not issue its first value copy
  float* partial_out;  // not null: leave [n_layers * B * H_q][kRecordFloats] (max, sum, unnormalised out) instead of `out`
};

// Eq. 7 scores from hidden states: text_sum [B, d] (scratch) and saliency [B, l_v], both float32.
cudaError_t launch_saliency(int dtype, const void* x_v, const void* x_t, int64_t B, int64_t l_v, int64_t l_t, int64_t d,
                            float* text_sum, float* saliency, cudaStream_t stream);

// Variance / outlier count per (slab, channel) of a key tensor; stats [n_slabs][2][128] float64 scratch.
cudaError_t launch_channel_metrics(int dtype, const KSrc& src, int64_t n_slabs, int64_t T_tokens, int metric, double M,
                                   double* stats, float* out, cudaStream_t stream);

// Test hook (vidkv_debug_withhold_once): 1 = the next key-encode launch withholds the tensor-core
// products of every block's first tile, 2 = the next stream-kernel launch withholds every warp's
// first value copy; the launch that honours it clears it.  0 = off.
extern int g_debug_withhold;

// Number of kernels launched by this library since it was loaded (host counter).
extern unsigned long long g_launch_count;
inline void count_launches(int n) { g_launch_count += static_cast<unsigned long long>(n); }

// Attention over the packed cache + residual: the block kernel alone, or the query preparation, the stream kernel and
// the merge of the partial records, which also attends to the residual.
cudaError_t launch_decode(const DecodeArgs& a, cudaStream_t stream);
cudaError_t launch_decode_block(const DecodeArgs& a, cudaStream_t stream);
// Log-sum-exp merge of n_parts partial sets [n_parts][n_rows][kRecordFloats] into out [n_rows][128].
cudaError_t launch_merge_partials(const float* parts, int64_t n_parts, int64_t n_rows, void* out, int out_dtype,
                                  cudaStream_t stream);
// Query preparation (and the step's append) for a.plan.n_chunks chunk-table entries per slab.
cudaError_t launch_decode_prep(const DecodeArgs& a, cudaStream_t stream);
// Persistent warps over 160-token units: caches without / with protected tokens.
cudaError_t launch_decode_stream(const DecodeArgs& a, cudaStream_t stream);
cudaError_t launch_decode_stream_stp(const DecodeArgs& a, cudaStream_t stream);
size_t decode_prep_bytes(int64_t n_slabs, int64_t n_chunks);

// Test-only dequantizers (float32 [B, H_kv, n_quantized, D]).
cudaError_t launch_dequant_keys(const CacheView& cv, int layer, int64_t T_q0, int64_t n_flush, float* out,
                                cudaStream_t stream);
cudaError_t launch_dequant_values(const CacheView& cv, int layer, int64_t T_q0, int64_t n_flush, int64_t n_prot,
                                  float* out, cudaStream_t stream);

// Test-only exports: undo the bit packing of one layer into plain arrays (any pointer may be null).
cudaError_t launch_export_codes(const CacheView& cv, int layer, int64_t n_kgroups, int64_t n_tgroups, int64_t n_pgroups,
                                int8_t* k2, uint8_t* k1, uint16_t* ks2, uint16_t* kz2, uint16_t* ks1, int8_t* trits,
                                uint16_t* vs, int8_t* v2, uint16_t* v2s, uint16_t* v2z, cudaStream_t stream);
cudaError_t launch_export_selection(const CacheView& cv, int layer, int n_chunks, uint8_t* dmask, int64_t T, int64_t T_sel,
                                    uint8_t* E, cudaStream_t stream);

}  // namespace vidkv
