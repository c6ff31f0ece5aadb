// Device helpers shared by the decode attention kernels (decode_block.cu, decode_stream.cu): bulk copies with
// mbarrier completion and bounded waits.
#pragma once

#include "decode_common.cuh"

namespace vidkv {
namespace {

constexpr int kKBufBytes = kSGGroups * kKGroupBytes;          // 5760: the key groups of one unit
constexpr int kGenKBufBytes = kSGGroups * kMaxKGroupBytes;    // the same for the general key formats
constexpr int kVBufBytes = kSGBytes;                          // 5376: a ternary supergroup
constexpr uint32_t kWaitLimit = 1u << 19;                     // mbarrier polls before a warp gives up (about a second)
constexpr float kStaleLog2 = 6.0f;                            // the running maximum may lag a unit's maximum by this much
constexpr float kRefLag = 60.0f;                              // a unit's reference is no further below the largest maximum (its sums
                                                              // are then nothing beside the others'), so that running sums stay below 2^95
constexpr uint32_t kMinus5 = 0xc500c500u;                     // binary16 pair (-5.0, -5.0)
constexpr uint32_t kMinus4 = 0xc400c400u;                     // binary16 pair (-4.0, -4.0)

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
// One bulk copy global -> shared of `bytes` (multiple of 16, both addresses 16-byte aligned),
// completion counted on `bar`.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  const uint32_t b = smem_u32(bar), d = smem_u32(dst);
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(d),
               "l"(src), "r"(bytes), "r"(b)
               : "memory");
}
// Bounded wait for the phase with the given parity by a whole warp; false if it never completed.  All lanes get one
// answer: a copy that lands just as the polls run out may be seen by some of them only, and what follows a wait (matrix
// products, shuffles) needs the warp together.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  const uint32_t b = smem_u32(bar);
  for (uint32_t i = 0; i < kWaitLimit; ++i) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; vote.sync.all.pred p, p, 0xffffffff; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(b), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
// The same by one lane.
__device__ __forceinline__ bool mbar_wait_lane(uint64_t* bar, uint32_t parity) {
  const uint32_t b = smem_u32(bar);
  for (uint32_t i = 0; i < kWaitLimit; ++i) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(b), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

}  // namespace
}  // namespace vidkv
