// Device helpers of the persistent product kernels (spmm_pipe.cu,
// spmm_mma.cu): mbarriers with bounded waits, bulk copies, the stage header
// that the producer hands to the consumers, and sums in FP32 pairs.
#pragma once

#include <stdint.h>

#include "xct_internal.cuh"

namespace xct {
namespace {

// stage descriptors are requested this many stages before the stage's
// copies, into kDescSlots = kDescAhead + 1 slots
constexpr int kDescAhead = 3;
constexpr int kDescSlots = kDescAhead + 1;

struct __align__(16) Hdr {
  int32_t work;    // work item inside its product (tile * nblocks + block), -1 = no more work
  int32_t kstage;  // stage index inside the block
  int32_t last;    // last stage of the block
  int32_t np;      // staged rows (0: a block without entries)
  int32_t prod;    // product index in the launch
  int32_t pad[3];
};

__device__ __forceinline__ uint32_t su32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint64_t* bar, uint32_t tx) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(bar)), "r"(tx)
               : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t tx) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(su32(bar)), "r"(tx)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(su32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// non-blocking test of the phase of `parity`
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(su32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Wait for the phase of `parity` to complete; false once `limit_ns` of wall
// time has passed without it (checked every 256 tries; a limit of 0 only
// tests the phase once, without suspending).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  if (limit_ns == 0) return mbar_test(bar, parity);   // no waiting at all
  if (mbar_try(bar, parity)) return true;
  const uint64_t t0 = now_ns();
  for (uint32_t i = 1;; ++i) {
    if (mbar_try(bar, parity)) return true;
    if ((i & 255u) == 0 && now_ns() - t0 > limit_ns) return false;
  }
}
// the limit of the waits that let copies already issued land before a CTA
// that gave up exits (independent of the configurable limit)
constexpr uint64_t kDrainNs = 2000000000ull;
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          su32(dst)),
      "l"(src), "r"(bytes), "r"(su32(bar))
      : "memory");
}

// the same for data read once: its lines are the first to leave L2
__device__ __forceinline__ void bulk_g2s_once(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .b64 policy;\n\tcreatepolicy.fractional.L2::evict_first.b64 policy, 1.0;\n\t"
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], "
      "policy;\n\t}" ::"r"(su32(dst)),
      "l"(src), "r"(bytes), "r"(su32(bar))
      : "memory");
}

// a hint to bring `bytes` (a multiple of 16) at `src` (16-byte aligned) into
// L2; nothing waits for it
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ int ceil_log2_exp_p(float m) {
  if (!(m > 0.0f)) return 0;
  int ex;
  const float f = frexpf(m, &ex);
  return f == 0.5f ? ex - 1 : ex;
}

// An unevaluated sum h + l of two FP32 values: squares of FP32 values are
// exact in it (l from an FMA), and sums of such non-negative terms keep
// about 47 bits (two-sum of the high parts, then renormalisation), on the
// FP32 pipes.
struct Ff {
  float h, l;
};
__device__ __forceinline__ Ff ff_square(float r) {
  const float h = __fmul_rn(r, r);
  return {h, __fmaf_rn(r, r, -h)};
}
__device__ __forceinline__ Ff sum2(Ff a, Ff b) {
  const float s = __fadd_rn(a.h, b.h);
  const float v = __fsub_rn(s, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, v)), __fsub_rn(b.h, v));   // s's error, exact
  const float t = __fadd_rn(e, __fadd_rn(a.l, b.l));
  const float h = __fadd_rn(s, t);
  return {h, __fsub_rn(t, __fsub_rn(h, s))};
}
__device__ __forceinline__ double sum2(double a, double b) { return a + b; }
__device__ __forceinline__ Ff shfl_xor(Ff v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)};
}
__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }

}  // namespace
}  // namespace xct
