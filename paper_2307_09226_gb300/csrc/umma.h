// Device helpers shared by the tcgen05 contractions: mbarriers with bounded waits, bulk
// copies, tensor-memory and descriptor instructions, phasors and the 16-bit split.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "rsim_internal.h"

namespace rsim {
namespace umma {

constexpr unsigned long long kWaitNs = 2000000000ull;  // 2 s per wait, then give up

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(b))
               : "memory");
}

// Arrive on the barrier at the same place in the shared memory of the cluster's CTA `rank`.
__device__ __forceinline__ void mbar_arrive_at(uint64_t* b, uint32_t rank) {
  asm volatile(
      "{\n\t.reg .b32 r;\n\tmapa.shared::cluster.u32 r, %0, %1;\n\t"
      "mbarrier.arrive.shared::cluster.b64 _, [r];\n\t}" ::"r"(smem_u32(b)),
      "r"(rank)
      : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Probe without waiting.
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Wait for the phase of parity `parity` to complete; false on timeout or abort (`abort`: the
// block's shared flag, raised by the first wait that runs out).
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, int* abort, unsigned* status) {
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (mbar_try(b, parity)) return true;
    if ((it & 255u) == 255u) {
      if (*(volatile int*)abort) return false;
      const uint64_t now = globaltimer();
      if (t0 == 0) {
        t0 = now;
      } else if (now - t0 > kWaitNs) {
        atomicOr(status, kStatusTimeout);
        *(volatile int*)abort = 1;
        return false;
      }
    }
  }
}

// Warp-collective wait: all lanes poll, the decision is made uniform.
__device__ __forceinline__ bool warp_wait(uint64_t* b, uint32_t parity, int* abort, unsigned* status) {
  return __all_sync(0xffffffffu, mbar_wait(b, parity, abort, status));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(
                   smem_u32(b)),
               "r"(bytes)
               : "memory");
}

// L2 eviction priorities.  A chunk's B images are read by every row tile at about the
// same time and then never again, while the split partial sums wait in L2 for the
// reduction after the contraction: the B copies take evict_first and the partial-sum
// stores and reductions evict_last.  (The partial sums are found in L2 by the reduction
// with evict_normal stores too; what it pays for is that most of its reads are served by
// the other die's L2 partition, over the link between the two partitions.)
// bulk_g2s with a createpolicy policy for the source lines:
__device__ __forceinline__ void bulk_g2s_hint(void* dst, const void* src, uint32_t bytes, uint64_t* bar,
                                              uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
// 16-byte store and FP32 add-reduction with a policy (the reduction is one instruction,
// like atomicAdd on a float4, so each address's additions keep the issuing thread's order).
__device__ __forceinline__ void st_hint_v4(float4* a, float4 v, uint64_t policy) {
  asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(a), "f"(v.x), "f"(v.y), "f"(v.z),
               "f"(v.w), "l"(policy)
               : "memory");
}
// 1-D bulk copy global -> shared (16-byte aligned, size a multiple of 16) that
// completes `bytes` of the barrier's transaction count.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 128-byte-swizzled K-major shared-memory matrix descriptor (tcgen05 format): rows of
// 128 B, 8-row groups 1024 B apart (stride byte offset), version 1, swizzle mode 2.
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t addr) {
  uint64_t d = (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;              // leading byte offset (unused for this layout)
  d |= (uint64_t)(1024 >> 4) << 32;    // stride byte offset
  d |= (uint64_t)1 << 46;              // descriptor version
  d |= (uint64_t)2 << 61;              // 128-byte swizzle
  return d;
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                 "=r"(v[7])
               : "r"(taddr)
               : "memory");
}

__device__ __forceinline__ float2 cis_q32(uint32_t ph) {
  const float ang = (float)(int32_t)ph * 1.46291807926715968e-09f;  // 2 pi / 2^32
  float s, c;
  __sincosf(ang, &s, &c);
  return make_float2(c, s);
}

// exp(j 2 pi x) for a 2^-32-cycle phase, the fraction taken from the top 23 bits by
// placing them in the mantissa of a float in [1, 2) (no integer-to-float conversion);
// the quantisation to 2^-23 cycle adds at most 7.5e-7 rad.
__device__ __forceinline__ float2 cis_q32_fast(uint32_t ph) {
  const float x = __int_as_float(0x3F800000u | ((ph ^ 0x80000000u) >> 9)) - 1.5f;  // [-1/2, 1/2)
  float s, c;
  __sincosf(x * 6.28318530717958648f, &s, &c);
  return make_float2(c, s);
}

// (x, y) as a pair of 16-bit numbers, low = x, high = y.
template <int BF>
__device__ __forceinline__ uint32_t pack2(float x, float y) {
  if (BF) {
    __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    return *reinterpret_cast<uint32_t*>(&h);
  }
  __half2 h = __floats2half2_rn(x, y);
  return *reinterpret_cast<uint32_t*>(&h);
}

// Split (x, y) into 16-bit hi and lo pairs, packed low = x, high = y.
template <int BF>
__device__ __forceinline__ void split2(float x, float y, uint32_t& hi, uint32_t& lo) {
  if (BF) {
    __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    float2 hf = __bfloat1622float2(h);
    __nv_bfloat162 l = __floats2bfloat162_rn(x - hf.x, y - hf.y);
    hi = *reinterpret_cast<uint32_t*>(&h);
    lo = *reinterpret_cast<uint32_t*>(&l);
  } else {
    __half2 h = __floats2half2_rn(x, y);
    float2 hf = __half22float2(h);
    __half2 l = __floats2half2_rn(x - hf.x, y - hf.y);
    hi = *reinterpret_cast<uint32_t*>(&h);
    lo = *reinterpret_cast<uint32_t*>(&l);
  }
}

// The power of two of sigma_scaling undone, as two factors.
__device__ __forceinline__ float2 sigma_unscale(const FrameIO& fr, int scaled) {
  return pow2_factors(sigma_exponent(fr.meta[1], scaled));
}

}  // namespace umma
}  // namespace rsim
