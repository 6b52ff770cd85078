// Building blocks shared by the tensor-core kernels (ozaki_tc.cu, gemm_tc.cu):
// mbarriers with bounded waits, bulk copies, tcgen05 descriptors and
// instructions, and the integer-only rounding of an exact digit sum to FP64.
#pragma once

#include <stdint.h>

namespace dqmc {

constexpr unsigned long long TC_WAIT_NS = 2000000000ull;   // bound of every device-side wait

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait on a phase of an mbarrier; false after TC_WAIT_NS.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer();
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (globaltimer() - t0 > TC_WAIT_NS) return false;
  }
}

// One contiguous global -> shared copy, completion counted in bytes on bar.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// Shared-memory matrix descriptor of a K-major tile with 64-byte swizzle:
// rows of 64 bytes, 8-row groups 512 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);        // start address
  d |= (uint64_t)1 << 16;                          // leading byte offset (unused when swizzled)
  d |= (uint64_t)(512 >> 4) << 32;                 // stride byte offset: 8 rows x 64 B
  d |= (uint64_t)1 << 46;                          // descriptor version
  d |= (uint64_t)4 << 61;                          // swizzle mode: 64-byte
  return d;
}

__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                     uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum)
      : "memory");
}

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// (T 2^32 + r) 2^e correctly rounded to FP64, for |T| < 2^45 and 0 <= r < 2^32
// (the exact sum of the weight groups), with 64-bit integer operations only:
// the magnitude is split into (Ta, ra) the same way, the 53-bit mantissa taken
// from Ta and the top bits of ra, and the discarded bits of ra decide the
// round-to-nearest-even step.
__device__ __forceinline__ double split_times_pow2(long long T, unsigned int r, int e) {
  if (T == 0 && r == 0) return 0.0;
  const bool neg = T < 0;
  unsigned long long Ta;
  unsigned int ra;
  if (!neg) { Ta = (unsigned long long)T; ra = r; }
  else if (r) { Ta = (unsigned long long)(-(T + 1)); ra = (unsigned int)(0x100000000ull - r); }
  else { Ta = (unsigned long long)(-T); ra = 0u; }
  unsigned long long mant;
  int ex;
  if (Ta < (1ull << 21)) {   // below 2^53: exact
    const unsigned long long A = (Ta << 32) | ra;
    const int nb = 64 - __clzll((long long)A);
    mant = A << (53 - nb);
    ex = nb - 1 + e;
  } else {                   // 54..77 bits: drop sh = 1..24 bits of ra
    const int nb = 96 - __clzll((long long)Ta);
    const int sh = nb - 53;
    mant = (Ta << (32 - sh)) | (ra >> sh);
    const unsigned int rem = ra & ((1u << sh) - 1u), half = 1u << (sh - 1);
    ex = nb - 1 + e;
    if (rem > half || (rem == half && (mant & 1ull))) {
      if (++mant == (1ull << 53)) { mant >>= 1; ++ex; }
    }
  }
  const int be = ex + 1023;
  if (be <= 0 || be >= 2047)   // result outside the normal range: scale in FP64
    return ldexp((double)Ta * 4294967296.0 + (double)ra, e) * (neg ? -1.0 : 1.0);
  return __longlong_as_double((long long)((neg ? (1ull << 63) : 0ull) |
                                          ((unsigned long long)be << 52) |
                                          (mant & 0xFFFFFFFFFFFFFull)));
}

}  // namespace dqmc
