// Building blocks shared by the tensor-core kernels (ozaki_tc.cu, gemm_tc.cu,
// chain_tc.cu, qrp_tc.cu): mbarriers with bounded waits, bulk copies, tcgen05
// descriptors and instructions, digits of FP64 values, the integer-only rounding of an
// exact digit sum to FP64, and the square root and reciprocal of a reflector.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

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

// (T 2^32 + r) 2^e correctly rounded to FP64 (subnormal results too), for |T| < 2^62
// and 0 <= r < 2^32 (the exact sum of the weight groups), with 32-bit integer operations and no
// branch but for results outside the normal range: the FP64 pipe stays free, and
// a CTA's epilogue converts thousands of sums.  The magnitude's three words are
// moved up past leading zero words and shifted to a leading one; the 53 top bits
// and the biased exponent less one are added, so that the leading one completes
// the exponent, and the round-to-nearest-even increment may carry into it.
__host__ __device__ __forceinline__ double split_times_pow2(long long T, unsigned int r, int e) {
  const unsigned int neg = (unsigned int)((unsigned long long)T >> 63);
  const unsigned int w0n = neg ? 0u - r : r;
  const unsigned long long Tm = neg ? ~(unsigned long long)T + (r == 0u) : (unsigned long long)T;
  unsigned int w2 = (unsigned int)(Tm >> 32), w1 = (unsigned int)Tm, w0 = w0n;
  int be = e + 95 + 1022;                    // biased exponent of the leading bit, less one
  if (w2 == 0u) { w2 = w1; w1 = w0; w0 = 0u; be -= 32; }
  if (w2 == 0u) { w2 = w1; w1 = 0u; be -= 32; }
#ifdef __CUDA_ARCH__
  const int lz = __clz((int)w2);
  const unsigned int m1 = __funnelshift_l(w1, w2, lz), m0 = __funnelshift_l(w0, w1, lz);
#else
  const int lz = w2 ? __builtin_clz(w2) : 32;
  const unsigned long long h = ((unsigned long long)w2 << 32) | w1, q = ((unsigned long long)w1 << 32) | w0;
  const unsigned int m1 = lz < 32 ? (unsigned int)((h << lz) >> 32) : w1;
  const unsigned int m0 = lz < 32 ? (unsigned int)((q << lz) >> 32) : w0;
#endif
  const unsigned int low = w0 << (lz & 31);  // (w0 is zero wherever lz reaches 32)
  be -= lz;
  const unsigned int up = (m0 & 0x400u) && ((m0 & 0xBFFu) | low) ? 1u : 0u;
  unsigned long long bits = ((unsigned long long)((unsigned int)be << 20) << 32) +
                            (((unsigned long long)(m1 >> 11)) << 32) +
                            (unsigned long long)((m1 << 21) | (m0 >> 11)) + up;
  bits |= (unsigned long long)neg << 63;
  if (w2 == 0u) bits = 0ull;
  else if (be < 0 || be > 2045) {            // result outside the normal range
    const unsigned long long m = ((unsigned long long)m1 << 32) | m0;
    const int sh = 11 - be;                  // the last bit kept is 2^-1074
    if (be > 0) bits = 0x7ffull << 52;
    else if (sh > 64) bits = 0ull;
    else {
      const unsigned long long half = 1ull << (sh - 1), rem = sh < 64 ? m & (2 * half - 1) : m;
      bits = sh < 64 ? m >> sh : 0ull;
      bits += rem > half || (rem == half && (low || (bits & 1ull))) ? 1u : 0u;
    }
    bits |= (unsigned long long)neg << 63;
  }
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)bits);
#else
  double d;
  memcpy(&d, &bits, 8);
  return d;
#endif
}

// 1 / D for a normal D > 0 whose reciprocal is normal, within 2 units of 2^-53: an FP32
// seed (22 bits, scaled by exponent arithmetic) and one cubic Newton step.
__device__ __forceinline__ double recip_newton(double D) {
  const long long db = __double_as_longlong(D);
  const int de = (int)(db >> 52) - 1023;
  const uint32_t zu = __float_as_uint(
      __fdividef(1.0f, __uint_as_float((127u << 23) | (uint32_t)((db >> 29) & 0x7fffff))));
  const double z0 = __longlong_as_double(((long long)((int)(zu >> 23) - 127 + 1023 - de) << 52) |
                                         ((long long)(zu & 0x7fffff) << 29));
  const double e = fma(-D, z0, 1.0);
  return fma(z0, fma(e, e, e), z0);
}

// nrm = sqrt(sig) and gam = 1 / (sig + |alpha| nrm) for a normal sig > 0, |alpha| <=
// nrm (1 + eps): the library's square root and division are chains of some 20 FP64
// instructions on one warp, each holding the pipe for 64 cycles, with every other
// warp waiting.  FP32 seeds (22 bits, scaled by exponent arithmetic) and FP64
// corrections take 9 in a row: one Goldschmidt step and Markstein's residual
// correction for the root (P. Markstein, IBM J. Res. Dev. 34, 1990), one cubic
// Newton step for the reciprocal.  Over 2e7 random arguments the root was the
// correctly rounded one and gam within 1.93 units of 2^-53 (1.90 with IEEE operations;
// tests/test_gpu_digit_arithmetic.py).  32 steps on 32 rows: 106 -> 98 thousand cycles.
__device__ __forceinline__ void norm_and_gamma(double sig, double alpha, double& nrm, double& gam) {
  const long long sb = __double_as_longlong(sig);
  const int ex = (int)(sb >> 52) - 1023, half = ex >> 1;
  const float m = __uint_as_float(((uint32_t)(127 + (ex & 1)) << 23) | (uint32_t)((sb >> 29) & 0x7fffff));
  const uint32_t yu = __float_as_uint(rsqrtf(m));
  const double y0 = __longlong_as_double(((long long)((int)(yu >> 23) - 127 + 1023 - half) << 52) |
                                         ((long long)(yu & 0x7fffff) << 29));
  const double g0 = sig * y0, h0 = 0.5 * y0, r0 = fma(-g0, h0, 0.5);
  const double g1 = fma(g0, r0, g0), h1 = fma(h0, r0, h0);
  nrm = fma(fma(-g1, g1, sig), h1, g1);
  gam = recip_newton(fma(fabs(alpha), nrm, sig));
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Exponent e that brings entries whose largest biased exponent is E into
// (-1/4, 1/4) as x 2^{-e}; a column without a normal entry keeps 0, one with an
// inf or NaN gets TC_NONFINITE.
constexpr int TC_NONFINITE = 1 << 20;
__device__ __forceinline__ int tc_exponent(int E) {
  return E == 0 ? 0 : (E == 0x7ff ? TC_NONFINITE : E - 1020);
}

// The eight balanced base-256 digits of V (4 or 8) consecutive values (FP64
// bits, value k scaled by 2^{-ex(k)} into (-1/4, 1/4) and rounded to a multiple of 2^-64),
// as V BF16 per digit: store(q, words) with the digits q of the V values.
// Adding 0x80 to every byte of the fixed-point value turns its bytes into the
// digits plus 128, and a byte becomes BF16 through the FP32 number 2^23 + byte.
template <int V, class Load, class Exp, class Store>
__device__ __forceinline__ void tc_digits(Exp&& ex, Load&& load, Store&& store) {
  uint32_t glo[V], ghi[V];
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const long long bits = __double_as_longlong(load(k));
    const int E = (int)((bits >> 52) & 0x7ff);
    unsigned long long F = 0;              // |x| 2^{64 - e}, below 2^62
    const int e = ex(k);
    if (E != 0 && E != 0x7ff && e < TC_NONFINITE / 2) {
      const unsigned long long m53 = ((unsigned long long)bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
      const int sh = E - 1011 - e;         // at most 9
      F = sh >= 0 ? m53 << (sh < 10 ? sh : 10) : (sh > -55 ? (m53 + (1ull << (-sh - 1))) >> -sh : 0ull);
    }
    const unsigned long long G = (bits < 0 ? 0ull - F : F) + 0x8080808080808080ull;
    glo[k] = (uint32_t)G;
    ghi[k] = (uint32_t)(G >> 32);
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    uint32_t w[V / 2];
    const uint32_t sel = 0x7440u | (uint32_t)(q < 4 ? 3 - q : 7 - q);
#pragma unroll
    for (int k = 0; k < V; k += 2) {
      const float f0 =
          __uint_as_float(__byte_perm(q < 4 ? ghi[k] : glo[k], 0x4B000000u, sel)) - 8388736.0f;
      const float f1 =
          __uint_as_float(__byte_perm(q < 4 ? ghi[k + 1] : glo[k + 1], 0x4B000000u, sel)) - 8388736.0f;
      w[k >> 1] = __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632u);
    }
    store(q, w);
  }
}

template <class Load, class Store>
__device__ __forceinline__ void tc_digits8(int e, Load&& load, Store&& store) {
  tc_digits<8>([e](int) { return e; }, load, [&](int q, const uint32_t (&w)[4]) { store(q, make_uint4(w[0], w[1], w[2], w[3])); });
}

template <class Load, class Store>
__device__ __forceinline__ void tc_digits4(int e, Load&& load, Store&& store) {
  tc_digits<4>([e](int) { return e; }, load, [&](int q, const uint32_t (&w)[2]) { store(q, make_uint2(w[0], w[1])); });
}

// Four accumulators of adjacent weights as one integer in units of the last
// (|acc| <= 2^24: the conversions are exact).
__device__ __forceinline__ long long tc_group4(float a0, float a1, float a2, float a3) {
  long long v = (long long)__float2int_rn(a3);
  v += (long long)__float2int_rn(a2) * 256;
  v += (long long)__float2int_rn(a1) * 65536;
  v += (long long)__float2int_rn(a0) * 16777216;
  return v;
}

}  // namespace dqmc
