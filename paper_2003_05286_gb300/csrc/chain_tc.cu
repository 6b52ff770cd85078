// The k slice products of one chunk in one launch on the tensor cores, for
// CHAIN_TC_MIN_N <= N <= 128 (Sec. 2, Eq. (Ztr); the arguments are those of
// chain_small.cu, the arithmetic of a product that of gemm_tc.cu).
//
// Every slice multiplies from the left, so a block of columns evolves on its
// own.  As separate products a slice is a split and a product launch with some
// 20 us of fixed cost between them (launches, TMEM allocation, first copies, a
// round trip of the block through memory).  Here one CTA keeps 32 columns of one
// instance for the whole chunk: the digits of the block in shared memory, the
// digit tiles of E streamed from L2 through two 64 KB slots (resident when N <=
// 64), the accumulators in TMEM.  Per slice: MMAs over the 32-row K-blocks; each
// of 512 threads turns eight sums into FP64, applies the row scale of the next
// slice and stages them; column exponents; digits of the next right operand.
// 32 columns: all eight weight groups then lie in the 128 columns of two MMA
// blocks, and a single instance still spreads over ceil(N / 32) SMs.
//
// Bound by the serial chain of a slice (7 us, of which the MMAs are 0.8 at N =
// 64).  One chunk of ten slices, before -> after: N = 36 (FP64 pipe, chain_small)
// 1 instance 110 -> 70 us, 128 353 -> 332; N = 49 256 instances 560 -> 151; from
// N = 64 (splits and products) N = 64 32 instances 292 -> 73 us, 256 470 -> 145;
// N = 100 256 instances 1020 -> 378; N = 121 32 instances 308 -> 99.
//
// Warps 0-15 epilogue and digits, warp 16 copies, warp 17 TMEM and MMAs.
#include <cuda_bf16.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace dqmc {

namespace {

constexpr int CT_EPI = 512, CT_THREADS = CT_EPI + 64;
constexpr int CT_CB = 32;                       // columns per CTA
constexpr int CT_SLOT = 8 * 128 * 64;           // digits of a 128 x 32 tile of E
constexpr int CT_DT = CT_CB * 64;               // one digit of a 32 x 32 tile of the block
constexpr int CT_KB = 11 * CT_DT;               // 3 zero tiles, 8 digits
constexpr int CT_LD = CT_CB + 1;
// BF16 operands (K-major), FP32 accumulator, M = 128, N = 128
constexpr uint32_t CT_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) |
                              ((128u >> 4) << 24);

struct ChainTcArgs {
  ChainSmallArgs c;
  const __nv_bfloat16* Es;   // digits of E (or E^T) as a left operand
  const int* eEs;
  int* status;
  int status_div, nkb, b0;
};

// The staged block lies in the second slot when there is no room beside it.
__host__ __device__ constexpr bool ct_alias(int nkb) { return nkb == 4; }
__host__ __device__ constexpr int ct_smem(int nkb) {
  return 1024 + 2 * CT_SLOT + nkb * CT_KB + (ct_alias(nkb) ? 0 : 32 * nkb * CT_LD * 8) +
         (3 * CT_CB + 128) * 4 + 128;
}
static_assert(ct_smem(2) <= 227 * 1024 && ct_smem(3) <= 227 * 1024 && ct_smem(4) <= 227 * 1024,
              "shared memory of one CTA");

// Barrier of the epilogue warps: whether any thread brought a true predicate.
__device__ __forceinline__ bool bar_any(bool p) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.or.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)p), "n"(CT_EPI)
      : "memory");
  return r != 0;
}

}  // namespace

__global__ void __launch_bounds__(CT_THREADS, 1) chain_tc_kernel(const ChainTcArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int nkb = a.nkb, N = a.c.N;
  const bool alias = ct_alias(nkb), resident = nkb <= 2;
  unsigned char* bd = base + 2 * CT_SLOT;                         // digits of the block
  double* ct = reinterpret_cast<double*>(alias ? base + CT_SLOT : bd + nkb * CT_KB);
  int* ecol = reinterpret_cast<int*>(bd + nkb * CT_KB + (alias ? 0 : 32 * nkb * CT_LD * 8));  // [3][32]
  int* erow = ecol + 3 * CT_CB;                                   // [128]
  uint64_t* full = reinterpret_cast<uint64_t*>(erow + 128);       // [2]
  uint64_t* empty = full + 2;                                     // [2]
  uint64_t* acc = empty + 2;                                      // accumulators complete
  uint64_t* ready = acc + 1;                                      // the block's digits are written
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(ready + 1);
  int* s_fail = reinterpret_cast<int*>(tmem_holder + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b = a.b0 + blockIdx.y, c0 = blockIdx.x * CT_CB;
  if (!DQMC_CHECK(blockDim.x == CT_THREADS && N <= 32 * nkb && nkb >= 1 && nkb <= 4, N) ||
      !DQMC_CHECK(dyn_smem_bytes() >= (unsigned)(reinterpret_cast<unsigned char*>(s_fail + 1) - smem_raw),
                  dyn_smem_bytes()) ||
      !DQMC_CHECK((reinterpret_cast<uintptr_t>(a.Es) & 15) == 0, nkb))
    return;
  const double* X = a.c.X + (long long)b * a.c.sX;
  double* C = a.c.C + (long long)b * a.c.sC;
  const double* ev = a.c.expV + (long long)(b / a.c.divS) * a.c.sV + (long long)(b % a.c.divS) * a.c.sV_inner;
  int nsl = a.c.nslices;
  if (a.c.lim) {                                // slices past the instance's own chain end
    const int last = a.c.lim[b] - a.c.lim_base + 1;
    nsl = last < nsl ? (last > 0 ? last : 0) : nsl;
  }
  if (nsl == 0) {                               // the chain has ended: the block passes through
    for (int e = tid; e < N * CT_CB; e += CT_THREADS) {
      const int r = e / CT_CB, c = c0 + e % CT_CB;
      if (c < N) C[(long long)r * N + c] = X[(long long)r * N + c];
    }
    return;
  }
  // row scale of slice step s: forward in front of the product, backward behind it
  auto scales = [&](int s) {
    return ev + (long long)((a.c.dir > 0 ? a.c.lo + s : a.c.hi - s) - 1) * N;
  };

  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    mbar_init(acc, 1);
    mbar_init(ready, CT_EPI / 32);
    *s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 17) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_holder)),
                 "r"(256u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  for (int i = tid; i < nkb * 3 * CT_DT / 16; i += CT_THREADS) {
    const int kb = i / (3 * CT_DT / 16), o = i % (3 * CT_DT / 16);
    reinterpret_cast<uint4*>(bd + kb * CT_KB)[o] = make_uint4(0u, 0u, 0u, 0u);
  }
  if (tid < 3 * CT_CB) ecol[tid] = 0;
  if (tid < 128) erow[tid] = a.eEs[tid];
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_holder;

  if (warp == 16) {
    if (lane == 0) {
      // tile g = s nkb + kb goes to slot g & 1 once the MMAs of tile g - 2 have read it;
      // the second slot also waits for the digits when the block is staged in it
      const int total = resident ? nkb : nsl * nkb;
      int issued = 0;
      for (int g = 0; g < total; ++g) {
        const int st = g & 1, s = g / nkb, kb = g % nkb;
        bool ok = true;
        if (g >= 2) ok = mbar_wait(&empty[st], (g / 2 - 1) & 1);
        if (ok && alias && st == 1 && kb == 1) ok = mbar_wait(ready, s & 1);
        if (!ok) atomicOr(s_fail, 1);
        if (*(volatile int*)s_fail) break;
        mbar_arrive_expect_tx(&full[st], CT_SLOT);
        bulk_load(base + st * CT_SLOT, reinterpret_cast<const unsigned char*>(a.Es) + (long long)kb * CT_SLOT,
                  CT_SLOT, &full[st]);
        issued = g + 1;
      }
      // after a failure the copies still in flight land before the CTA exits
      if (*(volatile int*)s_fail)
        for (int g = issued > 2 ? issued - 2 : 0; g < issued; ++g) mbar_wait(&full[g & 1], (g / 2) & 1);
    }
    __syncwarp();
  } else if (warp == 17) {
    if (lane == 0) {
      bool ok = true;
      for (int s = 0; s < nsl && ok; ++s) {
        ok = mbar_wait(ready, s & 1);
        for (int kb = 0; kb < nkb && ok; ++kb) {
          const int g = resident ? kb : s * nkb + kb, st = g & 1;
          if (!resident || s == 0) ok = mbar_wait(&full[st], (g / 2) & 1);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t da = smem_desc_sw64(smem_u32(base + st * CT_SLOT));
          const uint64_t db = smem_desc_sw64(smem_u32(bd + kb * CT_KB));
          for (int r = 0; r < 2; ++r)
            for (int kk = 0; kk < 2; ++kk)
              for (int q = 0; q <= 4 * r + 3; ++q)
                umma(tmem + 128u * r, da + (uint64_t)(kk * 2 + q * ((128 * 64) >> 4)),
                     db + (uint64_t)(kk * 2 + (3 + 4 * r - q) * (CT_DT >> 4)), CT_IDESC,
                     kb == 0 && kk == 0 && q == 0 ? 0u : 1u);
          if (!resident) umma_commit(&empty[st]);
        }
        if (ok) umma_commit(acc);
        if (*(volatile int*)s_fail) break;
      }
      if (!ok) atomicOr(s_fail, 1);
    }
    __syncwarp();
  } else {
    const int rl = (warp & 3) * 32 + lane, cb = 8 * (warp >> 2);
    // digits of the staged block, eight rows of one column per thread
    auto digits = [&](const int* e) {
      const int kb = tid >> 7, c = (tid >> 2) & 31, ch = tid & 3;
      if (kb < nkb) {
        const double* src = ct + (32 * kb + 8 * ch) * CT_LD + c;
        unsigned char* dst = bd + kb * CT_KB + 3 * CT_DT + c * 64 + ((ch ^ ((c >> 1) & 3)) << 4);
        tc_digits8(tc_exponent(e[c]), [&](int k) { return src[k * CT_LD]; },
                   [&](int q, uint4 w) { *reinterpret_cast<uint4*>(dst + q * CT_DT) = w; });
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(ready);
    };
    // the block as it comes in, with the first slice's scale
    {
      const double* sc = a.c.dir > 0 ? scales(0) : nullptr;
      for (int r = warp; r < 32 * nkb; r += 16) {
        double v = r < N && c0 + lane < N ? X[(long long)r * N + c0 + lane] : 0.0;
        if (sc && r < N) v *= sc[r];
        ct[r * CT_LD + lane] = v;
        atomicMax(&ecol[lane], (int)((__double_as_longlong(v) >> 52) & 0x7ff));
      }
      asm volatile("bar.sync 1, %0;" ::"n"(CT_EPI) : "memory");
      digits(ecol);
    }
    const bool live = (warp & 3) * 32 < 32 * nkb;   // this warp's rows exist
    bool ok = true;
    int i0 = 0, i1 = 1, i2 = 2;
    for (int s = 0; s < nsl && ok; ++s) {
      // column exponents of this product's right operand, of the next one's, and
      // those of the last one, which nothing reads any more
      int *e0 = ecol + i0 * CT_CB, *e1 = ecol + i1 * CT_CB, *e2 = ecol + i2 * CT_CB;
      const bool last = s + 1 == nsl;
      if (tid < CT_CB) e2[tid] = 0;
      // the scale behind this product (backward) or in front of the next (forward)
      double f = 1.0;
      const bool scaled = a.c.dir < 0 || !last;
      if (scaled && rl < N) f = scales(a.c.dir > 0 ? s + 1 : s)[rl];
      ok = mbar_wait(acc, s & 1);
      ok = __all_sync(0xffffffffu, ok);
      if (live && ok) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int ea = erow[rl];
        uint32_t r[8][8];
#pragma unroll
        for (int g = 0; g < 8; ++g)
          tmem_ld8_nowait(tmem + ((uint32_t)((warp & 3) * 32) << 16) + 32 * g + cb, r[g]);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const long long hi = tc_group4(__uint_as_float(r[0][j]), __uint_as_float(r[1][j]),
                                         __uint_as_float(r[2][j]), __uint_as_float(r[3][j]));
          const long long lo = tc_group4(__uint_as_float(r[4][j]), __uint_as_float(r[5][j]),
                                         __uint_as_float(r[6][j]), __uint_as_float(r[7][j]));
          const int eb = tc_exponent(e0[cb + j]);
          double v = split_times_pow2(hi + (lo >> 32), (unsigned int)(lo & 0xFFFFFFFFll), ea + eb - 72);
          if (ea >= TC_NONFINITE || eb >= TC_NONFINITE) v = __longlong_as_double(0x7ff8000000000000ll);
          if (scaled) v *= f;
          ct[rl * CT_LD + cb + j] = v;
          const int mx = __reduce_max_sync(0xffffffffu, (int)((__double_as_longlong(v) >> 52) & 0x7ff));
          if (lane == 0) atomicMax(&e1[cb + j], mx);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      }
      // all 16 warps go on or none does
      ok = !bar_any(!ok || *(volatile int*)s_fail);
      if (ok && !last) digits(e1);
      const int t = i2;
      i2 = i0; i0 = i1; i1 = t;
    }
    if (ok) {
      for (int r = warp; r < N; r += 16)
        if (c0 + lane < N) C[(long long)r * N + c0 + lane] = ct[r * CT_LD + lane];
    } else if (tid == 0) {
      atomicOr(s_fail, 1);                         // ends the other two warps' loops
      if (a.status) atomicOr(&a.status[b / a.status_div], DQMC_STATUS_TIMEOUT);
    }
  }
  __syncthreads();
  if (warp == 17) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u)
                 : "memory");
  }
}

cudaError_t chain_tc(const ChainSmallArgs& c, const __nv_bfloat16* Es, const int* eEs, int* status,
                     int status_div, cudaStream_t st) {
  if (c.batch <= 0 || c.nslices <= 0) return cudaSuccess;
  if (c.N < CHAIN_TC_MIN_N || c.N > 128) return cudaErrorInvalidValue;
  ChainTcArgs a;
  a.c = c;
  a.Es = Es; a.eEs = eEs;
  a.status = status; a.status_div = status_div;
  a.nkb = (c.N + 31) / 32;
  const cudaError_t e = allow_dyn_smem(chain_tc_kernel);
  if (e != cudaSuccess) return e;
  for (a.b0 = 0; a.b0 < c.batch; a.b0 += 65535) {
    const int nb = c.batch - a.b0 < 65535 ? c.batch - a.b0 : 65535;
    chain_tc_kernel<<<dim3((c.N + CT_CB - 1) / CT_CB, nb), CT_THREADS, ct_smem(a.nkb), st>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace dqmc

DQMC_CHECK_UNIT(chain_tc)
