// Batched FP64 products on the tcgen05 tensor cores.
//
// GB300 runs FP64 FMAs at 1.25 TFLOP/s and dense BF16 at about 1.9 PFLOP/s, so
// an N x N FP64 product evaluated as 36 exact BF16 digit products has a 40
// times higher ceiling than the FP64 pipe.  The evaluation is the error-free
// splitting of Ozaki et al. (Numer. Algorithms 59, 2012) with 8-bit digits:
//
//   * every row i of the left and every column j of the right operand is
//     scaled by a power of two so that its entries lie in (-1/4, 1/4), rounded
//     to a multiple of 2^-64 (61 to 62 bits below the largest entry, where
//     FP64 holds 53 below each entry) and written as eight digits in
//     [-128, 127]: x = sum_p d_p 2^{-8(p+1)}, exact in BF16;
//   * digit products are at most 2^14; those of equal weight p + q = g share a
//     TMEM accumulator, and the FP32 accumulation is exact while
//     K (pairs in the group) 2^14 <= 2^24: groups 0..3 (at most 4 pairs) may
//     sum over 256 values of k, groups 4..7 over 128, after which they are
//     drained into 64-bit integers and start again from zero;
//   * pairs with p + q >= 8 are dropped: 7.03 2^{-66} a term at most in scaled
//     units, with the rounding of both operands 8.03 2^{-66}.  The maxima of row
//     and column are at least 1/8 there: K 2^{-57} of (row max x column max) at
//     worst and some sqrt(K) 2^{-62} for digits of random sign, against K 2^{-53}
//     and sqrt(K) 2^{-54} for K FP64 FMAs (tests/test_gpu_digit_arithmetic.py);
//   * the epilogue adds the groups exactly in integers and rounds once to FP64.
// So the result is at least as accurate as the FMA chain normwise (against
// row max x column max); entries far below their row's and column's largest
// lose relative digits, as they do in the QR that consumes the products.
// A row or column with a non-finite entry gives NaN throughout.
//
// Measured against DFMA tiles at 92% of the FP64 pipe's rate: one product of 128
// instances at N = 256 takes 170 us (and its operand's split 43) instead of 3430,
// with the same error of the whole chain against 64-bit references.  A CTA of
// that product spends 29 thousand cycles in the MMAs (95% of their rate at N =
// 256 columns, a quarter of it on zero tiles), 10 in the conversion of the sums
// (21 with eight epilogue warps and branches in the rounding) and 5 around them.
//
// Digits are stored as tiles (128 rows x 32 k for the left operand, 64 x 32
// for the right), the eight planes of a tile adjacent, each in the 64-byte
// swizzled byte order the tensor core reads: one cp.async.bulk moves all
// digits of a tile.
#include <cuda_bf16.h>

#include <type_traits>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace dqmc {

namespace {

constexpr int TC_S = 8;            // digits per operand
constexpr int TC_BM = 128, TC_BN = 64, TC_BK = 32;
constexpr int TC_STAGES = 2;
constexpr int TC_EPI = 512;        // epilogue threads (16 warps); + producer and MMA warps
constexpr int TC_THREADS = TC_EPI + 64;
constexpr int TC_A_TILE = TC_BM * TC_BK * 2, TC_B_TILE = TC_BN * TC_BK * 2;   // bytes of one digit
constexpr int TC_BZERO = 3;        // zero tiles in front of the right operand's digits
constexpr int TC_BSLOTS = TC_BZERO + TC_S;
constexpr int TC_STAGE = TC_S * TC_A_TILE + TC_BSLOTS * TC_B_TILE;            // 108 KB
constexpr int TC_COPY = TC_S * (TC_A_TILE + TC_B_TILE);
constexpr int TC_C_LD = TC_BN + 1;
constexpr int TC_SMEM = TC_STAGES * TC_STAGE + 1024 + 128;
static_assert(TC_BM * TC_C_LD * 8 <= TC_STAGES * TC_STAGE, "result tile fits the stages");
static_assert(TC_SMEM <= 227 * 1024, "shared memory of one CTA");

// BF16 A and B (K-major), FP32 accumulator, M = 128, N = 256
constexpr uint32_t TC_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((256u >> 3) << 17) |
                              ((uint32_t)(TC_BM >> 4) << 24);

}  // namespace

// One CTA: a 128 x 64 tile of one product.  Warps 0-15 epilogue (four per
// TMEM lane quarter), warp 16 copies, warp 17 allocates TMEM and issues the MMAs.
// An accumulator block r holds groups 4r .. 4r + 3 in 256 TMEM columns; each
// MMA has N = 256 and adds, for one left digit p, the right digits 4r - p ..
// 4r - p + 3 (zero tiles where there is none), so consecutive MMAs write the
// same aligned block: MMAs into partially overlapping column ranges wait for
// one another and run at a third of the rate.  Shared-memory bandwidth bounds
// the loop (12 KB read per 128-cycle MMA, 96 KB copied per 24 of them).
// WIN: 1 when K <= 128 (no drain), 2 when K <= 256 (block 1 drains once), 3 else.
// STACK: the left operands of all instances form one tall matrix, whose 32-row
// groups (one per epilogue warp) fill the tiles; the right operand is shared.
// 1: C_b = A_b B, 2: C_b = (A_b B)^T, for products whose shared operand is the left one.
// At N = 144 an instance then takes 160 rows of tiles instead of 256, 3.75 tiles
// instead of 6, and K stops at the last 16 values that hold any: the wraps of a
// gradient of 64 instances (1344 checkpoints) and its chains 94.7 -> 80.1 ms.
template <int WIN, int STACK>
__global__ void __launch_bounds__(TC_THREADS, 1) tc_gemm_kernel(const TcGemmArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(base + TC_STAGES * TC_STAGE);   // [2]
  uint64_t* empty = full + TC_STAGES;        // [2]
  uint64_t* acc_full = empty + TC_STAGES;    // [2] block r of a window complete
  uint64_t* acc_free = acc_full + 2;         // [2] block r drained
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(acc_free + 2);
  int* s_fail = reinterpret_cast<int*>(tmem_holder + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n0 = blockIdx.x * TC_BN, m0 = blockIdx.y * TC_BM;
  const int z = STACK ? 0 : blockIdx.z;   // operand slot
  const int b = a.b0 + z;              // instance
  const int N = a.N;
  const int kb0 = a.upperA ? m0 / TC_BK : 0, nk = a.nkb - kb0;
  if (!DQMC_CHECK(blockDim.x == TC_THREADS && nk >= 1 && (WIN > 1 || nk <= 4) &&
                      (WIN > 2 || nk <= 8) && a.ldc >= N, nk) ||
      !DQMC_CHECK(dyn_smem_bytes() >= (unsigned)TC_SMEM, dyn_smem_bytes()) ||
      !DQMC_CHECK((reinterpret_cast<uintptr_t>(a.A) & 15) == 0 &&
                      (reinterpret_cast<uintptr_t>(a.B) & 15) == 0 && a.sA % 8 == 0 &&
                      a.sB % 8 == 0, a.sA))
    return;
  // an instance whose chain has ended: its source passes through (uniform over
  // the CTA, before any barrier or TMEM allocation)
  if (!STACK && a.lim && a.lim[b] < a.lim_at) {
    const double* src = a.csrc + (long long)b * a.scsrc;
    double* dst = a.C + (long long)b * a.sC;
    for (int e = tid; e < TC_BM * TC_BN; e += TC_THREADS) {
      const int r = m0 + e / TC_BN, c = n0 + e % TC_BN;
      if (r < N && c < N) dst[(long long)r * a.ldc + c] = src[(long long)r * a.ldcsrc + c];
    }
    return;
  }
  if (tid == 0) {
    for (int i = 0; i < TC_STAGES; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int r = 0; r < 2; ++r) {
      mbar_init(&acc_full[r], 1);
      mbar_init(&acc_free[r], TC_EPI / 32);
    }
    *s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 17) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_holder)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // zero tiles in front of the digits (the copies never write them)
  for (int st = 0; st < TC_STAGES; ++st) {
    uint4* zb = reinterpret_cast<uint4*>(base + st * TC_STAGE + TC_S * TC_A_TILE);
    for (int i = tid; i < TC_BZERO * TC_B_TILE / 16; i += TC_THREADS) zb[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_holder;

  if (warp == 16) {
    if (lane == 0) {
      const __nv_bfloat16* a0 = a.A + (long long)z * a.sA +
                                ((long long)blockIdx.y * a.nkb + kb0) * (TC_S * TC_BM * TC_BK);
      const __nv_bfloat16* b0 = a.B + (long long)z * a.sB +
                                ((long long)blockIdx.x * a.nkb + kb0) * (TC_S * TC_BN * TC_BK);
      int issued = 0;
      for (int i = 0; i < nk; ++i) {
        const int st = i % TC_STAGES;
        if (i >= TC_STAGES && !mbar_wait(&empty[st], (i / TC_STAGES - 1) & 1)) {
          atomicOr(s_fail, 1);
          break;
        }
        if (*(volatile int*)s_fail) break;
        unsigned char* sb = base + st * TC_STAGE;
        mbar_arrive_expect_tx(&full[st], TC_COPY);
        bulk_load(sb, a0 + (long long)i * (TC_S * TC_BM * TC_BK), TC_S * TC_A_TILE, &full[st]);
        bulk_load(sb + TC_S * TC_A_TILE + TC_BZERO * TC_B_TILE,
                  b0 + (long long)i * (TC_S * TC_BN * TC_BK), TC_S * TC_B_TILE, &full[st]);
        issued = i + 1;
      }
      // after a failure the copies still in flight land before the CTA exits
      if (*(volatile int*)s_fail)
        for (int i = issued > TC_STAGES ? issued - TC_STAGES : 0; i < issued; ++i)
          mbar_wait(&full[i % TC_STAGES], (i / TC_STAGES) & 1);
    }
    __syncwarp();
  } else if (warp == 17) {
    if (lane == 0) {
      bool ok = true;
      for (int i = 0; i < nk && ok; ++i) {
        const int st = i % TC_STAGES;
        if (!mbar_wait(&full[st], (i / TC_STAGES) & 1)) {
          ok = false;
          break;
        }
        // start-address fields of the stage's tiles (address >> 4; shared
        // addresses stay below 256 KB, so the field never carries)
        const uint64_t dA = smem_desc_sw64(smem_u32(base + st * TC_STAGE));
        const uint64_t dB = dA + (uint64_t)((TC_S * TC_A_TILE) >> 4);
        for (int r = 0; r < 2 && ok; ++r) {
          const int every = r ? 4 : 8;         // K-blocks a block may sum exactly
          const bool start = i % every == 0;
          if (start && i > 0 && !mbar_wait(&acc_free[r], (i / every - 1) & 1)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const int nkk = (kb0 + i) * TC_BK + 16 < N ? 2 : 1;   // all k beyond are zero
          for (int kk = 0; kk < nkk; ++kk) {
            const uint64_t dAk = dA + (uint64_t)(kk * 2), dBk = dB + (uint64_t)(kk * 2);
            for (int p = 0; p <= 4 * r + 3; ++p)
              umma(tmem + (uint32_t)(256 * r), dAk + (uint64_t)(p * (TC_A_TILE >> 4)),
                   dBk + (uint64_t)((TC_BZERO + 4 * r - p) * (TC_B_TILE >> 4)), TC_IDESC,
                   start && kk == 0 && p == 0 ? 0u : 1u);   // p = 0 reaches all four groups first
          }
        }
        if (!ok) break;
        umma_commit(&empty[st]);
        if (i == nk - 1 || i % 4 == 3) umma_commit(&acc_full[1]);
        if (i == nk - 1 || i % 8 == 7) umma_commit(&acc_full[0]);
        if (*(volatile int*)s_fail) break;
      }
      if (!ok) atomicOr(s_fail, 1);
    }
    __syncwarp();
  } else {
    // ---- epilogue ------------------------------------------------------------
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const int cbase = (warp >> 2) * 16;
    const int rl = (warp & 3) * 32 + lane;
    const int grp = 4 * blockIdx.y + (warp & 3);         // 32-row group of the stack
    const int zs = STACK ? grp / a.groups : z;
    const int row = STACK ? (grp - zs * a.groups) * 32 + lane : m0 + rl;
    const int nwin = (nk + 3) / 4;             // windows of block 1 (block 0: every second)
    long long lo[WIN >= 2 ? 16 : 1], hi[WIN >= 3 ? 16 : 1];
    bool ok = true;
    auto group4 = [](const uint32_t (&r)[4][8], int j) {
      return tc_group4(__uint_as_float(r[0][j]), __uint_as_float(r[1][j]), __uint_as_float(r[2][j]),
                       __uint_as_float(r[3][j]));
    };
    if (WIN >= 2) {
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        lo[WIN >= 2 ? j : 0] = 0;
        if (WIN >= 3) hi[WIN >= 3 ? j : 0] = 0;
      }
      for (int t = 0; t + 1 < nwin && ok; ++t) {
        const bool both = WIN >= 3 && (t & 1);
        ok = mbar_wait(&acc_full[1], t & 1);
        if (ok && both) ok = mbar_wait(&acc_full[0], (t >> 1) & 1);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t r[4][8];
#pragma unroll
          for (int g = 0; g < 4; ++g)
            tmem_ld8_nowait(tmem + lane_addr + (4 + g) * TC_BN + cbase + 8 * c, r[g]);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 8; ++j) lo[WIN >= 2 ? 8 * c + j : 0] += group4(r, j);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_free[1]);
        if (WIN >= 3 && both) {
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t r[4][8];
#pragma unroll
            for (int g = 0; g < 4; ++g)
              tmem_ld8_nowait(tmem + lane_addr + g * TC_BN + cbase + 8 * c, r[g]);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 8; ++j) hi[WIN >= 3 ? 8 * c + j : 0] += group4(r, j);
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_free[0]);
        }
      }
    }
    if (ok) ok = mbar_wait(&acc_full[1], (nwin - 1) & 1);
    if (ok) ok = mbar_wait(&acc_full[0], ((nwin - 1) >> 1) & 1);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok && lane == 0) atomicOr(s_fail, 1);
    asm volatile("bar.sync 1, %0;" ::"r"(TC_EPI) : "memory");
    ok = *(volatile int*)s_fail == 0;          // uniform over the epilogue warps
    if (ok) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int bs = a.b0 + zs;
      const bool have = row < N && zs < a.slots;
      const int ea = have ? a.eA[(long long)zs * a.seA + row] : 0;
      const bool ended = STACK == 2 && have && a.lim && a.lim[bs] < a.lim_at;
      const int* eB = a.eB + (long long)z * a.seB;
      double rscale = a.alpha;
      if (STACK != 2 && a.rs && have) rscale *= a.rs[(long long)(bs / a.divS) * a.srs + row];
      const double* crs = STACK == 2 && a.rs && have ? a.rs + (long long)(bs / a.divS) * a.srs : nullptr;
      double* cst = a.C + (long long)bs * a.sC + row;
      const double* cend = ended ? a.csrc + (long long)bs * a.scsrc + row : nullptr;
      double* ctile = reinterpret_cast<double*>(base);   // the stages are idle now
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t r[4][8];
        long long l8[8];
#pragma unroll
        for (int g = 0; g < 4; ++g) tmem_ld8_nowait(tmem + lane_addr + (4 + g) * TC_BN + cbase + 8 * c, r[g]);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          l8[j] = group4(r, j);
          if (WIN >= 2) l8[j] += lo[WIN >= 2 ? 8 * c + j : 0];
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) tmem_ld8_nowait(tmem + lane_addr + g * TC_BN + cbase + 8 * c, r[g]);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          long long h = group4(r, j);
          const long long l = l8[j];
          if (WIN >= 3) h += hi[WIN >= 3 ? 8 * c + j : 0];
          const int col = n0 + cbase + 8 * c + j;
          const int eb = col < N ? eB[col] : 0;
          // (h 2^32 + l) 2^{-8 (7 + 2)}: the lowest kept weight is g = 7
          double v = split_times_pow2(h + (l >> 32), (unsigned int)(l & 0xFFFFFFFFll),
                                      ea + eb - 8 * (TC_S + 1));
          if (ea >= TC_NONFINITE || eb >= TC_NONFINITE) v = __longlong_as_double(0x7ff8000000000000ll);
          if (STACK == 2) {                      // lanes along the rows of C
            if (have && col < N) {
              if (a.scaled) v *= crs ? rscale * crs[col] : rscale;
              cst[(long long)col * a.ldc] = ended ? cend[(long long)col * a.ldcsrc] : v;
            }
          } else {
            ctile[rl * TC_C_LD + cbase + 8 * c + j] = v;
          }
        }
      }
      if (STACK != 2 && a.scaled) {   // row scale (and alpha): one FP64 multiply per entry
#pragma unroll 4
        for (int j = 0; j < 16; ++j) ctile[rl * TC_C_LD + cbase + j] *= rscale;
      }
      if (STACK != 2) {
        asm volatile("bar.sync 1, %0;" ::"r"(TC_EPI) : "memory");
        for (int e = tid; e < TC_BM * TC_BN; e += TC_EPI) {
          const int r = e / TC_BN, c = e % TC_BN;
          const int g = 4 * blockIdx.y + (r >> 5), zr = STACK ? g / a.groups : z;
          const int cr = STACK ? (g - zr * a.groups) * 32 + (r & 31) : m0 + r;
          if (zr < a.slots && cr < N && n0 + c < N)
            a.C[(long long)(a.b0 + zr) * a.sC + (long long)cr * a.ldc + n0 + c] = ctile[r * TC_C_LD + c];
        }
      }
    } else if (a.status && (STACK ? lane == 0 && warp < 4 && zs < a.slots : tid == 0)) {
      atomicOr(&a.status[(a.b0 + zs) / a.status_div], DQMC_STATUS_TIMEOUT);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  if (warp == 17) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// Splitter: element (m, j) of the operand at X[gm(m) ldm + j ldj] (gm the
// optional row gather), times an optional scale sc[m], into digit tiles of R
// rows j x 32 columns m (planes of a tile adjacent) and exponents e[j].
// One CTA per 32 rows j of one instance.  Phase 1 stages them in shared memory
// (lanes along the contiguous index: j when ldj = 1, else m) and finds each
// row's largest exponent; phase 2 gives every thread eight consecutive m of one
// j, i.e. one 16-byte store per digit: about 30 integer and FP32 instructions
// per entry, and the kernel is bound by its stores (16 bytes per entry).
// ---------------------------------------------------------------------------
template <bool ALONG_M>
__global__ void __launch_bounds__(256) tc_split_kernel(const TcSplitArgs a) {
  extern __shared__ double tile[];   // [PM][33]
  __shared__ int emax[8][32];
  const int z = blockIdx.y, b = a.b0 + z;
  const int j0 = blockIdx.x * 32, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int N = a.N, PM = a.PM;
  if (!DQMC_CHECK(blockDim.x == 256 && PM % 32 == 0 && a.R >= 32 && a.R % 32 == 0, PM) ||
      !DQMC_CHECK(dyn_smem_bytes() >= (unsigned)PM * 33u * 8u, dyn_smem_bytes()))
    return;
  if (a.lim && a.lim[b] < a.lim_at) return;   // this instance's chain has ended
  const double* X = a.X + (long long)b * a.sX;
  const double* sc = a.sc ? a.sc + (long long)(b / a.divS) * a.ssc +
                                (long long)(b % a.divS) * a.ssc_inner
                          : nullptr;
  const int* gm = a.gm ? a.gm + (long long)b * a.sgm : nullptr;
  auto row_of = [&](int m) {
    if (m >= N) return -1;
    const int r = gm ? gm[m] : m;
    return DQMC_CHECK(r >= 0 && r < N, r) ? r : -1;
  };
  if (!ALONG_M) {
    const int j = j0 + lane;
    int mx = 0;
    for (int mb = wid; mb < PM; mb += 64) {   // eight loads in flight per thread
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = row_of(mb + 8 * u);
        v[u] = r >= 0 && j < N && !(a.upper && r < j) ? X[(long long)r * a.ldm + (long long)j * a.ldj] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int m = mb + 8 * u;
        if (sc && m < N) v[u] *= sc[m];
        if (m < PM) tile[m * 33 + lane] = v[u];
        mx = max(mx, (int)((__double_as_longlong(v[u]) >> 52) & 0x7ff));
      }
    }
    emax[wid][lane] = mx;
  } else {
    // warp w holds rows j0 + w, w + 8, w + 16, w + 24; lanes along m
    int mx[4] = {0, 0, 0, 0};
    for (int mb = 0; mb < PM; mb += 32) {
      const int m = mb + lane, r = row_of(m);
      const double s = sc && m < N ? sc[m] : 1.0;
      double v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = j0 + wid + 8 * u;
        v[u] = r >= 0 && j < N && !(a.upper && r < j) ? X[(long long)r * a.ldm + (long long)j * a.ldj] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (sc) v[u] *= s;
        tile[m * 33 + wid + 8 * u] = v[u];
        mx[u] = max(mx[u], (int)((__double_as_longlong(v[u]) >> 52) & 0x7ff));
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int m2 = __reduce_max_sync(0xffffffffu, mx[u]);
      if (lane == 0) emax[0][wid + 8 * u] = m2;
    }
  }
  __syncthreads();
  if (tid < 32) {
    int m2 = emax[0][tid];
    if (!ALONG_M)
      for (int r = 1; r < 8; ++r) m2 = max(m2, emax[r][tid]);
    const int e = tc_exponent(m2);
    emax[0][tid] = e;
    a.e[(long long)z * a.se + j0 + tid] = e;
  }
  __syncthreads();
  __nv_bfloat16* S = a.S + (a.stack ? 0 : (long long)z * a.sS);
  const int jt = (a.stack ? z * a.PJ : 0) + j0;   // the CTA's first row of the stack
  const int ch = tid & 3, nkb = PM / 32;
  const int plane = a.R * 32;
  for (int it = tid >> 2; it < 32 * nkb; it += 64) {
    const int jj = it & 31, kb = it >> 5;
    const int e = emax[0][jj];
    const int mb = kb * 32 + ch * 8;
    const int jr = (jt + jj) % a.R;
    __nv_bfloat16* out = S + ((long long)((jt + jj) / a.R) * nkb + kb) * (TC_S * (long long)plane) +
                         jr * 32 + ((ch ^ ((jr >> 1) & 3)) << 3);   // 64-byte swizzle
    tc_digits8(e, [&](int k) { return tile[(mb + k) * 33 + jj]; }, [&](int q, uint4 w) {
      if (DQMC_CHECK((reinterpret_cast<uintptr_t>(out + q * plane) & 15) == 0, q))
        *reinterpret_cast<uint4*>(out + q * plane) = w;
    });
  }
}

cudaError_t tc_split(const TcSplitArgs& a, int batch, cudaStream_t st) {
  if (batch <= 0) return cudaSuccess;
  if (batch > 65535 || a.PM % 32 || a.PJ % (a.stack ? 32 : a.R) || a.R % 32 || a.PM < a.N || a.PJ < a.N ||
      a.sS % 8 || (reinterpret_cast<uintptr_t>(a.S) & 15) || (a.ldm != 1 && a.ldj != 1))
    return cudaErrorInvalidValue;
  const size_t sm = (size_t)a.PM * 33 * sizeof(double);
  const dim3 grid(a.PJ / 32, batch);
  cudaError_t e;
  if (a.ldj == 1) {
    if ((e = allow_dyn_smem(tc_split_kernel<false>)) != cudaSuccess) return e;
    tc_split_kernel<false><<<grid, 256, sm, st>>>(a);
  } else {
    if ((e = allow_dyn_smem(tc_split_kernel<true>)) != cudaSuccess) return e;
    tc_split_kernel<true><<<grid, 256, sm, st>>>(a);
  }
  return cudaGetLastError();
}

cudaError_t tc_gemm(const TcGemmArgs& args, int batch, cudaStream_t st) {
  if (batch <= 0) return cudaSuccess;
  TcGemmArgs a = args;
  if (batch > 65535 || a.nkb < 1 || a.nkb * TC_BK < a.N || a.N > TC_MAX_N || (a.lim && !a.csrc) ||
      (a.stack && (a.upperA || a.sB != 0)) || (a.stack == 1 && a.lim))
    return cudaErrorInvalidValue;
  a.slots = batch;
  a.groups = (a.N + 31) / 32;
  const long long rows = a.stack ? ((long long)batch * a.groups + 3) / 4 : (a.N + TC_BM - 1) / TC_BM;
  if (rows > 65535) return cudaErrorInvalidValue;
  const dim3 grid((a.N + TC_BN - 1) / TC_BN, (int)rows, a.stack ? 1 : batch);
  auto go = [&](auto kern) {
    const cudaError_t e = allow_dyn_smem(kern);
    if (e != cudaSuccess) return e;
    kern<<<grid, TC_THREADS, TC_SMEM, st>>>(a);
    return cudaGetLastError();
  };
  auto pick = [&](auto win) {
    constexpr int W = decltype(win)::value;
    if (a.stack == 1) return go(tc_gemm_kernel<W, 1>);
    if (a.stack == 2) return go(tc_gemm_kernel<W, 2>);
    return go(tc_gemm_kernel<W, 0>);
  };
  if (a.nkb <= 4) return pick(std::integral_constant<int, 1>{});
  if (a.nkb <= 8) return pick(std::integral_constant<int, 2>{});
  return pick(std::integral_constant<int, 3>{});
}

}  // namespace dqmc

DQMC_CHECK_UNIT(gemm_tc)
