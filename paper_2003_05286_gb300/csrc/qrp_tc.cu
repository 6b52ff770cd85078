// Blocked column-pivoted Householder QR with its large products on the tensor
// cores, for N in QRTC_MIN_N .. QRTC_MAX_N (Sec. 4.2.2, "QR (UDT)"; outputs as
// in qrp_f64.cu).
//
// The one-CTA kernels of qrp_f64.cu do all 8/3 N^3 flops of a factorisation on
// one SM's FP64 pipe (two FMAs per clock: 5.4 ms at N = 256) and add a serial
// chain per pivot step.  Here only the 32-column panels stay on that pipe:
//
//   qr_init     W^T (columns contiguous) and the column norms of A.
//   qr_panel    one CTA per instance and panel.  Pivots: the 128 (N > 256: 64)
//               remaining columns of largest D_c ||a_c|| run 32 steps of pivoted
//               Householder reduction in FP32 in registers (residual norms
//               recomputed at every step), which fixes the
//               order; at each panel the FP32 columns start from the FP64 ones,
//               so no error carries over, and the choice of a pivot does not
//               enter the accuracy of the factorisation.  The chosen columns
//               are then reduced in FP64: H_j = 1 - gamma_j u_j u_j^T,
//               u = x - beta e_j, gamma = 1 / (beta (beta - alpha)); one pass of
//               dot products with the raw column x gives ||x||^2 and, through
//               u^T a = x^T a - beta a_j, every u^T a.  The products
//               H_0 ... H_31 = 1 - V T V^T (Schreiber and Van Loan, 1989): V^T V
//               on the tensor cores, T by block inversion.
//   qr_apply    A <- A - V T^T (V^T A) for 32 remaining columns per CTA: both
//               products as exact 8-digit products (gemm_tc.cu), V's digits from
//               the panel kernel, A's and W's digits made on chip; then the
//               residual norms for the next choice.  For Q the same kernel
//               applies all panels backwards to 32 columns of the identity that
//               stay in shared memory.
//   qr_out      D, T = D^{-1} R and the pivot order.
//
// Measured against the one-CTA kernels, whole factorisation, random graded
// columns: N = 64 0.476 -> 0.265 ms (one instance) and 0.479 -> 0.301 (128), N =
// 100 1.03 -> 0.55 and 1.03 -> 0.77, N = 256 7.76 -> 1.64 and 7.85 -> 2.95, N =
// 324 22.6 -> 2.37 and 25.4 -> 7.67; same pivots, residuals no larger.  What is
// left at N = 256 (thousand cycles per panel of 256 rows): pivot search 140, FP64
// panel 255 (the FP64 pipe, plus a square root, a division and two barriers per
// column), digits and V^T V 27, T 12; an apply of 256 rows 55.
//
// V's columns are scaled by powers of two into (-1/4, 1/4) (|u_r| <= |u_j|), so
// V needs no exponents and T takes up the scales.  A column whose entries differ by many
// orders (or has zeros) is divided by its leading entry first: H_j = 1 - tau_j v_j v_j^T,
// v_j = u_j / u_jj, tau_j = (beta_j - alpha_j) / beta_j, which are exact for a multiple of a
// unit vector, as are its digits, T and Q, and decoupled sites stay decoupled.  (The
// rounding of gamma put 2^-53 into Q's zeros, times the grading of the next chunk: K = 0,
// fields of variance 4, N = 160, M = 40, k = 10, error of G 6e-8 -> 1e-15.)  Every
// product is then accurate column by column against the column's largest entry, as
// Householder's method is.  When the rows of A are graded too (Drow: the levels of the tree fold, whose
// factor D_2 sits on the left), Householder QR with column pivoting is accurate
// row by row (Cox and Higham, 1998), and so must be the update of A: it then uses
// a second set of digits in which u_rj has the size s_r of row r: V W2 has row
// exponents, its columns u_j 2^{-h_j} with max_r u_rj 2^{-rho_r - h_j} of order one,
// 2^{rho_r} ~ s_r = Drow_r (a pivot column that D_1 puts in front of larger ones would
// otherwise meet the others' W2 at its own size), and V^T A multiplies 2^{rho_r} u_rj
// by 2^{-rho_r} a_rc, so that both factors' largest entries meet in the same row.  Q
// needs only the first set.
// T is the first set's in both (the scales go in and out as exponents), so that
// nothing squares a column's scale: norms over FP64's whole range are taken.
#include <cuda_bf16.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace dqmc {

namespace {

constexpr int NB = 32;                    // panel width = k extent of a digit tile
constexpr int DT = 32 * 64;               // bytes of one digit of a 32 x 32 tile
constexpr int VT_TILE = 8 * DT;           // V^T: 8 digits x 32 panel columns x 32 rows
constexpr int V_TILE = 8 * 128 * 64;      // V: 8 digits x 128 rows x 32 panel columns
constexpr int RING = 4 * VT_TILE;         // staging of both kernels (64 KB)
constexpr int TLD = 33;
// Columns whose entries span more than 2^UNIT_SPAN get reflectors with leading entry one
// (the head of this file).  A zero has exponent 0; a dense column of 256 random entries
// spans some 2^12 and gains nothing, while the division, one multiplication an entry on the
// FP64 pipe, takes up to 1% of an N = 256 factorisation (1.618 -> 1.631 ms with all columns).
constexpr int UNIT_SPAN = 30;
constexpr int QF = 2 * 8 * 52;             // floats of two staged FP32 columns (8 x 52 >= 4 x 68)
constexpr int XS = QRTC_MAX_N;            // rows of a staged FP64 column
enum { QP_SMALL, QP_MID, QP_BIG };        // forms of the panel kernel
__host__ __device__ constexpr int xs_rows(bool small) { return small ? 64 : XS; }
// BF16 operands (K-major), FP32 accumulator, M = 128, N = 128
constexpr uint32_t IDESC_128 = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) |
                               ((128u >> 4) << 24);

__device__ __forceinline__ float log2_wide_f(double x) {
  if (!(x > 0.0)) return -INFINITY;
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((bits >> 52) & 0x7ff);
  if (e == 0) return -1074.0f;
  return (float)(e - 1023) + __log2f(__int_as_float(0x3f800000 | (int)((bits >> 29) & 0x7fffff)));
}

// x 2^{-e} as FP32 (mantissa truncated) with integer operations; below the
// normal range 0, and e is such that the result stays below 2.
__device__ __forceinline__ float scaled_f32(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int fe = (int)((b >> 52) & 0x7ff) - 1023 - e + 127;
  if (fe <= 0) return 0.0f;
  return __uint_as_float((uint32_t)(b >> 32 & 0x80000000u) | ((uint32_t)(fe < 254 ? fe : 254) << 23) |
                         (uint32_t)((b >> 29) & 0x7fffff));
}

// log2 of the norm of rows r0 .. r1 - 1 of a column (contiguous), by one warp;
// bad is set when an entry is not finite.
__device__ __forceinline__ float warp_log2_norm(const double* col, int r0, int r1, bool& bad) {
  const int lane = threadIdx.x & 31;
  int mx = 0;
  for (int r = r0 + lane; r < r1; r += 32)
    mx = max(mx, (int)((__double_as_longlong(col[r]) >> 52) & 0x7ff));
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (mx == 0x7ff) { bad = true; return -INFINITY; }
  if (mx == 0) return -INFINITY;
  const int e = mx - 1022;                // entries below 2^e
  float s = 0.0f;
  for (int r = r0 + lane; r < r1; r += 32) {
    const float f = scaled_f32(col[r], e);
    s = fmaf(f, f, s);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return (float)e + 0.5f * __log2f(s);
}

// Position of 16-byte chunk ch of row r in a tile of 64-byte rows (64-byte swizzle).
__device__ __forceinline__ int swz(int r, int ch) { return r * 64 + ((ch ^ ((r >> 1) & 3)) << 4); }

// Exponent rho_r of a row scale: 2^{rho_r} ~ Drow_r (rho = 0 without scales).
__device__ __forceinline__ int row_rho(const double* Drow, int r, int N) {
  if (!Drow || r >= N) return 0;
  const int E = (int)((__double_as_longlong(Drow[r]) >> 52) & 0x7ff);
  return E == 0x7ff ? 0 : E - 1022;
}

// nb steps of pivoted Householder reduction in FP32 on the 512 / TPC candidate
// columns (row g + TPC k in register k of thread g); the winners' candidate
// numbers go to s_sel.  Keys are log2(D_c) + log2 of the residual norm, which is
// summed anew at every step.  With row scales (GR) the registers hold x_r
// 2^{-rho_r}, and products are weighted by 2^{2 (rho_r - rho_s)} at step s: rows
// far below the current one drop out of them without leaving FP32's range.
// Bound by shared-memory reads of the pivot column and FP32 issue; two columns
// per thread, which halve those reads, took twice as long (263 against 125
// thousand cycles for 32 steps of 256 rows).
template <int TPC, int KM, bool GR, bool SMALL>
__device__ __noinline__ void pivot_search(const double* W, const double* Din, const float* lnrm,
                                          const int* s_rem, const int* s_cand, int N, int j0,
                                          int m, int nb, float* qf, float* s_inv,
                                          unsigned* s_max, int* s_sel, const int* s_rho) {
  static_assert(KM % 8 == 0 && KM * TPC >= 32, "float4 rows, batches of loads");
  constexpr int CN = 512 / TPC, QS = KM + 4;   // row groups land in distinct banks
  constexpr int KT = 32 / TPC;                 // registers that hold the panel's rows
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const unsigned FULL = 0xffffffffu;
  const int ci = tid / TPC, g = tid % TPC;
  const bool have = ci < m;                 // m <= CN or all CN candidates exist
  const int col = have ? s_rem[s_cand[ci]] : 0;
  const float ln = have && !GR ? lnrm[col] : -INFINITY;
  const int e = ln > -2000.0f ? (int)floorf(ln) + 1 : 0;   // the norm (graded: its rows' scales) out
  const float lead = have ? log2_wide_f(Din[col]) + (float)e : 0.0f;
  // two buffers each of u, u times the weights, the next step's weights
  float* su = qf;
  float* sw = qf + QF;
  float* sv = qf + 2 * QF;
  auto weight = [&](int r, int s) {          // 2^{2 (rho_r - rho_s)}
    const int w = r < m ? 2 * (s_rho[r] - s_rho[s < m ? s : m - 1]) : 0;
    return r < m ? __uint_as_float((uint32_t)(min(max(w, -126), 60) + 127) << 23) : 0.0f;
  };
  float x[KM];
  {
    const double* src = W + (long long)col * N + j0;
    constexpr int LB = KM % 16 == 0 ? 16 : 8;   // loads in flight
#pragma unroll
    for (int k0 = 0; k0 < KM; k0 += LB) {
      double v[LB];
#pragma unroll
      for (int k = 0; k < LB; ++k) {
        const int r = g + TPC * (k0 + k);
        v[k] = have && r < m ? src[r] : 0.0;
      }
#pragma unroll
      for (int k = 0; k < LB; ++k) {
        const int r = g + TPC * (k0 + k);
        x[k0 + k] = scaled_f32(v[k], GR ? (r < m ? s_rho[r] : 0) : e);
      }
    }
  }
  if (GR) {                                  // weights of step 0
    if (tid < TPC * KM) sv[QS * TPC + tid % TPC * QS + tid / TPC] = weight(tid, 0);
    __syncthreads();
  }
  // squared norm of the rows left (finished ones are zero), weights in buffer bf
  auto sum_sq = [&](int bf) {
    const float* wv = sv + bf * QS * TPC + g * QS;
    float n[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < KM; ++k) {
      n[k & 3] = fmaf(x[k], GR ? x[k] * wv[k] : x[k], n[k & 3]);
    }
    float t = (n[0] + n[1]) + (n[2] + n[3]);
#pragma unroll
    for (int o = 1; o < TPC; o <<= 1) t += __shfl_xor_sync(FULL, t, o);
    return t;
  };
  float ns = sum_sq(1);
  bool act = have;
  for (int s = 0; s < nb; ++s) {
    // key in the high bits (order-preserving), candidate in the low ones
    float key = lead + 0.5f * __log2f(ns);
    if (!(key == key)) key = -INFINITY;
    const unsigned u = __float_as_uint(key);
    const unsigned ord = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    const unsigned pk = act ? ((ord & ~(unsigned)(CN - 1)) | (unsigned)(CN - 1 - ci)) : 0u;
    const unsigned wm = __reduce_max_sync(FULL, pk);
    if (lane == 0) s_max[(s & 1) * 16 + wid] = wm;
    __syncthreads();
    const unsigned best = __reduce_max_sync(FULL, s_max[(s & 1) * 16 + (lane & 15)]);
    const int win = CN - 1 - (int)(best & (unsigned)(CN - 1));
    const int bo = (s & 1) * QS * TPC + g * QS;
    // row s of this column, selected by the row number: a select on s / TPC alone is
    // an index into x, which then lives in local memory (twice the time)
    float xs = 0.0f;
#pragma unroll
    for (int k = 0; k < KT; ++k)
      if (g + TPC * k == s) xs = x[k];
    xs = __shfl_sync(FULL, xs, lane / TPC * TPC + s % TPC);
    if (ci == win) {
      act = false;
      const float nrm = ns * rsqrtf(fmaxf(ns, 1e-37f)), us = xs >= 0.0f ? xs + nrm : xs - nrm;
      // the weights of step s are in buffer (s + 1) & 1
      const float* wv = sv + ((s + 1) & 1) * QS * TPC + g * QS;
#pragma unroll
      for (int k = 0; k < KM; k += 4) {
        *reinterpret_cast<float4*>(su + bo + k) = make_float4(x[k], x[k + 1], x[k + 2], x[k + 3]);
        if (GR)
          *reinterpret_cast<float4*>(sw + bo + k) =
              make_float4(x[k] * wv[k], x[k + 1] * wv[k + 1], x[k + 2] * wv[k + 2], x[k + 3] * wv[k + 3]);
      }
      if (g == s % TPC) {
        su[bo + s / TPC] = us;
        if (GR) sw[bo + s / TPC] = us;       // weight one
      }
      if (g == 0) {
        s_inv[s & 1] = ns > 0.0f ? __fdividef(-1.0f, fmaf(fabsf(xs), nrm, ns)) : 0.0f;   // -gamma
        s_sel[s] = win;
      }
    }
    if (GR && tid < TPC * KM)                // weights of step s + 1
      sv[(s & 1) * QS * TPC + tid % TPC * QS + tid / TPC] = weight(tid, s + 1);
    __syncthreads();
    const float* qu = su + bo;
    const float* qw = GR ? sw + bo : qu;
    float d[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < KM; k += 4) {
      const float4 q = *reinterpret_cast<const float4*>(qw + k);
      d[0] = fmaf(q.x, x[k], d[0]); d[1] = fmaf(q.y, x[k + 1], d[1]);
      d[2] = fmaf(q.z, x[k + 2], d[2]); d[3] = fmaf(q.w, x[k + 3], d[3]);
    }
    float t = (d[0] + d[1]) + (d[2] + d[3]);
#pragma unroll
    for (int o = 1; o < TPC; o <<= 1) t += __shfl_xor_sync(FULL, t, o);
    const float w = t * s_inv[s & 1];
#pragma unroll
    for (int k = 0; k < KM; k += 4) {
      const float4 q = *reinterpret_cast<const float4*>(qu + k);
      x[k] = fmaf(q.x, w, x[k]); x[k + 1] = fmaf(q.y, w, x[k + 1]);
      x[k + 2] = fmaf(q.z, w, x[k + 2]); x[k + 3] = fmaf(q.w, w, x[k + 3]);
    }
    // row s is finished
#pragma unroll
    for (int k = 0; k < KT; ++k) x[k] = g + TPC * k == s ? 0.0f : x[k];
    ns = sum_sq(s & 1);
  }
}

// FP64 Householder reduction of the chosen columns by the first LPC warps, LPC
// lanes a column (row l + LPC k in register k).  Every FP64 warp instruction
// holds its sub-partition's pipe for 64 cycles: short panels take 8 lanes (few
// reduction levels, few warps), tall ones 16 (the columns left spread evenly
// over the sub-partitions; N = 256, 32 columns: 323 -> 240 thousand cycles).  A
// warp whose columns are done drops out.  Leaves R in W^T and in out[0] (zeros above j)
// u_j, or where s_unit[j] is set v_j 2^{E_j}, v_j = u_j / u_jj, 2^{E_j} <= |u_jj| < 2^{E_j + 1};
// out[1]: two columns of workspace.
// s_gam[j] is the gamma of u_j 2^{-s_ex[j]}.  Squares of the columns as they are
// (s_ex = 0) serve while they stay inside FP64's range.  Where one of a panel's steps
// met one outside (gamma is left at zero) the first form returns true and writes
// nothing, and WIDE does the panel again from W^T with every pivot column scaled to
// order one by its largest exponent: one more reduction on the serial chain of a step,
// which the first form does without.
template <int LPC, int KR, bool SMALL, bool WIDE>
__device__ __noinline__ bool panel_factor(double* W, const int* s_rem, const int* s_sel, int N,
                                          int j0, int m, int nb, int LDU, double* const* out,
                                          double* s_beta, double* s_gam, double* s_uj, int* s_ex,
                                          int* s_unit) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned FULL = 0xffffffffu;
  constexpr int CPW = 32 / LPC;             // columns per warp
  static_assert(LPC * KR >= 32 && LPC * KR <= XS && KR % 2 == 0, "a panel's triangle fits the lanes' rows");
  const int l8 = lane % LPC, pc = CPW * wid + lane / LPC;   // this lane's panel column
  const bool own = pc < nb;
  double* col = W + (long long)(own ? s_rem[s_sel[pc]] : 0) * N + j0;
  double* us = out[0] + pc * LDU;
  const int rows = LDU - 1;                // rows of us
  double x[KR];
#pragma unroll
  for (int k = 0; k < KR; ++k) {
    const int r = l8 + LPC * k;
    x[k] = own && r < m ? col[r] : 0.0;
  }
  for (int j = 0; j < nb; ++j) {
    double* xj = out[1] + (j & 1) * (LPC * KR);
    const bool owner = wid == j / CPW;
    double down = 1.0;                     // the owner's 2^{-ex}, a power of two
    int mx = 0;
    if (WIDE && owner) {
      if (pc == j) {
#pragma unroll
        for (int k = 0; k < KR; ++k)
          if (l8 + LPC * k >= j) mx = max(mx, (int)((__double_as_longlong(x[k]) >> 52) & 0x7ff));
      }
      mx = __reduce_max_sync(FULL, mx);
      down = mx > 0 && mx < 0x7ff ? scalbn(1.0, 1023 - mx) : 1.0;
      if (lane == 0) s_ex[j] = mx > 0 && mx < 0x7ff ? mx - 1023 : 0;
    }
    if (owner && pc == j) {                // the column as it is now, zeros above row j
#pragma unroll
      for (int k = 0; k < KR; ++k)
        xj[l8 + LPC * k] = l8 + LPC * k >= j ? (WIDE ? x[k] * down : x[k]) : 0.0;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * LPC) : "memory");
    double d = 0.0, ajc = 0.0;
    if (CPW * wid + CPW - 1 >= j) {                // dots of the warps with columns >= j
      double d0 = 0.0, d1 = 0.0;
#pragma unroll
      for (int k = 0; k < KR; k += 2) {
        d0 = fma(xj[l8 + LPC * k], x[k], d0);
        d1 = fma(xj[l8 + LPC * (k + 1)], x[k + 1], d1);
      }
      d = d0 + d1;
#pragma unroll
      for (int o = 1; o < LPC; o <<= 1) d += __shfl_xor_sync(FULL, d, o);
#pragma unroll
      for (int k = 0; k < 32 / LPC; ++k)     // row j of the column (by row number, as above)
        if (l8 + LPC * k == j) ajc = x[k];
      ajc = __shfl_sync(FULL, ajc, lane / LPC * LPC + j % LPC);
      if (owner) {                         // the column's own dot is ||x||^2 (2^{-ex} of it)
        const double own_d = __shfl_sync(FULL, d, j % CPW * LPC);
        const double own_a = __shfl_sync(FULL, ajc, j % CPW * LPC);
        const double sig = WIDE ? own_d * down : own_d, alpha = WIDE ? own_a * down : own_a;
        double beta = 0.0, gam = 0.0;
        if (WIDE ? mx > 0 && mx < 0x7ff : sig > 1e-290 && sig < 1e300) {
          double nrm;
          norm_and_gamma(sig, alpha, nrm, gam);
          beta = alpha >= 0.0 ? -nrm : nrm;
        } else {
          // nothing to reduce (no normal entry), or a NaN or inf that is to reach D (without
          // WIDE the panel is done again)
          if (WIDE) beta = mx == 0 ? alpha : __longlong_as_double(0x7ff8000000000000ll);
          else beta = sig < 1e300 ? alpha : sig;
        }
        if (lane == 0) { s_beta[j] = beta; s_gam[j] = gam; s_uj[j] = gam > 0.0 ? alpha - beta : 0.0; }
      }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * LPC) : "memory");
    if (CPW * wid + CPW - 1 > j) {                 // a_c -= u (gamma u^T a_c), c > j
      const double w = pc > j ? -s_gam[j] * fma(-s_beta[j], ajc, d) : 0.0;
      const double uj = s_uj[j];
#pragma unroll
      for (int k = 0; k < KR; ++k) {
        double u = xj[l8 + LPC * k];
        if (k < 32 / LPC && l8 + LPC * k == j) u = uj;
        x[k] = fma(u, w, x[k]);
      }
    }
  }
  // (written before the last barrier of the loop: every warp sees the same)
  if (!WIDE && __any_sync(FULL, lane < nb && s_gam[lane] == 0.0)) return true;
  const double up = WIDE && own ? scalbn(1.0, s_ex[pc]) : 1.0;
  const bool on = own && s_gam[pc] > 0.0;
  const double beta = own ? s_beta[pc] : 0.0, uj = on ? s_uj[pc] : 1.0, u = WIDE ? uj * up : uj;
  const long long ub = __double_as_longlong(u), top = 0x7ffll << 52;
  int least = 0x7ff;                       // exponent of the smallest entry below the leading one
#pragma unroll
  for (int k = 0; k < KR; ++k) {
    const int r = l8 + LPC * k;
    if (r > pc && r < m) least = min(least, (int)((__double_as_longlong(x[k]) >> 52) & 0x7ff));
  }
#pragma unroll
  for (int o = 1; o < LPC; o <<= 1) least = min(least, __shfl_xor_sync(FULL, least, o));
  const bool unit = on && least < (int)((ub & top) >> 52) - UNIT_SPAN;
  const bool some = __any_sync(FULL, unit);
  double mu = 1.0;
  if (some && unit) {
    const double mant = __longlong_as_double((ub & ~top) | (1023ll << 52));
    mu = copysign(recip_newton(fabs(mant)), mant);
  }
#pragma unroll
  for (int k = 0; k < KR; ++k) {
    const int r = l8 + LPC * k;
    if (r < rows) {
      double v = r == pc ? u : x[k];
      if (some) {                          // the leading entry, and one as large, exactly +-2^{E_j}
        const long long xb = __double_as_longlong(v) ^ ub;
        v = unit && (xb << 1) == 0 ? __longlong_as_double((ub & top) | (xb & (1ll << 63))) : v * mu;
      }
      us[r] = on && r < m && r >= pc ? v : 0.0;
      if (own && r <= pc && r < m) col[r] = r == pc ? (WIDE ? beta * up : beta) : x[k];
    }
  }
  if (l8 == 0) s_unit[pc] = unit;
  return false;
}

// Waits on a phase unless an earlier wait of this CTA already gave up.
__device__ __forceinline__ void wait_or_fail(uint64_t* bar, uint32_t parity, int* s_fail) {
  if (*(volatile int*)s_fail) return;
  if (!mbar_wait(bar, parity)) atomicOr(s_fail, 1);
}

// D (two blocks of 128 TMEM columns) += left^T right over one 32-row K-block.
// Left: 8 digits x 32 rows stacked four digits to an M = 128 tile; right: 8
// digits x 32 columns.  Lane block d of the result holds, in its columns
// 32 c .., the digit products of weight g = d + c (g <= 7 is used): digits
// 0-3 against right digits 0-7, digits 4-7 against 0-3 added at c = 4 .. 7.
__device__ __forceinline__ void mma_stacked(uint32_t tmem, uint32_t left, uint32_t right, bool first) {
  const uint64_t dl = smem_desc_sw64(left), dr = smem_desc_sw64(right);
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
    const uint64_t l0 = dl + kk * 2, l1 = l0 + ((4 * DT) >> 4);
    const uint64_t r0 = dr + kk * 2, r1 = r0 + ((4 * DT) >> 4);
    umma(tmem, l0, r0, IDESC_128, first && kk == 0 ? 0u : 1u);
    umma(tmem + 128, l0, r1, IDESC_128, first && kk == 0 ? 0u : 1u);
    umma(tmem + 128, l1, r0, IDESC_128, 1u);
  }
}

// Result (i, c) of mma_stacked, exact in (hi 2^32 + lo): each lane block's sum
// goes to exchange memory (hi at ex, lo at ex + 4096), eight columns at a time.
__device__ __forceinline__ void stacked_partial(uint32_t tmem, int warp, int c0, long long* ex) {
  const int lane = threadIdx.x & 31, d = warp & 3;
  uint32_t r[8][8];
#pragma unroll
  for (int c = 0; c < 8; ++c)
    if (c + d <= 7) tmem_ld8_nowait(tmem + ((uint32_t)(d * 32) << 16) + 32 * c + c0, r[c]);
  tmem_wait_ld();
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    long long hi = 0, lo = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int g = c + d;
      if (g > 7) continue;
      const long long v = (long long)__float2int_rn(__uint_as_float(r[c][j]));
      if (g < 4) hi += v << (8 * (3 - g)); else lo += v << (8 * (7 - g));
    }
    ex[(d * 32 + c0 + j) * 32 + lane] = hi;
    ex[4096 + (d * 32 + c0 + j) * 32 + lane] = lo;
  }
}

// Entry (i, c) from the four lane blocks' sums; e: exponent of the operands.
__device__ __forceinline__ double stacked_value(const long long* ex, int i, int c, int e) {
  long long hi = 0, lo = 0;
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    hi += ex[(d * 32 + c) * 32 + i];
    lo += ex[4096 + (d * 32 + c) * 32 + i];
  }
  return split_times_pow2(hi + (lo >> 32), (unsigned int)(lo & 0xFFFFFFFFll), e - 72);
}

// acc (256 TMEM columns, 32 per weight) = left (8 digits x 128 rows x 32 k) times
// right (3 zero tiles, then 8 digits x 32 columns x 32 k).
__device__ __forceinline__ void mma_rows(uint32_t acc, uint32_t left, uint32_t right) {
  const uint64_t dv = smem_desc_sw64(left), dw = smem_desc_sw64(right);
  for (int r = 0; r < 2; ++r)
    for (int kk = 0; kk < 2; ++kk)
      for (int q = 0; q <= 4 * r + 3; ++q)
        umma(acc + 128u * r, dv + (uint64_t)(kk * 2 + q * ((128 * 64) >> 4)),
             dw + (uint64_t)(kk * 2 + (3 + 4 * r - q) * (DT >> 4)), IDESC_128,
             kk == 0 && q == 0 ? 0u : 1u);
}

// a2[c LD + row] -= the product's entry for eight columns of warp wid (of 16), row
// below `rows`; er: the row's exponent, ew: biased exponents of the columns.
__device__ __forceinline__ void rows_subtract(uint32_t acc, int wid, int row, int rows, int er,
                                              const int* ew, double* a2, int LD) {
  const int cb = 8 * (wid >> 2);
  const uint32_t la = acc + ((uint32_t)((wid & 3) * 32) << 16);
  uint32_t r[8][8];
#pragma unroll
  for (int g = 0; g < 8; ++g) tmem_ld8_nowait(la + 32 * g + cb, r[g]);
  tmem_wait_ld();
  if (row >= rows) return;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const long long hi = tc_group4(__uint_as_float(r[0][j]), __uint_as_float(r[1][j]),
                                   __uint_as_float(r[2][j]), __uint_as_float(r[3][j]));
    const long long lo = tc_group4(__uint_as_float(r[4][j]), __uint_as_float(r[5][j]),
                                   __uint_as_float(r[6][j]), __uint_as_float(r[7][j]));
    const int E = ew[cb + j];
    const double v = E == 0x7ff || er >= TC_NONFINITE / 2
                         ? __longlong_as_double(0x7ff8000000000000ll)
                         : split_times_pow2(hi + (lo >> 32), (unsigned int)(lo & 0xFFFFFFFFll),
                                            tc_exponent(E) + er - 72);
    a2[(cb + j) * LD + row] -= v;
  }
}

struct QrTc {
  QrpArgs q;
  int np, nkb, nmt, b0;      // panels, 32-row blocks, 128-row tiles, instance of slot 0
  int sets;                  // digit sets: 2 with row scales
  int nc;                    // columns of W^T (the solver: N + right-hand sides)
  unsigned char* ws;         // per slot: see the pointers below
  long long slot_bytes;
  __host__ __device__ long long set_bytes() const {
    return (long long)np * (nkb * VT_TILE + nmt * V_TILE + NB * NB * 8 + 2 * NB * 4 + 32 * nkb * 4);
  }
  __host__ __device__ unsigned char* slot(int z) const { return ws + (long long)z * slot_bytes; }
  __host__ __device__ unsigned char* vt(int z, int p, int set) const {   // V^T tiles of panel p
    return slot(z) + set * set_bytes() + (long long)p * nkb * VT_TILE;
  }
  __host__ __device__ unsigned char* v(int z, int p, int set) const {    // V tiles of panel p
    return vt(z, np, set) + (long long)p * nmt * V_TILE;
  }
  __host__ __device__ double* T(int z, int p, int set) const {
    return reinterpret_cast<double*>(v(z, np, set)) + p * (NB * NB);
  }
  // exponents: f_j of V^T's rows (in the first set the scales of its vectors), in the
  // second set also e_r of V's rows and h_j of its columns
  __host__ __device__ int* f(int z, int p, int set) const {
    return reinterpret_cast<int*>(T(z, np, set)) + p * NB;
  }
  __host__ __device__ int* er(int z, int p, int set) const {
    return f(z, np, set) + p * 32 * nkb;
  }
  __host__ __device__ int* h(int z, int p, int set) const { return er(z, np, set) + p * NB; }
  // the column scales, kept here because D may be written over Din
  __host__ __device__ double* din(int z) const {
    return reinterpret_cast<double*>(slot(z) + sets * set_bytes());
  }
  __host__ __device__ float* lnrm(int z) const { return reinterpret_cast<float*>(din(z) + 32 * nkb); }
  __host__ __device__ int* rem(int z, int which) const {        // remaining columns, ping-pong
    return reinterpret_cast<int*>(lnrm(z) + 32 * nkb) + which * 32 * nkb;
  }
  // the solver: digits of R (128-row tiles x 32 columns, as V) and their row exponents
  __host__ __device__ unsigned char* r(int z) const { return slot(z) + set_bytes(); }
  __host__ __device__ long long r_bytes() const { return (long long)nmt * nkb * V_TILE; }
  __host__ __device__ int* r_exp(int z) const { return reinterpret_cast<int*>(r(z) + r_bytes()); }
};

void qr_geometry(QrTc& a, int N, int row_graded) {
  a.np = a.nkb = (N + NB - 1) / NB;
  a.nmt = (N + 127) / 128;
  a.sets = row_graded ? 2 : 1;
  a.nc = N;
  a.slot_bytes = (a.sets * a.set_bytes() + 5LL * 32 * a.nkb * 4 + 1023) & ~1023LL;
}

// The solver's slot: one digit set, R's digits and exponents.
void solve_geometry(QrTc& a, int N, int nrhs) {
  qr_geometry(a, N, 0);
  a.nc = N + nrhs;
  a.slot_bytes = (a.set_bytes() + a.r_bytes() + 128LL * a.nmt * 4 + 1023) & ~1023LL;
}

__device__ __forceinline__ bool qr_skip(const QrTc& a, int b) {
  return a.q.lim && a.q.lim[b] < a.q.lim_at;   // chain of this instance already finished
}

}  // namespace

// ---- W^T and norms -----------------------------------------------------------
__global__ void __launch_bounds__(256) qr_init_kernel(const QrTc a) {
  extern __shared__ double qi_tile[];   // 32 columns x LD
  const int z = blockIdx.y, b = a.b0 + z, N = a.q.N, LD = 32 * a.nkb + 1;
  if (qr_skip(a, b)) return;
  if (!DQMC_CHECK(blockDim.x == 256 && dyn_smem_bytes() >= 32u * LD * 8u, LD)) return;
  const int c0 = blockIdx.x * 32, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const double* A = a.q.A + (long long)b * a.q.sA;
  const int c = c0 + lane;
  for (int r0 = wid; r0 < N; r0 += 64) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      v[u] = r0 + 8 * u < N && c < N ? A[(long long)(r0 + 8 * u) * N + c] : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (r0 + 8 * u < N) qi_tile[lane * LD + r0 + 8 * u] = v[u];
  }
  __syncthreads();
  double* W = a.q.W + (long long)b * a.q.sW;
  const double* Din = a.q.Din ? a.q.Din + (long long)b * a.q.sDin : nullptr;
  bool bad = false;
  for (int u = 0; u < 4; ++u) {
    const int cc = wid + 8 * u, col = c0 + cc;
    if (col >= N) break;
    const float ln = warp_log2_norm(qi_tile + cc * LD, 0, N, bad);
    for (int r = lane; r < N; r += 32) W[(long long)col * N + r] = qi_tile[cc * LD + r];
    if (lane == 0) {
      a.lnrm(z)[col] = ln;
      a.rem(z, 0)[col] = col;
      const double d = Din ? Din[col] : 1.0;
      a.din(z)[col] = d;
      bad |= !(isfinite(d) && d >= 0.0);
    }
  }
  if (lane == 0 && bad && a.q.status)
    atomicOr(&a.q.status[b / a.q.status_div], DQMC_STATUS_NONFINITE_SCALE);
}

// ---- panel ---------------------------------------------------------------------
// QP_BIG (N > 256): 64 instead of 128 candidates of the pivot search.  QP_SMALL (N <=
// 64, many instances): two CTAs an SM (64 registers a thread, 112 KB), as the chain of
// a step leaves an SM's FP64 pipe idle for two thirds of its 3 to 4 thousand cycles;
// the same arithmetic.  QP_MID otherwise.
// PIV: with the pivot search; otherwise the columns in their order (the solver).
template <int SIZE, bool PIV>
__global__ void __launch_bounds__(512, SIZE == QP_SMALL ? 2 : 1) qr_panel_kernel(const QrTc a, int p) {
  constexpr int CN = SIZE == QP_BIG ? 64 : 128;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int z = blockIdx.x, b = a.b0 + z, N = a.q.N;
  if (qr_skip(a, b)) return;
  const int j0 = NB * p, m = N - j0, nb = m < NB ? m : NB;     // m rows and columns remain
  const int nkl = a.nkb - p, LDU = 32 * nkl + 1;
  double* us = reinterpret_cast<double*>(base + RING);         // [32][LDU]
  double* gm = us + NB * LDU;                                  // V^T V
  double* tm = gm + NB * TLD;                                  // T
  double* xs = tm + NB * TLD;                                  // [2][XS]
  double* s_beta = xs + 2 * xs_rows(SIZE == QP_SMALL);
  double* s_gam = s_beta + NB;
  double* s_uj = s_gam + NB;
  float* qf = reinterpret_cast<float*>(s_uj + NB);             // [3][2][row groups][68 or 52]
  float* s_inv = qf + 3 * QF;                                      // [2]
  float* s_key = s_inv + 2;                                    // [m]
  int* s_rem = reinterpret_cast<int*>(s_key + N);              // [m]
  int* s_cand = s_rem + N;                                     // [CN] positions in rem
  int* s_sel = s_cand + CN;                                    // [32] candidate numbers
  int* s_ex = s_sel + NB;                                      // [32] exponents of gamma's vectors
  int* s_unit = s_ex + NB;                                     // [32] columns with leading entry one
  int* s_f0 = s_unit + NB;                                       // [32] the first set's s_f
  int* s_f = s_f0 + NB;                                        // [32] exponents of V^T's rows
  int* s_h = s_f + NB;                                         // [32] of V's columns times 2^{-rho_r}
  int* s_rho = s_h + NB;                                       // [32 nkl]
  int* s_er = s_rho + 32 * nkl;                                // [32 nkl] exponents of V's rows
  unsigned* s_max = reinterpret_cast<unsigned*>(s_er + 32 * nkl);    // [2][16]
  uint64_t* bar = reinterpret_cast<uint64_t*>(
      (reinterpret_cast<uintptr_t>(s_max + 32) + 7) & ~(uintptr_t)7);
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bar + 1);
  int* s_fail = reinterpret_cast<int*>(tmem_holder + 1);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (!DQMC_CHECK(blockDim.x == 512 && N <= (SIZE == QP_BIG ? QRTC_MAX_N : (SIZE == QP_SMALL ? 64 : 256)), N) ||
      !DQMC_CHECK(dyn_smem_bytes() >=
                      (unsigned)(reinterpret_cast<unsigned char*>(s_fail + 1) - smem_raw), m))
    return;
  double* W = a.q.W + (long long)b * a.q.sW;
  const double* Din = a.din(z);
  int* perm = PIV ? a.q.perm + (long long)b * a.q.sperm : nullptr;

  if (tid == 0) {
    mbar_init(bar, 1);
    *s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (wid == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_holder)),
                 "r"(256u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // ---- candidates: the CN remaining columns of largest key (ties: lowest place)
  const double* Drow = a.q.Drow ? a.q.Drow + (long long)b * a.q.sDrow : nullptr;
  if (tid < 32 * nkl) s_rho[tid] = row_rho(Drow, j0 + tid, N);
  if (tid < NB) s_ex[tid] = 0;
  if (!PIV && tid < NB) {
    s_rem[tid] = j0 + tid;
    s_sel[tid] = tid;
  }
  if (PIV && tid < m) {
    const int col = a.rem(z, p & 1)[tid];
    const float k = log2_wide_f(Din[col]) + a.lnrm(z)[col];
    s_rem[tid] = col;
    s_key[tid] = k == k ? k : -INFINITY;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_holder;
  if (PIV && tid < m) {
    const float k = s_key[tid];
    int rank = 0;
    for (int u = 0; u < m; ++u) rank += s_key[u] > k || (s_key[u] == k && u < tid);
    if (rank < CN) s_cand[rank] = tid;
  }
  __syncthreads();
  // ---- FP32 pivoted reduction of the candidates: nb pivots -------------------------
  if constexpr (PIV) {
    // rows per thread rounded up: straight-line loops
#define DQMC_SEARCH(TPC_, KM_)                                                                 \
  do {                                                                                         \
    if (Drow)                                                                                  \
      pivot_search<TPC_, KM_, true, SIZE == QP_SMALL>(W, Din, a.lnrm(z), s_rem, s_cand, N, j0, m, nb, qf, s_inv, \
                                    s_max, s_sel, s_rho);                                      \
    else                                                                                       \
      pivot_search<TPC_, KM_, false, SIZE == QP_SMALL>(W, Din, a.lnrm(z), s_rem, s_cand, N, j0, m, nb, qf, s_inv, \
                                     s_max, s_sel, s_rho);                                     \
  } while (0)
    if constexpr (SIZE == QP_SMALL) {
      if (m <= 32) DQMC_SEARCH(4, 8);
      else DQMC_SEARCH(4, 16);
    } else if constexpr (SIZE == QP_BIG) {
      if (m <= 64) DQMC_SEARCH(8, 8);
      else if (m <= 128) DQMC_SEARCH(8, 16);
      else if (m <= 256) DQMC_SEARCH(8, 32);
      else DQMC_SEARCH(8, 48);
    } else {
      if (m <= 32) DQMC_SEARCH(4, 8);
      else if (m <= 64) DQMC_SEARCH(4, 16);
      else if (m <= 128) DQMC_SEARCH(4, 32);
      else if (m <= 192) DQMC_SEARCH(4, 48);
      else DQMC_SEARCH(4, 64);
    }
#undef DQMC_SEARCH
  }
  __syncthreads();
  // ---- pivot order and the columns that remain (their order kept) ------------------
  if (PIV && tid < nb) {
    const int pos = s_cand[s_sel[tid]];
    perm[j0 + tid] = s_rem[pos];
    s_sel[tid] = pos;
  }
  __syncthreads();
  if (PIV && tid < m) {
    int before = 0;
    bool taken = false;
    for (int s = 0; s < nb; ++s) {
      before += s_sel[s] < tid;
      taken |= s_sel[s] == tid;
    }
    if (!taken) a.rem(z, (p + 1) & 1)[tid - before] = s_rem[tid];
  }
  // ---- FP64 Householder panel (rows per lane rounded up: straight-line loops, as a
  // predicated FP64 instruction holds the pipe like any other) ---------------------
#define DQMC_FACTOR(LPC_, KR_)                                                                    \
  do {                                                                                            \
    bool redo = false;                                                                            \
    if (wid < LPC_)                                                                               \
      redo = panel_factor<LPC_, KR_, SIZE == QP_SMALL, false>(W, s_rem, s_sel, N, j0, m, nb, LDU, \
                                                              out, s_beta, s_gam, s_uj, s_ex, s_unit); \
    if (redo) {                             /* (alike in these warps) */                          \
      asm volatile("bar.sync 1, %0;" ::"n"(32 * LPC_) : "memory");                                \
      panel_factor<LPC_, KR_, SIZE == QP_SMALL, true>(W, s_rem, s_sel, N, j0, m, nb, LDU, out,    \
                                                      s_beta, s_gam, s_uj, s_ex, s_unit);         \
    }                                                                                             \
  } while (0)
  {
    double* out[2] = {us, xs};
    if constexpr (SIZE == QP_SMALL) {
      if (m <= 32) DQMC_FACTOR(8, 4);
      else DQMC_FACTOR(8, 8);
    } else {
      if (m <= 32) DQMC_FACTOR(8, 4);
      else if (m <= 64) DQMC_FACTOR(8, 8);
      else if (m <= 128) DQMC_FACTOR(16, 8);
      else if (m <= 192) DQMC_FACTOR(16, 12);
      else if (m <= 256) DQMC_FACTOR(16, 16);
      else DQMC_FACTOR(16, 24);
    }
  }
#undef DQMC_FACTOR
  __syncthreads();
  uint32_t nm = 0;                          // MMA groups waited for
  for (int set = 0; set < a.sets; ++set) {
    // ---- exponents: first set of the columns alone, second set with the row scales and
    // of the rows ---------------------------------------------------------------------
    if (tid < 32 * nkl) s_rho[tid] = set ? row_rho(Drow, j0 + tid, N) : 0;
    __syncthreads();
    {
      const int c = tid >> 4, l = tid & 15;
      int mf = 0, mh = -100000;
      bool bad = false;
      for (int r = l; r < 32 * nkl; r += 16) {
        const int E = (int)((__double_as_longlong(us[c * LDU + r]) >> 52) & 0x7ff);
        if (E == 0) continue;
        bad |= E == 0x7ff;
        mf = max(mf, E + s_rho[r] + 100000);
        mh = max(mh, E - s_rho[r]);
      }
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
        mf = max(mf, __shfl_xor_sync(0xffffffffu, mf, o));
        mh = max(mh, __shfl_xor_sync(0xffffffffu, mh, o));
        bad |= __shfl_xor_sync(0xffffffffu, (int)bad, o) != 0;
      }
      if (l == 0) {
        s_f[c] = bad ? TC_NONFINITE : (mf == 0 ? 0 : mf - 100000 - 1020);
        s_h[c] = bad ? TC_NONFINITE : (mf == 0 ? 0 : mh - 1020);
        if (!set) s_f0[c] = s_f[c];
        a.f(z, p, set)[c] = s_f[c];
        if (set) a.h(z, p, 1)[c] = s_h[c];
      }
    }
    __syncthreads();
    if (set && tid < 32 * nkl) {            // (NaN and inf come in with f_j)
      int mx = 0;
      for (int c = 0; c < NB; ++c) {
        const int E = (int)((__double_as_longlong(us[c * LDU + tid]) >> 52) & 0x7ff);
        if (E != 0 && E != 0x7ff && s_h[c] < TC_NONFINITE / 2) mx = max(mx, E - s_h[c] + 100000);
      }
      s_er[tid] = mx == 0 ? 0 : mx - 100000 - 1020;
      a.er(z, p, 1)[j0 + tid] = s_er[tid];
    }
    if (set) __syncthreads();
    // ---- digits of V^T (to the tiles and the staging ring) and V^T V: four 32-row
    // blocks at a time, in the second set two with their own left operands ------------
    {
      bool first = true;
      unsigned char* gvt = a.vt(z, p, set) + (long long)p * VT_TILE;
      const int slot = tid >> 7, c = (tid >> 2) & 31, ch = tid & 3;
      const int side = set ? slot >> 1 : 0, kq = set ? slot & 1 : slot, per = set ? 2 : 4;
      for (int kb = 0; kb < nkl; kb += per) {
        if (kb > 0) wait_or_fail(bar, nm++ & 1, s_fail);
        if (kb + kq < nkl) {
          const int r0 = 32 * (kb + kq) + 8 * ch;
          const double* uc = us + c * LDU + r0;
          unsigned char* gt = gvt + (long long)(kb + kq) * VT_TILE;
          unsigned char* st = base + slot * VT_TILE + swz(c, ch);
          const int e0 = side ? s_h[c] : s_f[c], sg = side ? 1 : -1;
          tc_digits<8>([&](int k) { return e0 + sg * s_rho[r0 + k]; }, [&](int k) { return uc[k]; },
                       [&](int q, const uint32_t (&w)[4]) {
                         const uint4 v = make_uint4(w[0], w[1], w[2], w[3]);
                         *reinterpret_cast<uint4*>(st + q * DT) = v;
                         if (side == 0) *reinterpret_cast<uint4*>(gt + q * DT + swz(c, ch)) = v;
                       });
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          for (int q = 0; q < per && kb + q < nkl; ++q) {
            // G_ij, i < j, sums rows r >= j: in the second set u_ri 2^{-rho_r} (of order
            // one) goes left and u_rj 2^{rho_r} (largest at r = j) right
            mma_stacked(tmem, smem_u32(base + (q + (set ? 2 : 0)) * VT_TILE), smem_u32(base + q * VT_TILE), first);
            first = false;
          }
          umma_commit(bar);
        }
      }
    }
    // digits of V (128-row tiles from the one that holds row j0) meanwhile
    for (int t = j0 / 128; t < a.nmt; ++t) {
      unsigned char* gv = a.v(z, p, set) + (long long)t * V_TILE;
      const int rr = tid >> 2, ch = tid & 3, r = 128 * t + rr - j0;
      const int er = set && r >= 0 && r < m ? s_er[r] : 0;
      tc_digits<8>([&](int k) { return set ? er + s_h[8 * ch + k] : s_f[8 * ch + k]; },
                   [&](int k) { return r >= 0 && r < m ? us[(8 * ch + k) * LDU + r] : 0.0; },
                   [&](int q, const uint32_t (&w)[4]) {
                     *reinterpret_cast<uint4*>(gv + q * (128 * 64) + swz(rr, ch)) =
                         make_uint4(w[0], w[1], w[2], w[3]);
                   });
    }
    wait_or_fail(bar, nm++ & 1, s_fail);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    __syncthreads();
    long long* ex = reinterpret_cast<long long*>(base);
    if (wid < 8)
      for (int c0 = 16 * (wid >> 2); c0 < 16 * (wid >> 2) + 16; c0 += 8) stacked_partial(tmem, wid, c0, ex);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    // V^T V of the vectors the first set holds, u_j 2^{-f_j} (in that set exponent 0), in
    // the second one too: entries and T's stay of order one whatever the columns' scales
    for (int e = tid; e < NB * NB; e += 512) {
      const int i = e & 31, c = e >> 5;
      gm[i * TLD + c] = stacked_value(ex, i, c, set ? s_h[i] + s_f[c] - s_f0[i] - s_f0[c] : 0);
    }
    double* s_g = xs;                       // (xs is free) gamma of u_j 2^{-f_j}, tau_j of v_j 2^{E_j - f_j}
    if (!set && tid < NB) {
      double g = tid < nb && s_f[tid] < TC_NONFINITE / 2 ? s_gam[tid] : 0.0;
      int e = s_ex[tid];
      if (g > 0.0 && s_unit[tid]) {         // tau_j = -u_jj / beta_j, a quotient in (1, 2]
        const double b1 = fabs(s_beta[tid]), zb = recip_newton(b1), n = fabs(s_uj[tid]), q = n * zb;
        g = fma(fma(-q, b1, n), zb, q);
        e = (int)((__double_as_longlong(us[tid * LDU + tid]) >> 52) & 0x7ff) - 1023;
      }
      s_g[tid] = scalbn(g, 2 * (s_f[tid] - e));
    }
    for (int e = tid; e < NB * TLD; e += 512) tm[e] = 0.0;
    __syncthreads();
    // ---- T: T_jj = gamma_j, T(:j, j) = -gamma_j T(:j,:j) G(:j, j); 8 x 8 blocks by one
    // warp each, then T12 = -T11 (G12 T22) twice ---------------------------------------
    if (wid < 4 && lane < 8) {
      const int o = 8 * wid;
      const unsigned M8 = 0xffu;
      for (int j = 0; j < 8; ++j) {
        const double gj = s_g[o + j];
        double s = 0.0;
        for (int l = 0; l < j; ++l) s = fma(tm[(o + lane) * TLD + o + l], gm[(o + l) * TLD + o + j], s);
        if (lane <= j) tm[(o + lane) * TLD + o + j] = lane == j ? gj : -gj * s;
        __syncwarp(M8);
      }
    }
    __syncthreads();
    double* tx = reinterpret_cast<double*>(base);   // G12 T22 (the exchange memory is free)
    for (int w = 8; w <= 16; w <<= 1) {
      const int nblk = NB / (2 * w), per = w * w;
      const int bl = tid / per, i = (tid % per) / w, j = tid % w;
      const int o = 2 * w * bl;
      if (bl < nblk) {
        // T22 and T11 are zero below their diagonals: whole rows, four chains
        double s[4] = {0.0, 0.0, 0.0, 0.0};
        for (int l = 0; l < w; l += 4)
#pragma unroll
          for (int t = 0; t < 4; ++t)
            s[t] = fma(gm[(o + i) * TLD + o + w + l + t], tm[(o + w + l + t) * TLD + o + w + j], s[t]);
        tx[bl * per + i * w + j] = (s[0] + s[1]) + (s[2] + s[3]);
      }
      __syncthreads();
      if (bl < nblk) {
        double s[4] = {0.0, 0.0, 0.0, 0.0};
        for (int l = 0; l < w; l += 4)
#pragma unroll
          for (int t = 0; t < 4; ++t)
            s[t] = fma(tm[(o + i) * TLD + o + l + t], tx[bl * per + (l + t) * w + j], s[t]);
        tm[(o + i) * TLD + o + w + j] = -((s[0] + s[1]) + (s[2] + s[3]));
      }
      __syncthreads();
    }
    for (int e = tid; e < NB * NB; e += 512) a.T(z, p, set)[e] = tm[(e >> 5) * TLD + (e & 31)];
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
  }
  if (tid == 0 && *(volatile int*)s_fail && a.q.status)
    atomicOr(&a.q.status[b / a.q.status_div], DQMC_STATUS_TIMEOUT);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (wid == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u)
                 : "memory");
  }
}

// ---- block reflectors on 32 columns --------------------------------------------
// APPLY_REM: the remaining columns 32 blockIdx.x .. of rem after panel p get
// (1 - V T V^T)^T; APPLY_NEXT (the solver): the columns right of panel p in W^T;
// APPLY_Q: columns 32 blockIdx.x .. of Q, all panels backwards.
enum { APPLY_REM, APPLY_NEXT, APPLY_Q };
template <int MODE>
__global__ void __launch_bounds__(512, 1) qr_apply_kernel(const QrTc a, int p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int z = blockIdx.y, b = a.b0 + z, N = a.q.N;
  if (qr_skip(a, b)) return;
  const int LD = 32 * a.nkb + 1;
  unsigned char* wz = base + RING;                              // 3 zero tiles, 8 digits of W
  double* a2 = reinterpret_cast<double*>(wz + 11 * DT);         // [32][LD]
  double* w1 = a2 + 32 * LD;                                    // V^T A
  double* w2 = w1 + NB * TLD;                                   // T^T V^T A
  double* tt = w2 + NB * TLD;
  int* ecol = reinterpret_cast<int*>(tt + NB * TLD);            // [32]
  int* ew = ecol + 32;
  int* s_f = ew + 32;                                           // [32]
  int* s_f0 = s_f + 32;                                         // [32]
  double* s_dn = reinterpret_cast<double*>(s_f0 + 32);          // [32] 2^{h - f0}
  int* s_rho = reinterpret_cast<int*>(s_dn + 32);               // [32 nkb]
  int* s_er = s_rho + 32 * a.nkb;                               // [32 nkb]
  uint64_t* full = reinterpret_cast<uint64_t*>(s_er + 32 * a.nkb);
  uint64_t* done = full + 1;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(done + 1);
  int* s_fail = reinterpret_cast<int*>(tmem_holder + 1);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (!DQMC_CHECK(blockDim.x == 512 && a.nkb <= 12, a.nkb) ||
      !DQMC_CHECK(dyn_smem_bytes() >=
                      (unsigned)(reinterpret_cast<unsigned char*>(s_fail + 1) - smem_raw), LD))
    return;
  double* W = a.q.W + (long long)b * a.q.sW;
  constexpr bool FORMQ = MODE == APPLY_Q;
  const int j0 = NB * p, c0 = 32 * blockIdx.x;
  const int next = j0 + NB < N ? j0 + NB : N;   // first column right of the panel
  const int left = (FORMQ ? N : (MODE == APPLY_REM ? N : a.nc) - next) - c0;
  const int ncols = left < 32 ? left : 32;
  const int* rem = MODE == APPLY_REM ? a.rem(z, (p + 1) & 1) + c0 : nullptr;
  auto column = [&](int c) { return MODE == APPLY_REM ? rem[c] : next + c0 + c; };

  if (tid == 0) {
    mbar_init(full, 1);
    mbar_init(done, 1);
    *s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (wid == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_holder)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  for (int i = tid; i < 3 * DT / 16; i += 512) reinterpret_cast<uint4*>(wz)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int u = 0; u < 2; ++u) {             // a warp per column, four loads in flight
    const int c = wid + 16 * u;
    double* dst = a2 + c * LD;
    const double* src = W + (long long)(!FORMQ && c < ncols ? column(c) : 0) * N;
    for (int r0 = lane; r0 < 32 * a.nkb; r0 += 128) {
      double v[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int r = r0 + 32 * t;
        if (FORMQ) v[t] = r == c0 + c && r < N ? 1.0 : 0.0;
        else v[t] = c < ncols && r < N && r >= j0 ? src[r] : 0.0;
      }
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (r0 + 32 * t < 32 * a.nkb) dst[r0 + 32 * t] = v[t];
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_holder;
  uint32_t nfull = 0, ndone = 0;            // phases waited for (uniform over the CTA)
  long long* ex = reinterpret_cast<long long*>(base);

  const int p_first = FORMQ ? (int)blockIdx.x : p, p_last = FORMQ ? 0 : p;
  const int set = FORMQ ? 0 : a.sets - 1;   // the second set has row exponents
  const double* Drow = a.q.Drow ? a.q.Drow + (long long)b * a.q.sDrow : nullptr;
  for (int pp = p_first; pp >= p_last; --pp) {
    for (int e = tid; e < NB * NB; e += 512) tt[(e >> 5) * TLD + (e & 31)] = a.T(z, pp, set)[e];
    if (tid < 32) {
      ew[tid] = 0;
      s_f[tid] = set ? a.f(z, pp, 1)[tid] : 0;
      s_f0[tid] = set ? a.f(z, pp, 0)[tid] : 0;
      s_dn[tid] = set ? scalbn(1.0, a.h(z, pp, 1)[tid] - s_f0[tid]) : 1.0;
    }
    for (int r = tid; r < 32 * a.nkb; r += 512) {
      s_rho[r] = set ? row_rho(Drow, r, N) : 0;
      s_er[r] = set && r >= 32 * pp ? a.er(z, pp, 1)[r] : 0;
    }
    __syncthreads();
    for (int u = 0; u < 2; ++u) {           // exponents of the columns over rows >= 32 pp
      const int c = wid + 16 * u;
      int mx = -100000;
      bool bad = false;
      for (int r = 32 * pp + lane; r < 32 * a.nkb; r += 32) {
        const int E = (int)((__double_as_longlong(a2[c * LD + r]) >> 52) & 0x7ff);
        bad |= E == 0x7ff;
        if (E != 0) mx = max(mx, E - s_rho[r]);
      }
      mx = __reduce_max_sync(0xffffffffu, mx);
      bad = __any_sync(0xffffffffu, bad);
      if (lane == 0) ecol[c] = bad ? TC_NONFINITE : (mx == -100000 ? 0 : mx - 1020);
    }
    __syncthreads();
    // ---- W1 = V^T A, two 32-row blocks at a time --------------------------------
    const unsigned char* gvt = a.vt(z, pp, set);
    for (int kb = pp; kb < a.nkb; kb += 2) {
      const int ng = a.nkb - kb < 2 ? 1 : 2;
      if (kb > pp) { wait_or_fail(done, ndone & 1, s_fail); ++ndone; }
      if (tid == 0) {
        mbar_arrive_expect_tx(full, (uint32_t)(ng * VT_TILE));
        bulk_load(base, gvt + (long long)kb * VT_TILE, (uint32_t)(ng * VT_TILE), full);
      }
      const int kq = tid >> 8, c = (tid >> 3) & 31, ch = (tid >> 1) & 3, hf = tid & 1;
      if (kq < ng) {                        // four rows of one column per thread
        const int r0 = 32 * (kb + kq) + 8 * ch + 4 * hf, ec = ecol[c];
        const double* ac = a2 + c * LD + r0;
        unsigned char* dst = base + (2 + kq) * VT_TILE + swz(c, ch) + 8 * hf;
        tc_digits<4>([&](int k) { return ec + s_rho[r0 + k]; }, [&](int k) { return ac[k]; },
                     [&](int q, const uint32_t (&w)[2]) {
                       *reinterpret_cast<uint2*>(dst + q * DT) = make_uint2(w[0], w[1]);
                     });
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
      if (tid == 0) {
        wait_or_fail(full, nfull & 1, s_fail);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        for (int q = 0; q < ng; ++q)
          mma_stacked(tmem, smem_u32(base + q * VT_TILE), smem_u32(base + (2 + q) * VT_TILE),
                      kb == pp && q == 0);
        umma_commit(done);
      }
      ++nfull;
    }
    wait_or_fail(done, ndone & 1, s_fail);
    ++ndone;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    __syncthreads();
    stacked_partial(tmem, wid, 8 * (wid >> 2), ex);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    for (int e = tid; e < NB * NB; e += 512) {
      const int i = e & 31, c = e >> 5, ec = ecol[c] + s_f[i];
      w1[i * TLD + c] = ec >= TC_NONFINITE / 2 ? __longlong_as_double(0x7ff8000000000000ll)
                                           : stacked_value(ex, i, c, ec - s_f0[i]);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    // ---- W2 = T^T W1 (T W1 for Q); the first V tile is on its way -------------------
    int t = 32 * pp / 128;
    const unsigned char* gv = a.v(z, pp, set);
    if (tid == 0) {
      mbar_arrive_expect_tx(full, V_TILE);
      bulk_load(base, gv + (long long)t * V_TILE, V_TILE, full);
    }
    {
      // rows w and 31 - w of warp w: the triangle's lengths even out
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int i = u ? 31 - wid : wid;
        double s0 = 0.0, s1 = 0.0;
        if (FORMQ) {
          int l = i;
          for (; l + 1 < NB; l += 2) {
            s0 = fma(tt[i * TLD + l], w1[l * TLD + lane], s0);
            s1 = fma(tt[i * TLD + l + 1], w1[(l + 1) * TLD + lane], s1);
          }
          if (l < NB) s0 = fma(tt[i * TLD + l], w1[l * TLD + lane], s0);
        } else {
          int l = 0;
          for (; l + 1 <= i; l += 2) {
            s0 = fma(tt[l * TLD + i], w1[l * TLD + lane], s0);
            s1 = fma(tt[(l + 1) * TLD + i], w1[(l + 1) * TLD + lane], s1);
          }
          if (l <= i) s0 = fma(tt[l * TLD + i], w1[l * TLD + lane], s0);
        }
        double s = s0 + s1;
        if (set) s *= s_dn[i];               // V's digits are those of u_i 2^{-h_i}
        w2[i * TLD + lane] = s;
        atomicMax(&ew[lane], (int)((__double_as_longlong(s) >> 52) & 0x7ff));
      }
    }
    __syncthreads();
    if (tid < 256) {
      const int c = tid >> 3, ch = (tid >> 1) & 3, hf = tid & 1;
      unsigned char* dst = wz + 3 * DT + swz(c, ch) + 8 * hf;
      tc_digits4(tc_exponent(ew[c]), [&](int k) { return w2[(8 * ch + 4 * hf + k) * TLD + c]; },
                 [&](int q, uint2 w) { *reinterpret_cast<uint2*>(dst + q * DT) = w; });
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    // ---- A -= V W2, 128 rows at a time ------------------------------------------------
    for (; t < a.nmt; ++t) {
      const uint32_t acc = tmem + 256u * (uint32_t)(t & 1);
      if (tid == 0) {
        wait_or_fail(full, nfull & 1, s_fail);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        mma_rows(acc, smem_u32(base), smem_u32(wz));
        umma_commit(done);
      }
      ++nfull;
      wait_or_fail(done, ndone & 1, s_fail);
      ++ndone;
      if (tid == 0 && t + 1 < a.nmt) {
        mbar_arrive_expect_tx(full, V_TILE);
        bulk_load(base, gv + (long long)(t + 1) * V_TILE, V_TILE, full);
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int row = 128 * t + (wid & 3) * 32 + lane;
      rows_subtract(acc, wid, row, 32 * a.nkb, row < 32 * a.nkb ? s_er[row] : 0, ew, a2, LD);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
    }
  }
  // ---- results --------------------------------------------------------------------
  if (FORMQ) {
    double* U = a.q.U + (long long)b * a.q.sU;
    for (int r = wid; r < N; r += 16)
      if (lane < ncols) U[(long long)r * N + c0 + lane] = a2[lane * LD + r];
  } else {
    bool bad = false;
    for (int u = 0; u < 2; ++u) {
      const int c = wid + 16 * u;
      if (c >= ncols) break;
      const int col = column(c);
      for (int r = j0 + lane; r < N; r += 32) W[(long long)col * N + r] = a2[c * LD + r];
      if (MODE == APPLY_REM) {
        const float ln = warp_log2_norm(a2 + c * LD, j0 + NB, N, bad);
        if (lane == 0) a.lnrm(z)[col] = ln;
      }
    }
    if (lane == 0 && bad && a.q.status)
      atomicOr(&a.q.status[b / a.q.status_div], DQMC_STATUS_NONFINITE_SCALE);
  }
  if (*(volatile int*)s_fail && tid == 0) {
    // a copy still in flight lands before the CTA exits (bounded)
    mbar_wait(full, nfull & 1);
    if (a.q.status) atomicOr(&a.q.status[b / a.q.status_div], DQMC_STATUS_TIMEOUT);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (wid == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
}

// ---- D, T = D^{-1} R in pivot order -----------------------------------------------
// One CTA per 32 columns of T of one instance: columns read along W^T, written
// as rows through a shared tile.
__global__ void __launch_bounds__(256) qr_out_kernel(const QrTc a) {
  __shared__ double tile[32][33];
  __shared__ double s_d[32], s_i[32];
  const int z = blockIdx.y, b = a.b0 + z, N = a.q.N;
  if (qr_skip(a, b)) return;
  const double* W = a.q.W + (long long)b * a.q.sW;
  const double* Din = a.din(z);
  const int* perm = a.q.perm + (long long)b * a.q.sperm;
  double* T = a.q.T + (long long)b * a.q.sT;
  const int c0 = blockIdx.x * 32, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid < 32 && c0 + tid < N) {
    const int c = c0 + tid, col = perm[c];
    s_d[tid] = Din[col];
    const double d = fabs(W[(long long)col * N + c]) * s_d[tid];
    int flag = 0;
    if (!(d > 0.0)) flag |= DQMC_STATUS_SINGULAR;
    if (!isfinite(d)) flag |= DQMC_STATUS_NONFINITE_SCALE;
    a.q.D[(long long)b * a.q.sD + c] = d;
    if (flag && a.q.status) atomicOr(&a.q.status[b / a.q.status_div], flag);
  }
  __syncthreads();
  for (int r0 = 0; r0 < N; r0 += 32) {
    const bool any = r0 <= c0 + 31;         // rows at or above some diagonal entry
    if (any && tid < 32 && r0 + tid < N) {
      const int i = r0 + tid, col = perm[i];
      const double rii = fabs(W[(long long)col * N + i]), d = Din[col];
      // two factors, as |r_ii| and D_i each may be far from one
      s_i[tid] = rii > 0.0 ? 1.0 / rii : 0.0;
      tile[tid][32] = d > 0.0 ? 1.0 / d : 0.0;
    }
    __syncthreads();
    if (any)
      for (int u = wid; u < 32; u += 8) {
        const int c = c0 + u, i = r0 + lane;
        double v = 0.0;
        if (c < N && i <= c)
          v = W[(long long)perm[c] * N + i] * s_i[lane] * (s_d[u] * tile[lane][32]);
        tile[lane][u] = v;
      }
    __syncthreads();
    for (int u = wid; u < 32; u += 8) {
      const int i = r0 + u;
      if (i < N && c0 + lane < N) T[(long long)i * N + c0 + lane] = any ? tile[u][lane] : 0.0;
    }
    __syncthreads();
  }
}

namespace {
size_t apply_smem(int nkb) {
  return 1024 + RING + 11 * DT + (size_t)32 * (32 * nkb + 1) * 8 + 3 * NB * TLD * 8 + 64 * nkb * 4 + 896;
}
size_t panel_smem(int N, int nkb, bool small = false) {
  return 1024 + RING + ((size_t)NB * (32 * nkb + 1) + 2 * NB * TLD + 2 * xs_rows(small) + 3 * NB) * 8 +
         (3 * QF + 2 + 2 * N + 128 + 6 * NB + 64 * nkb + 32) * 4 + 64;
}
}  // namespace

// ===========================================================================
// Solver: opA(A) Z = opR(R) by the same panels and reflectors without pivoting
// (Householder QR of [A | R], stable as it is), then blocked back substitution.
// Takes the place of lu_kernel (one CTA per instance on its SM's FP64 pipe)
// where that is the slower one.  det A = (-1)^{reflectors} prod r_ii.
// ===========================================================================
// [opA(A) | opR(R)] by columns into W^T; one CTA per 32 columns of one instance
__global__ void __launch_bounds__(256) solve_init_kernel(const QrTc a, const LuArgs l) {
  __shared__ double tile[32][33];
  const int b = a.b0 + blockIdx.y, N = a.q.N, c0 = blockIdx.x * 32;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (!DQMC_CHECK(blockDim.x == 256 && l.nrhs == a.nc - N, l.nrhs)) return;
  double* W = a.q.W + (long long)b * a.q.sW;
  const double* A = l.A + (long long)b * l.sA;
  const double* R = l.R ? l.R + (long long)b * l.sR : nullptr;
  const double* Rd = l.Rdiag ? l.Rdiag + (long long)b * l.sRdiag : nullptr;
  for (int r0 = 0; r0 < N; r0 += 32) {
    // entries that are contiguous along the column come in along it, the others along rows
    for (int u = wid; u < 32; u += 8) {
      const int cr = c0 + lane, rr = r0 + u;      // along a row
      const int cc = c0 + u, rc = r0 + lane;      // along a column
      if (cr < a.nc && rr < N) {
        if (cr < N) { if (!l.transA) tile[lane][u] = A[(long long)rr * N + cr]; }
        else if (!Rd && !l.transR) tile[lane][u] = R[(long long)rr * l.ldr + cr - N];
      }
      if (cc < a.nc && rc < N) {
        if (cc < N) { if (l.transA) tile[u][lane] = A[(long long)cc * N + rc]; }
        else if (Rd) tile[u][lane] = rc == cc - N ? (l.invRdiag ? 1.0 / Rd[rc] : Rd[rc]) : 0.0;
        else if (l.transR) tile[u][lane] = R[(long long)(cc - N) * l.ldr + rc];
      }
    }
    __syncthreads();
    for (int u = wid; u < 32; u += 8)
      if (c0 + u < a.nc && r0 + lane < N) W[(long long)(c0 + u) * N + r0 + lane] = tile[u][lane];
    __syncthreads();
  }
}

// log|det|, sign and singular pivots of one instance: lanes along the diagonal,
// sums in a fixed order
__global__ void __launch_bounds__(32) solve_det_kernel(const QrTc a, const LuArgs l) {
  const int z = blockIdx.x, b = a.b0 + z, N = a.q.N, lane = threadIdx.x;
  const double* W = a.q.W + (long long)b * a.q.sW;
  double ls = 0.0;
  int neg = 0;
  bool zero = false;
  for (int i = lane; i < N; i += 32) {
    const double r = W[(long long)i * N + i];
    zero |= r == 0.0;
    neg ^= (r < 0.0) ^ (a.T(z, i / NB, 0)[(i % NB) * (NB + 1)] > 0.0);
    if (l.logabsdet) ls += log(fabs(r));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ls += __shfl_xor_sync(0xffffffffu, ls, o);
    neg ^= __shfl_xor_sync(0xffffffffu, neg, o);
  }
  zero = __any_sync(0xffffffffu, zero);
  if (lane == 0) {
    if (l.logabsdet) l.logabsdet[b] = ls;
    if (l.sign) l.sign[b] = neg ? -1 : 1;
    if (zero && l.status) atomicOr(&l.status[b / l.status_div], DQMC_STATUS_SINGULAR);
  }
}

// R Z = Q^T R.h.s. for 32 right-hand sides per CTA, in shared memory: per 32-row
// block from the last, substitution in the block (a warp per two rows, lanes
// along the right-hand sides), then Y -= R(above, block) Z as exact digit products.
__global__ void __launch_bounds__(512, 1) solve_back_kernel(const QrTc a, const LuArgs l) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int z = blockIdx.y, b = a.b0 + z, N = a.q.N;
  const int LD = 32 * a.nkb + 1;
  unsigned char* wz = base + RING;                              // 3 zero tiles, 8 digits of Z
  double* y = reinterpret_cast<double*>(wz + 11 * DT);          // [32][LD]
  double* zs = y + 32 * LD;                                     // block of Z [32][TLD]
  double* rpp = zs + NB * TLD;                                  // diagonal block of R
  double* rinv = rpp + NB * TLD;                                // [32 nkb]
  int* er = reinterpret_cast<int*>(rinv + 32 * a.nkb);          // [32 nkb]
  int* ew = er + 32 * a.nkb;                                    // [32]
  uint64_t* full = reinterpret_cast<uint64_t*>(ew + 32);
  uint64_t* done = full + 1;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(done + 1);
  int* s_fail = reinterpret_cast<int*>(tmem_holder + 1);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (!DQMC_CHECK(blockDim.x == 512 && a.nkb <= 12, a.nkb) ||
      !DQMC_CHECK(dyn_smem_bytes() >=
                      (unsigned)(reinterpret_cast<unsigned char*>(s_fail + 1) - smem_raw), LD))
    return;
  const double* W = a.q.W + (long long)b * a.q.sW;
  const int c0 = 32 * blockIdx.x, ncols = l.nrhs - c0 < 32 ? l.nrhs - c0 : 32;
  if (tid == 0) {
    mbar_init(full, 1);
    mbar_init(done, 1);
    *s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (wid == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_holder)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  for (int i = tid; i < 3 * DT / 16; i += 512) reinterpret_cast<uint4*>(wz)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int u = 0; u < 2; ++u) {
    const int c = wid + 16 * u;
    const double* src = W + (long long)(N + c0 + (c < ncols ? c : 0)) * N;
    for (int r0 = lane; r0 < 32 * a.nkb; r0 += 128) {
      double v[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) v[t] = c < ncols && r0 + 32 * t < N ? src[r0 + 32 * t] : 0.0;
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (r0 + 32 * t < 32 * a.nkb) y[c * LD + r0 + 32 * t] = v[t];
    }
  }
  for (int r = tid; r < 32 * a.nkb; r += 512) {
    const double d = r < N ? W[(long long)r * N + r] : 0.0;
    rinv[r] = d != 0.0 ? 1.0 / d : 0.0;
    er[r] = a.r_exp(z)[r];
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_holder;
  uint32_t nfull = 0, ndone = 0;
  const unsigned char* gr = a.r(z);
  for (int p = a.np - 1; p >= 0; --p) {
    const int j0 = NB * p;
    if (tid == 0 && p > 0) {
      mbar_arrive_expect_tx(full, V_TILE);
      bulk_load(base, gr + (long long)p * V_TILE, V_TILE, full);
    }
    for (int e = tid; e < NB * NB; e += 512) {       // along the columns of W^T
      const int i = e & 31, j = e >> 5;
      rpp[i * TLD + j] = i < j && j0 + j < N ? W[(long long)(j0 + j) * N + j0 + i] : 0.0;
    }
    if (tid < 32) ew[tid] = 0;
    const int i0 = wid, i1 = 31 - wid;               // this warp's rows of the block
    double y0 = y[lane * LD + j0 + i0], y1 = y[lane * LD + j0 + i1];
    __syncthreads();
    for (int i = NB - 1; i >= 0; --i) {
      if (i == i0 || i == i1) zs[i * TLD + lane] = (i == i0 ? y0 : y1) * rinv[j0 + i];
      __syncthreads();
      if (i0 < i) {                                  // (i1 < i implies i0 < i)
        const double zi = zs[i * TLD + lane];
        y0 = fma(-rpp[i0 * TLD + i], zi, y0);
        if (i1 < i) y1 = fma(-rpp[i1 * TLD + i], zi, y1);
      }
    }
    {
      const double z0 = zs[i0 * TLD + lane], z1 = zs[i1 * TLD + lane];
      y[lane * LD + j0 + i0] = z0;
      y[lane * LD + j0 + i1] = z1;
      atomicMax(&ew[lane], max((int)((__double_as_longlong(z0) >> 52) & 0x7ff),
                               (int)((__double_as_longlong(z1) >> 52) & 0x7ff)));
    }
    __syncthreads();
    if (p == 0) break;
    if (tid < 256) {
      const int c = tid >> 3, ch = (tid >> 1) & 3, hf = tid & 1;
      unsigned char* dst = wz + 3 * DT + swz(c, ch) + 8 * hf;
      tc_digits4(tc_exponent(ew[c]), [&](int k) { return zs[(8 * ch + 4 * hf + k) * TLD + c]; },
                 [&](int q, uint2 w) { *reinterpret_cast<uint2*>(dst + q * DT) = w; });
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    const int nt = (j0 + 127) / 128;
    for (int t = 0; t < nt; ++t) {
      const uint32_t acc = tmem + 256u * (uint32_t)(t & 1);
      if (tid == 0) {
        wait_or_fail(full, nfull & 1, s_fail);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        mma_rows(acc, smem_u32(base), smem_u32(wz));
        umma_commit(done);
      }
      ++nfull;
      wait_or_fail(done, ndone & 1, s_fail);
      ++ndone;
      if (tid == 0 && t + 1 < nt) {
        mbar_arrive_expect_tx(full, V_TILE);
        bulk_load(base, gr + ((long long)(t + 1) * a.nkb + p) * V_TILE, V_TILE, full);
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int row = 128 * t + (wid & 3) * 32 + lane;
      rows_subtract(acc, wid, row, j0, row < 32 * a.nkb ? er[row] : 0, ew, y, LD);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
    }
  }
  double* Z = l.Z + (long long)b * l.sZ;
  if (!l.transZ) {
    for (int r = wid; r < N; r += 16)
      if (lane < ncols) Z[(long long)r * l.ldz + c0 + lane] = y[lane * LD + r];
  } else {
    for (int c = wid; c < ncols; c += 16)
      for (int r = lane; r < N; r += 32) Z[(long long)(c0 + c) * l.ldz + r] = y[c * LD + r];
  }
  if (*(volatile int*)s_fail && tid == 0) {
    mbar_wait(full, nfull & 1);   // a copy still in flight lands before the CTA exits (bounded)
    if (l.status) atomicOr(&l.status[b / l.status_div], DQMC_STATUS_TIMEOUT);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (wid == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
}

size_t solve_tc_slot_bytes(int N) {
  QrTc a;
  solve_geometry(a, N, 0);
  return (size_t)a.slot_bytes;
}

cudaError_t solve_tc(const LuArgs& l, void* ws, int slots, cudaStream_t st) {
  if (l.batch <= 0) return cudaSuccess;
  if (l.N < SOLVETC_MIN_N || l.N > QRTC_MAX_N || !ws || slots < 1) return cudaErrorInvalidValue;
  const int N = l.N;
  QrTc a;
  solve_geometry(a, N, l.nrhs);
  a.q.N = N; a.q.batch = l.batch;
  a.q.W = l.W; a.q.sW = l.sW;
  a.q.status = l.status; a.q.status_div = l.status_div;
  a.ws = static_cast<unsigned char*>(ws);
  const int LD = 32 * a.nkb + 1;
  const size_t sm_apply = apply_smem(a.nkb), sm_panel = panel_smem(N, a.nkb);
  const size_t sm_back = 1024 + RING + 11 * DT + ((size_t)32 * LD + 2 * NB * TLD + 32 * a.nkb) * 8 +
                         32 * a.nkb * 4 + 512;
  cudaError_t e;
  if ((e = allow_dyn_smem(qr_apply_kernel<APPLY_NEXT>)) != cudaSuccess) return e;
  if ((e = allow_dyn_smem(qr_panel_kernel<QP_MID, false>)) != cudaSuccess) return e;
  if ((e = allow_dyn_smem(qr_panel_kernel<QP_BIG, false>)) != cudaSuccess) return e;
  if ((e = allow_dyn_smem(solve_back_kernel)) != cudaSuccess) return e;
  if (slots > 65535) slots = 65535;
  const int passes = (l.batch + slots - 1) / slots;
  slots = (l.batch + passes - 1) / passes;   // passes of equal size
  for (a.b0 = 0; a.b0 < l.batch; a.b0 += slots) {
    const int nz = l.batch - a.b0 < slots ? l.batch - a.b0 : slots;
    solve_init_kernel<<<dim3((a.nc + 31) / 32, nz), 256, 0, st>>>(a, l);
    for (int p = 0; p < a.np; ++p) {
      if (N <= 256) qr_panel_kernel<QP_MID, false><<<nz, 512, sm_panel, st>>>(a, p);
      else qr_panel_kernel<QP_BIG, false><<<nz, 512, sm_panel, st>>>(a, p);
      const int left = a.nc - (NB * (p + 1) < N ? NB * (p + 1) : N);
      if (left > 0) qr_apply_kernel<APPLY_NEXT><<<dim3((left + 31) / 32, nz), 512, sm_apply, st>>>(a, p);
    }
    if (l.logabsdet || l.sign || l.status) solve_det_kernel<<<nz, 32, 0, st>>>(a, l);
    if (l.nrhs > 0) {
      TcSplitArgs r;                        // digits of R's rows, zero below the diagonal
      r.X = l.W; r.ldm = N; r.ldj = 1; r.sX = l.sW;
      r.N = N; r.R = 128; r.PJ = 128 * a.nmt; r.PM = 32 * a.nkb; r.upper = 1;
      r.S = reinterpret_cast<__nv_bfloat16*>(a.r(0)); r.sS = a.slot_bytes / 2;
      r.e = a.r_exp(0); r.se = a.slot_bytes / 4;
      r.b0 = a.b0;
      if ((e = tc_split(r, nz, st)) != cudaSuccess) return e;
      solve_back_kernel<<<dim3((l.nrhs + 31) / 32, nz), 512, sm_back, st>>>(a, l);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

size_t qrp_tc_slot_bytes(int N, int row_graded) {
  QrTc a;
  qr_geometry(a, N, row_graded);
  return (size_t)a.slot_bytes;
}

cudaError_t qrp_tc(const QrpArgs& q, void* ws, int slots, cudaStream_t st) {
  if (q.batch <= 0) return cudaSuccess;
  if (q.N < QRTC_MIN_N || q.N > QRTC_MAX_N || !ws || slots < 1) return cudaErrorInvalidValue;
  QrTc a;
  a.q = q;
  const int N = q.N;
  qr_geometry(a, N, q.Drow != nullptr);
  a.ws = static_cast<unsigned char*>(ws);
  const int LD = 32 * a.nkb + 1;
  const size_t sm_init = (size_t)32 * LD * 8;
  const size_t sm_apply = apply_smem(a.nkb);
  cudaError_t e;
  if ((e = allow_dyn_smem(qr_init_kernel)) != cudaSuccess) return e;
  if ((e = allow_dyn_smem(qr_apply_kernel<APPLY_REM>)) != cudaSuccess) return e;
  if ((e = allow_dyn_smem(qr_apply_kernel<APPLY_Q>)) != cudaSuccess) return e;
  if ((e = allow_dyn_smem(qr_panel_kernel<QP_SMALL, true>)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(qr_panel_kernel<QP_SMALL, true>,
                                cudaFuncAttributePreferredSharedMemoryCarveout, 100)) != cudaSuccess)
    return e;
  if ((e = allow_dyn_smem(qr_panel_kernel<QP_MID, true>)) != cudaSuccess) return e;
  if ((e = allow_dyn_smem(qr_panel_kernel<QP_BIG, true>)) != cudaSuccess) return e;
  if (slots > 65535) slots = 65535;
  for (a.b0 = 0; a.b0 < q.batch; a.b0 += slots) {
    const int nz = q.batch - a.b0 < slots ? q.batch - a.b0 : slots;
    // Two CTAs an SM where the launch alone covers three quarters of them (another one
    // runs beside it).  N = 64, M = 100: equal-time chains of 256 instances (128 a launch)
    // 8.82 -> 8.18 ms, both stacks of the time-displaced call 22.0 -> 20.2 ms; with 96 a
    // launch 16.1 -> 16.3 ms and with 16, where a CTA's own chain counts, 4.65 -> 4.93.
    const bool small = N <= 64 && 4 * nz > 3 * device_sms();
    const size_t sm_panel = panel_smem(N, a.nkb, small);
    qr_init_kernel<<<dim3(a.nkb, nz), 256, sm_init, st>>>(a);
    for (int p = 0; p < a.np; ++p) {
      if (small) qr_panel_kernel<QP_SMALL, true><<<nz, 512, sm_panel, st>>>(a, p);
      else if (N <= 256) qr_panel_kernel<QP_MID, true><<<nz, 512, sm_panel, st>>>(a, p);
      else qr_panel_kernel<QP_BIG, true><<<nz, 512, sm_panel, st>>>(a, p);
      const int left = N - NB * (p + 1);
      if (left > 0) qr_apply_kernel<APPLY_REM><<<dim3((left + 31) / 32, nz), 512, sm_apply, st>>>(a, p);
    }
    qr_apply_kernel<APPLY_Q><<<dim3(a.nkb, nz), 512, sm_apply, st>>>(a, 0);
    qr_out_kernel<<<dim3(a.nkb, nz), 256, 0, st>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace dqmc

DQMC_CHECK_UNIT(qrp_tc)
