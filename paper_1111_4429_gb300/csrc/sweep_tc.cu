// Trailing update of the Hermitian sweep on the tensor cores with FP64-level
// accuracy (error-free splitting of the operands, the Ozaki scheme).  The
// sweep inverts eps~ = I - v^1/2 chi v^1/2 (Eq. epsilon in its symmetric
// form; the paper inverts eps with LAPACK's ZGESV, Section "RPA Dielectric
// Matrix: epsilon").
//
// Each sweep step subtracts the rank-kb product P C^H from the lower triangle
// (kb <= 32).  With u_i = [Re P_i, Im P_i] and v_j = [Re C_j, Im C_j] (64 real
// values each), Re(P_i C_j^H) = u_i . v_j and
// Im(P_i C_j^H) = u_i[32:64] . v_j[0:32] - u_i[0:32] . v_j[32:64].
// Every row is scaled by a power of two sigma_i (>= its largest entry) and cut
// into S slices of 8 bits: u_i = sigma_i sum_a 2^{-8(a+1)} h_a, with integer
// h_a (|h_0| <= 256, |h_a| <= 128 for a >= 1) held exactly in FP16.  The
// slice products h_a . g_b are integers whose sums over 64 terms and over
// the pairs of one level L = a + b stay below 2^24, so the tensor cores'
// FP32 accumulation is exact: one FP32 accumulator per level (Re and Im) in
// tensor memory.  The levels a + b < S are kept; they are combined in
// double-FP32 (two-sum); the pair, scaled by the power of two
// sigma_i tau_j 2^-16, is subtracted from A in FP64.  The dropped levels and the double-FP32 sum
// bound the error near 2^-48 of |u_i| |v_j| 64.
//
// FP64 inputs (the plain path) join the seven exact level sums in integers
// instead: a 64-bit integer of unit 2^-55 sigma_i tau_j holds the sum but for
// its last nine bits, and is rounded to FP64 once.  What is left of the error
// is the dropped levels' and the operands' last bits (near 2^-55 sigma_i tau_j, at
// worst 2^-49).  An FMA chain errs relative to the sum of |P_ik C_jk|, which is
// smaller where the large entries of rows i and j lie at different k, so the inner
// indices are balanced before the cut (panel_slice_kernel, slice_general_kernel).
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <vector>

#include "runtime.h"
#include "sweep_common.cuh"
#include "sweep_items.cuh"
#include "tc_common.cuh"

namespace bgw {

namespace oz {

constexpr int S = 7;             // slices per value
constexpr int BETA = 8;          // bits per slice
constexpr int KR = 64;           // real inner length (32 complex)
constexpr int NB = 32;           // sweep block width
constexpr int kUTile = BM * KR * 2;    // 16 KiB
constexpr int kVTile = BN * KR * 2;    // 4 KiB
using tc::globaltimer;
using tc::kWaitNs;
using tc::mbar_try_wait;
using tc::mbar_wait;
using tc::mma;
using tc::smem_u32;
using tc::tma_load_2d;

// K-major operand, 128-byte swizzle: rows of 128 bytes, 8-row groups 1024
// bytes apart.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1u << 16;
  d |= (uint64_t)((1024u >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1u << 46;
  d |= (uint64_t)2u << 61;  // SWIZZLE_128B
  return d;
}
__host__ __device__ constexpr uint32_t idesc(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}
// 16 lanes x 256 bits: register pair (0, 1) holds lane base + l / 4, columns
// 2 (l % 4) and 2 (l % 4) + 1; pair (2, 3) the same columns of lane base + 8 + l / 4.
__device__ __forceinline__ void tmem_ld16x256(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

// Per-matrix description of one batched sweep (device pointers).
struct OzMat {
  double2* A;
  const double2* C;   // [ng][NB]
  const double2* P;   // [ng][NB]
  double2* Dinv;      // [NB][NB] D^-1 of the next diagonal block (written by mode 1)
  float4* Dff;        // [NB][NB] the same as double-FP32 pairs (re hi, re lo, im hi, im lo)
  int ng;
  int row_off;        // first slice row of this matrix (multiple of BM)
};
constexpr int kBatch = 96;
struct OzBatch {
  int n;
  OzMat m[kBatch];
};

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Two consecutive complex values in one 256-bit access (p 32-byte aligned).
__device__ __forceinline__ void ld_pair(const double2* p, double2& a, double2& b) {
  asm("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(a.x), "=d"(a.y), "=d"(b.x), "=d"(b.y) : "l"(p));
}
__device__ __forceinline__ void st_pair(double2* p, double2 a, double2 b) {
  asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(p), "d"(a.x), "d"(a.y), "d"(b.x), "d"(b.y) : "memory");
}

// two_sum(a, x w) for a power of two w (x w exact): the products enter fused
// multiply-adds, the results are those of two_sum(a, x w) bit for bit.
__device__ __forceinline__ void two_sum_scaled(float a, float x, float w, float& s, float& e) {
  s = __fmaf_rn(x, w, a);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fmaf_rn(x, w, -bb));
}

__device__ __forceinline__ double ff2d_scaled(float h, float l, int ex) {
  float s, t;
  two_sum(h, l, s, t);
  return ff2d_pair(s, t, ex);
}


// Balanced base-256 digits of a 56-bit fixed-point value: x = sum_a h_a
// 2^{-8(a+1)} for |x| < 1, |h_0| <= 256 and |h_a| <= 128 (a >= 1).  X is
// rint(x 2^56); integer arithmetic only.
__device__ __forceinline__ void digits7(long long X, __half* out, size_t stride) {
  int d[S];
#pragma unroll
  for (int p = 0; p < S - 1; ++p) {
    const long long dp = ((X + 128) & 255) - 128;
    d[S - 1 - p] = (int)dp;
    X = (X - dp) >> 8;
  }
  d[0] = (int)X;
  // |d| <= 256: FP16 bits 0x6600 + d are 1536 + d exactly (unit spacing in
  // [1024, 2048)); one FP16 subtraction leaves d, with no conversion
  // instruction
#pragma unroll
  for (int a = 0; a < S; ++a)
    out[a * stride] = __hsub(__ushort_as_half((unsigned short)(0x6600 + d[a])), __ushort_as_half(0x6600));
}

// Slices of one row of 64 values held by a warp (lane: value k and k + 32);
// all lanes call it.  VROW false: a row of U, re | im.  VROW true: the two
// rows a column of the product reads (vrow): re | im for the real part of
// P C^H and -im | re for the imaginary part, so that one MMA makes both.
// *exp_out: the row's exponent.  FP64 (FP64 inputs): the lane's value counts as
// value 2^t, and a row that holds an infinity or NaN gets kBadExp, which makes
// NaN of every element it updates.
template <bool VROW, bool FP64>
__device__ __forceinline__ void slice_row(double re, double im, int lane, __half* base, size_t stride, int* exp_out,
                                          int t = 0) {
  // e = frexp exponent of the row's largest magnitude, from the biased
  // exponent fields (integer max over the warp; 0 for a zero row, and rows
  // of subnormals alone are cut to zero)
  int top = max(exponent_field(re), exponent_field(im));
  if constexpr (FP64) top = top == 0x7FF ? kBadExp : top ? max(top + t, 1) : 0;
  const int emax = __reduce_max_sync(0xffffffffu, top);
  const int e = emax ? emax - 1022 : 0;   // |value| 2^(t - e) < 1
  const long long Xr = fixed56(re, e - t), Xi = fixed56(im, e - t);
  digits7(Xr, base + lane, stride);
  digits7(Xi, base + lane + 32, stride);
  if constexpr (VROW) {
    __half* second = base + 16 * KR;   // the imaginary part's row of the same column
    digits7(-Xi, second + lane, stride);
    digits7(Xr, second + lane + 32, stride);
  }
  if (lane == 0) *exp_out = FP64 && emax == kBadExp ? kBadExp : e;
}

// Row of V planes that holds column j's real-part row (its imaginary-part row
// lies 16 further): 16 columns' pairs of rows are contiguous, one TMA box.
__device__ __forceinline__ size_t vrow(size_t j) { return (j >> 4) * 32 + (j & 15); }

// The Hermitian sweep's panel and its slices in one launch (the look-ahead
// chain's critical path): for every row i outside the block K (warp per
// row, lane k = column k), C_i = A_iK (read from the stored lower triangle),
// P_i = C_i D^-1, the panel buffers and A_iK <- P_i written as the panel
// kernel of the FP64 sweep does, then P_i and C_i cut into their slices.
// Rows of K and padding rows get zero slices.  grid (ngpad/8, nmat).
// FP64 inputs: P_ik 2^t_k and C_jk 2^-t_k are cut, 2^t_k near (D^-1)_kk^-1/2.
// A row's entries are held to 2^-57 of its largest, and where the diagonal of
// eps~ is graded (a macroscopic constant of 1e6 or 1e8 in the head) P_ik falls
// and C_jk grows with the k-th diagonal entry: unscaled, the inverse of such a
// matrix was off by 2e-15 and 2e-14 against 5e-16.
// FF: P_i = C_i D^-1 in double FP32 (the five-slice update, whose target
// precision, near 2^-34, is far above the pair arithmetic's 2^-43): the
// products as exact pairs, their high words two-summed and the errors
// gathered in the low word; the FP64 pipe keeps only the conversions.
template <bool FF, bool FFD>
__global__ void __launch_bounds__(256) panel_slice_kernel(const __grid_constant__ OzBatch b, int k0, int rows_total,
                                                          int buf, int vpair, __half* __restrict__ U,
                                                          __half* __restrict__ V, int* __restrict__ sig,
                                                          int* __restrict__ tau) {
  __shared__ double2 Ds[NB][NB];   // FF: float4 (re hi, re lo, im hi, im lo)
  __shared__ double2 Cs[8][NB];
  const OzMat& M = b.m[blockIdx.y];
  const int ng = M.ng;
  const int ngpad = (ng + BM - 1) / BM * BM;
  if (blockIdx.x * 8 >= ngpad) return;
  const int kb = min(NB, ng - k0);
  double2* A = M.A;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // FFD: the look-ahead CTA that swept the block (every step after the
  // first) left D^-1 as double-FP32 pairs; the first step's block comes in
  // FP64 (a template flag: a runtime test would leave the conversions
  // predicated in every launch)
  for (int e = threadIdx.x; e < NB * NB; e += 256) {
    if constexpr (FF) {
      if constexpr (FFD) {
        reinterpret_cast<float4*>(&Ds[0][0])[e] = M.Dff[e];
      } else {
        const double2 d = M.Dinv[e];
        const float2 r = ff_from(d.x), m = ff_from(d.y);
        reinterpret_cast<float4*>(&Ds[0][0])[e] = make_float4(r.x, r.y, m.x, m.y);
      }
    } else {
      Ds[e / NB][e % NB] = M.Dinv[e];
    }
  }
  const int i = blockIdx.x * 8 + warp;
  const bool row_ok = k0 < ng && i < ng && (i < k0 || i >= k0 + kb);
  double2 cv = make_double2(0.0, 0.0);
  if (row_ok && lane < kb) {
    if (i >= k0 + kb) {
      cv = A[(size_t)i * ng + k0 + lane];
    } else {
      const double2 t = A[(size_t)(k0 + lane) * ng + i];
      cv = make_double2(t.x, neg_bits(t.y));
    }
  }
  // FF: the conversions in the integer pipe (the FP64 pipe bounds this kernel)
  if constexpr (FF) {
    const float2 r = ff_from_int(cv.x), m = ff_from_int(cv.y);
    reinterpret_cast<float4*>(&Cs[0][0])[warp * NB + lane] = make_float4(r.x, r.y, m.x, m.y);
  } else {
    Cs[warp][lane] = cv;
  }
  __syncthreads();
  double2 pv = make_double2(0.0, 0.0);
  if (row_ok) {
    if constexpr (FF) {
      const float4* Cf = reinterpret_cast<const float4*>(&Cs[0][0]) + warp * NB;
      const float4* Df = reinterpret_cast<const float4*>(&Ds[0][0]);
      float sr = 0.f, cr = 0.f, si = 0.f, ci = 0.f;   // high word, gathered low terms
      auto acc = [](float& S, float& c, float ah, float al, float bh, float bl) {
        const float p = __fmul_rn(ah, bh);
        float e = __fmaf_rn(ah, bh, -p);
        e = __fmaf_rn(ah, bl, e);
        e = __fmaf_rn(al, bh, e);
        const float2 t = ff_two_sum(S, p);
        S = t.x;
        c = __fadd_rn(c, __fadd_rn(t.y, e));
      };
      for (int t = 0; t < kb; ++t) {
        const float4 a = Cf[t], d = Df[t * NB + lane];
        acc(sr, cr, a.x, a.y, d.x, d.y);     // + a_r d_r
        acc(sr, cr, -a.z, -a.w, d.z, d.w);   // - a_i d_i
        acc(si, ci, a.x, a.y, d.z, d.w);     // + a_r d_i
        acc(si, ci, a.z, a.w, d.x, d.y);     // + a_i d_r
      }
      pv = make_double2(ff_to_any(sr, cr), ff_to_any(si, ci));
    } else {
      for (int t = 0; t < kb; ++t) {
        const double2 a = Cs[warp][t], d = Ds[t][lane];
        pv.x = fma(a.x, d.x, fma(-a.y, d.y, pv.x));
        pv.y = fma(a.x, d.y, fma(a.y, d.x, pv.y));
      }
    }
    if (lane < kb) {
      const_cast<double2*>(M.C)[(size_t)i * NB + lane] = cv;
      const_cast<double2*>(M.P)[(size_t)i * NB + lane] = pv;
      if (i >= k0 + kb)
        A[(size_t)i * ng + k0 + lane] = pv;
      else
        A[(size_t)(k0 + lane) * ng + i] = make_double2(pv.x, neg_bits(pv.y));
    }
  }
  if (lane >= kb) pv = cv = make_double2(0.0, 0.0);
  const int t = FF ? 0 : (1023 - exponent_field(Ds[lane][lane].x)) >> 1;
  const size_t row = (size_t)M.row_off + i;
  slice_row<false, !FF>(pv.x, pv.y, lane, U + ((size_t)buf * S * rows_total + row) * KR, (size_t)rows_total * KR,
                        sig + (size_t)buf * rows_total + row, t);
  if (vpair)
    slice_row<true, !FF>(cv.x, cv.y, lane, V + ((size_t)buf * S * 2 * rows_total + vrow(row)) * KR,
                         (size_t)2 * rows_total * KR, tau + (size_t)buf * rows_total + row, -t);
  else   // real values: the real part's rows alone
    slice_row<false, !FF>(cv.x, cv.y, lane, V + ((size_t)buf * S * rows_total + row) * KR, (size_t)rows_total * KR,
                          tau + (size_t)buf * rows_total + row, -t);
}

// Slices for the general (Gauss-Jordan) update A -= Cp R of the pivoted
// inverse: z = 0 slices the column panel Cp [ng][NB] (rows of the block K
// zero: they are overwritten with R afterwards), z = 1 slices R^H, read
// transposed from R [NB][ng] (every row live: the block's columns receive
// -Cp D^-1).  M.P holds Cp, M.C holds R.  FP64 inputs (sizes): Cp_ik 2^t_k and
// R_kj 2^-t_k, which brings both operands' largest entries of inner index k to
// the same size, as in the Hermitian panel (head 1e6 / 1e8: 1e-14 / 1e-13 without
// it, 4e-16 by FP64 FMA); sizes[m][0 / 1][k] are the exponent fields of the
// largest entries of row k of R and of column k of Cp.
template <bool FP64>
__global__ void __launch_bounds__(256) slice_general_kernel(const __grid_constant__ OzBatch b, int k0,
                                                            int rows_total, int buf,
                                                            const int* __restrict__ sizes,
                                                            __half* __restrict__ U, __half* __restrict__ V,
                                                            int* __restrict__ sig, int* __restrict__ tau) {
  const OzMat& M = b.m[blockIdx.y];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + warp;
  const int ngpad = (M.ng + BM - 1) / BM * BM;
  if (i >= ngpad) return;
  const int kb = min(NB, M.ng - k0);
  double re = 0.0, im = 0.0;
  if (blockIdx.z == 0) {
    if (i < M.ng && (i < k0 || i >= k0 + kb) && lane < kb) {
      const double2 v = M.P[(size_t)i * NB + lane];
      re = v.x;
      im = v.y;
    }
  } else if (i < M.ng && lane < kb) {
    const double2 v = M.C[(size_t)lane * M.ng + i];
    re = v.x;
    im = -v.y;
  }
  int t = 0;
  if constexpr (FP64) {
    const int r = sizes[blockIdx.y * 2 * NB + lane], q = sizes[blockIdx.y * 2 * NB + NB + lane];
    if (r && q) t = (r - q) >> 1;
  }
  const size_t row = (size_t)M.row_off + i;
  if (blockIdx.z == 0)
    slice_row<false, FP64>(re, im, lane, U + ((size_t)buf * S * rows_total + row) * KR, (size_t)rows_total * KR,
                           sig + (size_t)buf * rows_total + row, t);
  else
    slice_row<true, FP64>(re, im, lane, V + ((size_t)buf * S * 2 * rows_total + vrow(row)) * KR,
                          (size_t)2 * rows_total * KR, tau + (size_t)buf * rows_total + row, -t);
}

// Rows of the block K after the general update: A[k0 + r][j] = R[r][j].
__global__ void rows_from_r_kernel(const __grid_constant__ OzBatch b, int k0) {
  const OzMat& M = b.m[blockIdx.y];
  const int kb = min(NB, M.ng - k0);
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k0 >= M.ng || e >= (long long)kb * M.ng) return;
  const int r = (int)(e / M.ng), j = (int)(e - (long long)r * M.ng);
  M.A[(size_t)(k0 + r) * M.ng + j] = M.C[(size_t)r * M.ng + j];
}


// ---------------------------------------------------------------------------
// Persistent, pipelined form of the update.  A CTA takes work items of up to
// kJPI column tiles of one row tile I: the row's U slices are loaded once per
// item.  A complex tile is worked on as two halves of 16 columns, each with its
// own accumulators in tensor memory (SL levels x 16 columns, real and imaginary
// parts side by side: 224 of 512 columns) and its own group of 8 epilogue
// warps, so the tensor cores fill one half's sums while the other half's are
// used; tiles of real values alternate between the two sets and groups.  One
// control thread (warp 16) issues the TMA copies (V double-buffered) and the
// MMAs.  An epilogue thread reads its old values of A while the MMAs run, joins
// the levels as it reads them out of tensor memory and subtracts at once.
//
// Per 128 x 32 tile and SM: 1.9 us of MMAs (4 KB of U from shared memory per MMA),
// 2.0 us of FP64 adds (one per word), 1.9 us of instruction issue (level sums and
// conversions); 2.9 us of HBM where the matrix exceeds L2.  Measured 4.6 us:
// stamps show the control thread (2.3 us a half: MMA issue 1.1, the wait for the
// half before and its copies 0.7) and the reads of tensor memory (1.9 us, slower
// beside MMAs) in turn.  Bulk launch at N_G 7180 254 -> 232 us, six matrices of
// 2120 157 -> 142 us, with FP64 inputs 308 -> 261 and 193 -> 162 us, against one
// set of accumulators drained before the FP64 part.  Separate warps for copies
// and MMAs with lists of tiles in shared memory (MMAs of one half always beside
// reads of the other, both twice as slow) measured 240 and 148 us; a third V
// buffer leaves less shared memory to other streams' kernels (three concurrent
// solves 1 to 8% slower).
constexpr int kPipeEpiWarps = 16;
constexpr int kPipeThreads = (kPipeEpiWarps + 1) * 32;
static_assert(kPipeThreads == kDiagThreads, "the look-ahead CTA sweeps the next diagonal block");
constexpr int kVRing = 2;              // V units in flight

// A segment's seven level sums (integers below 2^23.2 in FP32) joined in units
// of 2^-55: adjacent levels in 32 bits, the rest in 64.
__device__ __forceinline__ long long join_levels(const uint32_t (&x)[7][4], int q) {
  auto f = [&](int L) { return __float2int_rn(__uint_as_float(x[L][q])); };
  const int p01 = f(0) * 256 + f(1), p23 = f(2) * 256 + f(3), p45 = f(4) * 256 + f(5);
  const long long hi = (long long)p01 * 65536 + p23, lo = (long long)p45 * 256 + f(6);   // units 2^-40, 2^-64
  return (hi << 15) + ((lo + 256) >> 9);
}

// The level sums of accumulator q as a double-FP32 pair: level L enters scaled
// by 2^-8L (exact), folded into fused multiply-adds (the roundings of scaling
// first).  Levels 1 .. two_sum that reach the running sum's last bits are
// two-summed into the high word (with seven slices the target is near 2^-48:
// levels 1 and 2; with five near 2^-34: level 1); deeper levels lie below
// the sum's last bit at the target precision and go to the low word.
template <int SL>
__device__ __forceinline__ void sum_levels(const uint32_t (&x)[SL][4], int q, float& h, float& l) {
  constexpr int two_sum = SL >= 7 ? 2 : 1;
  h = __uint_as_float(x[0][q]);
  l = 0.f;
#pragma unroll
  for (int L = 1; L < SL; ++L) {
    const float w = ldexpf(1.f, -BETA * L), v = __uint_as_float(x[L][q]);
    if (L <= two_sum) {
      float sm, e;
      two_sum_scaled(h, v, w, sm, e);
      h = sm;
      l = __fadd_rn(l, e);
    } else {
      l = __fmaf_rn(v, w, l);
    }
  }
}

// SL: slices used per value (the most significant SL of the S stored): 7
// gives an update error near 2^-48 of its scale, 5 near 2^-34.  FFC: the
// look-ahead CTA sweeps the next diagonal block in double FP32 (about 2^-46
// per operation, on the FP32 pipe) instead of FP64; without it (FP64 inputs)
// the level sums are joined in integers and rounded to FP64 once.
template <bool realv, int SL, bool FFC, bool NARROW>
__global__ void __launch_bounds__(kPipeThreads, 1)   // 17 warps: at most 5 per sub-partition, 96 registers
    update_pipe_kernel(const __grid_constant__ CUtensorMap umap, const __grid_constant__ CUtensorMap vmap,
                       const __grid_constant__ OzBatch b, int k0, int rows_total, int buf, int mode,
                       const int* __restrict__ sig, const int* __restrict__ tau, int* __restrict__ status) {
  // column tiles per bulk work item, a compile-time constant (a runtime
  // width costs 2% in the item decode)
  constexpr int wide = NARROW ? 2 : (SL < 7 ? 3 : kJPI);
  // Units of a tile: its two halves (16 columns, real and imaginary parts: 32
  // accumulator columns a level; accumulators h), or for real values the tile
  // itself (32 columns; accumulators of the tile's parity).
  constexpr int UN = realv ? 1 : 2, UC = BN / UN;
  const OzMat& M = b.m[blockIdx.y];
  const int ng = M.ng;
  if (k0 >= ng) return;
  const int kb = min(NB, ng - k0);
  const int nI = (ng + BM - 1) / BM, nJ = (ng + BN - 1) / BN;
  const int k1 = k0 + NB;
  const bool has_next = k1 < ng;
  const int In = k1 / BM, Jn = k1 / BN;
  if (mode == 1 && !has_next) return;
  const int nitems = pipe_items(mode, wide, nI, nJ, In, has_next);
  const int slice_base = buf * S * rows_total;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* us = smem;                          // SL x 16 KiB
  unsigned char* vs = smem + SL * kUTile;            // kVRing x SL x 4 KiB
  uint64_t* u_full = reinterpret_cast<uint64_t*>(vs + kVRing * SL * kVTile);
  uint64_t* v_full = u_full + 1;                     // [kVRing]
  uint64_t* v_empty = v_full + kVRing;               // [kVRing]
  uint64_t* t_full = v_empty + kVRing;               // [2] a half's sums are complete
  uint64_t* t_empty = t_full + 2;                    // [2] a half's sums have been read
  uint64_t* u_empty = t_empty + 2;                   // an item's MMAs are complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(u_empty + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  __shared__ DiagSmem dsm;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool control = warp == kPipeEpiWarps;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(u_full)) : "memory");
    for (int q = 0; q < kVRing; ++q) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(v_full + q)) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(v_empty + q)) : "memory");
    }
    for (int q = 0; q < 2; ++q) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(t_full + q)) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(t_empty + q)), "r"(kPipeEpiWarps / 2)
                   : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(u_empty)) : "memory");
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  int t = 0;           // tiles processed by this CTA (buffer and phase bookkeeping)
  int items_done = 0;  // items processed
  int u_loads = 0;     // U loads issued (control; phase of u_full)
  int vissued = 0;     // V units issued (control)
  PipeCursor cursor;
  for (int item = blockIdx.x; item < nitems; item += gridDim.x, ++items_done) {
    int I, J0, J1;
    pipe_decode_next(cursor, mode, wide, item, nI, nJ, In, Jn, has_next, I, J0, J1);
    const int i0 = I * BM;
    // tiles of the item that are not skipped, in order
    int Js[kJPI], nt = 0;
    for (int J = J0; J < J1; ++J)
      if (!pipe_skip(mode, item, I, J, ng, k0, kb, In, Jn, has_next)) Js[nt++] = J;
    if (control) {
      if (lane == 0 && nt > 0 && !*abort_flag) {
        // U slices of the row tile, once the previous item's MMAs have read
        // the last ones (its epilogue may still run: items are independent)
        bool ok = u_loads == 0 || mbar_wait(u_empty, (u_loads - 1) & 1, abort_flag);
        const int u_phase = u_loads & 1;
        if (ok) {
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(u_full)),
                       "r"((uint32_t)(SL * kUTile))
                       : "memory");
          for (int a = 0; a < SL; ++a)
            tma_load_2d(us + a * kUTile, &umap, u_full, 0, slice_base + a * rows_total + M.row_off + i0);
          ++u_loads;
        }
        // unit uu (counted over the CTA's life) of the item: columns UC (uu % UN) .. of tile Js[(uu - uu0) / UN]
        const int uu0 = UN * t, uu1 = UN * (t + nt);
        auto issue_v = [&](int uu) {
          const int bq = uu % kVRing;
          if (uu >= kVRing && !mbar_wait(&v_empty[bq], (uu / kVRing - 1) & 1, abort_flag)) return false;
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(v_full + bq)),
                       "r"((uint32_t)(SL * kVTile))
                       : "memory");
          const int j = Js[(uu - uu0) / UN] * BN + (uu % UN) * UC;
          for (int a = 0; a < SL; ++a)
            tma_load_2d(vs + (bq * SL + a) * kVTile, &vmap, v_full + bq, 0,
                        UN * (slice_base + a * rows_total + M.row_off + j));
          vissued = uu + 1;
          return true;
        };
        ok = ok && issue_v(uu0);
        for (int uu = uu0; uu < uu1 && ok; ++uu) {
          if (uu + 1 < uu1 && !issue_v(uu + 1)) {
            ok = false;
            break;
          }
          const int tt = uu / UN, bq = uu % kVRing;
          const int acc = realv ? tt & 1 : uu & 1, use = realv ? tt >> 1 : tt;   // accumulators, and how often used before
          if ((uu == uu0 && !mbar_wait(u_full, u_phase, abort_flag)) ||
              !mbar_wait(&v_full[bq], (uu / kVRing) & 1, abort_flag) ||
              (use > 0 && !mbar_wait(&t_empty[acc], (use - 1) & 1, abort_flag))) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          // Level L of the unit's sums lies in columns 32 L (16 of the real
          // parts, then 16 of the imaginary parts; real values: 32).  The V
          // slices lie one after the other in shared memory, so for one U slice
          // a the products with V slices 0 .. SL-1-a are one MMA of N = 32
          // (SL - a) columns into levels a .. SL-1, and the two rows of a column
          // (vrow) make both parts: each U chunk is read once per slice.  A
          // descriptor's start address is its low 14 bits (address / 16, no
          // carry below 256 KiB), so every operand descriptor is the base's plus
          // a constant; slice a = 0 writes every level first.
          const uint64_t du = sdesc(smem_u32(us)), dv = sdesc(smem_u32(vs + bq * SL * kVTile));
#pragma unroll
          for (int a = 0; a < SL; ++a) {
            const uint32_t d = tmem + (acc * SL + a) * 32;
            const uint64_t ua = du + (uint64_t)((a * kUTile) >> 4);
            const uint32_t id = idesc(32 * (SL - a));
            // byte offsets 32 q along K: +2 q in the descriptor; real values fill the first half of the row
#pragma unroll
            for (int q = 0; q < (realv ? 2 : 4); ++q) mma(d, ua + 2 * q, dv + 2 * q, id, a == 0 && q == 0 ? 0u : 1u);
          }
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                           smem_u32(v_empty + bq))
                       : "memory");
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                           smem_u32(t_full + acc))
                       : "memory");
        }
        if (ok)
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                           smem_u32(u_empty))
                       : "memory");
        if (!ok) {
          *abort_flag = 1;
          atomicExch(status, (int)kDevTimeout);
        }
      }
      __syncwarp();
    } else {
      // ---------------- epilogue warps: group warp / 8 takes one half of every tile (real values: every other tile),
      // its warps rows 32 (warp % 4) .. + 31 and eight columns (real values:
      // sixteen, eight at a time).  The accumulators are read in the 16x256b
      // shape: lane l holds rows g, g + 8, g + 16, g + 24 (g = l / 4) and
      // columns 2 (l % 4), + 1, so one warp-wide access of A touches 8 rows of
      // 128 contiguous bytes instead of 32 rows of 16 (four times fewer cache
      // lines).
      const int group = warp >> 3, quad = warp & 3, part = (warp >> 2) & 1;
      const int g = lane >> 2, cl = 2 * (lane & 3);
      const int c0 = realv ? part * 16 : group * UC + part * 8;
      // rows r0 + 8 m (m = 0 .. 3) and their exponents sigma
      const int r0 = i0 + quad * 32 + g;
      auto row_ok = [&](int i) { return i < ng && !(i >= k0 && i < k0 + kb); };
      int ei[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) ei[m] = row_ok(r0 + 8 * m) ? sig[buf * rows_total + M.row_off + r0 + 8 * m] : 0;
      // 128 bytes of A for tile kk (row g + 8 (lane % 4), the warp's eight
      // columns) into L2, one tile ahead
      const int prow = i0 + quad * 32 + g + 8 * (lane & 3);
      const bool prow_ok = prow < ng;
      auto prefetch_a = [&](int kk) {
        if (!prow_ok || kk >= nt) return;
        const int j = Js[kk] * BN + c0;
        if (j >= ng) return;
        const double2* row = M.A + (size_t)prow * ng;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(row + j));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(row + min(j + 7, ng - 1)));
        if constexpr (realv) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + min(j + 15, ng - 1)));
      };
      // the exponents of tile kk's columns from c (complex tiles: read one tile ahead)
      auto load_tau = [&](int kk, int c, int (&tv)[2]) {
#pragma unroll
        for (int n = 0; n < 2; ++n) {
          const int j = kk < nt ? Js[kk] * BN + c + cl + n : ng;
          tv[n] = j < ng ? tau[buf * rows_total + M.row_off + j] : 0;
        }
      };
      // element e = 2 m + n of tile kk from column c: row r0 + 8 m, column Js[kk] BN + c + cl + n,
      // scale exponent ei[m] + tv[n] - 16.  Bit e of the mask: the element is
      // updated; bit 8 + e: its old value is read (columns of the block K
      // start from zero in the Gauss-Jordan form).
      int tv[2];
      // a lane's pair of columns starts at an even index: 32-byte aligned in every row
      const bool paired = (ng & 1) == 0 && (reinterpret_cast<uintptr_t>(M.A) & 31u) == 0;
      unsigned mask = 0;
      auto tile_mask = [&](int kk, int c) {
        const int j0 = Js[kk] * BN;
        // inside the matrix, below the diagonal and clear of the block's rows
        // and columns: every element is live
        if (i0 + BM <= ng && (mode == 3 ? j0 + BN <= ng : j0 + BN <= i0) && (i0 >= k0 + kb || i0 + BM <= k0) &&
            (j0 >= k0 + kb || j0 + BN <= k0))
          return 0xFFFFu;
        unsigned mk = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int i = r0 + 8 * (e >> 1), j = j0 + c + cl + (e & 1);
          const bool jblock = j >= k0 && j < k0 + kb;
          const bool live = row_ok(i) && j < ng && (mode == 3 ? true : (j <= i && !jblock));
          mk |= (live ? 1u : 0u) << e;
          mk |= (live && !jblock ? 1u : 0u) << (8 + e);
        }
        return mk;
      };
      if (nt > 0 && !realv) {
        load_tau(0, c0, tv);
        mask = tile_mask(0, c0);
      }
      prefetch_a(0);
      for (int k = 0; k < nt; ++k) {
        const int tt = t + k;
        const int j0 = Js[k] * BN;
        if constexpr (realv) {
          prefetch_a(k + 2);
          if ((tt & 1) != group) continue;
        } else {
          prefetch_a(k + 1);
        }
        bool have = true;
#pragma unroll 1
        for (int ch = 0; ch < (realv ? 2 : 1) && have; ++ch) {
        const int c = c0 + 8 * ch;
        if constexpr (realv) {
          load_tau(k, c, tv);
          mask = tile_mask(k, c);
        }
        // the tile's old values, read while its MMAs run: a lane's two columns
        // are adjacent, one 256-bit access per row where both are read
        // (written) and the pair is 32-byte aligned (every row for an even N_G
        // and an aligned matrix), else one 128-bit access per element
        double2 av[8];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const size_t off = (size_t)(r0 + 8 * m) * ng + j0 + c + cl;
          const unsigned rd = (mask >> (8 + 2 * m)) & 3u;
          av[2 * m] = av[2 * m + 1] = make_double2(0.0, 0.0);
          if (rd == 3u && paired) {
            ld_pair(M.A + off, av[2 * m], av[2 * m + 1]);
          } else {
            if (rd & 1u) av[2 * m] = M.A[off];
            if (rd & 2u) av[2 * m + 1] = M.A[off + 1];
          }
        }
        // the next tile's column exponents, used after this tile
        int tnext[2];
        if constexpr (!realv) load_tau(k + 1, c0, tnext);
        have = mbar_wait(&t_full[group], (realv ? tt >> 1 : tt) & 1, abort_flag);
        have = __all_sync(0xffffffffu, have) != 0;
        if (have) {
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          // Four rounds (two 16-row halves, real then imaginary parts): each
          // issues the loads of all SL levels before one wait, joins the
          // levels, applies the scale 2^e2 (sigma_i tau_j 2^-16) in the
          // conversion and subtracts: one FP64 add per word.
#pragma unroll
          for (int rb = 0; rb < (realv ? 2 : 4); ++rb) {
            const int hb = realv ? rb : rb >> 1, im = realv ? 0 : rb & 1;
            const uint32_t tl = tmem + ((uint32_t)(quad * 32 + 16 * hb) << 16) + group * SL * 32 + im * UC + (realv ? c : part * 8);
            uint32_t x[SL][4];
#pragma unroll
            for (int L = 0; L < SL; ++L) tmem_ld16x256(tl + 32 * L, x[L]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (realv ? (ch == 1 && rb == 1) : rb == 3) {
              // every sum is read: the accumulators are free for the next MMAs
              asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
              __syncwarp();
              if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(t_empty + group)) : "memory");
            }
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) {
              const int e = 4 * hb + qq, m = e >> 1;
              const int e2 = ei[m] + tv[e & 1] - 2 * BETA;
              double& dst = im ? av[e].y : av[e].x;
              if constexpr (FFC) {
                float hs, ls;
                sum_levels<SL>(x, qq, hs, ls);
                dst -= ff2d_scaled(hs, ls, e2);
              } else {   // unit 2^-55 against the pairs' 2^-16
                dst -= i64_to_scaled(join_levels(x, qq), e2 - 39);
              }
            }
          }
        } else if (lane == 0) {
          *abort_flag = 1;
          atomicExch(status, (int)kDevTimeout);
        }
        if (!have) break;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const size_t off = (size_t)(r0 + 8 * m) * ng + j0 + c + cl;
          const unsigned wr = (mask >> (2 * m)) & 3u;
          if (wr == 3u && paired) {
            st_pair(M.A + off, av[2 * m], av[2 * m + 1]);
          } else {
            if (wr & 1u) M.A[off] = av[2 * m];
            if (wr & 2u) M.A[off + 1] = av[2 * m + 1];
          }
        }
        if (!realv && k + 1 < nt) {
          tv[0] = tnext[0];
          tv[1] = tnext[1];
          mask = tile_mask(k + 1, c0);
        }
        }
      }
    }
    t += nt;
    // Items of the bulk launches are independent and the barriers order the
    // buffers' reuse, so the next item's copies and MMAs overlap this item's
    // last epilogue.  The look-ahead launch's first item is followed by the
    // next diagonal block's sweep (all threads, U as scratch).
    if (mode == 1) __syncthreads();
    // The tile holding the next diagonal block (rows and columns k1 .. k1+31)
    // has its final values: sweep it here (next step's D^-1 into Dinv, -D^-1
    // into A_K1K1) without a separate launch.
    if (mode == 1 && item == 0 && !*abort_flag) {
      const int kb1 = min(NB, ng - k1);
      for (int e = threadIdx.x; e < NB * NB; e += kPipeThreads) {
        const int rr = e / NB, c2 = e % NB;
        if (rr < kb1 && c2 <= rr) dsm.L[rr][c2] = M.A[(size_t)(k1 + rr) * ng + k1 + c2];
      }
      // double-FP32 chain: the block's sweep in double FP32 (about 2^-46),
      // off the SM's slow FP64 pipe; else FP64
      if constexpr (FFC)
        diag_sweep_ff(dsm, reinterpret_cast<float4*>(us), kb1, threadIdx.x, status, M.Dff);
      else
        diag_sweep_f64(dsm, kb1, threadIdx.x, status);
      for (int e = threadIdx.x; e < NB * NB; e += kPipeThreads) {
        const int rr = e / NB, c2 = e % NB;
        if (rr >= kb1 || c2 >= kb1) continue;
        const double2 v = (rr >= c2) ? dsm.L[rr][c2] : make_double2(dsm.L[c2][rr].x, -dsm.L[c2][rr].y);
        M.Dinv[rr * NB + c2] = make_double2(-v.x, -v.y);
        if (rr >= c2) M.A[(size_t)(k1 + rr) * ng + k1 + c2] = v;
      }
      __syncthreads();
    }
  }
  // no copies in flight at exit (bounded waits on the last loads issued)
  if (control && lane == 0 && u_loads > 0) {
    const uint64_t t0 = globaltimer();
    while (!mbar_try_wait(u_full, (u_loads - 1) & 1) && globaltimer() - t0 < kWaitNs) {
    }
    const uint64_t t2 = globaltimer();
    while (!*abort_flag && !mbar_try_wait(u_empty, (u_loads - 1) & 1) && globaltimer() - t2 < kWaitNs) {
    }
    for (int uu = max(0, vissued - kVRing); uu < vissued; ++uu) {
      const uint64_t t1 = globaltimer();
      while (!mbar_try_wait(&v_full[uu % kVRing], (uu / kVRing) & 1) && globaltimer() - t1 < kWaitNs) {
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

}  // namespace oz

// Dynamic shared memory of update_pipe_kernel with SL slices: U, the ring of
// V halves, alignment slack and the barriers.
size_t pipe_smem(int slices) { return (size_t)slices * (oz::kUTile + oz::kVRing * oz::kVTile) + 1024 + 128; }

// State of one batched sweep that uses the tensor-core update.
struct OzPlan {
  bool general = false;   // Gauss-Jordan update (mode 3) of the pivoted inverse
  int slices = 7;         // slices per value the update uses (5 or 7)
  bool ff_chain = false;  // next diagonal block and panel product in double FP32
  bool real_values = false;  // every matrix real (real flavor): only the real-part MMAs
  int bulk_narrow = -1;   // bulk items: -1 SM-count rule, 0 wide, 1 two column tiles
  int nmat = 0;
  int buffers = 2;        // sets of slices
  int rows_total = 0;
  oz::OzBatch batch;
  CUtensorMap umap, vmap;
  Scratch U, V, sig, tau, dff;
};

int oz_prepare(Ctx* c, int nmat, const int* ng, double2* const* A, const double2* const* C, const double2* const* P,
               double2* const* D, OzPlan* plan, bool general, bool real_values, int slices, bool ff_chain, int buffers) {
  using namespace oz;
  if (slices != 5 && slices != 7) return fail(c, BGW_EINVAL, "tensor-core inverse: 5 or 7 slices");
  plan->slices = slices;
  plan->ff_chain = ff_chain || slices < 7;   // five slices always use the double-FP32 chain
  if (nmat > kBatch) return fail(c, BGW_EUNSUPPORTED, "tensor-core inverse: at most %d matrices per batch", kBatch);
  TensorMapEncode encode;
  if (int erc = tensor_map_encode(c, &encode)) return erc;
  plan->nmat = nmat;
  plan->general = general;
  plan->real_values = real_values;
  plan->batch.n = nmat;
  int rows = 0;
  for (int m = 0; m < nmat; ++m) {
    plan->batch.m[m].A = A[m];
    plan->batch.m[m].C = C[m];
    plan->batch.m[m].P = P[m];
    plan->batch.m[m].Dinv = D ? D[m] : nullptr;
    plan->batch.m[m].ng = ng[m];
    plan->batch.m[m].row_off = rows;
    rows += (ng[m] + BM - 1) / BM * BM;
  }
  plan->rows_total = rows;
  plan->U.pool = plan->V.pool = plan->sig.pool = plan->tau.pool = plan->dff.pool = &c->pool;
  int rc;
  // two sets of slices: a step may slice while the previous step's update still
  // reads its own
  for (plan->buffers = buffers > 0 ? buffers : general ? 1 : 2;; plan->buffers = 1) {
    const size_t sb = (size_t)plan->buffers * S * rows * KR * sizeof(__half);
    if ((rc = c->pool.alloc(sb, &plan->U.ptr)) == BGW_OK &&
        (rc = c->pool.alloc(real_values ? sb : 2 * sb, &plan->V.ptr)) == BGW_OK &&
        (rc = c->pool.alloc((size_t)2 * rows * sizeof(int), &plan->sig.ptr)) == BGW_OK &&
        (rc = c->pool.alloc((size_t)2 * rows * sizeof(int), &plan->tau.ptr)) == BGW_OK &&
        (rc = c->pool.alloc((size_t)nmat * NB * NB * sizeof(float4), &plan->dff.ptr)) == BGW_OK)
      break;
    for (Scratch* x : {&plan->U, &plan->V, &plan->sig, &plan->tau, &plan->dff}) {
      if (x->ptr) c->pool.release(x->ptr);
      x->ptr = nullptr;
    }
    if (rc != BGW_ENOMEM || plan->buffers == 1)
      return fail(c, rc, "tensor-core inverse: slice buffers (%zu B) could not be allocated", real_values ? 2 * sb : 3 * sb);
  }
  for (int m = 0; m < nmat; ++m) plan->batch.m[m].Dff = plan->dff.as<float4>() + (size_t)m * NB * NB;
  cuuint64_t gdim[2] = {(cuuint64_t)KR, (cuuint64_t)plan->buffers * S * rows};
  cuuint64_t gstride[1] = {(cuuint64_t)KR * sizeof(__half)};
  cuuint32_t estr[2] = {1, 1};
  cuuint32_t ubox[2] = {(cuuint32_t)KR, (cuuint32_t)BM};
  // 16 columns of two rows each (vrow); real values: 32 of one
  cuuint32_t vbox[2] = {(cuuint32_t)KR, (cuuint32_t)BN};
  cuuint64_t vdim[2] = {(cuuint64_t)KR, (cuuint64_t)(real_values ? 1 : 2) * plan->buffers * S * rows};
  if (encode(&plan->umap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, plan->U.ptr, gdim, gstride, ubox, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
      encode(&plan->vmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, plan->V.ptr, vdim, gstride, vbox, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return fail(c, BGW_ECUDA, "tensor-core inverse: tensor map encoding failed");
  // U slices, V ring, alignment and barriers: about 170 KiB dynamic (7 slices)
  const size_t psmem = pipe_smem(slices);
#define BGW_PIPE_ATTR(RV, SLC, FF)                                                                        \
  BGW_CUDA(c, cudaFuncSetAttribute(update_pipe_kernel<RV, SLC, FF, false>,                                       \
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psmem));                    \
  BGW_CUDA(c, cudaFuncSetAttribute(update_pipe_kernel<RV, SLC, FF, true>,                                        \
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psmem))
  if (slices == 7 && !plan->ff_chain) {
    BGW_PIPE_ATTR(false, 7, false);
    BGW_PIPE_ATTR(true, 7, false);
  } else if (slices == 7) {
    BGW_PIPE_ATTR(false, 7, true);
    BGW_PIPE_ATTR(true, 7, true);
  } else {
    BGW_PIPE_ATTR(false, 5, true);
    BGW_PIPE_ATTR(true, 5, true);
  }
#undef BGW_PIPE_ATTR
  return BGW_OK;
}

// Slices of one pivoted Gauss-Jordan step (column panel and R^H of every matrix) into buffer buf.
int oz_slice(Ctx* c, OzPlan* plan, int k0, int ngmax, int buf, const int* sizes, cudaStream_t st) {
  using namespace oz;
  const int rpad = (ngmax + BM - 1) / BM * BM;
  if (!plan->general) return fail(c, BGW_EINVAL, "oz_slice: the Hermitian sweep slices in oz_panel_slice");
  const dim3 g(rpad / 8, plan->nmat, 2);
  __half *U = plan->U.as<__half>(), *V = plan->V.as<__half>();
  int *sig = plan->sig.as<int>(), *tau = plan->tau.as<int>();
  if (plan->ff_chain)
    slice_general_kernel<false><<<g, 256, 0, st>>>(plan->batch, k0, plan->rows_total, buf, nullptr, U, V, sig, tau);
  else
    slice_general_kernel<true><<<g, 256, 0, st>>>(plan->batch, k0, plan->rows_total, buf, sizes, U, V, sig, tau);
  BGW_CUDA(c, cudaGetLastError());
  return BGW_OK;
}

// Panel and slices of one Hermitian sweep step in one launch (buffer buf).
int oz_panel_slice(Ctx* c, OzPlan* plan, int k0, int ngmax, int buf, cudaStream_t st) {
  using namespace oz;
  const int rpad = (ngmax + BM - 1) / BM * BM;
  // the look-ahead launches of the double-FP32 chain leave D^-1 as pairs
  // for every step after the first
  if (plan->ff_chain && k0 > 0)
    panel_slice_kernel<true, true><<<dim3(rpad / 8, plan->nmat), 256, 0, st>>>(
        plan->batch, k0, plan->rows_total, buf, plan->real_values ? 0 : 1, plan->U.as<__half>(), plan->V.as<__half>(),
        plan->sig.as<int>(), plan->tau.as<int>());
  else if (plan->ff_chain)
    panel_slice_kernel<true, false><<<dim3(rpad / 8, plan->nmat), 256, 0, st>>>(
        plan->batch, k0, plan->rows_total, buf, plan->real_values ? 0 : 1, plan->U.as<__half>(), plan->V.as<__half>(),
        plan->sig.as<int>(), plan->tau.as<int>());
  else
    panel_slice_kernel<false, false><<<dim3(rpad / 8, plan->nmat), 256, 0, st>>>(
        plan->batch, k0, plan->rows_total, buf, plan->real_values ? 0 : 1, plan->U.as<__half>(), plan->V.as<__half>(),
        plan->sig.as<int>(), plan->tau.as<int>());
  BGW_CUDA(c, cudaGetLastError());
  return BGW_OK;
}

// The trailing update of one sweep step from slice buffer buf: mode 0 all
// tiles, 1 the tiles touching the next block, 2 the others; a general plan
// runs mode 3 (every tile) and then writes R into the block's rows.
int oz_update(Ctx* c, OzPlan* plan, int k0, int ngmax, int buf, int mode, cudaStream_t st) {
  using namespace oz;
  if (mode == 1 && k0 + NB >= ngmax) return BGW_OK;
  if (plan->general) mode = 3;
  // Column tiles per bulk work item: 4 with seven slices, 3 with five; 2
  // where those items would not exceed the SMs (each CTA then pipelines two
  // items instead of running one alone; measured with seven slices: N_G 2120
  // 3.10 -> 2.95 ms per inverse, while at 7180 items of 4 stay best), unless
  // the plan fixes the width (the context's timed choice or its option).
  const int nsm = sm_count(c);
  int wide = plan->slices < 7 ? 3 : kJPI, grid;
  {
    // the most items of a matrix that has not finished: a smaller one at its
    // last step has items (no next row tile to leave out) where the largest
    // may have none
    auto most_items = [&](int w) {
      int n = 0;
      for (int m = 0; m < plan->nmat; ++m) {
        const int ng = plan->batch.m[m].ng, k1 = k0 + NB;
        if (k0 < ng && (mode != 1 || k1 < ng))
          n = std::max(n, pipe_items(mode, w, (ng + BM - 1) / BM, (ng + BN - 1) / BN, k1 / BM, k1 < ng));
      }
      return n;
    };
    grid = most_items(wide);
    const bool narrow = plan->bulk_narrow >= 0 ? plan->bulk_narrow == 1 : (long long)grid * plan->nmat <= nsm;
    if (mode != 1 && narrow) {
      wide = 2;
      grid = most_items(wide);
    }
  }
  if (grid <= 0) return BGW_OK;
  // Bulk launches with more items than SMs run persistent CTAs (items taken
  // round-robin): the next item's copies and MMAs then overlap the last
  // epilogue of the one before, and a CTA's start-up is paid once.  Only when
  // the matrices of the batch share the SMs evenly; the look-ahead launch
  // (on the critical path, few items) keeps one item per CTA.
  if (mode != 1) {
    const int per = nsm / plan->nmat;
    if (per >= 1 && (long long)grid * plan->nmat > nsm && 10 * per * plan->nmat >= 9 * nsm)
      grid = std::min(grid, per);
  }
  const size_t smem = pipe_smem(plan->slices);
  const dim3 g(grid, plan->nmat);
#define BGW_PIPE_LAUNCH(RV, SLC, FF)                                                                          \
  do {                                                                                                         \
    if (wide == 2)                                                                                             \
      update_pipe_kernel<RV, SLC, FF, true><<<g, kPipeThreads, smem, st>>>(                                     \
          plan->umap, plan->vmap, plan->batch, k0, plan->rows_total, buf, mode, plan->sig.as<int>(),           \
          plan->tau.as<int>(), c->d_status);                                                                   \
    else                                                                                                       \
      update_pipe_kernel<RV, SLC, FF, false><<<g, kPipeThreads, smem, st>>>(                                    \
          plan->umap, plan->vmap, plan->batch, k0, plan->rows_total, buf, mode, plan->sig.as<int>(),           \
          plan->tau.as<int>(), c->d_status);                                                                   \
  } while (0)
  const bool rv = plan->real_values;
  if (plan->slices == 7 && !plan->ff_chain) {
    if (rv)
      BGW_PIPE_LAUNCH(true, 7, false);
    else
      BGW_PIPE_LAUNCH(false, 7, false);
  } else if (plan->slices == 7) {
    if (rv)
      BGW_PIPE_LAUNCH(true, 7, true);
    else
      BGW_PIPE_LAUNCH(false, 7, true);
  } else {
    if (rv)
      BGW_PIPE_LAUNCH(true, 5, true);
    else
      BGW_PIPE_LAUNCH(false, 5, true);
  }
#undef BGW_PIPE_LAUNCH
  if (plan->general) {
    const long long ne = (long long)NB * ngmax;
    rows_from_r_kernel<<<dim3((unsigned)((ne + 255) / 256), plan->nmat), 256, 0, st>>>(plan->batch, k0);
  }
  BGW_CUDA(c, cudaGetLastError());
  return BGW_OK;
}

int oz_buffers(const OzPlan* plan) { return plan->buffers; }

void oz_set_bulk_items(OzPlan* plan, int narrow) { plan->bulk_narrow = narrow < 0 ? -1 : (narrow ? 1 : 0); }

OzPlan* oz_plan_new() { return new OzPlan(); }
void oz_plan_delete(OzPlan* p) { delete p; }

}  // namespace bgw
