// Sweep of one diagonal block in shared memory (the diagonal step of both
// sweeps in epsinv.cu, which invert eps~ of Eq. epsilon).
//
// D (Hermitian positive definite, kb <= 32) is held as its lower triangle
// L[i][j], i >= j.  Pivot s: every lower element outside row/column s loses
// col_i conj(col_j) / d (col = column s of the full matrix, d = L[s][s]), the
// pivot column is divided by d and the pivot becomes -1/d.  After kb pivots
// L holds -D^-1.
#pragma once
#include "runtime.h"

namespace bgw {

// -x by the sign bit (no FP64 instruction)
__device__ __forceinline__ double neg_bits(double x) {
  return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ull);
}

__device__ __forceinline__ int exponent_field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

constexpr int kSwNB = 32;
constexpr int kDiagThreads = 17 * 32;   // a thread per lower element, and the pivot's warp

struct DiagSmem {
  double2 L[kSwNB][kSwNB + 1];
  double2 col[kSwNB];    // column s of the current matrix
  double2 ncolr[kSwNB];  // -conj(col) / d
  double rpiv;
};

// Lower element handled by thread t (triangular order); low = t owns one.
__device__ __forceinline__ void diag_thread_element(int t, int kb, int& i, int& j, bool& low) {
  i = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  while (i * (i + 1) / 2 > t) --i;
  j = t - i * (i + 1) / 2;
  low = t < kSwNB * (kSwNB + 1) / 2 && i < kb;
}

// ---------------------------------------------------------------------------
// Double-FP32 arithmetic for the same sweep (a value is hi + lo, two floats,
// about 2^-46 relative per operation) for updates whose target precision is
// far coarser than FP64 (the five-slice tensor-core update, near 2^-34).
// GB300's FP32 pipe issues 64 times the FP64 pipe's operations, so the
// double-FP32 sweep, about 12 FP32 operations per FP64 multiply-add, leaves
// the FP64 pipe, the sweep's limit, out of the step.  The error-free
// transformations are Knuth's two-sum, the fast two-sum for |a| >= |b| and
// the FMA product error.
__device__ __forceinline__ float2 ff_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}
__device__ __forceinline__ float2 ff_fast(float a, float b) {   // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return make_float2(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ float2 ff_from(double x) {
  const float h = __double2float_rn(x);
  return make_float2(h, __double2float_rn(x - (double)h));
}
__device__ __forceinline__ double ff_to(float2 a) { return (double)a.x + (double)a.y; }

// (h + l) 2^ex as one double for the level sums of the update, built in the
// integer pipe without branches (the SM's FP64 pipe is the epilogue's
// bottleneck, and straight-line code lets the compiler interleave a thread's
// sixteen conversions).  h and l are finite and, where nonzero, far inside
// FP32's normal range (sums of level values, integers times 2^-8L, and their
// rounding errors: |h + l| >= 2^-90 or 0); |ex| < 900.  A two-sum first
// makes the pair non-overlapping: s = fl(h + l), |t| <= ulp(s) / 2, and
// |t| <= ulp(s) / 4 when s is a power of two and t lowers it.  The bits of
// s 2^ex as a double are s's own fields re-biased; t, counted in units of
// that double's last place (half that unit where t takes s below a power of
// two) and rounded, is added to the bit pattern as an integer: s + t stays
// inside the binade of s otherwise, and the pattern is monotonic in the
// magnitude.  The result is within half a unit in the last place of the
// exact (h + l) 2^ex plus the rounding of t to that unit.
__device__ __forceinline__ double ff2d_pair(float s, float t, int ex) {
  const unsigned us = __float_as_uint(s), ut = __float_as_uint(t);
  const unsigned k = (us << 1) != 0u ? (unsigned)(896 + ex) << 20 : 0u;
  const unsigned hi = (us & 0x80000000u) | (((us & 0x7FFFFFFFu) >> 3) + k);
  const unsigned lo = us << 29;
  const bool lowers = (int)(us ^ ut) < 0;   // t's sign differs from s's
  const int ge = (int)((us >> 23) & 0xFFu) - (int)((ut >> 23) & 0xFFu) - ((lowers && (us << 9) == 0u) ? 1 : 0);
  const unsigned mt = (ut & 0x7FFFFFu) | 0x800000u;
  const unsigned d = ge <= 29 ? mt << (29 - ge) : (((mt >> min(ge - 30, 31)) + 1u) >> 1);
  const long long b =
      (long long)(((unsigned long long)hi << 32) | lo) + (lowers ? -(long long)d : (long long)d);
  return __longlong_as_double(b);
}
// X 2^ex rounded to FP64 (half away from zero) for |X| < 2^63, in the integer
// pipe: the magnitude is shifted up to its leading bit, rounded at the 53rd
// and the carry runs into the exponent.  Results below the normal range are
// zero, above it NaN: ex = kBadExp marks operands that are not finite.
constexpr int kBadExp = 1 << 20;
__device__ __forceinline__ double i64_to_scaled(long long X, int ex) {
  const long long s = X >> 63;
  const unsigned long long m0 = (unsigned long long)((X ^ s) - s);
  const int c = __clzll((long long)m0) & 63;
  const unsigned long long m = (m0 << c) + 0x400ull;   // a carry out of bit 63 is the next power of two
  const bool carry = m < 0x400ull;
  const unsigned long long mant = carry ? 0ull : (m << 1) >> 12;
  const int e = 1023 + 63 - c + ex + (carry ? 1 : 0);
  unsigned long long b =
      ((unsigned long long)s & 0x8000000000000000ull) | ((unsigned long long)(unsigned)e << 52) | mant;
  if (m0 == 0ull || e <= 0) b = 0ull;
  if (e >= 2047) b = 0x7FF8000000000000ull;
  return __longlong_as_double((long long)b);
}
// The rare FP64 forms, out of line: a short slow path inline would be
// predicated and its FP64 instructions issued on every call.
static __device__ __noinline__ double ff_to_slow(float hi, float lo) { return (double)hi + (double)lo; }
static __device__ __noinline__ float2 ff_from_slow(double x) { return ff_from(x); }
static __device__ __noinline__ double rcp_slow(double x) { return 1.0 / x; }

// hi + lo as a double for any finite pair: the integer form above where the
// sum lies in [2^-66, 2^123), else the FP64 pipe.
__device__ __forceinline__ double ff_to_any(float hi, float lo) {
  const float2 st = ff_two_sum(hi, lo);
  const unsigned es = (__float_as_uint(st.x) >> 23) & 0xFFu;
  if (es >= 61u && es <= 250u) return ff2d_pair(st.x, st.y, 0);
  return ff_to_slow(hi, lo);
}

// (hi + lo) 2^ex as a double for any finite pair and |ex| < 600: the integer
// form where the two-summed pair lies in [2^-66, 2^123), else the FP64 pipe.
static __device__ __noinline__ double ff_to_scaled_slow(float hi, float lo, int ex) {
  return ldexp((double)hi + (double)lo, ex);
}
__device__ __forceinline__ double ff_to_scaled_any(float hi, float lo, int ex) {
  const float2 st = ff_two_sum(hi, lo);
  const unsigned es = (__float_as_uint(st.x) >> 23) & 0xFFu;
  if (es >= 61u && es <= 250u) return ff2d_pair(st.x, st.y, ex);
  return ff_to_scaled_slow(hi, lo, ex);
}

// ff_from(x) (hi = x rounded to FP32, lo = the remainder rounded) from x's
// fields in the integer pipe for 2^-74 <= |x| < 2^126 (FP64 pipe otherwise):
// hi is x's 53-bit mantissa rounded to 24 bits (half to even, the carry runs
// into the exponent), lo the integer remainder d (|d| <= 2^28) converted and
// scaled by x's last place, exactly as the FP64 form rounds it.
__device__ __forceinline__ float2 ff_from_int(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7FFull);
  if (E < 949 || E > 1149) return ff_from_slow(x);
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  unsigned q = (unsigned)(m >> 29);
  const unsigned r = (unsigned)(m & 0x1FFFFFFFull);
  const unsigned up = (r > 0x10000000u || (r == 0x10000000u && (q & 1u))) ? 1u : 0u;
  q += up;
  const unsigned sgn = (unsigned)(b >> 32) & 0x80000000u;
  const float hi = __uint_as_float(sgn | (((unsigned)(E - 897) << 23) + q));
  const float lo = __int2float_rn((int)r - (int)(up << 29)) * __uint_as_float((unsigned)(E - 948) << 23);
  return make_float2(hi, sgn ? -lo : lo);
}

// rint(v 2^(56 - e)) for |v| < 2^e, rounded half to even, from v's own
// fields in the integer pipe (the FP64 scaling and conversion it replaces run
// on the SM's slow FP64 pipe): v = m 2^(E - 1075) with the 53-bit mantissa m
// (no implicit bit below the normal range), so the result is m shifted by
// E - 1019 - e (at most 3 to the left).
__device__ __forceinline__ long long fixed56(double v, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int E = (int)((b >> 52) & 0x7FFull);
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (E ? (1ull << 52) : 0ull);
  const int sh = (E ? E : 1) - 1019 - e;
  unsigned long long X;
  if (sh >= 0) {
    X = m << sh;
  } else if (sh > -64) {
    const int k = -sh;
    const unsigned long long q = m >> k, r = m & ((1ull << k) - 1ull), half = 1ull << (k - 1);
    X = q + ((r > half || (r == half && (q & 1ull))) ? 1ull : 0ull);
  } else {
    X = 0ull;
  }
  return (b >> 63) ? -(long long)X : (long long)X;
}

__device__ __forceinline__ float2 ff_neg(float2 a) { return make_float2(-a.x, -a.y); }
// a b
__device__ __forceinline__ float2 ff_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  float e = __fmaf_rn(a.x, b.x, -p);
  e = __fmaf_rn(a.x, b.y, e);
  e = __fmaf_rn(a.y, b.x, e);
  return ff_fast(p, e);
}
// 1 / d for d > 0: the FP32 reciprocal and one Newton step in double FP32
__device__ __forceinline__ float2 ff_rcp(float2 d) {
  const float r0 = __frcp_rn(d.x);
  const float2 t = ff_mul(d, make_float2(r0, 0.f));                     // d r0 = 1 - err
  const float2 e = ff_two_sum(1.f, -t.x);
  const float err = __fsub_rn(__fadd_rn(e.x, e.y), t.y);               // 1 - d r0 (small)
  return ff_fast(r0, __fmul_rn(r0, err));
}

// 1 / d for a pivot d > 0 (else 0 and *status): the double-FP32 reciprocal
// (2^-46) and one Newton step with a fused residual, two FP64 operations
// instead of a division's chain of them, each of which would queue behind the
// update's at the FP64 pipe.
__device__ __forceinline__ double rcp_f64_checked(double d, int* status) {
  if (!(d > 0.0) || !isfinite(d)) {
    atomicExch(status, (int)kDevZeroPivot);
    return 0.0;
  }
  const int ex = (int)((unsigned)__double2hiint(d) >> 20) - 1023;
  if (ex < -60 || ex > 60) return rcp_slow(d);   // outside double FP32's safe range
  const float2 r = ff_rcp(ff_from_int(d));
  const double r0 = ff_to_any(r.x, r.y);
  return fma(r0, fma(-d, r0, 1.0), r0);
}

// v + a1 b1 + a2 b2 with both products as exact pairs and the high words
// two-summed; the result is left unnormalized (hi, lo): lo gathers the
// error terms, so hi + lo carries the sum to about 2^-43 of the largest
// term, and consumers that need a leading word close to the value (the
// pivot's reciprocal) renormalize it first.
__device__ __forceinline__ float2 ff_dot2(float2 v, float2 a1, float2 b1, float2 a2, float2 b2) {
  const float p1 = __fmul_rn(a1.x, b1.x);
  float e1 = __fmaf_rn(a1.x, b1.x, -p1);
  e1 = __fmaf_rn(a1.x, b1.y, e1);
  e1 = __fmaf_rn(a1.y, b1.x, e1);
  const float p2 = __fmul_rn(a2.x, b2.x);
  float e2 = __fmaf_rn(a2.x, b2.x, -p2);
  e2 = __fmaf_rn(a2.x, b2.y, e2);
  e2 = __fmaf_rn(a2.y, b2.x, e2);
  const float2 s1 = ff_two_sum(v.x, p1);
  const float2 s2 = ff_two_sum(s1.x, p2);
  return make_float2(s2.x, __fadd_rn(__fadd_rn(v.y, __fadd_rn(e1, e2)), __fadd_rn(s1.y, s2.y)));
}

// The sweep, by 17 warps.  Pivot s, two barriers: warp 16
// (lane r: index r) copies the pivot's column and its scaled form
// -conj(col) / d and writes the pivot's row and column, which are multiples of
// them; then warps 0 .. 15 update the other lower elements, one per thread
// (thread q: element (x, y) of the 31 x 31 triangle, indices from s on moved up
// by one), without divergence, while the lane of the next pivot forms that
// pivot's reciprocal from its own registers.  Called by all the block's threads
// (kDiagThreads or more) after L (lower) is loaded; ends with a __syncthreads().  A non-positive or
// non-finite pivot sets *status.
//
// Bound by the two phases' latencies (double FP32) and by the FP64 pipe (496
// elements x 4 operations at 2 a clock: 0.5 us of 1.0 us a pivot).  A 32 x 32
// block takes 15.3 us in double FP32 and 31.7 us in FP64; with every lower
// element at a fixed thread (the pivot's row and column as divergent branches)
// and the reciprocal by the thread that also updates, 17.3 and 38.7 us; with
// one barrier a pivot and no shared scaled column, 21 us in double FP32.
//
// sweep_element: element (i, j) in step s of the thread that holds (x, y) of the
// smaller triangle.
__device__ __forceinline__ void sweep_element(int x, int y, int s, int& i, int& j) {
  i = x + (x >= s ? 1 : 0);
  j = y + (y >= s ? 1 : 0);
}

__device__ __forceinline__ void diag_sweep_f64(DiagSmem& sm, int kb, int t, int* status) {
  const int lane = t & 31;
  const bool head = (t >> 5) == 16;
  int x, y;
  bool low;
  diag_thread_element(t, kb - 1, x, y, low);
  auto rcp_checked = [&](double d) { return rcp_f64_checked(d, status); };
  __syncthreads();
  if (head && lane == 0) sm.rpiv = rcp_checked(sm.L[0][0].x);
  for (int s = 0; s < kb; ++s) {
    double2 cv = make_double2(0.0, 0.0), nc = cv;
    double v = 0.0;
    __syncthreads();
    if (head && lane < kb) {
      const double rr = sm.rpiv;
      const double2 z = lane < s ? sm.L[s][lane] : sm.L[lane][s];
      v = sm.L[lane][lane].x;
      cv = lane < s ? make_double2(z.x, neg_bits(z.y)) : z;
      nc = make_double2(neg_bits(cv.x * rr), cv.y * rr);
      sm.col[lane] = cv;
      sm.ncolr[lane] = nc;
      if (lane == s)
        sm.L[s][s] = make_double2(neg_bits(rr), 0.0);
      else if (lane > s)                                            // A_is / d
        sm.L[lane][s] = make_double2(neg_bits(nc.x), nc.y);
      else                                                          // conj(col_j) / d
        sm.L[s][lane] = make_double2(neg_bits(nc.x), neg_bits(nc.y));
    }
    __syncthreads();
    if (head) {
      if (lane == s + 1 && lane < kb) sm.rpiv = rcp_checked(fma(cv.x, nc.x, fma(-cv.y, nc.y, v)));
    } else if (low) {
      int i, j;
      sweep_element(x, y, s, i, j);
      const double2 a = sm.col[i], c = sm.ncolr[j];
      double2 e = sm.L[i][j];
      e.x = fma(a.x, c.x, fma(-a.y, c.y, e.x));
      e.y = fma(a.x, c.y, fma(a.y, c.x, e.y));
      sm.L[i][j] = e;
    }
  }
  __syncthreads();
}

// The same in double FP32.  The elements are held in sm.L as float4 (re hi, re
// lo, im hi, im lo), the pivot's column and its scaled form in scratch (64
// float4 the caller does not need meanwhile).  Converts sm.L from and back to
// double2; dff gets -(the result) = D^-1 as normalized pairs, both triangles
// (ld kSwNB): the next panel product reads it without FP64 conversions.
__device__ __forceinline__ void diag_sweep_ff(DiagSmem& sm, float4* scratch, int kb, int t, int* status, float4* dff) {
  typedef float4 Row[kSwNB + 1];
  Row* const B = reinterpret_cast<Row*>(sm.L);
  float4* const col = scratch;
  float4* const ncol = scratch + kSwNB;
  float2* const rpiv = reinterpret_cast<float2*>(&sm.rpiv);
  const int lane = t & 31;
  const bool head = (t >> 5) == 16;
  int i, j, x, y;
  bool low, all;
  diag_thread_element(t, kb, i, j, all);        // conversions: every lower element
  diag_thread_element(t, kb - 1, x, y, low);    // updates: the 31 x 31 triangle
  auto rcp_checked = [&](float2 d) {
    d = ff_two_sum(d.x, d.y);   // leading word first (the pair may be unnormalized)
    if (!(d.x > 0.f) || !isfinite(d.x)) {
      atomicExch(status, (int)kDevZeroPivot);
      return make_float2(0.f, 0.f);
    }
    return ff_rcp(d);
  };
  __syncthreads();   // the caller's loads of L are visible before the conversion
  if (all) {
    const double2 z = sm.L[i][j];
    const float2 re = ff_from_int(z.x), im = ff_from_int(z.y);
    B[i][j] = make_float4(re.x, re.y, im.x, im.y);
    if (i == 0) *rpiv = rcp_checked(re);
  }
  for (int s = 0; s < kb; ++s) {
    float4 cv = make_float4(0.f, 0.f, 0.f, 0.f), nc = cv, v = cv;
    __syncthreads();
    if (head && lane < kb) {
      const float2 rp = *rpiv;
      const float4 z = lane < s ? B[s][lane] : B[lane][s];
      const float g = lane < s ? -1.f : 1.f;
      v = B[lane][lane];
      const float2 cr = ff_mul(make_float2(z.x, z.y), rp), ci = ff_mul(make_float2(g * z.z, g * z.w), rp);
      cv = make_float4(z.x, z.y, g * z.z, g * z.w);
      nc = make_float4(-cr.x, -cr.y, ci.x, ci.y);
      col[lane] = cv;
      ncol[lane] = nc;
      if (lane == s)
        B[s][s] = make_float4(-rp.x, -rp.y, 0.f, 0.f);
      else if (lane > s)                                       // A_is / d
        B[lane][s] = make_float4(cr.x, cr.y, ci.x, ci.y);
      else                                                     // conj(col_j) / d
        B[s][lane] = make_float4(cr.x, cr.y, -ci.x, -ci.y);
    }
    __syncthreads();
    if (head) {
      if (lane == s + 1 && lane < kb)
        *rpiv = rcp_checked(ff_dot2(make_float2(v.x, v.y), make_float2(cv.x, cv.y), make_float2(nc.x, nc.y),
                                    make_float2(-cv.z, -cv.w), make_float2(nc.z, nc.w)));
    } else if (low) {
      int ii, jj;
      sweep_element(x, y, s, ii, jj);
      const float4 a = col[ii], c = ncol[jj], e = B[ii][jj];
      const float2 ar = make_float2(a.x, a.y), ai = make_float2(a.z, a.w);
      const float2 cr = make_float2(c.x, c.y), ci = make_float2(c.z, c.w);
      const float2 vr = ff_dot2(make_float2(e.x, e.y), ar, cr, ff_neg(ai), ci);   // + a_r c_r - a_i c_i
      const float2 vi = ff_dot2(make_float2(e.z, e.w), ar, ci, ai, cr);           // + a_r c_i + a_i c_r
      B[ii][jj] = make_float4(vr.x, vr.y, vi.x, vi.y);
    }
  }
  __syncthreads();
  if (all) {
    const float4 z = B[i][j];
    sm.L[i][j] = make_double2(ff_to_any(z.x, z.y), ff_to_any(z.z, z.w));
    const float2 re = ff_two_sum(z.x, z.y), im = ff_two_sum(z.z, z.w);
    dff[i * kSwNB + j] = make_float4(-re.x, -re.y, -im.x, -im.y);
    if (i != j) dff[j * kSwNB + i] = make_float4(-re.x, -re.y, im.x, im.y);
  }
  __syncthreads();
}

}  // namespace bgw
